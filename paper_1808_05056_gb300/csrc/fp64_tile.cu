// Plain FP64 tile contraction for sm_103a: the compute stage of the Section IV
// pipeline (its per-block update c_ij = alpha a_i b_j + beta c_ij) on the FP64
// tensor-core MMA (mma.sync m8n8k4 .f64), fed by TMA tile loads.
//
// Shape: CTA tile 16 x 16, K steps of 16, an 8-stage ring of TMA-filled shared
// memory stages guarded by full/empty mbarriers.  Warp 4 is the producer (one
// elected lane issues the tensor copies); warps 0-3 each own one 8 x 8 MMA
// fragment of the tile in registers.  The grid is persistent: each CTA walks tiles
// blockIdx.x, blockIdx.x + gridDim.x, ... with the stage ring running on across
// tile boundaries, so the copies of the next tile overlap the epilogue of the
// current one (tiles are taken in a grouped raster order, see raster_tile).
// Ragged edges come from the tensor maps: reads outside the operand are
// zero-filled by TMA, the epilogue masks stores, and fragments and K steps that
// lie wholly outside the operands are not multiplied.
//
// What bounds it: GB300's FP64 rate, 1.75 fused multiply-adds per clock and SM
// (1.10 TFLOP/s in all).  Even this small tile holds an SM for 1.1 us per K step
// with 4 KiB of operands, so copies, barriers and shared-memory conflicts do not
// show and the only thing left to lose is balance: an SM that gets one tile more
// than another keeps the whole launch waiting.  Measured against 64 x 64 and
// 32 x 32 tiles (TFLOP/s): 8192 x 8192 x 512 1.097 / 1.096 / 1.097, 704 x 5003 x
// 1024 1.092 / 1.031 / 1.034, 1536 x 1000 x 2000 1.071 / 0.900 / 0.984, 512^3 1.02
// / 0.45 / 0.89, 192 x 1024 x 256 0.87 / 0.34 / 0.65; the small tile is never the
// slower one.  Every output is accumulated in the same order (k ascending, four
// at a time) whatever the tile.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>

#include "device_sync.cuh"
#include "ooc_internal.hpp"

namespace ooc {

namespace {

constexpr int T = 16;   // edge of the CTA tile
constexpr int W = T / 2;  // edge of a warp's 8 x 8 fragment
constexpr int BK = 16, STAGES = 8;
constexpr int CONSUMER_WARPS = 4;
constexpr int THREADS = (CONSUMER_WARPS + 1) * 32;
constexpr int STAGE = T * BK;  // doubles per operand
constexpr uint32_t STAGE_BYTES = 2 * STAGE * 8;
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + 2 * STAGES * sizeof(uint64_t) + 1024;

// Tiles of a triangular update (GEMMT / SYRK blocks that straddle the
// diagonal).  With square tiles of side T, tile (tm, tn) holds an element with
// col - row <= off (lower) iff tn - tm <= floor((off + T - 1) / T), and one
// with col - row >= off (upper) iff tn - tm >= ceil((off - T + 1) / T).  So
// the kept tiles of tile row tm are one run of columns whose length is
//   lower: clamp(tm + a, 0, tiles_n), starting at column 0,
//   upper: clamp(a - tm, 0, tiles_n), ending at the last column,
// and the run lengths have closed-form prefix sums, which map a kept-tile
// index to its (tm, tn) by a binary search over tile rows.
struct TriTiles {
    int mode;  // 0 every tile, 1 lower, 2 upper
    int64_t a, tiles_m, tiles_n;
};

__host__ __device__ inline int64_t clamp64(int64_t v, int64_t lo, int64_t hi) { return v < lo ? lo : (v > hi ? hi : v); }
__host__ __device__ inline int64_t floor_div(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

__host__ __device__ inline int64_t tri_run(const TriTiles& t, int64_t tm)
{
    return t.mode == 1 ? clamp64(tm + t.a, 0, t.tiles_n) : clamp64(t.a - tm, 0, t.tiles_n);
}

// number of kept tiles in tile rows [0, x)
__host__ __device__ inline int64_t tri_prefix(const TriTiles& t, int64_t x)
{
    const int64_t T = t.tiles_n, a = t.a;
    if (t.mode == 1) {
        const int64_t z = clamp64(1 - a, 0, x);    // rows before z keep no tile
        const int64_t s = clamp64(T - a, z, x);    // rows from s on keep all T
        const int64_t n = s - z;
        return n * (z + s - 1) / 2 + n * a + (x - s) * T;
    }
    const int64_t s = clamp64(a - T + 1, 0, x);    // rows before s keep all T
    const int64_t z = clamp64(a, s, x);            // rows from z on keep none
    const int64_t n = z - s;
    return s * T + n * a - n * (s + z - 1) / 2;
}

__host__ __device__ inline TriTiles tri_tiles(int mode, int64_t off, int64_t tiles_m, int64_t tiles_n, int64_t T)
{
    TriTiles t{mode, 0, tiles_m, tiles_n};
    if (mode == 1) t.a = floor_div(off + T - 1, T) + 1;
    else if (mode == 2) t.a = tiles_n + floor_div(-(off - T + 1), T);  // tiles_n - ceil((off - T + 1) / T)
    return t;
}

struct Fp64Args {
    int64_t M, N, K;
    int64_t tiles_n, tiles;
    double alpha, beta;
    int read_c;
    double* C;
    int64_t ldc;
    int* err;
    int tri;          // 0 full update, 1 lower (col - row <= tri_off), 2 upper (col - row >= tri_off)
    int64_t tri_off;
    TriTiles tt;
};

// Tile order of a full update: groups of kRasterRows tile rows (256 matrix rows),
// column-major inside a group, so that the ~900 tiles in flight span few rows and
// columns and re-read their A and B tiles from L2 rather than DRAM.
constexpr int64_t kRasterRows = 16;

__host__ __device__ __forceinline__ void raster_tile(int64_t tile, int64_t tiles_m, int64_t tiles_n, int64_t& tm,
                                                     int64_t& tn)
{
    const int64_t per_group = kRasterRows * tiles_n;
    const int64_t g = tile / per_group, r = tile % per_group;
    const int64_t first = g * kRasterRows;
    const int64_t rows = tiles_m - first < kRasterRows ? tiles_m - first : kRasterRows;
    tm = first + r % rows;
    tn = r / rows;
}

__device__ __forceinline__ void tile_of(const Fp64Args& p, int64_t tile, int64_t& tm, int64_t& tn)
{
    if (p.tri == 0) {
        raster_tile(tile, p.tiles / p.tiles_n, p.tiles_n, tm, tn);
        return;
    }
    int64_t lo = 0, hi = p.tt.tiles_m - 1;  // largest tm with prefix(tm) <= tile
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (tri_prefix(p.tt, mid) <= tile) lo = mid;
        else hi = mid - 1;
    }
    tm = lo;
    const int64_t first = p.tri == 1 ? 0 : p.tiles_n - tri_run(p.tt, lo);
    tn = first + (tile - tri_prefix(p.tt, lo));
}

__device__ __forceinline__ bool kept(const Fp64Args& p, int64_t row, int64_t col)
{
    return p.tri == 0 || (p.tri == 1 ? col - row <= p.tri_off : col - row >= p.tri_off);
}

__device__ __forceinline__ void dmma_8x8x4(double& d0, double& d1, double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(d0), "+d"(d1)
                 : "d"(a), "d"(b));
}

// The stage ring of a CTA: T x BK tiles of A and B, their barriers, and this
// thread's position in the ring (advanced without division).
struct Ring {
    double* stages;
    uint64_t *full, *empty;
    int s = 0;
    uint32_t ph = 0;

    __device__ explicit Ring(unsigned char* smem)
    {
        unsigned char* base =
            reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem) + 1023) & ~uintptr_t(1023));
        stages = reinterpret_cast<double*>(base);
        full = reinterpret_cast<uint64_t*>(base + STAGES * STAGE_BYTES);
        empty = full + STAGES;
    }
    __device__ void init()
    {
        if (threadIdx.x == 0) {
            for (int q = 0; q < STAGES; ++q) {
                mbar_init(&full[q], 1);
                mbar_init(&empty[q], CONSUMER_WARPS);
            }
            mbar_fence_init();
        }
        __syncthreads();
    }
    __device__ __forceinline__ void next()
    {
        if (++s == STAGES) { s = 0; ph ^= 1u; }
    }
};

// Producer: the K steps of one tile into the ring; false when a wait gave up.
template <bool A_KMAJOR, bool B_KMAJOR>
__device__ __forceinline__ bool produce_tile(Ring& r, const CUtensorMap* ma, const CUtensorMap* mb, int64_t nk,
                                             int32_t row0, int32_t col0, int64_t& issued, int* err)
{
    for (int64_t ks = 0; ks < nk; ++ks) {
        if (!mbar_wait(&r.empty[r.s], r.ph ^ 1u, err, kErrWaitEmpty)) return false;
        double* sA = r.stages + (size_t)r.s * 2 * STAGE;
        double* sB = sA + STAGE;
        mbar_arrive_expect_tx(&r.full[r.s], STAGE_BYTES);
        const int32_t k0 = (int32_t)(ks * BK);
        if (A_KMAJOR) tma_load_2d(sA, ma, &r.full[r.s], k0, row0);
        else tma_load_2d(sA, ma, &r.full[r.s], row0, k0);
        if (B_KMAJOR) tma_load_2d(sB, mb, &r.full[r.s], k0, col0);
        else tma_load_2d(sB, mb, &r.full[r.s], col0, k0);
        r.next();
        ++issued;
    }
    return true;
}

// After a wait gave up: let the copies already issued land before the CTA exits.
__device__ __forceinline__ void drain_ring(const Ring& r, int64_t issued)
{
    constexpr int N = STAGES;
    for (int64_t w = issued > N ? issued - N : 0; w < issued; ++w) {
        const int s = (int)(w % N);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(smem_u32(&r.full[s]), (uint32_t)((w / N) & 1)) && globaltimer_ns() - t0 < kWaitLimitNs) {
        }
    }
}

// Consumer warp: multiply the K steps of one tile into its fragment.  inside: the
// fragment holds an element of C; K: inner dimension.  False when a wait gave up.
template <bool A_KMAJOR, bool B_KMAJOR>
__device__ __forceinline__ bool consume_tile(Ring& r, double (&acc)[2], int64_t nk, int64_t K, bool inside, int* err)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = (warp >> 1) * W + (lane >> 2), col = (warp & 1) * W + (lane >> 2);  // 2 x 2 warps
    const int fc = lane & 3;
    for (int64_t ks = 0; ks < nk; ++ks) {
        if (!mbar_wait(&r.full[r.s], r.ph, err, kErrWaitFull)) return false;
        const double* sA = r.stages + (size_t)r.s * 2 * STAGE;
        const double* sB = sA + STAGE;
        const int64_t left = K - ks * BK;
        if (inside) {
#pragma unroll
            for (int kk = 0; kk < BK; kk += 4) {
                if (kk >= left) break;  // the last K step: only what lies inside the operands
                const int k = kk + fc;
                const double a = A_KMAJOR ? sA[row * BK + k] : sA[k * T + row];
                const double b = B_KMAJOR ? sB[col * BK + k] : sB[k * T + col];
                dmma_8x8x4(acc[0], acc[1], a, b);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&r.empty[r.s]);
        r.next();
    }
    return true;
}

// C = alpha acc + beta C on this warp's fragment at (row0, col0), then acc = 0.
// keep(row, col) masks single elements of a triangular update (kMasked).
template <bool kMasked, class Keep>
__device__ __forceinline__ void store_tile(double (&acc)[2], int64_t row0, int64_t col0, int64_t M, int64_t N,
                                           double alpha, double beta, int read_c, double* C, int64_t ldc, Keep keep)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = row0 + (lane >> 2), col = col0 + (lane & 3) * 2;
    if (row < M) {
        double* c = C + row * ldc + col;
        if (!kMasked && col + 1 < N) {
            double2 v;
            v.x = alpha * acc[0];
            v.y = alpha * acc[1];
            if (read_c) {
                const double2 o = *reinterpret_cast<const double2*>(c);
                v.x += beta * o.x;
                v.y += beta * o.y;
            }
            *reinterpret_cast<double2*>(c) = v;
        } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (col + e >= N || (kMasked && !keep(row, col + e))) continue;
                double v = alpha * acc[e];
                if (read_c) v += beta * c[e];
                c[e] = v;
            }
        }
    }
    acc[0] = acc[1] = 0.0;
}

template <bool A_KMAJOR, bool B_KMAJOR>
__global__ void __launch_bounds__(THREADS) fp64_tile_kernel(const __grid_constant__ CUtensorMap tmA,
                                                            const __grid_constant__ CUtensorMap tmB,
                                                            Fp64Args p)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Ring r(smem_raw);
    r.init();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nk = (p.K + BK - 1) / BK;
    if (warp == CONSUMER_WARPS) {
        // ---------------- producer ----------------
        if (lane != 0 || nk == 0) return;
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        int64_t issued = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x) {
            int64_t tm, tn;
            tile_of(p, tile, tm, tn);
            ok = produce_tile<A_KMAJOR, B_KMAJOR>(r, &tmA, &tmB, nk, (int32_t)(tm * T), (int32_t)(tn * T), issued,
                                                     p.err);
        }
        if (!ok) drain_ring(r, issued);
        return;
    }
    // ---------------- consumers ----------------
    double acc[2] = {0.0, 0.0};
    for (int64_t tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) {
        int64_t tm, tn;
        tile_of(p, tile, tm, tn);
        const int64_t row0 = tm * T + (warp >> 1) * W, col0 = tn * T + (warp & 1) * W;
        if (!consume_tile<A_KMAJOR, B_KMAJOR>(r, acc, nk, p.K, row0 < p.M && col0 < p.N, p.err))
            return;
        auto keep = [&](int64_t row, int64_t col) { return kept(p, row, col); };
        if (p.tri) store_tile<true>(acc, row0, col0, p.M, p.N, p.alpha, p.beta, p.read_c, p.C, p.ldc, keep);
        else store_tile<false>(acc, row0, col0, p.M, p.N, p.alpha, p.beta, p.read_c, p.C, p.ldc, keep);
    }
}

// CTAs of a launch: as many as are resident, at most one per tile.
template <class Kernel>
int resident_ctas(Kernel kernel, size_t smem, int& occ, std::once_flag& once)
{
    std::call_once(once, [&] {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, THREADS, smem);
    });
    return occ * device_sm_count();
}

template <bool AK, bool BKM>
int launch_variant(const CUtensorMap& ma, const CUtensorMap& mb, const Fp64Args& a, cudaStream_t st,
                   std::string& why)
{
    static int occ = 0;
    static std::once_flag once;
    const int64_t room = resident_ctas(fp64_tile_kernel<AK, BKM>, SMEM_BYTES, occ, once);
    if (room <= 0) {
        why = "fp64 tile kernel cannot be resident (occupancy 0)";
        return OOC_ERR_CUDA;
    }
    const int64_t grid = std::min<int64_t>(a.tiles > 0 ? a.tiles : 1, room);
    fp64_tile_kernel<AK, BKM><<<(unsigned)grid, THREADS, SMEM_BYTES, st>>>(ma, mb, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        why = std::string("fp64 tile launch: ") + cudaGetErrorString(e);
        return OOC_ERR_CUDA;
    }
    return OOC_OK;
}

// ---------------------------------------------------------------- grouped --
// One launch over the tiles of up to kGroupMax independent problems whose
// operands are all resident (a batch of uneven GEMMs): the CTAs walk the
// concatenated list of (problem, tile) items -- each problem's tiles in the
// raster order of tile_of -- with the stage ring running on across items and
// problems, so one launch's tail and pipeline fill are paid once per group of
// problems instead of once per problem.  Each problem's tensor maps live in
// the kernel parameters (no device-side descriptor copy, so the launch can be
// captured in a CUDA graph).
struct GroupProb {
    CUtensorMap ma, mb;
    double* C;
    int64_t ldc, M, N, K;
    int64_t tiles_n, tile_begin;  // tiles per row of tiles; first item of this problem
    double alpha, beta;
    int read_c, pad;
};

struct GroupArgs {
    int count;
    int64_t tiles;  // items in all problems
    int* err;
    GroupProb p[kGroupMax];
};

// the problem holding item t (tile_begin ascending, first entry 0)
__device__ __forceinline__ int group_problem(const GroupArgs& g, int64_t t)
{
    int lo = 0, hi = g.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.p[mid].tile_begin <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <bool A_KMAJOR, bool B_KMAJOR>
__global__ void __launch_bounds__(THREADS) fp64_group_kernel(const __grid_constant__ GroupArgs g)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Ring r(smem_raw);
    r.init();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto item = [&](int64_t t, const GroupProb*& q, int64_t& tm, int64_t& tn) {
        q = &g.p[group_problem(g, t)];
        raster_tile(t - q->tile_begin, (q->M + T - 1) / T, q->tiles_n, tm, tn);
    };
    if (warp == CONSUMER_WARPS) {
        // ---------------- producer ----------------
        if (lane != 0) return;
        int64_t issued = 0;
        bool ok = true;
        for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
            const GroupProb* q;
            int64_t tm, tn;
            item(t, q, tm, tn);
            ok = produce_tile<A_KMAJOR, B_KMAJOR>(r, &q->ma, &q->mb, (q->K + BK - 1) / BK, (int32_t)(tm * T),
                                                     (int32_t)(tn * T), issued, g.err);
        }
        if (!ok) drain_ring(r, issued);
        return;
    }
    // ---------------- consumers ----------------
    double acc[2] = {0.0, 0.0};
    for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x) {
        const GroupProb* q;
        int64_t tm, tn;
        item(t, q, tm, tn);
        const int64_t row0 = tm * T + (warp >> 1) * W, col0 = tn * T + (warp & 1) * W;
        if (!consume_tile<A_KMAJOR, B_KMAJOR>(r, acc, (q->K + BK - 1) / BK, q->K, row0 < q->M && col0 < q->N, g.err))
            return;
        store_tile<false>(acc, row0, col0, q->M, q->N, q->alpha, q->beta, q->read_c, q->C, q->ldc,
                             [](int64_t, int64_t) { return true; });
    }
}

template <bool AK, bool BKM>
int launch_group_variant(const GroupArgs& a, cudaStream_t st, std::string& why)
{
    static int occ = 0;
    static std::once_flag once;
    const int64_t room = resident_ctas(fp64_group_kernel<AK, BKM>, SMEM_BYTES, occ, once);
    if (room <= 0) {
        why = "fp64 group kernel cannot be resident (occupancy 0)";
        return OOC_ERR_CUDA;
    }
    const int64_t grid = std::min<int64_t>(a.tiles > 0 ? a.tiles : 1, room);
    fp64_group_kernel<AK, BKM><<<(unsigned)grid, THREADS, SMEM_BYTES, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        why = std::string("fp64 group launch: ") + cudaGetErrorString(e);
        return OOC_ERR_CUDA;
    }
    return OOC_OK;
}

// Tensor map of one operand: K-major (rows x K) or K down the stored rows, in
// boxes of T rows by BK of K.
int operand_map(CUtensorMap* map, bool kmajor, const double* X, int64_t rows, int64_t K, int64_t ld, std::string& why)
{
    return kmajor ? encode_map_2d(map, 0, X, (uint64_t)K, (uint64_t)rows, (uint64_t)ld, BK, T, 0, why)
                  : encode_map_2d(map, 0, X, (uint64_t)rows, (uint64_t)K, (uint64_t)ld, T, BK, 0, why);
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

}  // namespace

int launch_fp64_tile(bool a_kmajor, bool b_kmajor, int64_t M, int64_t N, int64_t K, double alpha,
                     const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                     bool read_c, double* C, int64_t ldc, int* err, void* stream, std::string& why, int tri,
                     int64_t tri_off)
{
    if (M <= 0 || N <= 0) return OOC_OK;
    CUtensorMap ma, mbm;
    std::memset(&ma, 0, sizeof(ma));
    std::memset(&mbm, 0, sizeof(mbm));
    if (K > 0) {
        int rc = operand_map(&ma, a_kmajor, A, M, K, lda, why);
        if (rc == OOC_OK) rc = operand_map(&mbm, b_kmajor, B, N, K, ldb, why);
        if (rc != OOC_OK) return rc;
    }
    Fp64Args a;
    a.M = M; a.N = N; a.K = K;
    a.tiles_n = cdiv(N, T);
    a.tiles = cdiv(M, T) * a.tiles_n;
    a.alpha = alpha; a.beta = beta; a.read_c = read_c ? 1 : 0;
    a.C = C; a.ldc = ldc; a.err = err;
    a.tri = tri; a.tri_off = tri_off;
    a.tt = tri_tiles(tri, tri_off, cdiv(M, T), a.tiles_n, T);
    if (tri) a.tiles = tri_prefix(a.tt, a.tt.tiles_m);
    if (a.tiles == 0) return OOC_OK;  // nothing of C is updated
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (a_kmajor && b_kmajor) return launch_variant<true, true>(ma, mbm, a, st, why);
    if (a_kmajor && !b_kmajor) return launch_variant<true, false>(ma, mbm, a, st, why);
    if (!a_kmajor && b_kmajor) return launch_variant<false, true>(ma, mbm, a, st, why);
    return launch_variant<false, false>(ma, mbm, a, st, why);
}

int launch_fp64_group(bool a_kmajor, bool b_kmajor, const Fp64GroupSpec* probs, int count, int* err, void* stream,
                      std::string& why, int64_t* tiles_out)
{
    if (count <= 0 || count > kGroupMax) {
        why = "grouped launch: problem count outside 1.." + std::to_string(kGroupMax);
        return OOC_ERR_INVALID_ARG;
    }
    static GroupArgs a;  // 24 KB of kernel parameters: not on the stack
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    std::memset(&a, 0, sizeof(a));
    a.err = err;
    int n = 0;
    int64_t tiles = 0;
    for (int i = 0; i < count; ++i) {
        const Fp64GroupSpec& s = probs[i];
        if (s.M <= 0 || s.N <= 0) continue;
        GroupProb& q = a.p[n];
        if (s.K > 0) {
            int rc = operand_map(&q.ma, a_kmajor, s.A, s.M, s.K, s.lda, why);
            if (rc == OOC_OK) rc = operand_map(&q.mb, b_kmajor, s.B, s.N, s.K, s.ldb, why);
            if (rc != OOC_OK) return rc;
        }
        q.C = s.C; q.ldc = s.ldc;
        q.M = s.M; q.N = s.N; q.K = s.K;
        q.tiles_n = cdiv(s.N, T);
        q.tile_begin = tiles;
        q.alpha = s.alpha; q.beta = s.beta; q.read_c = s.read_c ? 1 : 0;
        tiles += cdiv(s.M, T) * q.tiles_n;
        ++n;
    }
    if (tiles_out) *tiles_out = tiles;
    if (n == 0) return OOC_OK;
    a.count = n;
    a.tiles = tiles;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (a_kmajor && b_kmajor) return launch_group_variant<true, true>(a, st, why);
    if (a_kmajor && !b_kmajor) return launch_group_variant<true, false>(a, st, why);
    if (!a_kmajor && b_kmajor) return launch_group_variant<false, true>(a, st, why);
    return launch_group_variant<false, false>(a, st, why);
}

}  // namespace ooc
