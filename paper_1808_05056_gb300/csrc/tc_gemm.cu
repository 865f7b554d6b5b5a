// The FP32-accurate BF16x3 form on the 5th-generation tensor cores (sm_103a): the
// compute stage of the out-of-core pipeline for ooc_sgemm.
//
// Each FP32 operand is split into three bf16 pieces x = h + m + l (each piece the
// bf16 rounding of what is left), and C = sum of the six products hh, hm, mh, hl, mm,
// lh (the dropped ml, lm, ll are below 2^-24 relative).  The tensor cores round
// their FP32 accumulator toward zero, so each accumulator addition is biased by up
// to one ulp: the leading product hh has its own accumulator, drained every 512 of K
// (32 additions) into an unbiased double-float (hi, lo) pair per output with TwoSum;
// the five small products, 2^-8 of hh and below, share a second accumulator drained
// every 2048 of K straight into lo.  The drains run on the epilogue warps, four of
// which share the MMA thread's sub-partition (TMEM lane quarters tie warps to
// sub-partitions): draining hh every 128 of K took enough of that thread's issue
// slots to cost a fifth of the tensor-core rate.
//
// Kernel shape: tile 128 x 128, 18 warps, persistent CTAs (one per SM).
//   warp 0      TMA producer: for each K block of 64 loads the three plane tiles of
//               A and of B (96 KiB, 128-byte swizzle) into a ring of two stages;
//   warp 1      allocates all 512 TMEM columns and issues tcgen05.mma, committing
//               stage releases and accumulator-full events to mbarriers;
//   warps 2-17  epilogue: drain finished accumulators with tcgen05.ld into packed
//               double-float FP32 registers, 32 columns of one row per thread,
//               release them, and after the last chunk write alpha * acc + beta *
//               C_old, each store covering 8 rows x 4 consecutive columns (4 x 4
//               transposes by shuffles inside groups of 4 lanes).
//
// Instructions: the B planes h and m lie back to back in a stage, so one N = 256
// instruction multiplies an A plane by both; h l and l h take N = 128 ones.  Four
// instructions per 16 of K instead of six, and 104 bytes of operands read from shared
// memory per clock instead of 128, which leaves room for the TMA writes.
// TMEM: leading accumulators X0 and X1 used in turn, with two small-product ones, Y0
// and Y1, between them (columns X0 Y0 Y1 X1).  h x (h, m) fills X0 and Y0 in one chunk;
// in the next the stage holds the planes in the order (m, h) and the same instruction
// fills Y1 and X1.  m x (h, m) fills both Y.
//
// Clusters: when a launch has fewer tiles than SMs, the CTAs of a cluster share each
// tile's K blocks and add their double-float partial sums through distributed shared
// memory, each CTA a share of the columns, from its own rank on (the order of a column's
// sums follows from the column alone).  Cluster barriers sit in loops that every thread walks
// whatever happens, so a CTA whose bounded wait gave up still arrives.
//
// The ring releases whole stages: finer slots (one 16 KiB plane tile each, with a wait
// and a release per tile) ran at half the rate.  CTA pairs (cta_group::2, 256 x 128
// tiles with half of each B tile per CTA) were measured slower (1216 vs 1384 bf16
// TFLOP/s) and are not built.  Every wait is bounded (device_sync.cuh); the epilogue
// warps wait with a sleep between tries so that they leave the issue slots to the TMA
// and MMA threads.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "ooc_internal.hpp"
#include "tc_common.cuh"

namespace ooc {

namespace {

constexpr int BM = 128, BN = 128, BK = 64;
constexpr uint32_t A_TILE = BM * BK * 2u;             // 128 rows x 64 bf16 of K (16 KiB)
constexpr uint32_t STAGE_BYTES = 6 * A_TILE;          // three planes of A, three of B
constexpr int STAGES = 2;
constexpr uint32_t RING_BYTES = STAGES * STAGE_BYTES;
constexpr int EPI_WARPS = 16;                         // 4 per TMEM lane quadrant, 32 columns each
constexpr int THREADS = (2 + EPI_WARPS) * 32;
constexpr size_t SMEM_BYTES = 1024 + RING_BYTES + 1024;
constexpr int KSTEPS = BK / 16;
// K blocks between drains of the leading product's round-toward-zero accumulator (512:
// 32 accumulations of up to one ulp each, 2^-18 of sum |x||y|) and chunks between
// drains of the small products' (2048 of K)
constexpr int CHUNK_KBLOCKS = 512 / BK;
constexpr int SMALL_EVERY = 4;
// TMEM columns: X0 Y0 Y1 X1
constexpr uint32_t kX0 = 0, kY0 = BN, kY1 = 2 * BN, kX1 = 3 * BN;
constexpr int MAX_CLUSTER = 8;
static_assert(RING_BYTES >= (uint32_t)BM * BN * 8, "the ring holds a tile of double-float partial sums");

struct TcArgs {
    int M, N;
    int kblocks;
    int cluster;      // CTAs that share a tile's K blocks
    int tiles_m, tiles_n, tiles;
    float alpha, beta;
    int read_c;
    float* C;
    int64_t ldc;
    int* err;
    int tri;          // 0 full update, 1 lower (col - row <= tri_off), 2 upper (col - row >= tri_off)
    int64_t tri_off;
};

__device__ __forceinline__ float unpack2(uint64_t v, int j) { return __uint_as_float((uint32_t)(v >> (32 * j))); }

// Drains of the small-product accumulators: every SMALL_EVERY chunks and at the last
// chunk of a tile (both the MMA issuer and the epilogue use this)
__device__ __forceinline__ bool small_drain_after(int c, int nchunks)
{
    return c == nchunks - 1 || (c % SMALL_EVERY) == SMALL_EVERY - 1;
}

// (hi, lo) += (h, l): the sum of the leading parts exactly (TwoSum), its error with the rest
__device__ __forceinline__ void add_double_float(float& hi, float& lo, float h, float l)
{
    const float s = __fadd_rn(hi, h), bp = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(l, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(h, bp))));
    hi = s;
}

__global__ void __launch_bounds__(THREADS, 1) bf16x3_tile_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                 const __grid_constant__ CUtensorMap tmB,
                                                                 const __grid_constant__ TcArgs p)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + RING_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* small_full = acc_empty + 2;
    uint64_t* small_empty = small_full + 1;
    uint64_t* done = small_empty + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

    // the shuffle tells the compiler that the warp index is the same in all lanes
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], EPI_WARPS);
        }
        mbar_init(small_full, 1);
        mbar_init(small_empty, EPI_WARPS);
        mbar_init(done, 1);
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int rank = (int)blockIdx.x % p.cluster;
    const int first = (int)blockIdx.x / p.cluster, stride = (int)gridDim.x / p.cluster;
    const int kb0 = (int)((int64_t)p.kblocks * rank / p.cluster), kb1 = (int)((int64_t)p.kblocks * (rank + 1) / p.cluster);
    const int nchunks = (kb1 - kb0 + CHUNK_KBLOCKS - 1) / CHUNK_KBLOCKS;

    Ring r, b;                   // stage ring (producer, MMA); leading accumulators in turn (producer, MMA, epilogue)
    uint32_t issued = 0;         // producer: stages issued
    uint32_t small_drains = 0;   // drains of the small accumulators so far (MMA, epilogue)
    bool small_pending = false;  // MMA: one not yet released by the epilogue
    bool ok = true;
    const uint32_t idesc2 = idesc_bf16_f32(BM, 2 * BN), idesc1 = idesc_bf16_f32(BM, BN);
    const bool leader = elect_one();  // the lane that issues copies and MMAs
    if (warp == 0 && leader) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }

    for (int tile = first; tile < p.tiles; tile += stride) {
        int tm, tn;
        tile_coords(tile, p.tiles_m, p.tiles_n, tm, tn);
        if (warp == 0) {
            // -------------------------------------------- TMA producer
            if (ok) {
                for (int c = 0; c < nchunks && ok; ++c) {
                    const int end = min(kb1, kb0 + (c + 1) * CHUNK_KBLOCKS);
                    for (int kb = kb0 + c * CHUNK_KBLOCKS; kb < end; ++kb) {
                        if (!wait_warp(&empty[r.s], r.ph ^ 1u, p.err, kErrWaitEmpty)) { ok = false; break; }
                        if (leader) {
                            unsigned char* st = ring + (size_t)r.s * STAGE_BYTES;
                            mbar_arrive_expect_tx(&full[r.s], STAGE_BYTES);
                            for (int a = 0; a < 3; ++a)
                                tma_load_3d(st + a * A_TILE, &tmA, &full[r.s], kb * BK, tm * BM, a);
                            // B planes (h, m, l) beside X0, (m, h, l) beside X1
                            tma_load_3d(st + 3 * A_TILE, &tmB, &full[r.s], kb * BK, tn * BN, b.s);
                            tma_load_3d(st + 4 * A_TILE, &tmB, &full[r.s], kb * BK, tn * BN, 1 - b.s);
                            tma_load_3d(st + 5 * A_TILE, &tmB, &full[r.s], kb * BK, tn * BN, 2);
                        }
                        r.next(STAGES);
                        ++issued;
                    }
                    b.next(2);
                }
                if (!ok) {
                    // let the copies already issued land before the CTA goes on
                    const uint32_t n = min(issued, (uint32_t)STAGES);
                    for (uint32_t q = 0; q < n; ++q) {
                        int s = r.s - 1 - (int)q;
                        uint32_t ph = r.ph;
                        if (s < 0) { s += STAGES; ph ^= 1u; }
                        const uint64_t t0 = globaltimer_ns();
                        while (!mbar_try_wait(smem_u32(&full[s]), ph) && globaltimer_ns() - t0 < kWaitLimitNs) {
                        }
                    }
                }
            }
        } else if (warp == 1) {
            // -------------------------------------------- MMA issuer
            if (ok) {
                uint32_t small_acc = 0;  // accumulate flag of the small-product accumulators
                for (int c = 0; c < nchunks && ok; ++c) {
                    const int end = min(kb1, kb0 + (c + 1) * CHUNK_KBLOCKS);
                    if (!wait_warp(&acc_empty[b.s], b.ph ^ 1u, p.err, kErrWaitAcc)) { ok = false; break; }
                    if (small_pending) {
                        // the epilogue has read the small accumulators before they restart
                        if (!wait_warp(small_empty, (small_drains - 1) & 1u, p.err, kErrWaitAcc)) { ok = false; break; }
                        small_pending = false;
                    }
                    tc_fence_after();
                    // h x (h, m) -> (X0, Y0) or h x (m, h) -> (Y1, X1)
                    const uint32_t dh = tmem_base + (b.s ? kY1 : kX0), dy = tmem_base + kY0;
                    const uint32_t dlead = tmem_base + (b.s ? kX1 : kX0), dsmall = tmem_base + (b.s ? kY1 : kY0);
                    const uint32_t bh = (uint32_t)(3 + b.s) * (A_TILE >> 4);  // plane h of B
                    bool fresh = true;
                    for (int kb = kb0 + c * CHUNK_KBLOCKS; kb < end; ++kb) {
                        if (!wait_warp(&full[r.s], r.ph, p.err, kErrWaitFull)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t A = sw128_kmajor_desc(smem_u32(ring + (size_t)r.s * STAGE_BYTES));
                        constexpr uint32_t T = A_TILE >> 4;
                        if (leader) {
                            // both small accumulators start with m x (h, m)
#pragma unroll
                            for (int k = 0; k < KSTEPS; ++k)
                                tc_mma_bf16(dy, A + T + 2 * k, A + 3 * T + 2 * k, idesc2, k > 0 ? 1u : small_acc);
                            if (fresh) {
                                // the chunk's first h x h restarts the leading accumulator, which an
                                // N = 256 instruction cannot do without restarting its neighbour
#pragma unroll
                                for (int k = 0; k < KSTEPS; ++k)
                                    tc_mma_bf16(dlead, A + 2 * k, A + bh + 2 * k, idesc1, k > 0 ? 1u : 0u);
#pragma unroll
                                for (int k = 0; k < KSTEPS; ++k)
                                    tc_mma_bf16(dsmall, A + 2 * k, A + (7 * T - bh) + 2 * k, idesc1, 1u);
                            } else {
#pragma unroll
                                for (int k = 0; k < KSTEPS; ++k)
                                    tc_mma_bf16(dh, A + 2 * k, A + 3 * T + 2 * k, idesc2, 1u);
                            }
#pragma unroll
                            for (int k = 0; k < KSTEPS; ++k)  // h x l
                                tc_mma_bf16(dy, A + 2 * k, A + 5 * T + 2 * k, idesc1, 1u);
#pragma unroll
                            for (int k = 0; k < KSTEPS; ++k)  // l x h
                                tc_mma_bf16(dy, A + 2 * T + 2 * k, A + bh + 2 * k, idesc1, 1u);
                            tc_commit(&empty[r.s]);
                        }
                        small_acc = 1u;
                        fresh = false;
                        r.next(STAGES);
                    }
                    if (!ok) break;
                    if (leader) tc_commit(&acc_full[b.s]);
                    b.next(2);
                    if (small_drain_after(c, nchunks)) {
                        if (leader) tc_commit(small_full);
                        ++small_drains;
                        small_pending = true;
                        small_acc = 0;
                    }
                }
            }
        } else {
            // -------------------------------------------- epilogue warps
            const int q4 = warp & 3;                 // TMEM lane quadrant this warp may access
            const int quarter = (warp - 2) >> 2;    // column quarter of the tile
            const int row_in_tile = q4 * 32 + lane;
            const uint32_t lane_off = ((uint32_t)(q4 * 32) << 16) + (uint32_t)(quarter * 32);
            uint64_t hi2[16], lo2[16];  // a packed double-float (hi, lo) per output
#pragma unroll
            for (int j = 0; j < 16; ++j) hi2[j] = lo2[j] = 0ull;
            for (int c = 0; c < nchunks && ok; ++c) {
                // every lane gives up together (the warp shuffles and syncs below need all 32)
                if (!__all_sync(0xffffffffu, mbar_wait_backoff(&acc_full[b.s], b.ph, p.err, kErrWaitMma))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t t0 = tmem_base + lane_off + (b.s ? kX1 : kX0);
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    uint32_t v[8];
                    tmem_ld_32x32b_x8(t0 + cc * 8, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        // TwoSum on pairs: hi + x = sum + e exactly, e added into lo
                        uint64_t& h = hi2[cc * 4 + j];
                        const uint64_t x = pair(v[2 * j], v[2 * j + 1]);
                        const uint64_t sum = f2add(h, x);
                        const uint64_t bp = f2sub(sum, h);
                        const uint64_t e = f2add(f2sub(h, f2sub(sum, bp)), f2sub(x, bp));
                        h = sum;
                        lo2[cc * 4 + j] = f2add(lo2[cc * 4 + j], e);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[b.s]);
                b.next(2);
                if (small_drain_after(c, nchunks)) {
                    // the small products (2^-8 of hh and below) go straight into lo
                    if (!__all_sync(0xffffffffu,
                                    mbar_wait_backoff(small_full, small_drains & 1u, p.err, kErrWaitMma))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
#pragma unroll
                    for (int cc = 0; cc < 8; ++cc) {
                        uint32_t v[8];
                        tmem_ld_32x32b_x8(tmem_base + lane_off + (cc < 4 ? kY0 : kY1) + (cc & 3) * 8, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            lo2[(cc & 3) * 4 + j] = f2add(lo2[(cc & 3) * 4 + j], pair(v[2 * j], v[2 * j + 1]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(small_empty);
                    ++small_drains;
                }
            }
            // the tile's result, 4 columns at a time: each lane forms its own row's values,
            // transpose4 hands lane 4g + j column j of rows 4g .. 4g + 3, and each store then
            // covers 8 rows x 4 consecutive columns of C.  alpha * (hi + lo) + beta * C_old in
            // FP32 double-float steps (TwoSum, products split with fma), rounded once at the
            // end: on this part the FP64 pipe would take ~18 us per tile for it, holding the
            // accumulators the MMAs wait for.  The old values of a pass are fetched together,
            // before its arithmetic (each loaded between two stores, which it may alias, waited
            // for the one before: 10 us more for a 128 x 128 tile that reads C)
            const int64_t row0 = (int64_t)tm * BM + q4 * 32 + (lane & ~3);
            auto emit = [&](int pass, const float (&h)[4], const float (&l)[4]) {
                const int64_t col = (int64_t)tn * BN + quarter * 32 + pass * 4 + (lane & 3);
                float* const cp = p.C + row0 * p.ldc + col;
                bool keep[4];
                float old[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int64_t row = row0 + i;
                    keep[i] = col < p.N && row < p.M &&
                              (p.tri == 0 || (p.tri == 1 ? col - row <= p.tri_off : col - row >= p.tri_off));
                    old[i] = 0.f;
                    if (p.read_c && keep[i]) old[i] = cp[i * p.ldc];
                }
                double v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // (ph, pl) = alpha * (hi + lo), packed
                    const float sh = __fadd_rn(h[j], l[j]), bp = __fsub_rn(sh, h[j]);
                    const float sl = __fadd_rn(__fsub_rn(h[j], __fsub_rn(sh, bp)), __fsub_rn(l[j], bp));
                    const float ph = __fmul_rn(p.alpha, sh);
                    const float pl = __fmaf_rn(p.alpha, sl, __fmaf_rn(p.alpha, sh, -ph));
                    v[j] = __longlong_as_double((long long)pair(__float_as_uint(ph), __float_as_uint(pl)));
                }
                transpose4(v, lane);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint64_t w = (uint64_t)__double_as_longlong(v[i]);
                    const float ph = unpack2(w, 0), pl = unpack2(w, 1);
                    float c;
                    if (p.read_c) {
                        // beta * c = qh + ql and ph + qh = th + tl exactly; one rounding left
                        const float qh = __fmul_rn(p.beta, old[i]), ql = __fmaf_rn(p.beta, old[i], -qh);
                        const float th = __fadd_rn(ph, qh), bq = __fsub_rn(th, ph);
                        const float tl = __fadd_rn(__fsub_rn(ph, __fsub_rn(th, bq)), __fsub_rn(qh, bq));
                        c = __fadd_rn(th, __fadd_rn(tl, __fadd_rn(pl, ql)));
                    } else {
                        c = __fadd_rn(ph, pl);
                    }
                    if (keep[i]) cp[i * p.ldc] = c;
                }
            };
            if (p.cluster == 1) {
                if (ok) {
#pragma unroll
                    for (int pass = 0; pass < 8; ++pass) {
                        float h[4], l[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            h[j] = unpack2(hi2[pass * 2 + (j >> 1)], j & 1);
                            l[j] = unpack2(lo2[pass * 2 + (j >> 1)], j & 1);
                        }
                        emit(pass, h, l);
                    }
                }
            } else {
                // the tile's stages are consumed: its ring carries the partial sums, [column][row]
                uint64_t* part = reinterpret_cast<uint64_t*>(ring);
                if (ok) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        part[(quarter * 32 + j) * BM + row_in_tile] =
                            pair(__float_as_uint(unpack2(hi2[j >> 1], j & 1)), __float_as_uint(unpack2(lo2[j >> 1], j & 1)));
                }
                cluster_sync();
                if (ok) {
                    for (int pass = rank; pass < 8; pass += p.cluster) {
                        float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
                        const uint32_t at = smem_u32(part + (quarter * 32 + pass * 4) * BM + row_in_tile);
                        for_each_rank<4>(at, BM * 8, rank, p.cluster, [&](int j, long long w) {
                            add_double_float(h[j], l[j], unpack2((uint64_t)w, 0), unpack2((uint64_t)w, 1));
                        });
                        emit(pass, h, l);
                    }
                }
                // the next tile's copies come after these reads and writes of the ring
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                cluster_sync();
            }
        }
        if (warp < 2 && p.cluster > 1) {
            cluster_sync();
            cluster_sync();
        }
    }
    if (warp == 1 && leader) {
        // every MMA issued so far has completed before TMEM is released
        tc_commit(done);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(smem_u32(done), 0u) && globaltimer_ns() - t0 < kWaitLimitNs) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------- splits --
// Operand views: element (r, k) of a slot is X[r * sr + k * sk] with either
// sk == 1 (K-major rows) or sr == 1 (K runs down the stored rows).  Planes are
// K-major [rows_pad x k_pad] bf16, zero outside rows x K.

constexpr int ST = 64;  // split tile: 64 rows x 64 K

// x = h + m + l, each the bf16 rounding of the remainder (the remainders are
// exact in FP32 because each bf16 rounding keeps the leading bits).
__global__ void __launch_bounds__(256) split_bf16x3_kernel(const float* __restrict__ X, int64_t sr, int64_t sk,
                                                           int rows, int K, int rows_pad, int k_pad,
                                                           __nv_bfloat16* __restrict__ planes)
{
    __shared__ float t[ST][ST + 1];
    const int r0 = blockIdx.y * ST, k0 = blockIdx.x * ST;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;  // 64 x 4
    for (int i = ty; i < ST; i += 4) {
        // coalesced along the stored contiguous dimension
        int r, k;
        if (sk == 1) { r = r0 + i; k = k0 + tx; } else { r = r0 + tx; k = k0 + i; }
        float v = 0.f;
        if (r < rows && k < K) v = X[(int64_t)r * sr + (int64_t)k * sk];
        if (sk == 1) t[i][tx] = v; else t[tx][i] = v;
    }
    __syncthreads();
    const size_t plane = (size_t)rows_pad * k_pad;
    for (int i = ty; i < ST; i += 4) {
        const int r = r0 + i, k = k0 + tx;
        if (r >= rows_pad || k >= k_pad) continue;
        const float x = t[i][tx];
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        const float r1 = x - __bfloat162float(h);
        const __nv_bfloat16 m = __float2bfloat16_rn(r1);
        const float r2 = r1 - __bfloat162float(m);
        const __nv_bfloat16 l = __float2bfloat16_rn(r2);
        const size_t o = (size_t)r * k_pad + k;
        planes[o] = h;
        planes[plane + o] = m;
        planes[2 * plane + o] = l;
    }
}

// The same split for a K-major source whose rows start on 16-byte boundaries
// (the A slots of row-major operands): thread (k8, row) splits 8 consecutive K
// with two 16-byte loads and one 16-byte store per piece plane; no staging.
// Grid: x over k_pad / 8 in blocks of 256 threads, y over rows_pad.
__device__ __forceinline__ uint32_t bf16_pair(float a, float b)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}

__global__ void __launch_bounds__(256) split_bf16x3_rows_kernel(const float* __restrict__ X, int64_t sr, int rows,
                                                                int K, int rows_pad, int k_pad,
                                                                __nv_bfloat16* __restrict__ planes)
{
    const int r = blockIdx.y;
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) * 8;
    if (k >= k_pad) return;
    float x[8];
    if (r < rows && k + 8 <= K) {
        const float4* src = reinterpret_cast<const float4*>(X + (int64_t)r * sr + k);
        const float4 a = __ldg(src), b = __ldg(src + 1);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = (r < rows && k + j < K) ? X[(int64_t)r * sr + k + j] : 0.f;
    }
    uint32_t hw[4], mw[4], lw[4];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        float h2[2], r1[2], m2[2], r2[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            h2[q] = __bfloat162float(__float2bfloat16_rn(x[j + q]));
            r1[q] = x[j + q] - h2[q];
            m2[q] = __bfloat162float(__float2bfloat16_rn(r1[q]));
            r2[q] = r1[q] - m2[q];
        }
        hw[j / 2] = bf16_pair(h2[0], h2[1]);
        mw[j / 2] = bf16_pair(m2[0], m2[1]);
        lw[j / 2] = bf16_pair(r2[0], r2[1]);
    }
    const size_t plane = (size_t)rows_pad * k_pad, o = (size_t)r * k_pad + k;
    *reinterpret_cast<uint4*>(planes + o) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    *reinterpret_cast<uint4*>(planes + plane + o) = make_uint4(mw[0], mw[1], mw[2], mw[3]);
    *reinterpret_cast<uint4*>(planes + 2 * plane + o) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

// CTAs per tile: the size whose busiest cluster finishes first, in K blocks; the exchange
// of the partial sums costs about as much as kExchange of them.
constexpr int64_t kExchange = 4;
int cluster_size(const ClusterCounts& n, int64_t tiles, int64_t kblocks)
{
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int c = 1; c <= MAX_CLUSTER; c *= 2) {
        if (n.at_once[c] <= 0) continue;
        const int64_t t = (tiles + n.at_once[c] - 1) / n.at_once[c] * ((kblocks + c - 1) / c + (c > 1 ? kExchange : 0));
        if (t < cost) { cost = t; best = c; }
    }
    return best;
}

}  // namespace

int launch_split_bf16x3(const float* X, int64_t sr, int64_t sk, int rows, int K, int rows_pad, int k_pad, void* planes,
                        void* stream, std::string& why)
{
    if (sk == 1 && sr % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0 && k_pad % 8 == 0 &&
        reinterpret_cast<uintptr_t>(planes) % 16 == 0 && rows_pad <= 65535) {
        dim3 grid((unsigned)((k_pad / 8 + 255) / 256), (unsigned)rows_pad);
        split_bf16x3_rows_kernel<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(
            X, sr, rows, K, rows_pad, k_pad, static_cast<__nv_bfloat16*>(planes));
    } else {
        dim3 grid((unsigned)((k_pad + ST - 1) / ST), (unsigned)((rows_pad + ST - 1) / ST));
        split_bf16x3_kernel<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(
            X, sr, sk, rows, K, rows_pad, k_pad, static_cast<__nv_bfloat16*>(planes));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { why = std::string("split_bf16x3: ") + cudaGetErrorString(e); return OOC_ERR_CUDA; }
    return OOC_OK;
}

int launch_bf16x3_tiles(const TcProblem& P, void* stream, std::string& why)
{
    if (P.M <= 0 || P.N <= 0) return OOC_OK;
    static const ClusterCounts counts = count_clusters((const void*)bf16x3_tile_kernel, THREADS, SMEM_BYTES);
    if (counts.at_once[1] <= 0) { why = "bf16x3 tile kernel: shared memory attribute"; return OOC_ERR_CUDA; }
    if (P.k_pad % BK) { why = "K padding not a multiple of the K block"; return OOC_ERR_INVALID_ARG; }
    TcArgs a;
    std::memset(&a, 0, sizeof(a));
    a.M = (int)P.M; a.N = (int)P.N;
    a.kblocks = (int)(P.k_pad / BK);
    a.tiles_n = (int)((P.N + BN - 1) / BN);
    a.tiles_m = (int)((P.M + BM - 1) / BM);
    a.tiles = a.tiles_m * a.tiles_n;
    a.alpha = P.alpha; a.beta = P.beta;
    a.read_c = P.read_c ? 1 : 0;
    a.C = P.C; a.ldc = P.ldc;
    a.err = P.err;
    a.tri = P.tri; a.tri_off = P.tri_off;
    CUtensorMap ma, mb;
    std::memset(&ma, 0, sizeof(ma));
    std::memset(&mb, 0, sizeof(mb));
    if (a.kblocks > 0) {  // K == 0 runs the epilogue only (C = beta * C)
        int rc = encode_map_3d_bf16(&ma, P.a_planes, (uint64_t)P.k_pad, (uint64_t)P.a_rows_pad, 3, BK, BM, why);
        if (rc) return rc;
        rc = encode_map_3d_bf16(&mb, P.b_planes, (uint64_t)P.k_pad, (uint64_t)P.b_rows_pad, 3, BK, BN, why);
        if (rc) return rc;
    }
    a.cluster = cluster_size(counts, a.tiles, a.kblocks);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    cluster_config(cfg, at, a.cluster, std::min(a.tiles, counts.at_once[a.cluster]), THREADS, SMEM_BYTES,
                   static_cast<cudaStream_t>(stream));
    const cudaError_t e = cudaLaunchKernelEx(&cfg, bf16x3_tile_kernel, ma, mb, a);
    if (e != cudaSuccess) cudaGetLastError();
    if (e != cudaSuccess) { why = std::string("bf16x3 tile launch: ") + cudaGetErrorString(e); return OOC_ERR_CUDA; }
    return OOC_OK;
}

}  // namespace ooc
