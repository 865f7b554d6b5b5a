// The FP64-accurate Ozaki form on the 5th-generation tensor cores (sm_103a): the
// compute stage of the out-of-core pipeline for OOC_FORM_OZAKI, after Ozaki, Ogita,
// Oishi and Rump's error-free splitting of matrix products.
//
// Digits.  Every row of A (column of B) is scaled by a power of two 2^e so that its
// largest entry is below 1 in magnitude; the value, rounded to a fixed-point number
// of 8 S bits, is cut into S balanced digits of 8 bits, x = 2^(e+1) sum_s d_s 2^(-8 s)
// with d_s in [-128, 128], each exact in bf16.  Products of digit planes accumulate
// exactly in FP32 over at most 1024 products of two digits (1024 x 128^2 = 2^24), and
// the products with s + t <= S + 1 are added with their weight 2^(-8 (s + t)).
// Eight balanced bits per digit carry what digits of 6 truncated bits (|d| <= 63,
// the width an exact sum over 4096 needs) carry in 4/3 of the planes: 6 planes and 21
// products where 8 and 36 were needed, 7 and 28 for 9 and 45.  Rounding to nearest
// leaves no bias, and the largest dropped product shrinks from 63^2 2^-6(S6+2) to
// 2^14 2^-(8(S+2)-2), so the error bound of the 6-bit digits holds with room.
//
// Sums.  The exact FP32 sums go into one 64-bit fixed-point integer per output (unit
// 2^-frac): to an integer by packed FP32 additions of large constants (the conversion
// unit is a quarter as wide as these pipes), then one wide multiply-add.  In FP64 the same drain is bound by the FP64 pipe
// (1.75 additions a clock and SM: 9400 clocks per 128 x 128 sum, which takes the
// tensor cores 4096 clocks to make).  Sums on diagonals 8 m <= frac are added exactly,
// finer ones are rounded to the unit first.  Where that would cost more than the dropped
// products (seven and eight planes but for short K, six beyond K 2^18; one_unit), the wide
// kernel takes the fine diagonals first, in a unit 2^16 times finer, puts the low 16 bits
// of their sums away in shared memory and goes on with the rest shifted to the unit: 80 bits
// in all, rounded once.  The order of integer additions does not matter, and rounded sums are
// cut where they are rounded (cut_stages), so the result does not depend on how a tile's
// work is cut.
//
// Kernel shape: tile 128 x 128, 64 of K per stage, 18 warps.
//   warp 0      TMA producer: the bf16 tiles of one A plane and of two neighbouring B
//               planes (48 KiB, 128-byte swizzle) into a ring of four stages;
//   warp 1      allocates all 512 TMEM columns and issues tcgen05.mma: the two B plane
//               tiles lie back to back, so one N = 256 instruction makes both products
//               (it reads A once for both: 96 bytes of shared memory a clock instead of
//               the 128 of two N = 128 ones, which leaves room for the TMA writes);
//   warps 2-17  drain: finished sums into the 64-bit integers in registers, 32
//               columns of one row per thread; after the tile's last sum they write
//               alpha 2^(e_i + f_j) sum + beta C, each store covering 8 rows x 4
//               consecutive columns (4 x 4 transposes by shuffles).
// TMEM: two buffers of two 128-column accumulators (neighbouring diagonals s + t).
//
// Order of the products: diagonals in pairs (d, d + 1); a group is one A plane s with
// the B planes d - s and d - s + 1, and one single product (A plane d, B plane 1)
// completes the pair.  When K is short the groups of a pair share one accumulator
// pair (their sum is still exact); when it is long each group has its own, drained
// every 1024 of K.  The host takes whichever drains less often (plan_units).
//
// Clusters: when a launch has fewer tiles than SMs, the CTAs of a cluster share each
// tile.  Each takes a contiguous share of the tile's stages, puts its 64-bit partial
// sums in shared memory, and the cluster adds them through distributed shared memory.
// Cluster barriers sit in loops that every thread walks whatever happens, so a CTA
// whose bounded wait gave up still arrives.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>

#include "ooc_internal.hpp"
#include "tc_common.cuh"

namespace ooc {

namespace {

constexpr int BM = 128, BN = 128, BK = 64;
constexpr int DIGIT = 8;                              // bits per digit
constexpr int EXACT_KBLOCKS = 1024 / BK;              // K blocks x products whose FP32 sum stays exact
constexpr uint32_t TILE_BYTES = BM * BK * 2u;         // one plane tile: 128 rows x 64 bf16 (16 KiB)
constexpr uint32_t STAGE_BYTES = 3 * TILE_BYTES;      // A plane, two B planes
constexpr int STAGES = 4;
constexpr uint32_t RING_BYTES = STAGES * STAGE_BYTES;
constexpr uint32_t LOW_BYTES = BM * BN * 2u;          // wide kernel: 16 low bits per output
constexpr size_t SMEM_BYTES = 1024 + RING_BYTES + 256;
constexpr int EPI_WARPS = 16;                         // 4 per TMEM lane quadrant, 32 columns each
constexpr int THREADS = (2 + EPI_WARPS) * 32;
constexpr int KSTEPS = BK / 16;
constexpr int MAX_PLANES = 8;
constexpr int MAX_GROUPS = 20;                        // 8 planes: 16 double and 4 single groups
constexpr int MAX_UNITS = MAX_GROUPS;
constexpr int MAX_CLUSTER = 8;
static_assert(RING_BYTES >= (uint32_t)BM * BN * 8, "the ring holds a tile of 64-bit partial sums");
static_assert(SMEM_BYTES + LOW_BYTES <= 227 * 1024, "the wide kernel fits an SM");

// One group: A plane a with B planes b and b + 1 (nb == 2), or with plane b alone, whose
// product goes into the second accumulator.
struct Group {
    int8_t a, b, nb, pad;
};

// A unit shares one accumulator pair: `ngroups` groups from `first`, drained every
// `chunk` K blocks.  The two accumulators' weights as a factor applied in FP32 (a
// power of two, sums are rounded to integers after it) and a left shift.  fine: in the wide
// kernel's finer unit; those units come first.
struct Unit {
    int16_t first, ngroups, chunk, fine;
    float scale[2];
    int32_t shift[2];
};

struct Args {
    int M, N;
    int kb0, kblocks;      // K blocks [kb0, kb0 + kblocks) of the planes
    int tiles_m, tiles_n, tiles;
    int nunits;
    int cluster;           // CTAs that share a tile
    int cut[MAX_CLUSTER + 1];  // CTA r of a cluster takes stages [cut[r], cut[r + 1]) of a tile
    int frac;              // the integers' unit is 2^-frac
    double alpha, beta;
    int alpha_one;         // 1: alpha is one, -1: minus one (no multiplication on the FP64 pipe)
    int read_c;
    double* C;
    int64_t ldc;
    const int* row_exp;
    const int* col_exp;
    int* err;
    int tri;               // 0 full update, 1 lower (col - row <= tri_off), 2 upper (col - row >= tri_off)
    int64_t tri_off;
    Unit unit[MAX_UNITS];
    Group group[MAX_GROUPS];
};

// The stages of a tile that this CTA takes, walked in order by every role: each call
// of fn(unit, group0, kb0, nk, lo, hi) is one drain -- the stages [lo, hi) of the
// ngroups x nk block of (group, K block) pairs of one unit and one K chunk.
template <class Fn>
__device__ __forceinline__ bool walk(const Args& p, int begin, int end, Fn fn)
{
    int pos = 0;
    for (int u = 0; u < p.nunits; ++u) {
        const Unit& un = p.unit[u];
        for (int k0 = 0; k0 < p.kblocks; k0 += un.chunk) {
            const int nk = min((int)un.chunk, p.kblocks - k0);
            const int n = un.ngroups * nk;
            const int lo = max(begin - pos, 0), hi = min(end - pos, n);
            pos += n;
            if (lo < hi && !fn(un, k0, nk, lo, hi)) return false;
            if (pos >= end) return true;
        }
    }
    return true;
}

__device__ __forceinline__ uint64_t f2fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// v * sc for two FP32 sums v, |v * sc| <= 2^24, rounded to the nearest integer (ties to
// even).  Adding 1.5 2^25 rounds to a multiple of 4, h, and leaves h / 4 in the low bits;
// the rest, exact and at most 2 in magnitude, is rounded by adding 1.5 2^23, and 4 being
// even the tie rule is that of the whole.
__device__ __forceinline__ void round_pair(uint64_t v, uint64_t sc, int& i0, int& i1)
{
    const uint64_t big = pair(50331648.0f), one = pair(12582912.0f);
    const uint64_t t = f2fma(v, sc, big);
    const uint64_t u = f2add(f2fma(v, sc, f2sub(big, t)), one);
    constexpr uint32_t bias = 0x4C400000u * 4u + 0x4B400000u;  // what the two constants leave
    i0 = (int)(((uint32_t)t << 2) + (uint32_t)u - bias);
    i1 = (int)(((uint32_t)(t >> 32) << 2) + (uint32_t)(u >> 32) - bias);
}

// Results outside the normal range, rounded by the library.
__device__ __noinline__ double scaled_slowly(long long t, int e) { return ldexp((double)t, e); }

// t * 2^e, rounded once (to nearest, ties to even) from the 64-bit integer, with 32-bit
// integer operations: every instruction per output on the FP64 pipe holds it for 9700
// clocks a tile, a comparison as much as a conversion, a scaling or a multiplication.
__device__ __forceinline__ double fixed_to_f64(long long t, int e)
{
    const long long sign = t >> 63;
    const unsigned long long a = (unsigned long long)((t ^ sign) - sign);
    const uint32_t h = (uint32_t)(a >> 32), l = (uint32_t)a;
    const uint32_t top = h ? h : l, next = h ? l : 0u;
    const int lz = __clz((int)top);
    const uint32_t x = __funnelshift_l(next, top, lz), y = next << (lz & 31);  // bit 31 of x set (t != 0)
    const int be = 1023 + 63 - lz - (h ? 0 : 32) + e;  // biased exponent before rounding
    if ((uint32_t)(be - 1) >= 2045u && top) return scaled_slowly(t, e);
    const uint32_t ml = __funnelshift_r(y, x, 11);      // the 53 bits of x : y above the 11 dropped ones
    const uint32_t up = ((y & 0x7FFu) + 0x3FFu + (ml & 1u)) >> 11;
    // the implicit bit of the mantissa (and a carry out of the rounding) adds to the exponent
    const uint32_t mh = ((uint32_t)(be - 1) << 20) + (x >> 11);
    const unsigned long long m = (((unsigned long long)mh << 32) | ml) + up;
    const uint32_t hi = (uint32_t)(m >> 32) | ((uint32_t)sign & 0x80000000u);
    return top ? __hiloint2double((int)hi, (int)(uint32_t)m) : 0.0;
}

// The leading bits of 2^16 t + r (0 <= r < 2^16) as one integer times 2^up, with room for its
// negation.  Bits that do not fit set the lowest one (rounding to odd): at least 60 bits are
// left then, so that rounding to 53 sees the same as from all of them.
__device__ __forceinline__ long long joined(long long t, uint32_t r, int& up)
{
    const int s = min(16, max(0, __clzll(t ^ (t >> 63)) - 2));
    up = 16 - s;
    return (long long)((unsigned long long)t << s) | (r >> up) | ((r & ((1u << up) - 1u)) != 0 ? 1 : 0);
}

template <bool kWide>
__global__ void __launch_bounds__(THREADS, 1) ozaki_tile_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                const __grid_constant__ CUtensorMap tmB,
                                                                const __grid_constant__ Args p)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + RING_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* done = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    uint64_t* low = reinterpret_cast<uint64_t*>(ring + RING_BYTES + 256);  // [4 columns][row], 16 bits each

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
        mbar_init(done, 1);
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int rank = (int)blockIdx.x % p.cluster;
    const int first = (int)blockIdx.x / p.cluster, stride = (int)gridDim.x / p.cluster;
    const int begin = p.cut[rank], end = p.cut[rank + 1];

    Ring r, b;               // stage ring (producer, MMA), accumulator buffers (MMA, drain)
    uint32_t issued = 0;     // producer: stages issued
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
                const int arow = tm * BM, brow = tn * BN;
                ok = walk(p, begin, end, [&](const Unit& un, int k0, int nk, int lo, int hi) {
                    int gi = lo / nk, kb = lo - gi * nk;
                    for (int i = lo; i < hi; ++i) {
                        const Group g = p.group[un.first + gi];
                        if (!wait_warp(&empty[r.s], r.ph ^ 1u, p.err, kErrWaitEmpty)) return false;
                        if (leader) {
                            unsigned char* st = ring + (size_t)r.s * STAGE_BYTES;
                            mbar_arrive_expect_tx(&full[r.s], (1 + g.nb) * TILE_BYTES);
                            const int x = (p.kb0 + k0 + kb) * BK;
                            tma_load_3d(st, &tmA, &full[r.s], x, arow, g.a);
                            tma_load_3d(st + TILE_BYTES, &tmB, &full[r.s], x, brow, g.b);
                            if (g.nb == 2) tma_load_3d(st + 2 * TILE_BYTES, &tmB, &full[r.s], x, brow, g.b + 1);
                        }
                        r.next(STAGES);
                        ++issued;
                        if (++kb == nk) { kb = 0; ++gi; }
                    }
                    return true;
                });
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
                ok = walk(p, begin, end, [&](const Unit& un, int, int nk, int lo, int hi) {
                    if (!wait_warp(&acc_empty[b.s], b.ph ^ 1u, p.err, kErrWaitAcc)) return false;
                    tc_fence_after();
                    const uint32_t d = tmem_base + (uint32_t)b.s * 2 * BN;
                    int gi = lo / nk, left = nk - (lo - gi * nk);
                    bool two = p.group[un.first + gi].nb == 2;
                    uint32_t acc = 0;
                    for (int i = lo; i < hi; ++i) {
                        if (!wait_warp(&full[r.s], r.ph, p.err, kErrWaitFull)) return false;
                        tc_fence_after();
                        const uint64_t da = sw128_kmajor_desc(smem_u32(ring + (size_t)r.s * STAGE_BYTES));
                        const uint64_t db = da + (TILE_BYTES >> 4);
                        if (leader) {
                            const uint32_t dst = two ? d : d + BN, idesc = two ? idesc2 : idesc1;
#pragma unroll
                            for (int k = 0; k < KSTEPS; ++k)
                                tc_mma_bf16(dst, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : acc);
                            tc_commit(&empty[r.s]);
                        }
                        acc = 1u;
                        r.next(STAGES);
                        if (--left == 0) {
                            left = nk;
                            ++gi;
                            if (i + 1 < hi) two = p.group[un.first + gi].nb == 2;
                        }
                    }
                    if (leader) tc_commit(&acc_full[b.s]);
                    b.next(2);
                    return true;
                });
            }
        } else {
            // -------------------------------------------- drain and epilogue
            const int q4 = warp & 3;                // TMEM lane quadrant this warp may access
            const int quarter = (warp - 2) >> 2;    // column quarter of the tile
            const int row_in_tile = q4 * 32 + lane;
            const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
            long long acc[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = 0;
            uint64_t* const low_me = low + quarter * 8 * BM + row_in_tile;
            auto put_away = [&] {
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    uint64_t w = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        w |= (uint64_t)(acc[j + i] & 0xFFFF) << (16 * i);
                        acc[j + i] >>= 16;
                    }
                    low_me[j / 4 * BM] = w;
                }
            };
            bool fine = kWide;  // the sums so far are in the finer unit
            if (ok)
                ok = walk(p, begin, end, [&](const Unit& un, int, int nk, int lo, int) {
                    // every lane gives up together (the warp shuffles and syncs below need all 32)
                    if (!__all_sync(0xffffffffu, mbar_wait_backoff(&acc_full[b.s], b.ph, p.err, kErrWaitMma)))
                        return false;
                    tc_fence_after();
                    const uint32_t t0 = tmem_base + lane_off + (uint32_t)(b.s * 2 * BN + quarter * 32);
                    if constexpr (kWide) {
                        if (fine && !un.fine) {
                            put_away();
                            fine = false;
                        }
                    }
                    // the pair's single product comes last: alone, it leaves the first accumulator unused
                    const int q0 = p.group[un.first + lo / nk].nb == 2 ? 0 : 1;
#pragma unroll 1
                    for (int q = q0; q < 2; ++q) {
                        const uint64_t sc = pair(un.scale[q]);
                        const int sh = un.shift[q], mul = 1 << (sh & 31);
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            uint32_t v[8];
                            tmem_ld_32x32b_x8(t0 + q * BN + cc * 8, v);
                            tmem_wait_ld();
#pragma unroll
                            for (int j = 0; j < 8; j += 2) {
                                int s0, s1;
                                round_pair(pair(v[j], v[j + 1]), sc, s0, s1);
                                long long &a0 = acc[cc * 8 + j], &a1 = acc[cc * 8 + j + 1];
                                if (sh < 32) {
                                    a0 += (long long)s0 * mul;
                                    a1 += (long long)s1 * mul;
                                } else {  // reaches the high word only
                                    a0 += (long long)((unsigned long long)((unsigned)s0 * mul) << 32);
                                    a1 += (long long)((unsigned long long)((unsigned)s1 * mul) << 32);
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[b.s]);
                    b.next(2);
                    return true;
                });
            if constexpr (kWide) {
                if (fine) put_away();
            }
            // the tile's result, 4 columns at a time: each lane forms its own row's values,
            // transpose4 hands lane 4g + j column j of rows 4g .. 4g + 3, and each store then
            // covers 8 rows x 4 consecutive columns of C (whole 32-byte sectors).  The old values
            // of a pass are fetched before its conversions, so that they arrive behind them.
            // One load per lane brings the exponents of its row and of column `lane` of the quarter
            // (none when K == 0).
            const int64_t row_me = (int64_t)tm * BM + row_in_tile, col_me = (int64_t)tn * BN + quarter * 32 + lane;
            const int ce_lane = p.col_exp && col_me < p.N ? p.col_exp[col_me] : 0;
            const int re = (p.row_exp && row_me < p.M ? p.row_exp[row_me] : 0) + 2 - p.frac;
            const int row0 = tm * BM + q4 * 32 + (lane & ~3), col0 = tn * BN + quarter * 32 + (lane & 3);
            double* const c_lane = p.C + (int64_t)row0 * p.ldc + col0;
            const int rows_left = p.M - row0;
            // read_c and scale are compile-time: a predicated-off instruction holds the FP64 pipe too
            // t: sums in the unit; r: the wide kernel's 16 bits below it
            auto emit = [&](auto read_c, auto scale, int pass, const long long (&t)[4], const uint32_t (&r)[4]) {
                const int col = col0 + pass * 4;
                double* const c = c_lane + pass * 4;
                bool keep[4];
                double old[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) keep[i] = col < p.N && i < rows_left;
                if (p.tri) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int64_t d = (int64_t)col - (row0 + i);
                        keep[i] = keep[i] && (p.tri == 1 ? d <= p.tri_off : d >= p.tri_off);
                    }
                }
                if constexpr (read_c.value) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) old[i] = keep[i] ? c[i * p.ldc] : 0.0;
                }
                double v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int up = 16;
                    const long long w = kWide ? joined(t[j], r[j], up) : t[j];
                    v[j] = fixed_to_f64(p.alpha_one < 0 ? -w : w,
                                        re + up - 16 + __shfl_sync(0xffffffffu, ce_lane, pass * 4 + j));
                }
                if constexpr (scale.value) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] *= p.alpha;
                }
                transpose4(v, lane);
                if constexpr (read_c.value) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = fma(p.beta, old[i], v[i]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (keep[i]) c[i * p.ldc] = v[i];
            };
            long long* part = reinterpret_cast<long long*>(ring);  // [column][row]
            if (p.cluster > 1) {
                // the tile's stages are consumed: its ring carries the partial sums
                if (ok) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) part[(quarter * 32 + j) * BM + row_in_tile] = acc[j];
                }
                cluster_sync();
            }
            auto store = [&](auto read_c, auto scale) {
                if (p.cluster == 1) {
#pragma unroll
                    for (int pass = 0; pass < 8; ++pass) {
                        const long long t[4] = {acc[pass * 4], acc[pass * 4 + 1], acc[pass * 4 + 2], acc[pass * 4 + 3]};
                        uint32_t r[4] = {0, 0, 0, 0};
                        if constexpr (kWide) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) r[j] = (uint32_t)(low_me[pass * BM] >> (16 * j)) & 0xFFFFu;
                        }
                        emit(read_c, scale, pass, t, r);
                    }
                    return;
                }
#pragma unroll 1
                for (int pass = rank; pass < 8; pass += p.cluster) {
                    long long t[4] = {0, 0, 0, 0};
                    const uint32_t at = smem_u32(part + (quarter * 32 + pass * 4) * BM + row_in_tile);
                    for_each_rank<4>(at, BM * 8, rank, p.cluster, [&](int j, long long w) { t[j] += w; });
                    uint32_t r[4] = {0, 0, 0, 0};
                    if constexpr (kWide) {
                        for_each_rank<1>(smem_u32(low_me + pass * BM), 0, rank, p.cluster, [&](int, long long w) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) r[j] += (uint32_t)((uint64_t)w >> (16 * j)) & 0xFFFFu;
                        });
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            t[j] += r[j] >> 16;
                            r[j] &= 0xFFFFu;
                        }
                    }
                    emit(read_c, scale, pass, t, r);
                }
            };
            if (ok) {
                if (p.alpha_one == 0) {
                    if (p.read_c) store(std::true_type{}, std::true_type{});
                    else store(std::false_type{}, std::true_type{});
                } else if (p.read_c) {
                    store(std::true_type{}, std::false_type{});
                } else {
                    store(std::false_type{}, std::false_type{});
                }
            }
            if (p.cluster > 1) {
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

constexpr int ST = 64;      // split tile: 64 rows x 64 K
constexpr int MAX_K = 2048; // K per block of the row-maximum kernel (K-major)

__device__ __forceinline__ unsigned long long abs_bits(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// max |x| over each row (as the bit pattern of a non-negative double, which orders
// like its value); rowmax must start at zero.  One row and MAX_K of K per block.
__global__ void __launch_bounds__(256) rowmax_rows_kernel(const double* __restrict__ X, int64_t sr, int K,
                                                          unsigned long long* __restrict__ rowmax)
{
    __shared__ unsigned long long wm[8];
    const double* x = X + (int64_t)blockIdx.x * sr;
    unsigned long long m = 0;
    for (int64_t b = (int64_t)blockIdx.y * MAX_K; b < K; b += (int64_t)gridDim.y * MAX_K) {
        const int64_t k1 = min((int64_t)K, b + MAX_K);
#pragma unroll 8
        for (int64_t k = b + threadIdx.x; k < k1; k += 256) m = max(m, abs_bits(__ldg(x + k)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = max(m, wm[w]);
        if (m) atomicMax(&rowmax[blockIdx.x], m);
    }
}

// The same with K down the stored rows: 64 rows and 256 of K per block, one row and
// 64 of K per thread.
__global__ void __launch_bounds__(256) rowmax_cols_kernel(const double* __restrict__ X, int64_t sk, int rows, int K,
                                                          unsigned long long* __restrict__ rowmax)
{
    __shared__ unsigned long long t[4][ST];
    const int c = threadIdx.x & 63, q = threadIdx.x >> 6;
    const int r = blockIdx.y * ST + c;
    const int64_t k0 = (int64_t)blockIdx.x * 256, k1 = min((int64_t)K, k0 + 256);
    unsigned long long m = 0;
    if (r < rows) {
#pragma unroll 8
        for (int64_t k = k0 + q; k < k1; k += 4) m = max(m, abs_bits(__ldg(X + k * sk + r)));
    }
    t[q][c] = m;
    __syncthreads();
    if (q == 0 && r < rows) {
        m = max(max(t[0][c], t[1][c]), max(t[2][c], t[3][c]));
        if (m) atomicMax(&rowmax[r], m);
    }
}

// exponent e with max|x| < 2^e (0 for an all-zero row)
__device__ __forceinline__ int exponent_of(unsigned long long rowmax)
{
    if (!rowmax) return 0;
    const int biased = (int)((rowmax >> 52) & 0x7FF);
    return (biased ? biased - 1023 : -1022) + 1;
}

// The fixed-point value x 2^(8 S - 1 - e), rounded to nearest.  |x| < 2^e, so it is at
// most 2^(8 S - 1) in magnitude; for S = 8 it has no bits to round off at that size
// and stays below 2^63.
__device__ __forceinline__ long long fixed_point(double x, int e, int S)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int biased = (int)((bits >> 52) & 0x7FF);
    unsigned long long mant = bits & ((1ull << 52) - 1ull);
    if (biased) mant |= 1ull << 52;
    const int ex = biased ? biased - 1023 : -1022;  // |x| = mant * 2^(ex - 52)
    const int shift = ex - 52 + DIGIT * S - 1 - e;
    unsigned long long F;
    if (shift >= 0) F = mant << shift;              // at most DIGIT S - 54 for entries of this row
    else F = shift > -64 ? (mant + (1ull << (-shift - 1))) >> -shift : 0ull;
    return (bits >> 63) ? -(long long)F : (long long)F;
}

// S balanced digits (most significant first) of 8 consecutive K of a row: one 16-byte
// store per plane at element offset o.
__device__ __forceinline__ void store_digits(const double (&x)[8], int e, int S, __nv_bfloat16* planes, size_t plane,
                                             size_t o)
{
    long long F[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) F[j] = fixed_point(x[j], e, S);
    for (int s = S - 1; s >= 0; --s) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            int d[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // the low 8 bits as a signed digit, the rest carried on; the top digit is what is left
                d[h] = s > 0 ? (int)(signed char)(F[j + h] & 0xFF) : (int)F[j + h];
                F[j + h] = (F[j + h] - d[h]) >> DIGIT;
            }
            const __nv_bfloat162 b = __floats2bfloat162_rn((float)d[0], (float)d[1]);
            w[j / 2] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(planes + (size_t)s * plane + o) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Digit planes and row exponents from the row maxima: 64 rows x 64 K per block.
__global__ void __launch_bounds__(256) split_kernel(const double* __restrict__ X, int64_t sr, int64_t sk, int rows,
                                                    int K, int rows_pad, int k_pad,
                                                    const unsigned long long* __restrict__ rowmax, int S,
                                                    __nv_bfloat16* __restrict__ planes, int* __restrict__ rowexp)
{
    __shared__ double t[ST][ST + 1];  // [k][row], operands with K down the stored rows
    const int r0 = blockIdx.y * ST, k0 = blockIdx.x * ST;
    if (sk != 1) {
        const int c = threadIdx.x & 63;
        for (int i = threadIdx.x >> 6; i < ST; i += 4)
            t[i][c] = (r0 + c < rows && k0 + i < K) ? __ldg(X + (int64_t)(k0 + i) * sk + r0 + c) : 0.0;
        __syncthreads();
    }
    const int g = threadIdx.x & 7;
    for (int i = threadIdx.x >> 3; i < ST; i += 32) {
        const int r = r0 + i, k = k0 + g * 8;
        if (r >= rows_pad || k >= k_pad) continue;
        const int e = r < rows ? exponent_of(rowmax[r]) : 0;
        if (k == 0) rowexp[r] = e;
        double x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (sk != 1) x[j] = t[g * 8 + j][i];
            else x[j] = (r < rows && k + j < K) ? __ldg(X + (int64_t)r * sr + k + j) : 0.0;
        }
        store_digits(x, e, S, planes, (size_t)rows_pad * k_pad, (size_t)r * k_pad + k);
    }
}

// The whole split in one launch, for short K: each block finds the maxima of FR rows over all
// of K and then cuts them, reading them again from L1 / L2.
constexpr int FR = 16, FK = 128;
template <bool kKMajor>
__global__ void __launch_bounds__(256) split_short_kernel(const double* __restrict__ X, int64_t ld, int rows, int K,
                                                          int rows_pad, int k_pad, int S,
                                                          __nv_bfloat16* __restrict__ planes, int* __restrict__ rowexp)
{
    __shared__ unsigned long long part[FR][17];
    __shared__ int ex[FR];
    __shared__ double t[kKMajor ? 1 : FK][FR + 1];  // [k][row], operands with K down the stored rows
    const int r0 = blockIdx.x * FR, tid = threadIdx.x;
    // 16 threads per row: along K when it is contiguous, along the rows when they are
    const int row = kKMajor ? tid >> 4 : tid & 15, q = kKMajor ? tid & 15 : tid >> 4;
    auto at = [&](int r, int64_t k) { return __ldg(X + (kKMajor ? (int64_t)r * ld + k : k * ld + r)); };
    unsigned long long m = 0;
    if (r0 + row < rows) {
#pragma unroll 8
        for (int k = q; k < K; k += 16) m = max(m, abs_bits(at(r0 + row, k)));
    }
    part[row][q] = m;
    __syncthreads();
    if (tid < FR) {
        m = part[tid][0];
#pragma unroll
        for (int i = 1; i < 16; ++i) m = max(m, part[tid][i]);
        ex[tid] = exponent_of(m);
        if (r0 + tid < rows_pad) rowexp[r0 + tid] = ex[tid];
    }
    __syncthreads();
    const int i = tid >> 4, g = tid & 15;  // this thread's row and group of 8 K
    for (int k0 = 0; k0 < k_pad; k0 += FK) {
        if (!kKMajor) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < FK; u += 16)
                t[u + q][row] = r0 + row < rows && k0 + u + q < K ? at(r0 + row, k0 + u + q) : 0.0;
            __syncthreads();
        }
        const int r = r0 + i, k = k0 + g * 8;
        if (r >= rows_pad || k >= k_pad) continue;
        double x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            x[j] = kKMajor ? (r < rows && k + j < K ? at(r, k + j) : 0.0) : t[kKMajor ? 0 : g * 8 + j][i];
        store_digits(x, ex[i], S, planes, (size_t)rows_pad * k_pad, (size_t)r * k_pad + k);
    }
}
// K up to which the one-launch split is taken: a block walks K serially, 16 rows at a time,
// so it pays while that walk is shorter than the clear, the maxima and the cut of the general
// one (both operands: K 64 43 -> 23 us, 512 81 -> 55, 1024 144 -> 119, but 1900 61 -> 103).
constexpr int kShortSplit = 1024;

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// The integers' unit of a launch over `kblocks` K blocks, 2^-frac: |sum| <= (128 / 255)^2 K <
// 0.253 K, so 2^(64 - ceil(log2 K)) units stay below 2^62.02.
int unit_bits(int64_t kblocks)
{
    int lg = 6;
    while (((int64_t)1 << lg) < kblocks * BK) ++lg;
    return 64 - lg;
}

// Whether that unit holds the sums of `planes` planes with room: all of them exactly, or what
// is rounded costs less than the products that S = 4/3 planes slices of 6 bits drop.  Those are
// sqrt(K) 2^(-6 S - 2.2) of the operands' scales; one rounding in 1024 of K of each sum finer
// than the unit, 11 to 22 of them, is sqrt(K) 2^(-frac - 4.5) or less.  So one unit does to K
// 2^18 for six planes, 4096 for seven, 64 for eight.  With one throughout, ten slices were 3 to
// 66 times less accurate than FP64 sums of the digit products from K 2048 to 65536 (N(0,1)
// 9.8e-16 for 1.2e-16 at 4096, 2.4e-14 for 3.7e-16 at 65536) and nine up to ten times from 16384
// (4.7e-14 for 4.8e-15 at 65536, sign 10^U(-4,4)); the wide kernel's error is half of those sums'
// or less throughout (below 1e-16 and 1e-15 at 65536) and costs 1-8 % (9 slices 4096 x 4096 x
// 8192 10.3 -> 10.6 ms, 3000 x 2000 x 16384 in 256 MiB 37.1 -> 40.0; 10 slices 4096 x 4096 x 2048
// 3.18 -> 3.30; a solve of order 12288 60.5 -> 61.9).  The same sums as two launches that add
// into C took 10.9, 40.6, 3.53 and 62.7 ms, and parts that overflow to opposite sides left NaN.
bool one_unit(int planes, int frac) { return frac >= std::min(6 * planes + 10, DIGIT * (planes + 1)); }

// First diagonal pair whose sums the wide kernel takes in the finer unit: from 5 on K products on
// each add up to less than 2^57 of 2^-(frac + 16), while pairs below stay at or under diagonal 5,
// which the unit holds exactly to K 2^24, the longest a launch takes.
constexpr int kFinePair = 5;
constexpr int64_t kStretch = 1 << 24;

// Groups and units of a launch (kernel comment, "Order of the products") for S planes and
// `kblocks` K blocks, and each accumulator's weight: a sum of digit products with s + t = m
// counts 2^(frac - 8 m) units.
void plan_units(Args& a, int S, bool wide)
{
    int ng = 0, nu = 0;
    auto weigh = [&](Unit& u, int q, int m) {
        // a left shift of the converted sum (at most 2^24 in magnitude); below 0: bits rounded
        // off in the conversion.  2^31 as a signed multiplier is -2^31, so the sum changes sign
        int sh = a.frac + (u.fine ? 16 : 0) - DIGIT * m;
        float sc = 1.0f;
        if (sh < 0) { sc = std::ldexp(1.0f, sh); sh = 0; }
        else if (sh == 31) sc = -1.0f;
        u.scale[q] = sc;
        u.shift[q] = sh;
    };
    auto add_unit = [&](int first, int n, int chunk, int d) {
        Unit& u = a.unit[nu++];
        u.first = (int16_t)first;
        u.ngroups = (int16_t)n;
        u.chunk = (int16_t)std::max(1, chunk);
        u.fine = wide && d >= kFinePair;
        weigh(u, 0, d);
        weigh(u, 1, d + 1);
    };
    // diagonals 2 .. S + 1 in pairs (d, d + 1); an odd number of them leaves 2 to itself, a
    // single product, which a pair (1, 2) describes
    auto add_pair = [&](int d) {
        const int first = ng;
        for (int s = 1; s < d; ++s) a.group[ng++] = Group{(int8_t)(s - 1), (int8_t)(d - s - 1), 2, 0};
        a.group[ng++] = Group{(int8_t)(d - 1), 0, 1, 0};
        const int shared = EXACT_KBLOCKS / d;  // the second accumulator adds d products
        if (cdiv(a.kblocks, shared) <= d * cdiv(a.kblocks, EXACT_KBLOCKS)) add_unit(first, d, shared, d);
        else
            for (int g = first; g < ng; ++g) add_unit(g, 1, EXACT_KBLOCKS, d);
    };
    for (int fine = wide ? 1 : 0; fine >= 0; --fine)
        for (int d = S % 2 ? 1 : 2; d <= S; d += 2)
            if (!wide || (d >= kFinePair) == (fine == 1)) add_pair(d);
    a.nunits = nu;
}

// Cost of a stage in clocks: the MMAs of one K block of a double or single group (at
// the rate shared memory lets through) -- only ratios matter here.
int stage_cost(const Group& g) { return g.nb == 2 ? 2 : 1; }

int64_t tile_cost(const Args& a)
{
    int64_t n = 0;
    for (int u = 0; u < a.nunits; ++u)
        for (int g = 0; g < a.unit[u].ngroups; ++g) n += stage_cost(a.group[a.unit[u].first + g]);
    return n * a.kblocks;
}

// Cut a tile's stages (in walk()'s order) into `cluster` shares of about equal cost; returns
// the largest.  Sums that are rounded to the integers' unit are cut at drains only, so that
// what is rounded, and with it the result, does not depend on the cut.
int64_t cut_stages(Args& a, int cluster)
{
    bool anywhere = true;
    for (int u = 0; u < a.nunits; ++u)
        anywhere = anywhere && std::min(std::fabs(a.unit[u].scale[0]), std::fabs(a.unit[u].scale[1])) == 1.0f;
    const int64_t total = tile_cost(a);
    int64_t cost = 0, largest = 0, begun = 0;
    int pos = 0, next = 1;
    a.cut[0] = 0;
    auto cut = [&](int at, int64_t cost_at) {
        a.cut[next++] = at;
        largest = std::max(largest, cost_at - begun);
        begun = cost_at;
    };
    for (int u = 0; u < a.nunits; ++u)
        for (int k0 = 0; k0 < a.kblocks; k0 += a.unit[u].chunk) {
            const int nk = std::min<int>(a.unit[u].chunk, a.kblocks - k0);
            int64_t drain = 0;
            for (int g = 0; g < a.unit[u].ngroups; ++g) drain += (int64_t)stage_cost(a.group[a.unit[u].first + g]) * nk;
            while (!anywhere && next < cluster && cost + drain / 2 >= total * next / cluster) cut(pos, cost);
            for (int g = 0; g < a.unit[u].ngroups; ++g) {
                const int64_t c = stage_cost(a.group[a.unit[u].first + g]);
                while (anywhere && next < cluster && cost + c * nk >= total * next / cluster) {
                    const int64_t n = std::min<int64_t>(nk, (total * next / cluster - cost + c - 1) / c);
                    cut(pos + (int)n, cost + c * n);
                }
                cost += c * nk;
                pos += nk;
            }
        }
    while (next < cluster) cut(pos, cost);
    largest = std::max(largest, cost - begun);
    while (next <= MAX_CLUSTER) a.cut[next++] = pos;
    return largest;
}

// CTAs per tile: the size whose busiest cluster finishes first.  The CTAs of a cluster share
// a tile's stages; the exchange of their partial sums costs about as much as kExchange
// stages.  Leaves the chosen size and its cuts in `a`.
constexpr int64_t kExchange = 16;
void choose_cluster(Args& a, const ClusterCounts& counts)
{
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int c = 1; c <= MAX_CLUSTER; c *= 2) {
        const int n = counts.at_once[c];
        if (n <= 0) continue;
        const int64_t t = cdiv(a.tiles, n) * (cut_stages(a, c) + (c > 1 ? kExchange : 0));
        if (t < cost) { cost = t; best = c; }
    }
    a.cluster = best;
    cut_stages(a, best);
}

template <bool kWide>
int launch_kernel(const CUtensorMap& ma, const CUtensorMap& mb, Args& a, cudaStream_t st, std::string& why)
{
    constexpr size_t smem = SMEM_BYTES + (kWide ? LOW_BYTES : 0);
    static const ClusterCounts counts = count_clusters((const void*)ozaki_tile_kernel<kWide>, THREADS, smem);
    if (counts.at_once[1] <= 0) { why = "ozaki tile kernel: shared memory attribute"; return OOC_ERR_CUDA; }
    choose_cluster(a, counts);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    cluster_config(cfg, at, a.cluster, std::min(a.tiles, counts.at_once[a.cluster]), THREADS, smem, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, ozaki_tile_kernel<kWide>, ma, mb, a);
    if (e != cudaSuccess) {
        cudaGetLastError();
        why = std::string("ozaki tile launch: ") + cudaGetErrorString(e);
        return OOC_ERR_CUDA;
    }
    return OOC_OK;
}

}  // namespace

int split_ozaki_launches(int64_t K) { return K > kShortSplit ? 2 : 1; }

int launch_split_ozaki(const double* X, int64_t sr, int64_t sk, int rows, int K, int rows_pad, int k_pad, int S,
                       void* planes, int* rowexp, unsigned long long* rowmax, void* stream, std::string& why)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto* pl = static_cast<__nv_bfloat16*>(planes);
    if (K <= kShortSplit) {
        const unsigned grid = (unsigned)cdiv(rows_pad, FR);
        if (sk == 1) split_short_kernel<true><<<grid, 256, 0, st>>>(X, sr, rows, K, rows_pad, k_pad, S, pl, rowexp);
        else split_short_kernel<false><<<grid, 256, 0, st>>>(X, sk, rows, K, rows_pad, k_pad, S, pl, rowexp);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) { why = std::string("split_ozaki: ") + cudaGetErrorString(e); return OOC_ERR_CUDA; }
        return OOC_OK;
    }
    if (cudaMemsetAsync(rowmax, 0, sizeof(unsigned long long) * (size_t)rows_pad, st) != cudaSuccess) {
        why = "rowmax clear";
        return OOC_ERR_CUDA;
    }
    if (K > 0 && rows > 0) {
        if (sk == 1)
            rowmax_rows_kernel<<<dim3((unsigned)rows, (unsigned)std::min<int64_t>(cdiv(K, MAX_K), 65535)), 256, 0,
                                 st>>>(X, sr, K, rowmax);
        else
            rowmax_cols_kernel<<<dim3((unsigned)cdiv(K, 256), (unsigned)cdiv(rows, ST)), 256, 0, st>>>(X, sk, rows, K,
                                                                                                       rowmax);
    }
    split_kernel<<<dim3((unsigned)cdiv(k_pad, ST), (unsigned)cdiv(rows_pad, ST)), 256, 0, st>>>(
        X, sr, sk, rows, K, rows_pad, k_pad, rowmax, S, pl, rowexp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { why = std::string("split_ozaki: ") + cudaGetErrorString(e); return OOC_ERR_CUDA; }
    return OOC_OK;
}

int launch_ozaki_tiles(const OzakiProblem& P, void* stream, std::string& why)
{
    if (P.M <= 0 || P.N <= 0) return OOC_OK;
    if (P.planes < 1 || P.planes > MAX_PLANES) { why = "digit plane count out of range"; return OOC_ERR_INVALID_ARG; }
    if (P.k_pad % BK) { why = "K padding not a multiple of the K block"; return OOC_ERR_INVALID_ARG; }
    CUtensorMap ma, mb;
    std::memset(&ma, 0, sizeof(ma));
    std::memset(&mb, 0, sizeof(mb));
    if (P.k_pad > 0) {  // K == 0 runs the epilogue only (C = beta * C)
        int rc = encode_map_3d_bf16(&ma, P.a_planes, (uint64_t)P.k_pad, (uint64_t)P.a_rows_pad, (uint64_t)P.planes,
                                    BK, BM, why);
        if (rc) return rc;
        rc = encode_map_3d_bf16(&mb, P.b_planes, (uint64_t)P.k_pad, (uint64_t)P.b_rows_pad, (uint64_t)P.planes, BK,
                                BN, why);
        if (rc) return rc;
    }
    Args a;
    std::memset(&a, 0, sizeof(a));
    a.M = (int)P.M; a.N = (int)P.N;
    a.tiles_m = (int)cdiv(P.M, BM);
    a.tiles_n = (int)cdiv(P.N, BN);
    a.tiles = a.tiles_m * a.tiles_n;
    a.alpha = P.alpha;
    a.alpha_one = P.alpha == 1.0 ? 1 : P.alpha == -1.0 ? -1 : 0;
    a.C = P.C; a.ldc = P.ldc;
    a.row_exp = P.row_exp; a.col_exp = P.col_exp;
    a.err = P.err;
    a.tri = P.tri; a.tri_off = P.tri_off;
    // Longer K in stretches, each added into C: sums must not go through C where that can be
    // helped, since parts that overflow to opposite sides leave NaN.
    const int64_t kb_total = P.k_pad / BK, kb_step = kStretch / BK;
    for (int64_t kb0 = 0; kb0 == 0 || kb0 < kb_total; kb0 += kb_step) {
        a.kb0 = (int)kb0;
        a.kblocks = (int)std::min(kb_step, kb_total - kb0);
        a.beta = kb0 == 0 ? P.beta : 1.0;
        a.read_c = kb0 == 0 ? (P.read_c ? 1 : 0) : 1;
        a.frac = unit_bits(a.kblocks);
        const bool wide = !one_unit(P.planes, a.frac);
        plan_units(a, P.planes, wide);
        cudaStream_t st = static_cast<cudaStream_t>(stream);
        const int rc = wide ? launch_kernel<true>(ma, mb, a, st, why) : launch_kernel<false>(ma, mb, a, st, why);
        if (rc) return rc;
    }
    return OOC_OK;
}

}  // namespace ooc
