// Blackwell tensor-core building blocks (sm_100a/sm_103a PTX): TMEM
// allocation, shared-memory matrix descriptors, the kind::f16 instruction
// descriptor, tcgen05.mma / commit / ld, and 3-D TMA tile loads.
//
// Conventions used by every kernel that includes this file:
//   * operand tiles are K-major bf16 written by TMA with the 128-byte swizzle
//     (64 elements of K per row, 1024-byte 8-row atoms) or the 64-byte swizzle
//     (32 elements of K per row, 512-byte atoms); tiles start on a 1024-byte
//     boundary;
//   * the MMA is cta_group::1 with M = 128, so accumulator row i lives in
//     TMEM lane i and column j in TMEM column (base + j), 32-bit each.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "device_sync.cuh"
#include "ooc_internal.hpp"

namespace ooc {

// --- shared-memory matrix descriptor (tcgen05 format) --------------------
// bits  0-13 start address >> 4
// bits 16-29 leading-dimension byte offset >> 4 (unused for swizzled K-major; 1)
// bits 32-45 stride-dimension byte offset >> 4 (8-row atom pitch: 1024 B)
// bits 46-47 descriptor version (1 on sm_100 family)
// bits 49-51 base offset (0: atoms 1024-byte aligned)
// bits 61-63 layout: 2 = 128-byte swizzle
__device__ __forceinline__ uint64_t sw128_kmajor_desc(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// --- instruction descriptor, kind::f16, bf16 x bf16 -> f32, both K-major --
// bits 4-5 D format (1 = f32), 7-9 A format (1 = bf16), 10-12 B format (1 = bf16),
// 15/16 A/B major (0 = K), 17-22 N >> 3, 24-28 M >> 4
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// --- TMEM allocation (one warp) --------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_result, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, M=128, N from idesc; accumulate when acc != 0
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
}

// One lane of a converged warp.  The TMA and MMA warps run their loops with all lanes
// (waits are voted, see wait_warp) and only issue under this lane's flag: the compiler
// then keeps descriptors and addresses in uniform registers.  With the loop inside an
// `if (lane == 0)` it moved every operand of every tcgen05.mma there one by one, and the
// issuing thread took 700 clocks for a stage of 450 clocks of MMAs.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// mbar_wait by a whole warp, with one answer for all lanes
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, int* err, int code)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, err, code)) != 0;
}

// arrive on an mbarrier once every tcgen05 operation issued so far by this thread completes
__device__ __forceinline__ void tc_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 lanes x 8 consecutive 32-bit columns: thread i of the warp gets lane (base lane + i)
__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 3-D TMA tile load (x innermost), completing on `bar`
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int32_t x, int32_t y,
                                            int32_t z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// --- shared by the tile kernels of both forms ------------------------------
// Packed pairs of FP32 values (element 2j in the low half): Blackwell's f32x2
// arithmetic does two of a drain's additions per instruction.
__device__ __forceinline__ uint64_t f2add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2sub(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t pair(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }
__device__ __forceinline__ uint64_t pair(float x) { return pair(__float_as_uint(x), __float_as_uint(x)); }

// Tile order: groups of kRasterRows tile rows, column-major inside a group, so that
// the tiles in flight at once span few rows and few columns and share their A and B
// plane tiles in L2.
constexpr int kRasterRows = 8;
__device__ __forceinline__ void tile_coords(int tile, int tiles_m, int tiles_n, int& tm, int& tn)
{
    const int per_group = kRasterRows * tiles_n;
    const int g = tile / per_group, r = tile % per_group;
    const int first = g * kRasterRows;
    const int rows = min(tiles_m - first, kRasterRows);
    tm = first + r % rows;
    tn = r / rows;
}

// ring position: slot and pass parity, advanced without division
struct Ring {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next(int n)
    {
        if (++s == n) { s = 0; ph ^= 1u; }
    }
};

// 4 x 4 transpose inside each group of 4 lanes: lane 4g + r holds row r of its
// group's block in v[0..3] on entry and column r on exit.  Each butterfly stage
// m swaps the off-diagonal m x m sub-blocks: the lane without bit m trades its
// elements with bit m set for its partner's elements without it.
__device__ __forceinline__ void transpose4(double (&v)[4], int lane)
{
#pragma unroll
    for (int m = 2; m >= 1; m >>= 1) {
        const bool upper = (lane & m) != 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (e & m) continue;
            const double send = upper ? v[e] : v[e | m];
            const double got = __shfl_xor_sync(0xffffffffu, send, m);
            if (upper) v[e] = got;
            else v[e | m] = got;
        }
    }
}

// How many clusters of 1, 2, 4 and 8 CTAs of a kernel the device holds at once (0: none);
// sets the kernel's shared-memory limit.
struct ClusterCounts {
    int at_once[9] = {0};
};

inline void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, int cluster, int clusters, int threads,
                           size_t smem, cudaStream_t st)
{
    cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * cluster));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

inline ClusterCounts count_clusters(const void* kernel, int threads, size_t smem)
{
    ClusterCounts n;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return n;
    }
    n.at_once[1] = device_sm_count();
    for (int c = 2; c <= 8; c *= 2) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        cluster_config(cfg, at, c, 1, threads, smem, nullptr);
        if (cudaOccupancyMaxActiveClusters(&n.at_once[c], kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n.at_once[c] = 0;
        }
    }
    return n;
}

}  // namespace ooc
