// cluster_run.cuh -- a whole small circuit's blocks on one thread-block cluster (FP32).
//
// Below about 2^15 amplitudes a pass is over before the next launch has reached the SMs; the CTAs
// of a cluster instead go through the blocks together, a cluster barrier (a few hundred ns) between
// two blocks.  The state stays in global memory, which at this size is the L2: every CTA owns a
// contiguous share of a block's groups, reads their members past the L1 (another CTA wrote them),
// multiplies them with the matrix in its shared memory and writes them back.  The next block's
// matrix is fetched into a second buffer meanwhile.  Products are summed in the order of the
// one-launch-per-block kernels (apply.cu), so the amplitudes are the same bit for bit.
//
// Two ways to spread a block over the threads: a group a thread (all 2^k rows, four at a time), and,
// while that would leave half of the threads idle, several threads to a group's rows, which shortens
// the chain of FMAs a thread goes through (a 12-qubit, 4-qubit block: 256 FMAs instead of 1024).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"

namespace sycsim {

constexpr int kClThreads = 256;  // 512: 1.3-1.9 times the time at 10-18 qubits (dearer barriers)
constexpr int kClMaxK = 5;

// CTAs of the cluster for a kernel of kClThreads threads on the current device: 16 (beyond the portable
// 8) where the device can place such a cluster, else 8.
template <typename Kern>
int cluster_ctas(Kern kern)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 16;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kClThreads);
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0)
        return 16;
    cudaGetLastError();  // not an error of the caller: the narrower cluster is used
    return 8;
}

struct ClBlock {
    int k;
    int tpos[kMaxK];   // ascending physical target bits
    uint32_t mat_off;  // float2 offset of the block's matrix in the table (a multiple of 2)
};

struct ClShared {
    alignas(16) float2 m[2][1 << (2 * kClMaxK)];
    uint32_t moff[2][1 << kClMaxK];
    int tpos[2][kMaxK];
    int k[2];
};

__device__ __forceinline__ uint64_t cl_insert_zero_bits(uint64_t x, const int *pos, int cnt)
{
    for (int i = 0; i < cnt; ++i) {
        const int p = pos[i];
        const uint64_t lo = x & ((1ull << p) - 1);
        x = ((x >> p) << (p + 1)) | lo;
    }
    return x;
}

// Rows r0 .. r0 + RB - 1 of one group: RB independent chains for each of Re and Im.
template <int K, int RB, typename Store>
__device__ __forceinline__ void cl_rows(const float2 (&x)[1 << K], const float2 *M, int r0, Store st)
{
    constexpr int D = 1 << K;
    float yr[RB], yi[RB];
#pragma unroll
    for (int b = 0; b < RB; ++b) yr[b] = yi[b] = 0.f;
#pragma unroll
    for (int c = 0; c < D; c += 2) {
        float4 m[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) m[b] = *reinterpret_cast<const float4 *>(M + (r0 + b) * D + c);
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            yr[b] = fmaf(m[b].x, x[c].x, yr[b]);
            yr[b] = fmaf(m[b].y, -x[c].y, yr[b]);
            yi[b] = fmaf(m[b].x, x[c].y, yi[b]);
            yi[b] = fmaf(m[b].y, x[c].x, yi[b]);
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            yr[b] = fmaf(m[b].z, x[c + 1].x, yr[b]);
            yr[b] = fmaf(m[b].w, -x[c + 1].y, yr[b]);
            yi[b] = fmaf(m[b].z, x[c + 1].y, yi[b]);
            yi[b] = fmaf(m[b].w, x[c + 1].x, yi[b]);
        }
    }
#pragma unroll
    for (int b = 0; b < RB; ++b) st(r0 + b, make_float2(yr[b], yi[b]));
}

// This CTA's groups g0 .. g0 + gc - 1 of one block (all threads of the CTA; gc a power of two).
template <int K>
__device__ __forceinline__ void cl_apply(float2 *psi, uint32_t g0, uint32_t gc, const int *tpos, const float2 *M,
                                         const uint32_t *moff)
{
    constexpr int D = 1 << K, RB = D < 4 ? D : 4;
    const uint32_t tid = threadIdx.x;
    if (gc * (D / RB) <= kClThreads || gc <= kClThreads / 2) {  // several threads share a group's rows
        const uint32_t gi = tid & (gc - 1), rb = tid / gc, step = kClThreads / gc;
        const bool on = rb < D / RB;
        float2 *p = psi + cl_insert_zero_bits(g0 + gi, tpos, K);
        float2 x[D];
        if (on) {
#pragma unroll
            for (int j = 0; j < D; ++j) x[j] = __ldcg(p + moff[j]);
        }
        __syncthreads();  // a group's threads have all read it before any of them writes
        auto st = [&](int r, float2 y) { p[moff[r]] = y; };
        if (step >= D / RB) {
            if (on) cl_rows<K, RB>(x, M, (int)rb * RB, st);
        } else {
#pragma unroll 1
            for (uint32_t q = rb; q < D / RB; q += step) cl_rows<K, RB>(x, M, (int)q * RB, st);
        }
        return;
    }
    for (uint32_t i = tid; i < gc; i += kClThreads) {
        float2 *p = psi + cl_insert_zero_bits(g0 + i, tpos, K);
        float2 x[D];
#pragma unroll
        for (int j = 0; j < D; ++j) x[j] = __ldcg(p + moff[j]);
#pragma unroll 1  // 4 x 4 x 2^k FMAs of code, not 4^(k+1): the instruction cache holds it
        for (int r0 = 0; r0 < D; r0 += RB) cl_rows<K, RB>(x, M, r0, [&](int r, float2 y) { p[moff[r]] = y; });
    }
}

// The next block's matrix on its way: read into registers before a block is applied, put into the
// buffer that block does not use after it, so that the reads' latency passes during the products.
// (Plain loads: the table may be in device memory or in a kernel's parameters.)
struct ClNext {
    float4 v[(1 << (2 * kClMaxK)) / 2 / kClThreads];
    int b;
};

__device__ __forceinline__ void cl_load_next(ClNext &nx, const ClBlock *blocks, const float2 *mats, int b)
{
    nx.b = b;
    const int n4 = 1 << (2 * blocks[b].k - 1);
    const float4 *src = reinterpret_cast<const float4 *>(mats + blocks[b].mat_off);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(nx.v) / sizeof(float4)); ++i)
        if ((int)threadIdx.x + i * kClThreads < n4) nx.v[i] = src[threadIdx.x + i * kClThreads];
}

__device__ __forceinline__ void cl_store_next(ClShared &sh, const ClNext &nx, const ClBlock *blocks)
{
    const int buf = nx.b & 1, k = blocks[nx.b].k, n4 = 1 << (2 * k - 1);
    float4 *dst = reinterpret_cast<float4 *>(sh.m[buf]);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(nx.v) / sizeof(float4)); ++i)
        if ((int)threadIdx.x + i * kClThreads < n4) dst[threadIdx.x + i * kClThreads] = nx.v[i];
    if ((int)threadIdx.x < (1 << k)) {
        uint32_t o = 0;
        for (int q = 0; q < k; ++q)
            if ((threadIdx.x >> q) & 1) o += 1u << blocks[nx.b].tpos[q];
        sh.moff[buf][threadIdx.x] = o;
    }
    if (threadIdx.x < kMaxK) sh.tpos[buf][threadIdx.x] = blocks[nx.b].tpos[threadIdx.x];
    if (threadIdx.x == 0) sh.k[buf] = k;
}

// Every block of a circuit on n <= 31 qubits; all threads of the cluster, which have finished with
// sh.  Ends with a cluster barrier: every CTA sees the final state.
__device__ __forceinline__ void cl_run_blocks(float2 *psi, int n, const ClBlock *blocks, const float2 *mats,
                                              int nblocks, ClShared &sh)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const uint32_t ncta = cl.num_blocks(), rank = cl.block_rank();
    ClNext nx;
    if (nblocks > 0) {
        cl_load_next(nx, blocks, mats, 0);
        cl_store_next(sh, nx, blocks);
    }
    for (int b = 0; b < nblocks; ++b) {
        // this block's matrix is in its buffer, every CTA's writes of the block before are visible,
        // and the other buffer is no longer read
        cl.sync();
        if (b + 1 < nblocks) cl_load_next(nx, blocks, mats, b + 1);
        const int buf = b & 1, k = sh.k[buf];
        const uint32_t groups = 1u << (n - k);
        const uint32_t gc = groups >= ncta ? groups / ncta : 1;
        const uint32_t g0 = rank * gc;
        if (g0 < groups) {  // uniform over the CTA
            switch (k) {
            case 1: cl_apply<1>(psi, g0, gc, sh.tpos[buf], sh.m[buf], sh.moff[buf]); break;
            case 2: cl_apply<2>(psi, g0, gc, sh.tpos[buf], sh.m[buf], sh.moff[buf]); break;
            case 3: cl_apply<3>(psi, g0, gc, sh.tpos[buf], sh.m[buf], sh.moff[buf]); break;
            case 4: cl_apply<4>(psi, g0, gc, sh.tpos[buf], sh.m[buf], sh.moff[buf]); break;
            default: cl_apply<5>(psi, g0, gc, sh.tpos[buf], sh.m[buf], sh.moff[buf]); break;
            }
        }
        if (b + 1 < nblocks) cl_store_next(sh, nx, blocks);
    }
    cl.sync();
}

}  // namespace sycsim
