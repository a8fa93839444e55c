// block_mat.cuh -- how a fused block's matrix (FP32, rows and columns in sorted-target order)
// reaches a kernel: by value in the kernel's parameters for k <= 5 (8 KiB; nothing to upload), from
// device memory for k = 6 (32 KiB, above the parameter space).
#pragma once

#include <cuda_runtime.h>

#include <cstring>

namespace sycsim {

template <int K>
struct BlockMat {
    alignas(16) float2 m[(1 << K) * (1 << K)];
};

template <>
struct BlockMat<6> {
    const float2 *p;
};

// host = the matrix; dev = its device copy (k = 6 only)
template <int K>
BlockMat<K> block_mat(const float2 *host, const float2 *dev)
{
    BlockMat<K> M;
    if constexpr (K == 6) {
        M.p = dev;
    } else {
        std::memcpy(M.m, host, sizeof(M.m));
    }
    return M;
}

// The matrix as memory that the threads of a CTA read at different places (M: a __grid_constant__
// parameter).  The address is made opaque so that parameters are read through the ordinary load
// path; as constants, 32 different addresses a warp would be served one after the other.
template <int K>
__device__ __forceinline__ const float2 *block_mat_ptr(const BlockMat<K> &M)
{
    if constexpr (K == 6) {
        return M.p;
    } else {
        const float2 *p = M.m;
        asm volatile("" : "+l"(p));
        return p;
    }
}

}  // namespace sycsim
