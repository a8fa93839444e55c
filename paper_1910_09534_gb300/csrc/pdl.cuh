// pdl.cuh -- programmatic dependent launch between the kernels of a handle's stream.
//
// A plan is a chain of passes over the same buffer.  Launched the ordinary way, a pass starts once
// the one before has drained and the launch has reached the SMs: 2-3 us a pass on GB300, as long as
// the pass itself below 2^20 amplitudes.  Kernels launched through launch_pdl may become resident
// while the one before still runs; they do what does not depend on it (the block's matrix into
// shared memory, barriers, tensor memory) and call pdl_wait before their first access to anything
// that earlier work of the stream writes or reads.  pdl_wait returns when every earlier kernel has
// completed and its writes are visible, so an early start changes no result.  A copy, a memset or
// an event between two kernels orders them fully, as ever.
#pragma once

#include <cuda_runtime.h>

#include <utility>

// The runtime call that launches a kernel in clusters, which a device may refuse: a test compiles
// one that refuses in its place.
#ifndef SYCSIM_CLUSTER_LAUNCH
#define SYCSIM_CLUSTER_LAUNCH cudaLaunchKernelEx
#endif

namespace sycsim {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// The next kernel of the stream may start, once every CTA of this one has got here or left.  A kernel
// of which several CTAs fit on an SM had better not call it, or at its last tile: the next one's CTAs
// are put where there is room, several on the SMs that are idle or done first, and share those while
// others stand empty.  Without it the next launch still reaches the SMs while this kernel drains.
// Replays of plans of FP32 blocks, us, launched the ordinary way / trigger at the start / at the last tile
// / none: 4 qubits a block on 19 qubits (128 CTAs a pass) 90 / 134 / 84 / 82, on 20 137 / 171 / 164 / 125,
// on 22 349 / 370 / 368 / 340; 3 qubits on 18 76 / 98 / 82 / 62, on 20 166 / 148 / 149 / 146.  A kernel of very
// many short CTAs pays for the instruction itself (permute.cu).
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// Whether a tensor-core pass over 2^nbits amplitudes lets the next one start early (the tcgen05 kernels
// at each CTA's last tile, 2 % faster on a 20-qubit plan than at the start, where the next kernel's
// CTAs crowd the SMs that are still idle).  Measured on plans, early / not: 22 qubits 266 / 290 us, 24
// qubits 849 / 869, 26 qubits 3.31 / 3.34 ms, 28 qubits 31.48 / 31.56; at 30 qubits, where a pass takes
// 2.7 ms and nothing is gained, 60.8 / 58.5 ms.
inline bool pdl_early(int nbits) { return nbits <= 28; }

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// The same with the grid in clusters of `cluster` CTAs.
template <typename... P, typename... A>
cudaError_t launch_cluster(void (*kern)(P...), unsigned grid, unsigned cluster, unsigned block, size_t smem,
                           cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return SYCSIM_CLUSTER_LAUNCH(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace sycsim
