// Compiled in front of a source file with -DSYCSIM_CLUSTER_LAUNCH=refused_launch: cluster launches wider
// than $REFUSE_ABOVE CTAs are refused, on the host, with the error a device gives that cannot place
// them; the first $REFUSE_AFTER of all launches go through.
#pragma once
#include <cuda_runtime.h>

#include <cstdlib>
#include <utility>

template <typename... P, typename... A>
cudaError_t refused_launch(const cudaLaunchConfig_t *cfg, void (*kern)(P...), A &&...args)
{
    static int after = getenv("REFUSE_AFTER") ? atoi(getenv("REFUSE_AFTER")) : 0;
    unsigned width = 1;
    for (unsigned i = 0; i < cfg->numAttrs; ++i)
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) width = cfg->attrs[i].val.clusterDim.x;
    if (width > (unsigned)atoi(getenv("REFUSE_ABOVE")) && after-- <= 0) return cudaErrorLaunchOutOfResources;
    return cudaLaunchKernelEx(cfg, kern, std::forward<A>(args)...);
}
