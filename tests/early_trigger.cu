// A kernel of a caller's own that lets the stream's next kernel start early and then runs on for a
// while (one CTA, bounded by the global timer and by its number of turns).
#include <cuda_runtime.h>

__global__ void k_trigger_then_run(unsigned long long ns, float2 *psi, unsigned long long count, float scale)
{
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (unsigned long long turn = 0; turn < ns / 1000; ++turn) {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > ns) break;
    }
    for (unsigned long long i = threadIdx.x; i < count; i += blockDim.x) {
        psi[i].x *= scale;
        psi[i].y *= scale;
    }
}

extern "C" int trigger_then_run(void *stream, double seconds, void *psi, unsigned long long count, float scale)
{
    k_trigger_then_run<<<1, 256, 0, (cudaStream_t)stream>>>((unsigned long long)(seconds * 1e9), (float2 *)psi, count,
                                                            scale);
    return (int)cudaGetLastError();
}
