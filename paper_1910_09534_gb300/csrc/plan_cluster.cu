// plan_cluster.cu -- a plan's blocks on a small state, many a launch (cluster_run.cuh).
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>

#include "cluster_run.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace sycsim {
namespace {

// A launch's blocks: as many as fit the parameter space (14 of 4 qubits, 3 of 5), so that nothing is
// uploaded and the launch can be captured; a longer plan takes several launches.
constexpr int kTableBlocks = 14;
constexpr int kTableElems = kTableBlocks * 256;
struct PlanTable {
    ClBlock blocks[kTableBlocks];
    alignas(16) float2 mats[kTableElems];
};

__global__ void __launch_bounds__(kClThreads, 1) k_plan_cluster(float2 *psi, int n, int nblocks,
                                                                const __grid_constant__ PlanTable t)
{
    __shared__ ClShared sh;
    pdl_launch_next();
    const float2 *mats = t.mats;
    asm volatile("" : "+l"(mats));  // read with ordinary loads, not as constants (block_mat.cuh)
    pdl_wait();
    cl_run_blocks(psi, n, t.blocks, mats, nblocks, sh);
}

}  // namespace

// CTAs of the cluster on the current device, looked up once per device
static int plan_ctas()
{
    static std::atomic<uint64_t> wide{0}, known{0};  // bit d: device d < 64
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
    const uint64_t bit = 1ull << dev;
    if (!(known.load(std::memory_order_acquire) & bit)) {
        if (cluster_ctas(k_plan_cluster) == 16) wide.fetch_or(bit, std::memory_order_acq_rel);
        known.fetch_or(bit, std::memory_order_acq_rel);
    }
    return wide.load(std::memory_order_acquire) & bit ? 16 : 8;
}

// Where one cluster is faster than a launch per block on all SMs.  Measured (20 cycles, us a plan, cluster
// of 16 / of 8 / separate launches): k_max 4: 12 qubits 37 / 39 / 59, 14 qubits 58 / 66 / 76, 15 qubits 81 /
// 105 / 90, 16 qubits 88 / 150 / 82; k_max 5, whose separate kernel keeps up with one tile a CTA: 12
// qubits 45 / 50 / 65, 13 qubits 51 / 67 / 52, 14 qubits 73 / 83 / 65; k_max 3: 13 qubits 57 / 63 / 65,
// 14 qubits 74 / 81 / 76, 15 qubits 90 / 129 / 83; k_max 2: 13 qubits 133 / 139 / 149, 14 qubits 158 / 181 /
// 169, 15 qubits 205 / 284 / 189.
bool plan_cluster_eligible(int n, int nblocks, int max_k)
{
    if (nblocks < 2 || max_k > kClMaxK) return false;
    const int top = max_k == 4 ? 15 : (max_k == 5 ? 13 : 14);
    return n <= top - 1 || (n <= top && plan_ctas() == 16);
}

int launch_plan_cluster(float2 *psi, int n, int nblocks, const int *k, const int *const *tpos,
                        const float2 *const *mats, cudaStream_t st, int *launches)
{
    static thread_local PlanTable t;
    *launches = 0;
    int ctas = plan_ctas();
    for (int i = 0; i < nblocks;) {
        int c = 0;
        uint32_t off = 0;
        for (; i < nblocks && c < kTableBlocks && off + (1u << (2 * k[i])) <= (uint32_t)kTableElems; i++, c++) {
            ClBlock &b = t.blocks[c];
            b.k = k[i];
            for (int q = 0; q < kMaxK; q++) b.tpos[q] = q < k[i] ? tpos[i][q] : 0;
            b.mat_off = off;
            std::memcpy(t.mats + off, mats[i], sizeof(float2) << (2 * k[i]));
            off += 1u << (2 * k[i]);
        }
        cudaError_t e = launch_cluster(k_plan_cluster, ctas, ctas, kClThreads, 0, st, psi, n, c, t);
        if (e != cudaSuccess && ctas > 8) {  // the occupancy query's answer does not bind the launch
            cudaGetLastError();
            ctas = 8;
            e = launch_cluster(k_plan_cluster, ctas, ctas, kClThreads, 0, st, psi, n, c, t);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            return i - c;
        }
        ++*launches;
    }
    return nblocks;
}

}  // namespace sycsim
