// apply.cu -- aggregated k-qubit gate apply on CUDA cores, FP32 (Sect. 5: gates are
// aggregated into k-qubit kernels, each a 2^k x 2^k unitary applied to the state).
//
// For targets t_0 < ... < t_{k-1} (physical bits), a "group" is the 2^k amplitudes that
// share every non-target bit; member j of a group sits at base + sum_b bit_b(j) 2^{t_b}.
// Each group is replaced by M times itself.  One pass reads and writes every amplitude
// once: 16 bytes per amplitude of HBM traffic, 8 * 2^k - 2 real flops per amplitude.
//
// Five kernels:
//  * reg (default for k <= 4, n >= k + 5) -- see the comment above k_apply_reg: persistent warps,
//    register-resident groups, an exchange through the warp's own shared memory for targets
//    below bit 5.
//  * rtile (k = 5, 6, n >= k + 6) -- see above k_apply_rtile: tiles in shared memory, each thread a
//    register tile of rows x groups, the matrix in shared memory.
//  * direct -- every target >= 5: thread = group; the 32 threads of a warp take 32
//    consecutive groups, so each member load/store is one contiguous 256-byte run.
//    Amplitudes go straight to registers; no shared memory.  Used for k <= 3.
//  * cta -- k = 5, 6 on fewer qubits than that: one CTA, several threads to a group's rows.
//  * tiled -- k <= 4 on fewer than k + 5 qubits: a CTA stages a tile of 2^(F+k) amplitudes (2^h rows of
//    2^m contiguous amplitudes, the rows indexed by the h targets >= m) through shared
//    memory with coalesced loads, each of its 2^F threads applies M to one group, and
//    the tile is written back.  An XOR swizzle maps the low target bits onto free bits
//    so that shared-memory accesses stay conflict-free for any target set.
//
// The matrix (FP32, complex64) is a kernel parameter for k <= 5: up to k = 4 (2 KiB) the FMAs read it
// straight from the constant bank; k = 5, 6 (8, 32 KiB, more than the constant cache keeps) are
// copied to shared memory once per CTA, k = 6 from device memory.
//
// Early starts: reg and direct do not trigger the next launch, rtile does at its last tile (pdl.cuh has
// the figures; rtile on 18-19 qubits, trigger at the start / at the last tile: 76, 115 / 62, 96 us a replay).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "cluster_run.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace sycsim {
namespace {

// The CUDA-core kernels' matrix: a parameter that the FMAs read as constants (BlockMat's 16-byte
// alignment, for wide loads, moved it in the constant bank and cost k = 4, 5 passes 1-1.5 %).
template <int K>
struct MatP {
    float2 m[(1 << K) * (1 << K)];
};

struct MatPtr {
    const float2 *p;
};

struct DirectGeom {
    float2 *psi;
    uint64_t n_groups;
    int tpos[kMaxK];     // ascending physical target bits
    uint64_t moff[8];    // offset of member j (k <= 3)
};

struct TiledGeom {
    float2 *psi;
    int F;               // log2(threads per CTA) = log2(groups per tile)
    int m;               // log2(row length) = F + nlow
    int nlow, nhigh;     // targets below / at-or-above m
    int ltpos[kMaxK];    // low target bits (ascending, < m)
    int hpos[kMaxK];     // high target bits (ascending, >= m)
    int nsw;             // swizzle pairs: bit sw_src[i] of a tile position is XORed into bit sw_dst[i]
    int sw_src[4], sw_dst[4];
    uint32_t soff[16];   // tile-local offset of member j (k <= 4)
    uint64_t rowoff[16]; // global offset of tile row r
};

__device__ __forceinline__ uint64_t insert_zero_bits(uint64_t x, const int *pos, int cnt)
{
#pragma unroll
    for (int i = 0; i < kMaxK; ++i) {
        if (i >= cnt) break;
        const int p = pos[i];
        const uint64_t lo = x & ((1ull << p) - 1);
        x = ((x >> p) << (p + 1)) | lo;
    }
    return x;
}

// 8-byte asynchronous global -> shared copy (no register staging) and its completion wait.
__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gmem_src)
{
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Opaque copies: stop the compiler from keeping load-phase addresses alive through the
// compute phase (it would otherwise reuse them for the stores and spill).
__device__ __forceinline__ float2 *opaque(float2 *p)
{
    float2 *q;
    asm volatile("mov.b64 %0, %1;" : "=l"(q) : "l"(p));
    return q;
}

__device__ __forceinline__ uint32_t opaque_tid()
{
    uint32_t t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

__device__ __forceinline__ uint32_t swizzle(uint32_t p, const TiledGeom &g)
{
    uint32_t x = p;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (i < g.nsw) x ^= ((p >> g.sw_src[i]) & 1u) << g.sw_dst[i];
    return x;
}

// y = M x for one group; rows are produced RB at a time (RB independent FMA chains per
// real/imag part) and handed to `st(row, value)`.
template <int K, typename MatAt, typename Store>
__device__ __forceinline__ void apply_group(const float2 (&x)[1 << K], MatAt M, Store st)
{
    constexpr int D = 1 << K;
    constexpr int RB = D >= 4 ? 4 : D;
#pragma unroll
    for (int r0 = 0; r0 < D; r0 += RB) {
        float yr[RB], yi[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) yr[b] = yi[b] = 0.f;
#pragma unroll
        for (int c = 0; c < D; ++c) {
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                const float2 mm = M(r0 + b, c);
                yr[b] = fmaf(mm.x, x[c].x, yr[b]);
                yr[b] = fmaf(mm.y, -x[c].y, yr[b]);
                yi[b] = fmaf(mm.x, x[c].y, yi[b]);
                yi[b] = fmaf(mm.y, x[c].x, yi[b]);
            }
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) st(r0 + b, make_float2(yr[b], yi[b]));
    }
}

// Occupancy target (CTAs per SM) that bounds the register count of each width.
constexpr int tiled_min_blocks(int k) { return k == 4 ? 2 : 4; }

template <int K>
__global__ void __launch_bounds__(256, 4) k_apply_direct(DirectGeom g, MatP<K> M)
{
    constexpr int D = 1 << K;
    const uint64_t gi = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.n_groups) return;
    pdl_wait();
    float2 *p = g.psi + insert_zero_bits(gi, g.tpos, K);
    float2 x[D];
#pragma unroll
    for (int j = 0; j < D; ++j) x[j] = __ldcs(p + g.moff[j]);
    float2 *const q = opaque(p);
    apply_group<K>(x, [&](int r, int c) { return M.m[r * D + c]; },
                         [&](int r, float2 y) { __stcs(q + g.moff[r], y); });
}

template <int K>
__global__ void __launch_bounds__(256, tiled_min_blocks(K)) k_apply_tiled(TiledGeom g, MatP<K> M)
{
    constexpr int D = 1 << K;
    extern __shared__ float2 tile[];
    pdl_launch_next();

    const uint32_t tid = threadIdx.x;
    const int F = g.F;
    const uint32_t lowmask = (1u << g.nlow) - 1;
    const uint64_t base = insert_zero_bits((uint64_t)blockIdx.x << g.m, g.hpos, g.nhigh);
    float2 *gp = g.psi + base;
    pdl_wait();

    // load: linear tile position p = tid + c 2^F; row r = c >> nlow, column ((c & lowmask) << F) | tid
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const uint32_t p = tid + ((uint32_t)c << F);
        const uint32_t col = ((c & lowmask) << F) | tid;
        cp_async8(&tile[swizzle(p, g)], gp + g.rowoff[c >> g.nlow] + col);
    }
    cp_async_wait_all();
    __syncthreads();

    // compute: thread tid owns group tid
    const uint32_t bg = (uint32_t)insert_zero_bits(tid, g.ltpos, g.nlow);
    const uint32_t sb = swizzle(bg, g);
    float2 x[D];
#pragma unroll
    for (int j = 0; j < D; ++j) x[j] = tile[sb ^ g.soff[j]];
    auto st = [&](int r, float2 y) { tile[sb ^ g.soff[r]] = y; };
    apply_group<K>(x, [&](int r, int c) { return M.m[r * D + c]; }, st);
    __syncthreads();

    // store
    const uint32_t tid2 = opaque_tid();
    float2 *const gq = opaque(gp);
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const uint32_t p = tid2 + ((uint32_t)c << F);
        const uint32_t col = ((c & lowmask) << F) | tid2;
        __stcs(gq + g.rowoff[c >> g.nlow] + col, tile[swizzle(p, g)]);
    }
}

constexpr int kTiledF = 8;  // most threads per CTA (log2) of the tiled kernel

template <typename Kern>
cudaError_t ensure_smem(Kern kern, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int K>
int launch_direct(float2 *psi, int nbits, const int *tpos, const MatP<K> &M, cudaStream_t st)
{
    constexpr int D = 1 << K;
    DirectGeom g{};
    g.psi = psi;
    g.n_groups = 1ull << (nbits - K);
    for (int i = 0; i < K; i++) g.tpos[i] = tpos[i];
    for (int j = 0; j < D; j++) {
        uint64_t o = 0;
        for (int b = 0; b < K; b++)
            if ((j >> b) & 1) o += 1ull << tpos[b];
        g.moff[j] = o;
    }
    const uint64_t blocks = (g.n_groups + 255) / 256;
    return launch_pdl(k_apply_direct<K>, (unsigned)blocks, 256, 0, st, g, M) == cudaSuccess ? 0 : -1;
}

template <int K>
int launch_tiled(float2 *psi, int nbits, const int *tpos, const MatP<K> &M, cudaStream_t st)
{
    constexpr int D = 1 << K;
    TiledGeom g{};
    g.psi = psi;
    g.F = std::min(kTiledF, nbits - K);
    int m = g.F;
    for (;;) {  // m = F + #(targets below m)
        int below = 0;
        for (int i = 0; i < K; i++) below += tpos[i] < m;
        if (g.F + below == m) break;
        m = g.F + below;
    }
    g.m = m;
    g.nlow = g.nhigh = 0;
    for (int i = 0; i < K; i++) {
        if (tpos[i] < m)
            g.ltpos[g.nlow++] = tpos[i];
        else
            g.hpos[g.nhigh++] = tpos[i];
    }
    // swizzle: the free (non-target) tile bits f0 < f1 < ... ; the first four of them at or
    // above bit 4 are XORed into the target bits below 4, in order.
    {
        int dsts[4], nd = 0, srcs[4], ns = 0;
        for (int i = 0; i < g.nlow; i++)
            if (g.ltpos[i] < 4) dsts[nd++] = g.ltpos[i];
        int free_seen = 0;
        for (int b = 0; b < m && free_seen < 4; b++) {
            bool is_t = false;
            for (int i = 0; i < g.nlow; i++) is_t |= g.ltpos[i] == b;
            if (is_t) continue;
            if (b >= 4 && ns < nd) srcs[ns++] = b;
            free_seen++;
        }
        g.nsw = std::min(nd, ns);
        for (int i = 0; i < g.nsw; i++) {
            g.sw_src[i] = srcs[i];
            g.sw_dst[i] = dsts[i];
        }
    }
    for (int j = 0; j < D; j++) {
        uint32_t o = 0;
        for (int b = 0; b < g.nlow; b++)
            if ((j >> b) & 1) o |= 1u << g.ltpos[b];
        o |= (uint32_t)(j >> g.nlow) << m;
        g.soff[j] = o;
    }
    for (int r = 0; r < (1 << g.nhigh); r++) {
        uint64_t o = 0;
        for (int b = 0; b < g.nhigh; b++)
            if ((r >> b) & 1) o += 1ull << g.hpos[b];
        g.rowoff[r] = o;
    }
    const uint64_t tiles = 1ull << (nbits - g.F - K);
    const size_t smem = sizeof(float2) << (g.F + K);
    auto kern = k_apply_tiled<K>;
    if (ensure_smem(kern, smem) != cudaSuccess) return -1;
    return launch_pdl(kern, (unsigned)tiles, 1u << g.F, smem, st, g, M) == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------------------
// k = 5, 6 on fewer qubits than a tile of k_apply_rtile (n < k + 6): at most 32 groups, one CTA.  Bound by
// one chain of FMAs: a thread a group is 4^(k+1) of them on one warp; 2^k / 4 threads a group (8 where
// 32 groups of 64 leave no more) take four rows each (cl_apply), the matrix read from shared memory.
// Sums in the order of the other kernels.  Replays of plans of 5-qubit blocks, 12 cycles: on 10 qubits 73 us
// by the register kernel, 97 by the tiled one, 27 by this; on 7 qubits 49, 68, 14.  One 6-qubit block, its
// upload included: 6 qubits 251 -> 15 us, 8 qubits 126 -> 16, 10 and 11 qubits 74, 64 -> 25.
// ---------------------------------------------------------------------------------------
template <int K>
struct CtaGeom {
    float2 *psi;
    uint32_t groups;
    int tpos[kMaxK];
    uint32_t moff[1 << K];
};

template <int K, typename MatSrc>
__global__ void __launch_bounds__(kClThreads) k_apply_cta(const __grid_constant__ CtaGeom<K> g,
                                                          const __grid_constant__ MatSrc mat)
{
    __shared__ __align__(16) float2 m[1 << (2 * K)];
    pdl_launch_next();  // one CTA: there is room for the next pass to fetch its matrix meanwhile
    const float2 *src;
    if constexpr (K == 6) {
        src = mat.p;
    } else {
        src = mat.m;
        asm volatile("" : "+l"(src));  // ordinary loads, not constants (32 addresses a warp)
    }
    for (int i = threadIdx.x; i < 1 << (2 * K); i += kClThreads) m[i] = src[i];
    __syncthreads();
    pdl_wait();
    cl_apply<K>(g.psi, 0, g.groups, g.tpos, m, g.moff);
}

template <int K, typename MatSrc>
int launch_cta(float2 *psi, int nbits, const int *tpos, const MatSrc &M, cudaStream_t st)
{
    CtaGeom<K> g{};
    g.psi = psi;
    g.groups = 1u << (nbits - K);
    std::copy(tpos, tpos + K, g.tpos);
    for (int j = 0; j < (1 << K); j++)
        for (int b = 0; b < K; b++)
            if ((j >> b) & 1) g.moff[j] += 1u << tpos[b];
    return launch_pdl(k_apply_cta<K, MatSrc>, 1, kClThreads, 0, st, g, M) == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------------------
// Register-resident apply for k <= 4 (the default path when n >= k + 5).
//
// A warp owns a "warp tile": 32 lanes (index bits 0..4) x 2^k registers.  Register bit
// j < J (J = number of targets below bit 5) first stands for a free index bit E_j >= 5,
// register bits j >= J for the high targets.  Loads and stores are therefore 256-byte runs
// per register.  Each low target t_j (a lane bit) is then exchanged with register bit j, after
// which every lane holds one complete group in registers and applies M with the matrix read from
// the constant bank; the same exchange undoes the transpose before the stores.  Warps are
// persistent.  (Double-buffering the next tile in registers was measured slower than simply
// running more CTAs per SM.)
//
// The exchange goes through 2^(k+5) amplitudes of shared memory that only this warp uses.  Register x
// of lane l is written at x 32 + (l ^ s(x)), s(x) = sum of bit j of x << t_j, and lane l's register r
// of the transpose is found at ((r without its J low bits) + (the J target bits of l)) 32 + (l ^ s(r)):
// for one register the 16 lanes of an access phase cover 16 distinct bank pairs either way, and each
// lane's results go back where it read its members, so two __syncwarp a tile are all the ordering.
// 2^(k+2) 8-byte accesses a tile whatever J is; exchanging by warp shuffles took 4 J 2^k instructions
// (two shuffles and four selects a pair, both ways), which made k = 4 issue-bound (79 % issue active).
// Measured on 2^28 amplitudes, J = 1 .. k targets below bit 5, us a pass (the traffic alone: 641):
// k = 4 831, 904, 988, 1074 by shuffles -> 818, 804, 803, 799 (708 with J = 0: the accesses and their
// addresses are still issued beside 1024 FMAs a tile); k = 3 673, 695, 777 -> 675, 688, 681; k = 1, 2
// with J = k 755, 681 -> 696, 652.  Staging whole tiles with cp.async instead, group a thread: k = 4
// 820-1030, k = 3 654-674.
// ---------------------------------------------------------------------------------------
struct RegGeom {
    float2 *psi;
    uint64_t n_wtiles;  // 2^(n - 5 - k)
    int J;              // targets below bit 5
    int lt[5];          // their bit positions (lane bits), ascending
    int nfix;           // index bits >= 5 owned by registers (high targets + E), ascending
    int fix[kMaxK];
    uint64_t xoff[16];  // offset of register x (pre-exchange meaning)
    uint32_t cw[16];    // byte address in the warp's exchange tile: (8 lane) ^ cw[x] before the
    uint32_t cr[16];    // exchange, (8 lane | 256 (its target bits)) ^ cr[r] after it
};

constexpr int reg_min_blocks(int k) { return k <= 3 ? 4 : 3; }

template <int K, bool kLow>
__global__ void __launch_bounds__(256, reg_min_blocks(K)) k_apply_reg(RegGeom g, MatP<K> M)
{
    constexpr int D = 1 << K;
    __shared__ float2 xch[kLow ? 8 * 32 * D : 1];
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= g.n_wtiles) return;
    auto tile_ptr = [&](uint64_t wt) {
        return g.psi + insert_zero_bits(wt << 5, g.fix, g.nfix) + lane;
    };
    auto MatAt = [&](int r, int c) { return M.m[r * D + c]; };
    uint8_t *const my = reinterpret_cast<uint8_t *>(xch + (kLow ? (threadIdx.x >> 5) * 32 * D : 0));
    const uint32_t bw = 8 * lane;
    uint32_t br = bw;
    if constexpr (kLow) {
#pragma unroll
        for (int b = 0; b < 5; ++b)
            if (b < g.J) br |= (uint32_t)((lane >> g.lt[b]) & 1) << (8 + b);
    }
    float2 x[D];
    {
        const float2 *p = tile_ptr(w);
#pragma unroll
        for (int j = 0; j < D; ++j) x[j] = __ldcs(p + g.xoff[j]);
    }
    for (; w < g.n_wtiles; w += nw) {
        const uint64_t wn = w + nw;
        float2 *const q = opaque(tile_ptr(w));
        if constexpr (kLow) {
#pragma unroll
            for (int j = 0; j < D; ++j) *reinterpret_cast<float2 *>(my + (bw ^ g.cw[j])) = x[j];
            __syncwarp();
#pragma unroll
            for (int j = 0; j < D; ++j) x[j] = *reinterpret_cast<const float2 *>(my + (br ^ g.cr[j]));
            apply_group<K>(x, MatAt,
                                 [&](int r, float2 v) { *reinterpret_cast<float2 *>(my + (br ^ g.cr[r])) = v; });
            __syncwarp();
#pragma unroll
            for (int j = 0; j < D; ++j)
                __stcs(q + g.xoff[j], *reinterpret_cast<const float2 *>(my + (bw ^ g.cw[j])));
        } else {
            apply_group<K>(x, MatAt, [&](int r, float2 v) { __stcs(q + g.xoff[r], v); });
        }
        if (wn < g.n_wtiles) {
            const float2 *pn = tile_ptr(wn);
#pragma unroll
            for (int j = 0; j < D; ++j) x[j] = __ldcs(pn + g.xoff[j]);
        }
    }
}

template <int K, bool kLow>
int launch_reg_kernel(const RegGeom &g, const MatP<K> &M, cudaStream_t st)
{
    auto kern = k_apply_reg<K, kLow>;
    // resident CTAs per SM for this instantiation (function-local static: initialised once,
    // thread-safe)
    static const LaunchCfg cfg = [&] {
        LaunchCfg c;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return c;
        if (cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return c;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c.occ, kern, 256, 0) != cudaSuccess || c.occ < 1)
            c.occ = 1;
        c.ok = true;
        return c;
    }();
    if (!cfg.ok) return -1;
    const uint64_t need = (g.n_wtiles + 7) / 8;  // 8 warps per CTA
    const uint64_t grid = std::min<uint64_t>(need, (uint64_t)cfg.sms * cfg.occ);
    return launch_pdl(kern, (unsigned)grid, 256, 0, st, g, M) == cudaSuccess ? 0 : -1;
}

template <int K>
int launch_reg(float2 *psi, int nbits, const int *tpos, const MatP<K> &M, cudaStream_t st)
{
    RegGeom g{};
    g.psi = psi;
    g.n_wtiles = 1ull << (nbits - 5 - K);
    g.J = 0;
    int high[kMaxK], nh = 0;
    for (int i = 0; i < K; i++) {
        if (tpos[i] < 5)
            g.lt[g.J++] = tpos[i];
        else
            high[nh++] = tpos[i];
    }
    int extra[5], ne = 0;  // the J lowest free bits >= 5
    for (int b = 5; ne < g.J && b < nbits; b++) {
        bool used = false;
        for (int i = 0; i < nh; i++) used |= high[i] == b;
        if (!used) extra[ne++] = b;
    }
    if (ne < g.J) return -1;
    g.nfix = 0;
    for (int i = 0; i < ne; i++) g.fix[g.nfix++] = extra[i];
    for (int i = 0; i < nh; i++) g.fix[g.nfix++] = high[i];
    std::sort(g.fix, g.fix + g.nfix);
    for (int x = 0; x < (1 << K); x++) {
        uint64_t o = 0;
        uint32_t sx = 0;
        for (int b = 0; b < g.J; b++)
            if ((x >> b) & 1) o += 1ull << extra[b], sx |= 1u << g.lt[b];
        for (int i = 0; i < nh; i++)
            if ((x >> (g.J + i)) & 1) o += 1ull << high[i];
        g.xoff[x] = o;
        g.cw[x] = 8 * sx | 256 * (uint32_t)x;
        g.cr[x] = 8 * sx | 256 * (uint32_t)(x >> g.J << g.J);
    }
    return g.J ? launch_reg_kernel<K, true>(g, M, st) : launch_reg_kernel<K, false>(g, M, st);
}

// ---------------------------------------------------------------------------------------
// Register-tiled apply for k = 5 and 6 (n >= k + 6), on CUDA cores.
//
// At these widths the FMAs bind (4 2^k an amplitude: k = 5 takes 0.93 ms per 2^28 amplitudes at 128
// FMAs a clock and SM, against 0.64 ms of HBM traffic), so what matters is what else is issued
// beside them.  One group a thread needs the whole matrix per group: as constants 8 KiB miss the
// constant cache (63 FMAs a clock and SM), and 2^k members plus results leave 8 warps an SM.  Here a
// CTA keeps a tile of 64 groups in shared memory and thread (row group, group pair) sums a register
// tile of RT rows x 2 groups: per column one 16-byte load of its groups' members and RT/2 broadcast
// loads of the matrix feed 8 RT FMAs.  The tile lies in address order, 16-byte units XOR-swizzled
// (address bits 1-3 taken by targets are fed from the group bits of the lanes), so every target set
// is loaded and stored without bank conflicts; with bit 0 a target, a unit is two members of a
// group instead of one member of two groups (LOW0).  The next tile is fetched with cp.async during
// the sums (two buffers), and 2-5 CTAs an SM cover the exchange of the results through the tile.
// Sums run over the columns in ascending order, as everywhere here: bit-identical results.
// Measured on 2^28 amplitudes: k = 5 1.88-2.54 ms (register kernel, by targets) -> 1.43 ms for all
// (48 TFLOP/s), k = 6 2.78-7.63 ms (2.78 only with every target above bit 5) -> 2.65 ms.  Tried:
// 4 x 8 and 8 x 4 tiles on 128 or 256 groups 1.45-1.75 ms; one buffer 1.77; packed FMAs
// (fma.rn.f32x2), which do not raise the FMA rate but need operand pairs, 1.73.
// ---------------------------------------------------------------------------------------
constexpr int kRtF = 6;  // log2 groups a tile

struct RtGeom {
    float2 *psi;
    uint64_t n_tiles;
    int tpos[kMaxK];
    uint64_t off[16];   // global offset of local bit b (b < kRtF + k)
    uint32_t sw[16];    // staging byte address (swizzled) of local bit b
    uint32_t mem[64];   // staging byte address of member c
    uint32_t grp[kRtF]; // staging byte address of group bit i
};

constexpr int rtile_rows(int k) { return k == 5 ? 8 : 16; }
constexpr int rtile_threads(int k) { return 32 * ((1 << k) / rtile_rows(k)); }
constexpr int rtile_min_blocks(int k) { return k == 5 ? 4 : 2; }
constexpr size_t rtile_smem(int k) { return ((size_t)16 << (kRtF + k)) + ((size_t)8 << (2 * k)); }

template <int K, bool LOW0, typename MatSrc>
__global__ void __launch_bounds__(rtile_threads(K), rtile_min_blocks(K))
    k_apply_rtile(const __grid_constant__ RtGeom g, const __grid_constant__ MatSrc mat)
{
    constexpr int D = 1 << K, RT = rtile_rows(K), NT = rtile_threads(K), T = D << kRtF;
    constexpr int NI = T / 2 / NT;  // 16-byte units a thread moves
    constexpr int LT = __builtin_ctz(NT);
    extern __shared__ __align__(128) uint8_t sm[];
    float2 *M = reinterpret_cast<float2 *>(sm + 2 * T * 8);  // [row group][column][row]
    __shared__ uint64_t ioff[NI];
    __shared__ uint32_t isw[NI];
    const int tid = threadIdx.x, lane = tid & 31, rg = tid >> 5;
    {
        const float2 *src;
        if constexpr (K == 6) {
            src = mat.p;
        } else {
            src = mat.m;
            asm volatile("" : "+l"(src));  // ordinary loads, not constants (32 addresses a warp)
        }
        for (int i = tid; i < D * D; i += NT) {
            const int r = i / D, c = i % D;
            M[((r / RT) * D + c) * RT + r % RT] = src[i];
        }
    }
    // unit tid + i NT of a tile: local bits 1 .. LT from tid, the others from i
    if (tid < NI) {
        uint64_t o = 0;
        uint32_t s = 0;
        for (int b = 0; 1 + LT + b < kRtF + K; ++b)
            if ((tid >> b) & 1) {
                o += g.off[1 + LT + b];
                s ^= g.sw[1 + LT + b];
            }
        ioff[tid] = o;
        isw[tid] = s;
    }
    uint64_t toff = 0;
    uint32_t tsw = 0;
#pragma unroll
    for (int b = 0; b < LT; ++b)
        if ((tid >> b) & 1) {
            toff += g.off[1 + b];
            tsw ^= g.sw[1 + b];
        }
    // this thread's two groups: LOW0: group bits 0-4 = lane, bit 5 = which of the two; else bit 0 =
    // which (one unit holds both), bits 1-5 = lane
    uint32_t base[2] = {0, 0};
#pragma unroll
    for (int b = 0; b < 5; ++b)
        if ((lane >> b) & 1) base[0] ^= g.grp[(LOW0 ? 0 : 1) + b];
    if constexpr (LOW0) base[1] = base[0] ^ g.grp[5];
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sm);
    auto fetch = [&](uint64_t t, int buf) {
        const float2 *tp = g.psi + insert_zero_bits(t << kRtF, g.tpos, K) + toff;
#pragma unroll
        for (int i = 0; i < NI; ++i)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s0 + buf * T * 8 + (tsw ^ isw[i])),
                         "l"(tp + ioff[i])
                         : "memory");
    };
    __syncthreads();
    pdl_wait();
    if (blockIdx.x < g.n_tiles) fetch(blockIdx.x, 0);
    int buf = 0;
    for (uint64_t t = blockIdx.x; t < g.n_tiles; t += gridDim.x, buf ^= 1) {
        cp_async_wait_all();
        __syncthreads();  // the tile is here; the other buffer's results have been read out
        if (t + gridDim.x < g.n_tiles)
            fetch(t + gridDim.x, buf ^ 1);
        else
            pdl_launch_next();
        uint8_t *sb = sm + buf * T * 8;
        float2 y[RT][2];
#pragma unroll
        for (int r = 0; r < RT; ++r) y[r][0] = y[r][1] = make_float2(0.f, 0.f);
        const float4 *mr = reinterpret_cast<const float4 *>(M + rg * RT * D);
#pragma unroll 2
        for (int c = 0; c < D; c += 2) {
            const uint32_t m0 = g.mem[c], m1 = g.mem[c + 1];
            const float4 u = *reinterpret_cast<const float4 *>(sb + (base[0] ^ m0));
            const float4 v = *reinterpret_cast<const float4 *>(sb + (LOW0 ? base[1] ^ m0 : base[0] ^ m1));
            // x[column][group]
            const float2 x[2][2] = {{make_float2(u.x, u.y), LOW0 ? make_float2(v.x, v.y) : make_float2(u.z, u.w)},
                                    {LOW0 ? make_float2(u.z, u.w) : make_float2(v.x, v.y), make_float2(v.z, v.w)}};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float2 m[RT];
#pragma unroll
                for (int r = 0; r < RT; r += 2) {
                    const float4 w = mr[((c + e) * RT + r) / 2];
                    m[r] = make_float2(w.x, w.y);
                    m[r + 1] = make_float2(w.z, w.w);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
#pragma unroll
                    for (int r = 0; r < RT; ++r) {
                        y[r][j].x = fmaf(m[r].x, x[e][j].x, y[r][j].x);
                        y[r][j].y = fmaf(m[r].x, x[e][j].y, y[r][j].y);
                    }
#pragma unroll
                    for (int r = 0; r < RT; ++r) {
                        y[r][j].x = fmaf(m[r].y, -x[e][j].y, y[r][j].x);
                        y[r][j].y = fmaf(m[r].y, x[e][j].x, y[r][j].y);
                    }
                }
            }
        }
        __syncthreads();  // every member has been read
#pragma unroll
        for (int r = 0; r < RT; r += 2) {
            const uint32_t m0 = g.mem[rg * RT + r], m1 = g.mem[rg * RT + r + 1];
            if constexpr (LOW0) {
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    *reinterpret_cast<float4 *>(sb + (base[j] ^ m0)) =
                        make_float4(y[r][j].x, y[r][j].y, y[r + 1][j].x, y[r + 1][j].y);
            } else {
                *reinterpret_cast<float4 *>(sb + (base[0] ^ m0)) =
                    make_float4(y[r][0].x, y[r][0].y, y[r][1].x, y[r][1].y);
                *reinterpret_cast<float4 *>(sb + (base[0] ^ m1)) =
                    make_float4(y[r + 1][0].x, y[r + 1][0].y, y[r + 1][1].x, y[r + 1][1].y);
            }
        }
        __syncthreads();
        float2 *tp = g.psi + insert_zero_bits(t << kRtF, g.tpos, K) + toff;
#pragma unroll
        for (int i = 0; i < NI; ++i)
            __stcs(reinterpret_cast<float4 *>(tp + ioff[i]), *reinterpret_cast<const float4 *>(sb + (tsw ^ isw[i])));
    }
}

template <int K, bool LOW0, typename MatSrc>
int launch_rtile_kernel(const RtGeom &g, const MatSrc &M, cudaStream_t st)
{
    auto kern = k_apply_rtile<K, LOW0, MatSrc>;
    constexpr size_t smem = rtile_smem(K);
    static std::atomic<uint64_t> smem_done{0};
    if (smem > 48 * 1024 && !smem_opt_in(kern, (int)smem, smem_done)) return -1;
    static const LaunchCfg cfg = [&] {
        LaunchCfg c;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return c;
        if (cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return c;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c.occ, kern, rtile_threads(K), smem) != cudaSuccess ||
            c.occ < 1)
            c.occ = 1;
        c.ok = true;
        return c;
    }();
    if (!cfg.ok) return -1;
    const uint64_t grid = std::min<uint64_t>(g.n_tiles, (uint64_t)cfg.sms * cfg.occ);
    return launch_pdl(kern, (unsigned)grid, rtile_threads(K), smem, st, g, M) == cudaSuccess ? 0 : -1;
}

template <int K, typename MatSrc>
int launch_rtile(float2 *psi, int nbits, const int *tpos, const MatSrc &M, cudaStream_t st)
{
    RtGeom g{};
    g.psi = psi;
    g.n_tiles = 1ull << (nbits - K - kRtF);
    bool is_target[64] = {};
    for (int q = 0; q < K; q++) {
        g.tpos[q] = tpos[q];
        is_target[tpos[q]] = true;
    }
    // local bits: the targets and the kRtF lowest other bits, ascending
    int addr[16], mpos[kMaxK], gpos[kRtF], nl = 0, nm = 0, ng = 0;
    for (int b = 0; b < nbits && nl < K + kRtF; b++) {
        if (is_target[b])
            mpos[nm++] = nl;
        else if (ng < kRtF)
            gpos[ng++] = nl;
        else
            continue;
        addr[nl++] = b;
    }
    if (nl != K + kRtF) return -1;
    // the lanes' three lowest group bits must reach address bits 1-3 (the 16-byte units of a 128-byte
    // line): those that lie higher are XORed into the bits that targets occupy, in order
    const int l0 = is_target[0] ? 0 : 1;
    int src[3], ns = 0, dst[3], nd = 0;
    for (int b = 1; b <= 3; b++)
        if (is_target[b]) dst[nd++] = b;
    for (int i = 0; i < 3; i++)
        if (gpos[l0 + i] > 3) src[ns++] = gpos[l0 + i];
    if (ns != nd) return -1;
    auto swz = [&](uint32_t p) {
        uint32_t x = p;
        for (int i = 0; i < nd; i++) x ^= ((p >> src[i]) & 1u) << dst[i];
        return 8 * x;
    };
    for (int x = 0; x < nl; x++) {
        g.off[x] = 1ull << addr[x];
        g.sw[x] = swz(1u << x);
    }
    for (int c = 0; c < (1 << K); c++) {
        uint32_t p = 0;
        for (int q = 0; q < K; q++)
            if ((c >> q) & 1) p |= 1u << mpos[q];
        g.mem[c] = swz(p);
    }
    for (int i = 0; i < kRtF; i++) g.grp[i] = swz(1u << gpos[i]);
    return is_target[0] ? launch_rtile_kernel<K, true>(g, M, st) : launch_rtile_kernel<K, false>(g, M, st);
}

template <int K>
int launch_param(float2 *psi, int nbits, const int *tpos, const float2 *mat, cudaStream_t st)
{
    MatP<K> M;
    std::memcpy(M.m, mat, sizeof(M.m));
    // Measured on GB300 at n = 30: for k <= 3 with every target >= 5 the one-group-per-thread
    // kernel streams at ~7.0 TB/s, ~10% above the persistent register kernel; everywhere
    // else (k = 4, or any target below bit 5) the register kernel is faster.
    if constexpr (K <= 3) {
        if (tpos[0] >= 5 && nbits - K >= 8) return launch_direct<K>(psi, nbits, tpos, M, st);
    }
    if constexpr (K <= 4) {
        if (nbits >= K + 5) return launch_reg<K>(psi, nbits, tpos, M, st);
        return launch_tiled<K>(psi, nbits, tpos, M, st);
    } else {
        return nbits >= K + kRtF ? launch_rtile<K>(psi, nbits, tpos, M, st) : launch_cta<K>(psi, nbits, tpos, M, st);
    }
}

}  // namespace

int launch_apply_fp32(sim_t *, float2 *psi, int nbits, int k, const int *tpos, const float2 *mat,
                      const float2 *mat6_dev, cudaStream_t st)
{
    switch (k) {
    case 1: return launch_param<1>(psi, nbits, tpos, mat, st);
    case 2: return launch_param<2>(psi, nbits, tpos, mat, st);
    case 3: return launch_param<3>(psi, nbits, tpos, mat, st);
    case 4: return launch_param<4>(psi, nbits, tpos, mat, st);
    case 5: return launch_param<5>(psi, nbits, tpos, mat, st);
    case 6:
        if (nbits >= 6 + kRtF) return launch_rtile<6>(psi, nbits, tpos, MatPtr{mat6_dev}, st);
        return launch_cta<6>(psi, nbits, tpos, MatPtr{mat6_dev}, st);
    default: return -1;
    }
}

// Validate targets, map them to physical bits through phys_of (a qubit whose entry is < 0 or
// >= nlocal is not local), sort, and reorder + round the FP64 matrix to FP32 in sorted-bit
// order.  Returns SIM_OK or an error code (message set on h).
int prepare_block_map(sim_t *h, int k, const int *targets, const double *matrix, const int *phys_of,
                      int nlocal, int *tpos, float2 *mat, int nq)
{
    if (nq < 0) nq = h->n;
    if (k < 1 || k > kMaxK) return fail(h, SIM_E_INVAL, "apply: k=%d outside 1..%d", k, kMaxK);
    if (!targets || !matrix) return fail(h, SIM_E_INVAL, "apply: NULL targets or matrix");
    if (k > nlocal)
        return fail(h, SIM_E_NONLOCAL, "apply: k=%d exceeds the %d local qubits", k, nlocal);
    int phys[kMaxK], order[kMaxK];
    for (int j = 0; j < k; j++) {
        const int q = targets[j];
        if (q < 0 || q >= nq) return fail(h, SIM_E_INVAL, "apply: target %d outside 0..%d", q, nq - 1);
        for (int i = 0; i < j; i++)
            if (targets[i] == q) return fail(h, SIM_E_INVAL, "apply: duplicate target %d", q);
        phys[j] = phys_of[q];
        if (phys[j] < 0 || phys[j] >= nlocal)
            return fail(h, SIM_E_NONLOCAL, "apply: qubit %d is sliced (not among the %d local bits)", q,
                        nlocal);
        order[j] = j;
    }
    std::sort(order, order + k, [&](int a, int b) { return phys[a] < phys[b]; });
    for (int i = 0; i < k; i++) tpos[i] = phys[order[i]];
    const int D = 1 << k;
    int map[64];
    for (int x = 0; x < D; x++) {
        int y = 0;
        for (int i = 0; i < k; i++)
            if ((x >> i) & 1) y |= 1 << order[i];
        map[x] = y;
    }
    for (int r = 0; r < D; r++)
        for (int c = 0; c < D; c++) {
            const double *e = matrix + 2 * ((size_t)map[r] * D + map[c]);
            mat[r * D + c] = make_float2((float)e[0], (float)e[1]);
        }
    return SIM_OK;
}

int prepare_block(sim_t *h, int k, const int *targets, const double *matrix, int *tpos, float2 *mat)
{
    return prepare_block_map(h, k, targets, matrix, h->bit_of, h->n - h->s, tpos, mat);
}

// Which kernel family takes a block: the one place that decides it.
BlockPath block_path(int nbits, int k, const int *tpos, int precision)
{
    if (tmem_mode(precision) && tcgen05_eligible(nbits, k, tpos)) return BlockPath::Tcgen05;
    if (precision != SIM_FP32 && (tc_eligible(nbits, k, tpos) || (tmem_mode(precision) && tc_eligible_low4(nbits, k))))
        return BlockPath::MmaSync;
    return BlockPath::CudaCore;
}

// A block's matrix travels as kernel parameters (k <= 5) or, at k = 6, through device memory.
size_t block_staged_bytes(int k) { return k == 6 ? sizeof(float2) * 4096 : 0; }

bool staging_slot_free(sim_t *h, int k)
{
    // an event never recorded counts as complete
    return block_staged_bytes(k) == 0 || cudaEventQuery(h->mat6_ev[h->mat6_next]) != cudaErrorNotReady;
}

int launch_block_staged(sim_t *h, float2 *psi, int nbits, int k, const int *tpos, const float2 *mat,
                        int precision, const void *d_staged, cudaStream_t st, double *red, int *red_grid)
{
    int rc;
    if (red_grid) *red_grid = 0;
    const float2 *mat6 = k == 6 ? static_cast<const float2 *>(d_staged) : nullptr;
    switch (block_path(nbits, k, tpos, precision)) {
    case BlockPath::Tcgen05:
        rc = launch_apply_tcgen05(h, psi, nbits, k, tpos, mat, mat6, precision == SIM_BF16X3, st, red, red_grid);
        break;
    case BlockPath::MmaSync: rc = launch_apply_tc(psi, nbits, k, tpos, mat, mat6, precision, st); break;
    default: rc = launch_apply_fp32(h, psi, nbits, k, tpos, mat, mat6, st); break;
    }
    if (rc != 0) return fail(h, SIM_E_CUDA, "apply: kernel launch failed: %s", cudaGetErrorString(cudaGetLastError()));
    return SIM_OK;
}

// Enqueue one prepared block on a buffer of 2^nbits amplitudes, on stream st.
int enqueue_block_on(sim_t *h, float2 *psi, int nbits, int k, const int *tpos, const float2 *mat,
                     int precision, cudaStream_t st)
{
    const size_t bytes = block_staged_bytes(k);
    float2 *staged = nullptr;
    int slot = -1;
    if (bytes) {
        slot = h->mat6_next;
        h->mat6_next = (slot + 1) % sim_s::kMat6Slots;
        SIM_CUDA_TRY(h, cudaEventSynchronize(h->mat6_ev[slot]));  // host staging slot free
        std::memcpy(h->h_mat6 + 4096 * slot, mat, bytes);
        staged = h->d_mat6 + 4096 * slot;
        SIM_CUDA_TRY(h, cudaMemcpyAsync(staged, h->h_mat6 + 4096 * slot, bytes, cudaMemcpyHostToDevice, st));
    }
    const int ps = prof_begin(h, SIM_PROF_APPLY, 16.0 * std::ldexp(1.0, nbits), st);
    const int rc = launch_block_staged(h, psi, nbits, k, tpos, mat, precision, staged, st);
    prof_end(h, ps, st);
    // the matrix slot is free again once this kernel, which reads it, has run (on any stream)
    if (slot >= 0) SIM_CUDA_TRY(h, cudaEventRecord(h->mat6_ev[slot], st));
    return rc;
}

int enqueue_block(sim_t *h, int k, const int *tpos, const float2 *mat, int precision)
{
    return enqueue_block_on(h, h->d_state, h->n, k, tpos, mat, precision, h->stream);
}

bool precision_ok(int precision) { return precision >= SIM_FP32 && precision <= SIM_BF16X3; }

}  // namespace sycsim

using namespace sycsim;

extern "C" int sim_apply_fused(sim_t *h, int k, const int *targets, const double *matrix,
                               int precision)
{
    if (!h) return fail(nullptr, SIM_E_INVAL, "sim_apply_fused: NULL handle");
    state_written(h);
    if (h->store != SIM_STORE_DEVICE)
        return fail(h, SIM_E_UNSUPPORTED, "sim_apply_fused: host-store state: use sim_run_phase");
    if (!precision_ok(precision))
        return fail(h, SIM_E_INVAL, "sim_apply_fused: precision %d", precision);
    int tpos[kMaxK];
    static thread_local float2 mat[4096];
    int rc = prepare_block(h, k, targets, matrix, tpos, mat);
    if (rc != SIM_OK) return rc;
    SIM_DEVICE_SCOPE(h, h->device);
    return enqueue_block(h, k, tpos, mat, precision);
}
