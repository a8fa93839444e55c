// apply_tc.cu -- aggregated k-qubit gate apply on tensor cores (k = 4..6).
//
// The block y = M x (M complex 2^k x 2^k) is written over the reals: with x as 2^(k+1) reals,
// R = [[Re M, -Im M], [Im M, Re M]] (interleaved), and for a tile of 16 groups
//     W^T (16 x 2^(k+1)) = V^T (16 x 2^(k+1)) . R^T,
// one warp-level mma.sync m16n8k8 (TF32 in, FP32 accumulate) per 8x8 piece of R^T.
//
// Orderings are chosen so that every thread moves whole complex amplitudes:
//  * K (input reals) in steps of 8 = 4 members: column c < 4 is Re of member 4s + c, column
//    c >= 4 is Im of member 4s + c - 4.  A thread's A fragment (rows g, g+8; columns t, t+4)
//    is then the two complex values member 4s + t of groups g and g + 8: one 8-byte load each.
//  * N (output reals) in tiles of 8 = 4 members: columns 2t, 2t+1 are Re, Im of member 4n + t,
//    so a thread's accumulator pairs are whole output amplitudes: one 8-byte store each.
// The B fragments (R^T, permuted as above, split hi/lo for the 3xTF32 mode) are built from the
// FP32 matrix once per CTA, fragment-major in shared memory.
//
// Accumulation: chaining many MMAs through one FP32 accumulator was measured to shrink the
// state's norm systematically (the tensor cores' internal accumulation is not round-to-nearest):
// -4e-7 per k = 5 pass.  So each k-step's main product starts from a zero accumulator and is
// added with round-to-nearest FP32 adds, and the small hi*lo + lo*hi corrections (2^-11 of
// the main term) are chained in a second accumulator.  Outputs are produced in chunks of at
// most 4 n-tiles to bound the accumulator registers.
//
// Modes: TF32 (one MMA per piece; TF32 keeps 10 mantissa bits, so ~1e-3 relative error per
// pass) and 3xTF32 (a = a_hi + a_lo with both parts TF32; hi*hi + hi*lo + lo*hi recovers
// ~FP32 accuracy); see also 3xFP16 below.  Used for k >= 5.  A tile's 16 groups are 16
// consecutive group indices; with every target >= bit 4 each member load is a 64-byte run
// per 8 groups, with low targets the runs interleave members instead.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "block_mat.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace sycsim {
namespace {

struct MmaGeom {
    float2 *psi;
    uint64_t n_mtiles;      // tiles of 16 groups: 2^(nbits - k - 4)
    int tpos[kMaxK];        // ascending target bits
    uint64_t moff[64];      // offset of member j
    int early;              // the next kernel may start before this one ends (pdl_early)
};

__device__ __forceinline__ uint32_t to_tf32(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint64_t insert_zero_bits_t(uint64_t x, const int *pos, int cnt)
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

// Tuning constants (overridable at build time): CTAs per SM each width is compiled for, and
// the n-tiles per output chunk.
#ifndef SYCSIM_MMA_MINB5
#define SYCSIM_MMA_MINB5 3
#endif
#ifndef SYCSIM_MMA_NC
#define SYCSIM_MMA_NC 2
#endif
constexpr int mma_min_blocks(int k) { return k <= 4 ? 2 : (k == 5 ? SYCSIM_MMA_MINB5 : 1); }

// Round an FP32 value to TF32 (nearest, ties away from zero) with the dropped bits zero.
__device__ __forceinline__ uint32_t round_tf32(float x)
{
    uint32_t u = __float_as_uint(x);
    if ((u & 0x7f800000u) == 0x7f800000u) return u & 0xffffe000u;  // inf/nan: truncate
    u += 0x1000u;                                                  // half of the dropped 13 bits
    return u & 0xffffe000u;
}

// The B fragments of one block into shared memory (all threads): B[k][n] = R^T, permuted: k = (step
// s, column c): member 4s + (c & 3), Re for c < 4, Im for c >= 4; n = (tile m, column c'): member
// 4m + c'/2, Re for even c', Im for odd c'.  With the split, hi then lo.  Splitting on the device
// keeps the host's share of a block to copying its matrix (built there it cost 15-200 us a block).
template <int K, bool kSplit>
__device__ __forceinline__ void build_frag_tf32(const float2 *mat, uint32_t *sb)
{
    constexpr int D = 1 << K, NT = D / 4, PAIRS = (D / 4) * NT * 32;
    for (int i = threadIdx.x; i < PAIRS; i += blockDim.x) {
        const int lane = i & 31, n = (i >> 5) & (NT - 1), s = (i >> 5) / NT;
        const int gid = lane >> 2, t = lane & 3;
        const float2 m = mat[(4 * n + (gid >> 1)) * D + 4 * s + t];
        const bool out_im = gid & 1;
        const float b0 = out_im ? m.y : m.x;   // Re x -> (Re y: Mr, Im y: Mi)
        const float b1 = out_im ? m.x : -m.y;  // Im x -> (Re y: -Mi, Im y: Mr)
        const uint32_t h0 = round_tf32(b0), h1 = round_tf32(b1);
        *reinterpret_cast<uint2 *>(sb + 2 * i) = make_uint2(h0, h1);
        if constexpr (kSplit)
            *reinterpret_cast<uint2 *>(sb + 2 * PAIRS + 2 * i) =
                make_uint2(round_tf32(b0 - __uint_as_float(h0)), round_tf32(b1 - __uint_as_float(h1)));
    }
    __syncthreads();
}

template <int K, bool kSplit>
__global__ void __launch_bounds__(256, mma_min_blocks(K)) k_apply_mma(const __grid_constant__ MmaGeom g,
                                                                      const __grid_constant__ BlockMat<K> M)
{
    constexpr int D = 1 << K;
    constexpr int KS = D / 4;  // k-steps (4 input members each)
    constexpr int NT = D / 4;  // n-tiles (4 output members each)
    constexpr int NC = NT < SYCSIM_MMA_NC ? NT : SYCSIM_MMA_NC;  // n-tiles per output chunk
    constexpr int FRAG_WORDS = KS * NT * 64;
    extern __shared__ uint32_t sb[];
    if (g.early) pdl_launch_next();
    build_frag_tf32<K, kSplit>(block_mat_ptr(M), sb);
    pdl_wait();

    const int lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t mt = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; mt < g.n_mtiles;
         mt += nw) {
        const uint64_t grp = mt * 16 + gid;
        float2 *p0 = g.psi + insert_zero_bits_t(grp, g.tpos, K);
        float2 *p1 = g.psi + insert_zero_bits_t(grp + 8, g.tpos, K);
        float2 x0[KS], x1[KS];
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            x0[s] = __ldcs(p0 + g.moff[4 * s + t]);
            x1[s] = __ldcs(p1 + g.moff[4 * s + t]);
        }
#pragma unroll 1
        for (int c0 = 0; c0 < NT; c0 += NC) {
            float acc[NC][4], cor[NC][4];
#pragma unroll
            for (int n = 0; n < NC; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[n][i] = cor[n][i] = 0.f;
#pragma unroll
            for (int s = 0; s < KS; ++s) {
                const float av[4] = {x0[s].x, x1[s].x, x0[s].y, x1[s].y};
                uint32_t ahi[4], alo[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    ahi[i] = to_tf32(av[i]);
                    if constexpr (kSplit) alo[i] = to_tf32(av[i] - __uint_as_float(ahi[i]));
                }
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const int nt = c0 + n;
                    const uint2 bh = *reinterpret_cast<const uint2 *>(sb + ((s * NT + nt) * 32 + lane) * 2);
                    float part[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_tf32(part, ahi, bh.x, bh.y);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[n][i] += part[i];
                    if constexpr (kSplit) {
                        const uint2 bl = *reinterpret_cast<const uint2 *>(
                            sb + FRAG_WORDS + ((s * NT + nt) * 32 + lane) * 2);
                        mma_tf32(cor[n], ahi, bl.x, bl.y);
                        mma_tf32(cor[n], alo, bh.x, bh.y);
                    }
                }
            }
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int nt = c0 + n;
                __stcs(p0 + g.moff[4 * nt + t], make_float2(acc[n][0] + cor[n][0], acc[n][1] + cor[n][1]));
                __stcs(p1 + g.moff[4 * nt + t], make_float2(acc[n][2] + cor[n][2], acc[n][3] + cor[n][3]));
            }
        }
    }
}

// ---- 3xFP16: the same GEMM with m16n8k16 FP16 MMAs (twice the TF32 rate on this GPU) ----
// K steps of 16 reals = 8 members: columns 2t, 2t+1 are (Re, Im) of member 8s + t, columns
// 2t+8, 2t+9 of member 8s + 4 + t, so each A register is one packed half2 amplitude.  The
// state is scaled per warp tile by a power of two so that its largest component sits near
// 2^14 (FP16 keeps it normal), split as hi = fp16(a), lo = fp16(a - hi); the products
// hi*hi + hi*lo + lo*hi are accumulated in FP32 and the scale is removed exactly.
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void split_half2(float re, float im, uint32_t &hi, uint32_t &lo)
{
    const __half2 h = __floats2half2_rn(re, im);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(re - hf.x, im - hf.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// The B fragments (hi, lo) of one block into shared memory (all threads): k rows 2t, 2t+1 | 2t+8,
// 2t+9; n column gid, as half2 (Re-input, Im-input) of input member 8s + t (word 0) and 8s + 4 + t
// (word 1) for output member 4n + gid/2.
template <int K>
__device__ __forceinline__ void build_frag_f16(const float2 *mat, uint32_t *sb)
{
    constexpr int D = 1 << K, NT = D / 4, PAIRS = (D / 8) * NT * 32;
    for (int i = threadIdx.x; i < PAIRS; i += blockDim.x) {
        const int lane = i & 31, n = (i >> 5) & (NT - 1), s = (i >> 5) / NT;
        const int gid = lane >> 2, t = lane & 3;
        const bool out_im = gid & 1;
        uint32_t hi[2], lo[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 m = mat[(4 * n + (gid >> 1)) * D + 8 * s + 4 * j + t];
            // coefficients of Re x and Im x
            split_half2(out_im ? m.y : m.x, out_im ? m.x : -m.y, hi[j], lo[j]);
        }
        *reinterpret_cast<uint2 *>(sb + 2 * i) = make_uint2(hi[0], hi[1]);
        *reinterpret_cast<uint2 *>(sb + 2 * PAIRS + 2 * i) = make_uint2(lo[0], lo[1]);
    }
    __syncthreads();
}

template <int K>
__global__ void __launch_bounds__(256, mma_min_blocks(K)) k_apply_mma_f16x3(const __grid_constant__ MmaGeom g,
                                                                            const __grid_constant__ BlockMat<K> M)
{
    constexpr int D = 1 << K;
    constexpr int KS = D / 8;  // k-steps (8 input members each)
    constexpr int NT = D / 4;  // n-tiles (4 output members each)
    constexpr int NC = NT < SYCSIM_MMA_NC ? NT : SYCSIM_MMA_NC;
    constexpr int FRAG_WORDS = KS * NT * 64;
    extern __shared__ uint32_t sb[];
    if (g.early) pdl_launch_next();
    build_frag_f16<K>(block_mat_ptr(M), sb);
    pdl_wait();

    const int lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t mt = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; mt < g.n_mtiles;
         mt += nw) {
        const uint64_t grp = mt * 16 + gid;
        float2 *p0 = g.psi + insert_zero_bits_t(grp, g.tpos, K);
        float2 *p1 = g.psi + insert_zero_bits_t(grp + 8, g.tpos, K);
        float2 x0[2 * KS], x1[2 * KS];  // members 8s + t (even index) and 8s + 4 + t (odd index)
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            x0[2 * s] = __ldcs(p0 + g.moff[8 * s + t]);
            x0[2 * s + 1] = __ldcs(p0 + g.moff[8 * s + 4 + t]);
            x1[2 * s] = __ldcs(p1 + g.moff[8 * s + t]);
            x1[2 * s + 1] = __ldcs(p1 + g.moff[8 * s + 4 + t]);
        }
        float amax = 0.f;
#pragma unroll
        for (int i = 0; i < 2 * KS; ++i)
            amax = fmaxf(amax, fmaxf(fmaxf(fabsf(x0[i].x), fabsf(x0[i].y)), fmaxf(fabsf(x1[i].x), fabsf(x1[i].y))));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        int e = 0;
        frexpf(amax, &e);                       // amax < 2^e
        const int sh = amax > 0.f ? max(-100, min(100, 14 - e)) : 0;  // largest component < 2^14
        const float sc = ldexpf(1.f, sh), inv = ldexpf(1.f, -sh);
#pragma unroll 1
        for (int c0 = 0; c0 < NT; c0 += NC) {
            float acc[NC][4], cor[NC][4];
#pragma unroll
            for (int n = 0; n < NC; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[n][i] = cor[n][i] = 0.f;
#pragma unroll
            for (int s = 0; s < KS; ++s) {
                uint32_t ahi[4], alo[4];
                split_half2(x0[2 * s].x * sc, x0[2 * s].y * sc, ahi[0], alo[0]);
                split_half2(x1[2 * s].x * sc, x1[2 * s].y * sc, ahi[1], alo[1]);
                split_half2(x0[2 * s + 1].x * sc, x0[2 * s + 1].y * sc, ahi[2], alo[2]);
                split_half2(x1[2 * s + 1].x * sc, x1[2 * s + 1].y * sc, ahi[3], alo[3]);
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const int nt = c0 + n;
                    const uint2 bh = *reinterpret_cast<const uint2 *>(sb + ((s * NT + nt) * 32 + lane) * 2);
                    const uint2 bl =
                        *reinterpret_cast<const uint2 *>(sb + FRAG_WORDS + ((s * NT + nt) * 32 + lane) * 2);
                    float part[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_f16(part, ahi, bh.x, bh.y);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[n][i] += part[i];
                    mma_f16(cor[n], ahi, bl.x, bl.y);
                    mma_f16(cor[n], alo, bh.x, bh.y);
                }
            }
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int nt = c0 + n;
                __stcs(p0 + g.moff[4 * nt + t],
                       make_float2((acc[n][0] + cor[n][0]) * inv, (acc[n][1] + cor[n][1]) * inv));
                __stcs(p1 + g.moff[4 * nt + t],
                       make_float2((acc[n][2] + cor[n][2]) * inv, (acc[n][3] + cor[n][3]) * inv));
            }
        }
    }
}

template <int K>
constexpr size_t f16x3_bytes() { return sizeof(uint32_t) * 2 * ((1 << K) / 8) * ((1 << K) / 4) * 64; }

template <int K, bool kSplit>
constexpr size_t mma_bytes() { return sizeof(uint32_t) * (kSplit ? 2 : 1) * ((1 << K) / 4) * ((1 << K) / 4) * 64; }

template <int K, size_t kBytes, void (*kern)(const MmaGeom, const BlockMat<K>)>
int launch_mma(float2 *psi, int nbits, const int *tpos, const BlockMat<K> &M, int precision, cudaStream_t st)
{
    constexpr int D = 1 << K;
    MmaGeom g{};
    g.psi = psi;
    g.n_mtiles = 1ull << (nbits - K - 4);
    for (int i = 0; i < K; i++) g.tpos[i] = tpos[i];
    for (int j = 0; j < D; j++) {
        uint64_t o = 0;
        for (int b = 0; b < K; b++)
            if ((j >> b) & 1) o += 1ull << tpos[b];
        g.moff[j] = o;
    }
    static std::atomic<uint64_t> smem_done{0};
    if (kBytes > 48 * 1024 && !smem_opt_in(kern, (int)kBytes, smem_done)) return -1;
    static const LaunchCfg cfg = [&] {  // once per instantiation, thread-safe
        LaunchCfg c;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return c;
        if (cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return c;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c.occ, kern, 256, kBytes) != cudaSuccess || c.occ < 1)
            c.occ = 1;
        c.ok = true;
        return c;
    }();
    if (!cfg.ok) return -1;
    const uint64_t need = (g.n_mtiles + 7) / 8;
    const uint64_t most = (uint64_t)cfg.sms * cfg.occ, grid = std::min<uint64_t>(need, most);
    // With room left on the SMs, where several CTAs fit on one (k = 4, 5), the next pass's CTAs crowd
    // (pdl.cuh): early only with half of the SMs idle or all of the room taken.  Replays of 3xFP16 plans, k =
    // 5, early / not: 18 qubits (64 CTAs) 60 / 70 us, 19 100 / 76, 20 125 / 106, 21 (all taken) 165 / 174, 24
    // 864 / 874; k = 6, one CTA an SM, 19 qubits 98 / 112, 20 117 / 127.  In the tcgen05 modes the next pass
    // is mostly one of those kernels, of which one CTA fills an SM: always early (reset and plan, 14
    // cycles, k_max 6, 19 qubits 119 / 124, 20 146 / 148).
    g.early = pdl_early(nbits) && (tmem_mode(precision) || cfg.occ == 1 || 2 * grid <= (uint64_t)cfg.sms || grid == most);
    return launch_pdl(kern, (unsigned)grid, 256, kBytes, st, g, M) == cudaSuccess ? 0 : -1;
}

}  // namespace

// Measured on GB300 (n = 30, ms a pass): for k >= 5 the tensor cores win (3xFP16 k = 5 2.8-3.3, CUDA-core
// FP32 5.7; k = 6 4.5-5.1, 10.6).  k = 4 stays on CUDA cores in these modes (2.81 with every target at bit 5
// and above, 3.18-3.20 otherwise): the tensor-core kernels took 3.6 and more when the rule was made
// (3xFP16 with a low target: below).  Any target set works: groups map to amplitude offsets by bit insertion.
bool tc_eligible(int nbits, int k, const int *) { return k >= 5 && k <= 6 && nbits >= k + 4; }

// In SIM_FP16X3_TMEM mode the blocks the tcgen05 kernel leaves (targets in the low bits) come
// here for k = 4 too: measured on 2^30 amplitudes, targets {0,1,2,3}: 2.73 ms (CUDA-core FP32
// 3.18 ms), {0,2,6,8}: 2.60 ms (3.19), {1,6,7,12}: 2.61 ms (3.20).
bool tc_eligible_low4(int nbits, int k) { return k == 4 && nbits >= k + 4; }

int launch_apply_tc(float2 *psi, int nbits, int k, const int *tpos, const float2 *mat, const float2 *mat6_dev,
                    int precision, cudaStream_t st)
{
    auto go = [&](auto kc) {
        constexpr int K = decltype(kc)::value;
        const BlockMat<K> M = block_mat<K>(mat, mat6_dev);
        if (f16x3_mode(precision)) return launch_mma<K, f16x3_bytes<K>(), k_apply_mma_f16x3<K>>(psi, nbits, tpos, M, precision, st);
        if (precision == SIM_TF32X3)
            return launch_mma<K, mma_bytes<K, true>(), k_apply_mma<K, true>>(psi, nbits, tpos, M, precision, st);
        return launch_mma<K, mma_bytes<K, false>(), k_apply_mma<K, false>>(psi, nbits, tpos, M, precision, st);
    };
    switch (k) {
    case 4: return go(std::integral_constant<int, 4>{});
    case 5: return go(std::integral_constant<int, 5>{});
    case 6: return go(std::integral_constant<int, 6>{});
    default: return -1;
    }
}

}  // namespace sycsim
