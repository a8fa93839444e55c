// permute.cu -- in-place qubit-bit permutation of the state (Sect. 4: between phases the
// layout is reorganised so that a different set of qubits is local; on one GPU this is a
// permutation of the amplitude-index bits).  Pure data movement: bit-exact.
//
// A bit permutation pi is written as sigma2 o sigma1 with both sigmas involutions (products
// of disjoint bit transpositions): a cycle c_0 -> c_1 -> ... -> c_{L-1} is the reflection
// x -> 1 - x (mod L) after the reflection x -> -x (mod L).  Each involution is one pass:
//  * transpositions between two bits >= LB swap whole tiles (tile tau <-> tile sigma(tau));
//  * transpositions with one bit < LB make the other bit a "row" bit of the tile;
//  * transpositions inside [0, LB) act within the tile.
// A tile (or tile pair) of 2^(LB+q) amplitudes, rows of 2^LB contiguous amplitudes, is brought into
// shared memory, permuted there and written back.  Tiles that nothing moves are skipped, so a single
// high-bit swap touches half of the state.  Three kernels, chosen in launch_involution: a tensor-map
// pipeline (k_permute_tma), a bulk copy a row where rows are long (k_permute_tile_bulk), 16-byte loads
// and stores for the small states and the geometries left (k_permute_pass).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"
#include "pdl.cuh"

// Measured on 2^30 amplitudes: 16-byte accesses 13-17 % faster than 8-byte on every pattern;
// minimum tiles of 2^11-2^12 amplitudes help tiles that permute in place a little and tile pairs
// much less (persistent CTAs looping over tile pairs were slower still).
#ifndef SYCSIM_PERM_TILE
#define SYCSIM_PERM_TILE 10  // minimum tile: 2^SYCSIM_PERM_TILE amplitudes
#endif
#ifndef SYCSIM_PERM_TILE_SAME
#define SYCSIM_PERM_TILE_SAME 12  // the same when no tile pairs swap (measured best of 10..13)
#endif

namespace sycsim {
namespace {

constexpr int kMaxRow = 6;

struct PermGeom {
    float2 *psi;
    int LB, q;                    // low-block bits, row bits
    int rowpos[kMaxRow];          // global bit of row bit i (ascending)
    int sig[16];                  // in-tile involution on local bits 0..LB+q-1
    int nhh, hh_a[20], hh_b[20];  // high-high transpositions
    int trivial_in;               // sig is the identity
    uint32_t fsw[1 << kMaxRow];   // row r -> XOR applied to its low index (bank spreading)
    uint64_t rowoff[1 << kMaxRow];
    // the in-tile maps are XOR-linear in the local index p: their values on each single bit
    uint64_t lin_off[16];   // global offset of p (row offset + low index)
    uint32_t lin_sidx[16];  // shared-memory slot of p (row-XOR swizzle)
    uint32_t lin_src[16];   // shared-memory slot of the amplitude that lands at p (swizzle o sig)
    // bulk in-place path: local bit of thread-index bit j (bits 0-4: the lanes of a warp, chosen so
    // that p and sig(p) both spread over the shared-memory banks), then the iteration bits
    int8_t tbit[8], ibit[16];
};

__device__ __forceinline__ uint64_t insert_zero_bits_p(uint64_t x, const int *pos, int cnt)
{
    for (int i = 0; i < cnt; ++i) {
        const int p = pos[i];
        const uint64_t lo = x & ((1ull << p) - 1);
        x = ((x >> p) << (p + 1)) | lo;
    }
    return x;
}

__global__ void __launch_bounds__(256) k_permute_pass(PermGeom g)
{
    extern __shared__ float2 sm[];
    pdl_wait();
    const uint64_t baseA = insert_zero_bits_p((uint64_t)blockIdx.x << g.LB, g.rowpos, g.q);
    uint64_t baseB = baseA;
    for (int i = 0; i < g.nhh; ++i) {
        const uint64_t ba = (baseA >> g.hh_a[i]) & 1, bb = (baseA >> g.hh_b[i]) & 1;
        if (ba != bb) baseB ^= (1ull << g.hh_a[i]) | (1ull << g.hh_b[i]);
    }
    if (baseB < baseA) return;  // the partner CTA moves this pair
    const bool same = baseA == baseB;
    if (same && g.trivial_in) return;  // nothing in this tile moves

    // Thread t handles the amplitude pairs p = 2t + j * 2 * blockDim: the part of each map that
    // depends on 2t is computed once, the part that depends on j is uniform across the warp.
    const int nloc = g.LB + g.q, T = 1 << nloc;
    const uint32_t step = 2 * blockDim.x, p0 = 2 * threadIdx.x;
    int sbits = 0;
    while ((1u << sbits) < step) ++sbits;
    uint64_t off0 = 0;
    uint32_t ld0 = 0, st0 = 0;
    for (int x = 1; x < sbits && x < nloc; ++x)
        if ((p0 >> x) & 1) {
            off0 += g.lin_off[x];
            ld0 ^= g.lin_sidx[x];
            st0 ^= g.lin_src[x];
        }
    const uint32_t ld1 = g.lin_sidx[0], st1 = g.lin_src[0];  // the odd amplitude of the pair
    for (uint32_t hi = 0; p0 + hi < (uint32_t)T; hi += step) {
        uint64_t offj = 0;
        uint32_t ldj = 0;
        for (int x = sbits; x < nloc; ++x)
            if ((hi >> x) & 1) {
                offj += g.lin_off[x];
                ldj ^= g.lin_sidx[x];
            }
        const uint64_t off = off0 + offj;
        const uint32_t l = ld0 ^ ldj;
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(g.psi + baseA + off));
        sm[l] = make_float2(a.x, a.y);
        sm[l ^ ld1] = make_float2(a.z, a.w);
        if (!same) {
            const float4 b = __ldcs(reinterpret_cast<const float4 *>(g.psi + baseB + off));
            sm[T + l] = make_float2(b.x, b.y);
            sm[T + (l ^ ld1)] = make_float2(b.z, b.w);
        }
    }
    __syncthreads();
    for (uint32_t hi = 0; p0 + hi < (uint32_t)T; hi += step) {
        uint64_t offj = 0;
        uint32_t stj = 0;
        for (int x = sbits; x < nloc; ++x)
            if ((hi >> x) & 1) {
                offj += g.lin_off[x];
                stj ^= g.lin_src[x];
            }
        const uint64_t off = off0 + offj;
        const uint32_t s0 = st0 ^ stj, s1 = s0 ^ st1;
        const float2 x = sm[s0], y = sm[s1];
        if (same) {
            __stcs(reinterpret_cast<float4 *>(g.psi + baseA + off), make_float4(x.x, x.y, y.x, y.y));
        } else {
            const float2 u = sm[T + s0], v = sm[T + s1];
            __stcs(reinterpret_cast<float4 *>(g.psi + baseB + off), make_float4(x.x, x.y, y.x, y.y));
            __stcs(reinterpret_cast<float4 *>(g.psi + baseA + off), make_float4(u.x, u.y, v.x, v.y));
        }
    }
}

__device__ __forceinline__ uint64_t perm_now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Long rows: one CTA a tile (or tile pair), one bulk copy a row of 1 KiB and more into shared memory
// (completion counted in bytes on an mbarrier), the threads swap the pairs (p, sig(p)) the in-tile
// involution exchanges, one bulk store a row back, a pair's tiles to each other's rows.  sig is
// XOR-linear in the local index p: sig(p) = sig(p_thread) ^ sig(p_iter), the second from a per-CTA table.
// launch_involution takes it where it is the faster one; us a pass, this / k_permute_tma: 2^28
// amplitudes in place with 0-3 row bits 606-630 / 660-685, with 4, 5 (rows of 256-512 bytes) 727, 737 /
// 670-690; tile pairs with no row bits, 2^30 1225 / 1322, 2^28 575 / 590; pairs of 2^11 with rows of 1 KiB 687
// / 740, of 2^10 809 / 690, with shorter rows 973-1286 / 690-711.
// A CTA a tile, most of which may only find that nothing moves, and each pays for the trigger of the next
// launch: a swap of the two highest of 28 bits (2^18 CTAs) 497 us with it, 400 without, of 24 bits (2^14)
// 21.9, 17.6, of 22 bits (2^12) 8.7, 8.8; random permutations of 21-22 bits 1-3 % faster with it.
// The only wait (the copies' mbarrier) is bounded by %globaltimer: on a timeout the CTA records the
// failure, writes nothing back and waits (again bounded) for its copies before leaving.
constexpr unsigned kPermEarlyCtas = 4096;
__global__ void __launch_bounds__(256) k_permute_tile_bulk(PermGeom g, int *err)
{
    extern __shared__ __align__(128) float2 tile[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t p_it[64], sig_it[64];  // the iteration part of p, and its image under sig
    __shared__ int ok;
    if (gridDim.x <= kPermEarlyCtas) pdl_launch_next();
    const int nloc = g.LB + g.q, T = 1 << nloc;
    const uint32_t row_bytes = 8u << g.LB;
    const uint64_t base = insert_zero_bits_p((uint64_t)blockIdx.x << g.LB, g.rowpos, g.q);
    uint64_t baseB = base;
    for (int i = 0; i < g.nhh; ++i) {
        const uint64_t ba = (base >> g.hh_a[i]) & 1, bb = (base >> g.hh_b[i]) & 1;
        if (ba != bb) baseB ^= (1ull << g.hh_a[i]) | (1ull << g.hh_b[i]);
    }
    if (baseB < base) return;  // the partner CTA moves this pair
    const bool same = baseB == base;
    if (same && g.trivial_in) return;  // nothing in this tile moves
    const int ntile = same ? 1 : 2;
    const uint32_t sbar = (uint32_t)__cvta_generic_to_shared(&bar);
    const uint32_t stile = (uint32_t)__cvta_generic_to_shared(tile);
    auto sig_of = [&](uint32_t p) {
        uint32_t r = 0;
        for (int x = 0; x < nloc; ++x)
            if ((p >> x) & 1) r |= 1u << g.sig[x];
        return r;
    };
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        pdl_wait();  // this thread issues every access to the state
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(sbar),
                     "r"((uint32_t)(ntile * T) * 8u)
                     : "memory");
        for (int t = 0; t < ntile; ++t)
            for (int r = 0; r < (1 << g.q); ++r)
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        stile + (uint32_t)t * T * 8u + r * row_bytes),
                    "l"(g.psi + (t ? baseB : base) + g.rowoff[r]), "r"(row_bytes), "r"(sbar)
                    : "memory");
    }
    for (int it = threadIdx.x; it < (T >> 8); it += blockDim.x) {
        uint32_t p = 0;
        for (int j = 0; j < nloc - 8; ++j)
            if ((it >> j) & 1) p |= 1u << g.ibit[j];
        p_it[it] = p;
        sig_it[it] = sig_of(p);
    }
    if (threadIdx.x == 0) {
        const uint64_t t0 = perm_now_ns();
        uint32_t done = 0;
        while (!done) {
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0, 20000;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}\n"
                : "=r"(done)
                : "r"(sbar)
                : "memory");
            if (!done && perm_now_ns() - t0 > 4000000000ull) break;
        }
        ok = done;
        if (!done && err) atomicExch(err, 1);
    }
    __syncthreads();
    if (ok) {
        uint32_t p_t = 0;  // blockDim = 256: p = (thread bits deposited) | (iteration bits deposited)
        for (int j = 0; j < 8; ++j)
            if ((threadIdx.x >> j) & 1) p_t |= 1u << g.tbit[j];
        const uint32_t s_t = sig_of(p_t);
        for (int t = 0; t < ntile && !g.trivial_in; ++t) {
            float2 *tt = tile + t * T;
            for (int it = 0; it < (T >> 8); ++it) {
                const uint32_t p = p_t | p_it[it], q = s_t ^ sig_it[it];
                if (p < q) {
                    const float2 a = tt[p], c = tt[q];
                    tt[p] = c;
                    tt[q] = a;
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the bulk stores read the tile
        __syncthreads();
        if (threadIdx.x == 0) {  // a pair's tiles go to each other's rows
            for (int t = 0; t < ntile; ++t)
                for (int r = 0; r < (1 << g.q); ++r)
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(
                                     g.psi + ((t == 0) == same ? base : baseB) + g.rowoff[r]),
                                 "r"(stile + (uint32_t)t * T * 8u + r * row_bytes), "r"(row_bytes)
                                 : "memory");
            asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");  // the tile is read out
        }
    } else if (threadIdx.x == 0) {  // no copy may still be writing the tile when the CTA leaves
        const uint64_t t0 = perm_now_ns();
        uint32_t done = 0;
        while (!done && perm_now_ns() - t0 <= 4000000000ull)
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0, 20000;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}\n"
                : "=r"(done)
                : "r"(sbar)
                : "memory");
    }
}

// The same pass as a pipeline fed by tensor-map (TMA) copies.  A tile's local bits lie apart in the
// address (the low block and up to 5 row bits); a 5-dimensional tensor map whose dimensions begin at
// those bits moves a tile in at most four copies of 2 KiB and more, where one bulk copy a row of 256
// bytes ran into the copy engine's operation rate.  A stage is 2^11 amplitudes: a tile pair (high-high
// transpositions) or, without any, one tile of twice the size.
//  * warp 0, producer: its lanes look at up to 32 tiles at a time (the partner's base, whether anything
//    moves); the tiles that do are loaded into the stage ring, a copy a lane (bytes counted on an mbarrier);
//  * warps 2-9, swappers, two groups of 128 threads, a stage to each in turn: 16 amplitudes a
//    thread, read where the in-tile involution sig puts them from, a barrier among the group, written
//    to their places.  The maps are XOR-linear: a thread part computed once, an iteration part from
//    the parameters;
//  * warp 1, storer: stores the stage (a pair's tiles crosswise) and releases it once read.
// The copies lay a tile out with the 128-byte swizzle (16-byte unit bits ^= local bits 4-6), so lanes
// on two of bits 0-3 and two of the row bits find 16 bank pairs on both sides (choose_lane_bits).
// What bounds it: HBM, 16 bytes an amplitude that moves.  Measured on 2^28 amplitudes, us a pass
// (641 for a whole pass): every low bit with a high one and 9 high pairs 1286 -> 694, 5 low-high pairs
// 737 -> 673, 3 high pairs 587 -> 584; random permutations (two passes) of 2^29 3.2-4.5 -> 2.70-2.93 ms,
// of 2^24 127-141 -> 85-94 us.  The kernel before, one CTA a tile pair and 4 amplitudes a thread, was
// issue-bound (76 %) on setting up its maps.
// Every wait is bounded by %globaltimer, from when the kernels before have ended: on a timeout the
// kernel records the failure, every role leaves, and the CTA waits (again bounded) for its own copies.
constexpr int kPtRing = 98304;                    // bytes of stages (64 KiB: 10-20 % slower); a stage is one tile or a tile pair
constexpr int kPtMaxStages = 16;
constexpr int kPtGroups = 2;                      // swapper groups, a stage to each in turn
constexpr int kPtSwap = 128;                      // threads a group
constexpr int kPtThreads = 64 + kPtGroups * kPtSwap;
constexpr unsigned long long kPtWaitNs = 4000000000ull;

struct PermTma {
    CUtensorMap map;
    int LB, q;
    int rowpos[kMaxRow];
    int nhh, hh_a[20], hh_b[20];
    int trivial_in;
    uint64_t n_tiles;             // candidates: every value of the non-tile bits
    int per;                      // candidates the producer looks at together (<= 32)
    int nloc;                     // local bits of a tile (a pair has one more: which tile)
    int stages;                   // a multiple of kPtGroups: a stage belongs to one group, which sees every
                                  // phase of its barriers in turn (a wait for a parity would otherwise be
                                  // satisfied by the phase before the one before)
    uint32_t stage_bytes;
    int start[5];                 // first address bit of each tensor-map dimension
    uint32_t size_mask[5];
    int nops;                     // copies a tile
    uint32_t op_bytes;
    uint64_t op_off[4];           // address offset of copy i of a tile
    uint32_t tp[7], tq[7];        // stage byte of thread-index bit j, and of its image under sig
    uint32_t ip[16], iq[16];      // the same of iteration i
};

__device__ __forceinline__ bool perm_try(uint32_t bar, uint32_t parity, uint32_t hint_ns)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(hint_ns)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ bool perm_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    if (perm_try(bar, parity, 0)) return true;
    const uint64_t t0 = perm_now_ns();
    for (;;) {
        if (perm_try(bar, parity, 20000)) return true;
        if (*abort_flag || perm_now_ns() - t0 > kPtWaitNs) return false;
    }
}

__device__ __forceinline__ bool perm_bar_and(int id, int n, bool p)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\tsetp.ne.u32 pi, %1, 0;\n\tbar.red.and.pred po, %2, %3, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint32_t perm_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__global__ void __launch_bounds__(kPtThreads, 2) k_permute_tma(const __grid_constant__ PermTma g, int *err)
{
    extern __shared__ uint8_t sm_raw[];
    uint8_t *const sm = sm_raw + ((1024 - (perm_smem(sm_raw) & 1023)) & 1023);  // the swizzle's period
    __shared__ __align__(8) uint64_t full[kPtMaxStages], swapped[kPtMaxStages], empty[kPtMaxStages];
    __shared__ uint64_t dst_a[kPtMaxStages], dst_b[kPtMaxStages];  // where a stage's first and second tile go
    __shared__ int abort_flag, ntile_of[kPtMaxStages];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t S = (uint32_t)g.stages;
    pdl_launch_next();
    if (tid == 0) {
        for (uint32_t i = 0; i < S; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(perm_smem(&full[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(perm_smem(&swapped[i])), "r"(kPtSwap / 32) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(perm_smem(&empty[i])) : "memory");
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    volatile int *ab = &abort_flag;
    auto give_up = [&]() {
        *ab = 1;
        if (err) atomicExch(err, 1);
    };
    const uint32_t stage0 = perm_smem(sm);
    // one copy between a stage and the state, to each lane its own: copy `lane % nops` of tile `lane / nops`
    // (at address offset ta or tb).  Issued by one thread one after the other, the address arithmetic of up
    // to 8 copies took longer than the stage's share of HBM time.
    const int op = lane & (g.nops - 1), op_tile = lane / g.nops;
    const uint32_t tile_bytes = 8u << g.nloc;
    const uint32_t op_at = op_tile * tile_bytes + op * g.op_bytes;
    const uint64_t op_off = g.op_off[op];
    auto copy = [&](bool load, uint32_t at, uint64_t ta, uint64_t tb, uint32_t bar) {
        const uint64_t a = (op_tile ? tb : ta) + op_off;
        const int c0 = (int)(a & g.size_mask[0]), c1 = (int)((a >> g.start[1]) & g.size_mask[1]),
                  c2 = (int)((a >> g.start[2]) & g.size_mask[2]), c3 = (int)((a >> g.start[3]) & g.size_mask[3]),
                  c4 = (int)((a >> g.start[4]) & g.size_mask[4]);
        if (load)
            asm volatile(
                "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
                "%5, %6}], [%7];\n" ::"r"(at + op_at),
                "l"(&g.map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
                : "memory");
        else
            asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];\n" ::"l"(
                             &g.map),
                         "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(at + op_at)
                         : "memory");
    };

    uint32_t issued = 0, marked = 0;  // thread 0: items loaded, end marks behind them
    if (warp == 0) {
        // ---------------- producer ----------------
        // Every role waits for the work before first, each after its own set-up, so that its waits' time
        // limits do not count from an early start.
        pdl_wait();
        uint32_t it = 0;
        bool stop = false;
        for (uint64_t c0 = (uint64_t)blockIdx.x * g.per; c0 < g.n_tiles && !stop; c0 += (uint64_t)gridDim.x * g.per) {
            const uint64_t t = c0 + lane;
            uint64_t a = 0, b = 0;
            bool moves = false;
            if (lane < g.per && t < g.n_tiles) {
                a = insert_zero_bits_p(t << g.LB, g.rowpos, g.q);
                b = a;
                for (int i = 0; i < g.nhh; ++i) {
                    const uint64_t x = ((a >> g.hh_a[i]) ^ (a >> g.hh_b[i])) & 1;
                    b ^= (x << g.hh_a[i]) | (x << g.hh_b[i]);
                }
                moves = b > a || (b == a && !g.trivial_in);  // b < a: the partner's turn moves the pair
            }
            for (uint32_t m = __ballot_sync(0xffffffffu, moves); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const uint64_t ta = __shfl_sync(0xffffffffu, a, src), tb = __shfl_sync(0xffffffffu, b, src);
                const uint32_t st = it % S;
                bool ok = true;
                if (lane == 0 && it >= S) ok = perm_wait(perm_smem(&empty[st]), (it / S - 1) & 1, ab);
                if (!__shfl_sync(0xffffffffu, ok, 0)) {
                    if (lane == 0) give_up();
                    stop = true;
                    break;
                }
                const int nt = ta == tb ? 1 : 2;
                const uint32_t bar = perm_smem(&full[st]);
                if (lane == 0) {
                    dst_a[st] = tb;  // a pair's tiles go to each other's places
                    dst_b[st] = ta;
                    ntile_of[st] = nt;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(nt * tile_bytes)
                                 : "memory");  // before any of the copies can complete
                }
                __syncwarp();
                if (op_tile < nt) copy(true, stage0 + st * g.stage_bytes, ta, tb, bar);
                ++it;
            }
        }
        if (lane == 0) {
            // the end: items of no tiles, one for each swapper group, in order behind the loaded ones
            uint32_t marks = 0;
            for (; !stop && marks < (uint32_t)kPtGroups; ++marks) {
                const uint32_t e = it + marks;
                if (e >= S && !perm_wait(perm_smem(&empty[e % S]), (e / S - 1) & 1, ab)) break;
                ntile_of[e % S] = 0;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(perm_smem(&full[e % S])) : "memory");
            }
            if (marks < (uint32_t)kPtGroups) give_up();
            issued = it;
            marked = marks;
        }
    } else if (warp == 1) {
        // ---------------- storer ----------------
        pdl_wait();
        uint32_t it = 0;
        for (;; ++it) {
            const uint32_t st = it % S;
            bool ok = perm_wait(perm_smem(&full[st]), (it / S) & 1, ab);
            const int nt = ok ? ntile_of[st] : 0;
            if (ok && nt && !g.trivial_in) ok = perm_wait(perm_smem(&swapped[st]), (it / S) & 1, ab);
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) give_up();
                break;
            }
            if (nt == 0) break;
            if (op_tile < nt) copy(false, stage0 + st * g.stage_bytes, dst_a[st], dst_b[st], 0);
            asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
            if (it > 0) {  // every lane's copies of the stage before this one have been read out
                asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(perm_smem(&empty[(it - 1) % S]))
                                 : "memory");
            }
        }
        asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
        __syncwarp();
        if (lane == 0 && it > 0)  // the producer's end mark may wait for this stage
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(perm_smem(&empty[(it - 1) % S])) : "memory");
    } else if (!g.trivial_in) {
        // ---------------- swappers ----------------
        const int w = (tid - 64) & (kPtSwap - 1), grp = (tid - 64) / kPtSwap;
        uint32_t pt = 0, qt = 0;
#pragma unroll
        for (int j = 0; j < 7; ++j)
            if ((w >> j) & 1) {
                pt ^= g.tp[j];
                qt ^= g.tq[j];
            }
        pdl_wait();
        // a group takes the items congruent to its number, the last of them an end mark
        for (uint32_t it = grp;; it += kPtGroups) {
            const uint32_t st = it % S;
            const bool ok = perm_wait(perm_smem(&full[st]), (it / S) & 1, ab);
            if (!perm_bar_and(1 + grp, kPtSwap, ok)) {  // all leave together: the barrier below counts them
                give_up();
                break;
            }
            const int nt = ntile_of[st];
            if (nt == 0) break;
            uint8_t *sb = sm + st * g.stage_bytes;
            const int n = (nt << g.nloc) / kPtSwap;
            float2 v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < n) v[i] = *reinterpret_cast<const float2 *>(sb + (qt ^ g.iq[i]));
            asm volatile("bar.sync %0, 128;\n" ::"r"(1 + grp) : "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < n) *reinterpret_cast<float2 *>(sb + (pt ^ g.ip[i])) = v[i];
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the store reads the stage
            __syncwarp();
            if ((tid & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(perm_smem(&swapped[st])) : "memory");
        }
    }
    // No copy may still be writing a stage when the CTA leaves.  The storer has waited for every one, unless
    // a role gave up: then those whose barriers have not moved on (by later copies or end marks, which
    // waited until the older items were stored) are waited for here, after the last role.
    __syncthreads();
    if (tid == 0 && *ab)
        for (uint32_t j = issued + marked > S ? issued + marked - S : 0; j < issued; ++j) {
            const uint64_t t0 = perm_now_ns();
            while (!perm_try(perm_smem(&full[j % S]), (j / S) & 1, 20000) && perm_now_ns() - t0 <= kPtWaitNs) {
            }
        }
}

// One involution pass; inv[b] = partner of bit b (inv[b] == b: fixed).
// Geometry of one involution pass for tiles of at least 2^min_tile amplitudes.
int build_geom(float2 *psi, int nbits, const int *inv, int min_tile, PermGeom &g)
{
    // low block: smallest LB >= min(5, nbits) with LB + q >= min(min_tile, nbits)
    int LB = std::min(5, nbits), q = 0;
    for (;; LB++) {
        q = 0;
        for (int b = 0; b < LB; b++)
            if (inv[b] >= LB) q++;
        if (LB + q >= std::min(min_tile, nbits) || LB == nbits) break;
    }
    if (q > kMaxRow) return -2;

    g = PermGeom{};
    g.psi = psi;
    g.LB = LB;
    g.q = q;
    std::vector<std::pair<int, int>> rows;  // (global high bit, low partner)
    for (int b = 0; b < LB; b++)
        if (inv[b] >= LB) rows.push_back({inv[b], b});
    std::sort(rows.begin(), rows.end());
    for (int i = 0; i < q; i++) g.rowpos[i] = rows[i].first;
    for (int x = 0; x < 16; x++) g.sig[x] = x;
    g.trivial_in = 1;
    for (int b = 0; b < LB; b++) {
        if (inv[b] == b) continue;
        g.trivial_in = 0;
        if (inv[b] < LB) {
            g.sig[b] = inv[b];
        } else {
            int i = 0;
            while (rows[i].first != inv[b]) i++;
            g.sig[b] = LB + i;
            g.sig[LB + i] = b;
        }
    }
    g.nhh = 0;
    for (int b = LB; b < nbits; b++)
        if (inv[b] > b) {
            bool row = false;
            for (int i = 0; i < q; i++) row |= g.rowpos[i] == b || g.rowpos[i] == inv[b];
            if (!row) {
                g.hh_a[g.nhh] = b;
                g.hh_b[g.nhh] = inv[b];
                g.nhh++;
            }
        }
    for (int r = 0; r < (1 << q); r++) {
        uint64_t o = 0;
        uint32_t f = 0;
        for (int i = 0; i < q; i++)
            if ((r >> i) & 1) {
                o += 1ull << g.rowpos[i];
                f ^= 1u << rows[i].second;  // row bit i lands on bank bit of its low partner
            }
        g.rowoff[r] = o;
        g.fsw[r] = f & ((1u << LB) - 1);
    }
    // values of the XOR-linear in-tile maps on each single local bit
    const int nloc = LB + q;
    auto sidx_h = [&](uint32_t p) {
        const uint32_t r = p >> LB;
        return (r << LB) | ((p & ((1u << LB) - 1)) ^ g.fsw[r]);
    };
    for (int x = 0; x < nloc; x++) {
        const uint32_t p = 1u << x;
        g.lin_off[x] = x < LB ? (uint64_t)p : g.rowoff[p >> LB];
        g.lin_sidx[x] = sidx_h(p);
        g.lin_src[x] = sidx_h(1u << g.sig[x]);  // the amplitude landing at p came from slot sig(p)
    }
    return 0;
}

// ---- the tensor-map pass: geometry, tensor map, launch ----

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled()
{
    static const EncodeTiled fn = [] {  // the driver's entry: the library itself links only the runtime
        void *p = nullptr;
        cudaDriverEntryPointQueryResult st;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &st) != cudaSuccess ||
            st != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiled>(p);
    }();
    return fn;
}

// Bank pair (0-15, a vector of 4 bits) of local bit x in the swizzled stage: bit 0 as it is, bits 1-3
// the 16-byte unit, which local bits 4-6 are XORed into.
uint32_t bank_of(int x) { return x < 4 ? 1u << x : (x < 7 ? 1u << (x - 3) : 0u); }
uint32_t stage_byte(uint32_t p) { return 8 * p ^ (((p >> 4) & 7u) << 4); }

// Thread-index and iteration bits of the swappers over nl local bits with in-tile involution sig: the
// four bits of a half-warp's lanes are taken so that the ranks of their bank pairs, at p and at
// sig(p), are as large as can be (4 and 4: no conflicts), then the remaining bits ascending.
void swap_bits(PermTma &g, const int *sig, int nl)
{
    // the span of a set of bank vectors as a mask of 16 bits (bit v: v is in it)
    auto grown = [](uint32_t span, uint32_t v) {
        uint32_t x = span;
        if (v & 1) x = ((x & 0x5555u) << 1) | ((x >> 1) & 0x5555u);
        if (v & 2) x = ((x & 0x3333u) << 2) | ((x >> 2) & 0x3333u);
        if (v & 4) x = ((x & 0x0f0fu) << 4) | ((x >> 4) & 0x0f0fu);
        if (v & 8) x = ((x & 0x00ffu) << 8) | ((x >> 8) & 0x00ffu);
        return span | x;
    };
    const int nsel = std::min(nl, 11);
    int order[16], no = 4, pick[4], best = -1;
    // depth first, both ranks growing at every step; the best partial choice is completed greedily
    auto search = [&](auto &&self, int depth, uint32_t sp, uint32_t sq, int from) -> bool {
        if (depth > best) {
            best = depth;
            uint32_t p = sp, q = sq;
            std::copy(pick, pick + depth, order);
            for (int d = depth; d < 4; d++) {
                int bx = -1, bg = -1;
                for (int x = 0; x < nsel; x++) {
                    if (std::find(order, order + d, x) != order + d) continue;
                    const int gn = !((p >> bank_of(x)) & 1) + !((q >> bank_of(sig[x])) & 1);
                    if (gn > bg) bg = gn, bx = x;
                }
                order[d] = bx;
                p = grown(p, bank_of(bx));
                q = grown(q, bank_of(sig[bx]));
            }
        }
        if (depth == 4) return true;
        for (int x = from; x < nsel; x++) {
            const uint32_t vp = bank_of(x), vq = bank_of(sig[x]);
            if (((sp >> vp) & 1) || ((sq >> vq) & 1)) continue;
            pick[depth] = x;
            if (self(self, depth + 1, grown(sp, vp), grown(sq, vq), x + 1)) return true;
        }
        return false;
    };
    search(search, 0, 1u, 1u, 0);
    bool used[16] = {};
    for (int j = 0; j < 4; j++) used[order[j]] = true;
    for (int x = 0; x < nl; x++)
        if (!used[x]) order[no++] = x;  // a pair's tile bit, the highest, comes last
    for (int j = 0; j < 7; j++) {
        g.tp[j] = stage_byte(1u << order[j]);
        g.tq[j] = stage_byte(1u << sig[order[j]]);
    }
    for (int i = 0; i < 16; i++) {
        g.ip[i] = g.iq[i] = 0;
        for (int b = 0; 7 + b < nl; b++)
            if ((i >> b) & 1) {
                g.ip[i] ^= stage_byte(1u << order[7 + b]);
                g.iq[i] ^= stage_byte(1u << sig[order[7 + b]]);
            }
    }
}

// Everything but the encoded map; false if the involution has no such geometry.
bool permute_tma_geom(int nbits, const int *inv, PermTma &g, cuuint32_t *box, cuuint64_t *dim, cuuint64_t *stride)
{
    if (nbits < 11 || nbits > 35) return false;
    // the widest low block whose tile (2^11 amplitudes; 2^10 where tiles swap in pairs) fits a stage
    for (int LB = 5; LB <= 11; LB++) {
        int row[kMaxRow], q = 0, pairs = 0;
        for (int b = 0; b < LB && q <= 5; b++)
            if (inv[b] >= LB) row[q < kMaxRow ? q : 0] = inv[b], q++;
        if (q > 5) continue;
        std::sort(row, row + q);
        int hh_a[20], hh_b[20];
        for (int b = LB; b < nbits; b++)
            if (inv[b] > b) {
                bool is_row = false;
                for (int i = 0; i < q; i++) is_row |= row[i] == b || row[i] == inv[b];
                if (is_row) continue;
                if (pairs == 20) return false;
                hh_a[pairs] = b;
                hh_b[pairs++] = inv[b];
            }
        if (LB + q > (pairs ? 10 : 11)) continue;
        g.LB = LB;
        g.q = q;
        g.nhh = pairs;
        std::copy(row, row + q, g.rowpos);
        std::copy(hh_a, hh_a + pairs, g.hh_a);
        std::copy(hh_b, hh_b + pairs, g.hh_b);
    }
    if (g.LB == 0) return false;
    const int LB = g.LB, q = g.q;
    g.nloc = LB + q;
    if (g.nloc < 9) return false;
    g.stage_bytes = 8u << (g.nloc + (g.nhh ? 1 : 0));
    g.stages = std::min<int>(kPtMaxStages, kPtRing / g.stage_bytes) / kPtGroups * kPtGroups;
    g.n_tiles = 1ull << (nbits - g.nloc);
    // the involution on local bits: low bits, row bits, and (a pair) which tile
    int sig[16];
    g.trivial_in = 1;
    for (int x = 0; x < 16; x++) sig[x] = x;
    for (int b = 0; b < LB; b++) {
        if (inv[b] == b) continue;
        g.trivial_in = 0;
        if (inv[b] < LB) {
            sig[b] = inv[b];
        } else {
            int i = 0;
            while (g.rowpos[i] != inv[b]) i++;
            sig[b] = LB + i;
            sig[LB + i] = b;
        }
    }
    swap_bits(g, sig, g.nloc + (g.nhh ? 1 : 0));
    // tensor-map dimensions: bits 0-3 (128 bytes, the swizzle's rows), then one from each tile bit that
    // does not continue the dimension before it; tile bits beyond the fifth dimension are looped over
    int tile_bit[16], nt = 0;
    for (int b = 4; b < LB; b++) tile_bit[nt++] = b;
    for (int i = 0; i < q; i++) tile_bit[nt++] = g.rowpos[i];
    for (int d = 0; d < 5; d++) box[d] = d ? 1 : 16;
    int nd = 1, i = 0;
    for (; i < nt; i++) {
        if (nd > 1 && tile_bit[i] == tile_bit[i - 1] + 1) {
            box[nd - 1] *= 2;
            continue;
        }
        if (nd == 5) break;
        g.start[nd] = tile_bit[i];
        box[nd++] = 2;
    }
    const int looped = nt - i;
    if (looped > 2) return false;
    g.nops = 1 << looped;
    g.op_bytes = (8u << g.nloc) >> looped;
    for (int o = 0; o < g.nops; o++)
        for (int b = 0; b < looped; b++)
            if ((o >> b) & 1) g.op_off[o] += 1ull << tile_bit[i + b];
    for (int d = 0; d < 5; d++) {
        const int lo = d < nd ? g.start[d] : nbits, hi = d + 1 < nd ? g.start[d + 1] : nbits;
        if (hi - lo > 31) return false;
        dim[d] = 1ull << (hi - lo);
        g.start[d] = d < nd ? lo : 0;
        g.size_mask[d] = d < nd ? (uint32_t)(dim[d] - 1) : 0;
        if (d > 0) stride[d - 1] = 8ull << lo;
    }
    return true;
}

// The pass as tensor-map copies: 0 launched, 1 not a geometry for it, < 0 an error.
int launch_permute_tma(float2 *psi, int nbits, const int *inv, cudaStream_t st, int *err)
{
    PermTma g{};
    cuuint32_t box[5];
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    cuuint64_t dim[5], stride[4];
    if (((uintptr_t)psi & 15) != 0 || !encode_tiled() || !permute_tma_geom(nbits, inv, g, box, dim, stride)) return 1;
    if (encode_tiled()(&g.map, CU_TENSOR_MAP_DATA_TYPE_INT64, 5, psi, dim, stride, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return 1;
    constexpr int smem = kPtRing + 1024;
    static std::atomic<uint64_t> smem_done{0};
    if (!smem_opt_in(k_permute_tma, smem, smem_done)) return -1;
    static const LaunchCfg cfg = [] {
        LaunchCfg c;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return c;
        if (cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return c;
        c.ok = true;
        return c;
    }();
    if (!cfg.ok) return -1;
    // odd: which tiles lead a pair follows their address bits, and with 304 CTAs, a multiple of 16, the
    // low 4 bits of a CTA's turns would never change (a swap of bits 12 and 18 left half the CTAs idle)
    const uint64_t ctas = 2 * (uint64_t)cfg.sms - 1;
    // candidates a producer takes at a time: many, since evaluating them costs its warp the same for 1
    // and for 32, but at least 16 turns a CTA, so that the last one is not half empty (2^24 amplitudes:
    // 127-141 us two random passes with 32 at a time, 94-110 with 4)
    g.per = 32;
    while (g.per > 1 && g.n_tiles / g.per < 16 * ctas) g.per >>= 1;
    if (g.nhh == 0) g.per = std::min(g.per, 4);  // no pairs: little to evaluate, neighbours together
    const uint64_t grid = std::min<uint64_t>(ctas, (g.n_tiles + g.per - 1) / g.per);
    return launch_pdl(k_permute_tma, (unsigned)grid, kPtThreads, smem, st, g, err) == cudaSuccess ? 0 : -1;
}

// Bits of the local index the 32 lanes of a warp run over in k_permute_tile_bulk: a warp reads
// and writes both p and sig(p); with 8-byte elements the bank pair is bits 0-3 of the index, so a
// set of lane bits costs max(2, 32 >> |bits in 0-3|) wavefronts for p, the same for sig(p).  The
// cheapest 5-subset of the bits 0-4 and their images under sig is taken (ties: the lowest), then
// three more bits for the warps and the rest for the iterations, ascending.
void choose_lane_bits(PermGeom &g)
{
    const int nloc = g.LB + g.q;
    int cand[16], nc = 0;
    bool in[16] = {};
    for (int x = 0; x < 5 && x < nloc; x++) {
        for (int y : {x, g.sig[x]})
            if (!in[y]) in[y] = true, cand[nc++] = y;
    }
    std::sort(cand, cand + nc);
    auto wf = [](int low) { return std::max(2, 32 >> low); };
    int best_cost = 1 << 30;
    uint32_t best = 0;
    for (uint32_t m = 0; m < (1u << nc); m++) {
        if (__builtin_popcount(m) != 5) continue;
        int lp = 0, ls = 0;
        for (int i = 0; i < nc; i++)
            if ((m >> i) & 1) {
                lp += cand[i] < 4;
                ls += g.sig[cand[i]] < 4;
            }
        const int cost = wf(lp) + wf(ls);
        if (cost < best_cost) best_cost = cost, best = m;
    }
    bool used[16] = {};
    int j = 0;
    for (int i = 0; i < nc; i++)
        if ((best >> i) & 1) g.tbit[j++] = (int8_t)cand[i], used[cand[i]] = true;
    for (int x = 0; x < nloc && j < 8; x++)
        if (!used[x]) g.tbit[j++] = (int8_t)x, used[x] = true;
    int k = 0;
    for (int x = 0; x < nloc; x++)
        if (!used[x]) g.ibit[k++] = (int8_t)x;
}

int launch_involution(float2 *psi, int nbits, const int *inv, cudaStream_t st, int *err)
{
    bool any = false;
    for (int b = 0; b < nbits; b++) any |= inv[b] != b;
    if (!any) return 0;
    PermGeom g;
    const int rc = build_geom(psi, nbits, inv, SYCSIM_PERM_TILE, g);
    if (rc == 0 && g.nhh == 0) {  // tiles that only permute in place gain from more work per CTA
        PermGeom big;
        if (build_geom(psi, nbits, inv, SYCSIM_PERM_TILE_SAME, big) == 0) g = big;
    }
    // long rows (see k_permute_tile_bulk): in place with at most 3 row bits, pairs without row bits, pairs
    // of 2^11 amplitudes whose rows are 1 KiB and more
    const bool bulk = g.nhh == 0 ? g.q <= 3 : (g.q == 0 || (g.LB + g.q == 11 && g.LB >= 7));
    if (rc == 0 && bulk && g.LB >= 5 && g.LB + g.q >= 8 && g.LB + g.q <= (g.nhh ? 11 : 12) && ((uintptr_t)psi & 15) == 0) {
        const uint64_t tiles = 1ull << (nbits - g.LB - g.q);
        choose_lane_bits(g);
        return launch_pdl(k_permute_tile_bulk, (unsigned)tiles, 256,
                          (g.nhh ? 2 : 1) * (sizeof(float2) << (g.LB + g.q)), st, g, err) == cudaSuccess
                   ? 0
                   : -1;
    }
    const int tma = launch_permute_tma(psi, nbits, inv, st, err);
    if (tma <= 0) return tma;
    if (rc != 0) return rc;
    const int LB = g.LB, q = g.q;
    const uint64_t tiles = 1ull << (nbits - LB - q);
    const size_t smem = (g.nhh ? 2 : 1) * sizeof(float2) << (LB + q);  // a tile pair, or one tile
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(k_permute_pass, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
        return -1;
    const int threads = std::min(256, 1 << (LB + q));
    return launch_pdl(k_permute_pass, (unsigned)tiles, threads, smem, st, g) == cudaSuccess ? 0 : -1;
}

}  // namespace

// Amplitudes an involution moves: those whose bits differ across at least one transposition.
static double moved_fraction(int nbits, const int *inv)
{
    int pairs = 0;
    for (int b = 0; b < nbits; b++) pairs += inv[b] > b;
    return 1.0 - std::ldexp(1.0, -pairs);
}

int launch_permute(sim_t *h, float2 *psi, int nbits, const int *perm, cudaStream_t st)
{
    // split pi into cycles; sigma1 = reflection x -> -x, sigma2 = reflection x -> 1 - x
    int s1[kMaxQubits], s2[kMaxQubits];
    bool seen[kMaxQubits] = {};
    for (int b = 0; b < nbits; b++) s1[b] = s2[b] = b;
    for (int b = 0; b < nbits; b++) {
        if (seen[b]) continue;
        std::vector<int> cyc;
        for (int x = b; !seen[x]; x = perm[x]) {
            seen[x] = true;
            cyc.push_back(x);
        }
        const int L = (int)cyc.size();
        for (int x = 0; x < L; x++) {
            s1[cyc[x]] = cyc[(L - x) % L];
            s2[cyc[x]] = cyc[(L + 1 - x) % L];
        }
    }
    const double amps = std::ldexp(1.0, nbits);
    int rc = 0;
    for (const int *inv : {s1, s2}) {
        const double frac = moved_fraction(nbits, inv);
        if (frac == 0.0) continue;
        const int ps = h ? prof_begin(h, SIM_PROF_PERMUTE, 16.0 * amps * frac, st) : -1;
        rc = launch_involution(psi, nbits, inv, st, h ? h->d_errflag : nullptr);
        if (h) prof_end(h, ps, st);
        if (rc != 0) return rc;
    }
    return 0;
}

}  // namespace sycsim

using namespace sycsim;

extern "C" int sim_permute(sim_t *h, const int *perm)
{
    if (!h) return fail(nullptr, SIM_E_INVAL, "sim_permute: NULL handle");
    state_written(h);
    if (!perm) return fail(h, SIM_E_INVAL, "sim_permute: NULL perm");
    if (h->store != SIM_STORE_DEVICE)
        return fail(h, SIM_E_UNSUPPORTED, "sim_permute: the host store's layout is fixed by its sliced sets");
    bool used[kMaxQubits] = {};
    for (int q = 0; q < h->n; q++) {
        if (perm[q] < 0 || perm[q] >= h->n || used[perm[q]])
            return fail(h, SIM_E_INVAL, "sim_permute: perm is not a bijection on 0..%d", h->n - 1);
        used[perm[q]] = true;
    }
    // physical permutation: old bit bit_of[q] -> new bit perm[q]
    int phys[kMaxQubits];
    for (int q = 0; q < h->n; q++) phys[h->bit_of[q]] = perm[q];
    SIM_DEVICE_SCOPE(h, h->device);
    int rc = launch_permute(h, h->d_state, h->n, phys, h->stream);
    if (rc != 0)
        return fail(h, SIM_E_CUDA, "sim_permute: launch failed (%d): %s", rc,
                    cudaGetErrorString(cudaGetLastError()));
    for (int q = 0; q < h->n; q++) {
        h->bit_of[q] = perm[q];
        h->qubit_at[perm[q]] = q;
    }
    return SIM_OK;
}

extern "C" int sim_set_layout(sim_t *h, const int *perm)
{
    if (!h) return fail(nullptr, SIM_E_INVAL, "sim_set_layout: NULL handle");
    state_written(h);
    if (!perm) return fail(h, SIM_E_INVAL, "sim_set_layout: NULL perm");
    bool used[kMaxQubits] = {};
    for (int q = 0; q < h->n; q++) {
        if (perm[q] < 0 || perm[q] >= h->n || used[perm[q]])
            return fail(h, SIM_E_INVAL, "sim_set_layout: perm is not a bijection on 0..%d", h->n - 1);
        used[perm[q]] = true;
    }
    if (h->store == SIM_STORE_HOST) {
        if (!host_store_relabel(h, perm))
            return fail(h, SIM_E_INVAL, "sim_set_layout: a host store keeps sets A and B on their bits");
        return SIM_OK;
    }
    for (int q = 0; q < h->n; q++) {
        h->bit_of[q] = perm[q];
        h->qubit_at[perm[q]] = q;
    }
    return SIM_OK;
}
