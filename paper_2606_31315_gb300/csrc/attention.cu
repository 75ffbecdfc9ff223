// Block attention for the verify (causal-within-block) and drafter (bidirectional-
// within-block) passes of block-diffusion speculative decoding (Section 2.1,
// Figure 1 of the BlockPilot paper).
//
// bf16 tensor-core path (sm_103a):
//   * One work unit = (sequence, KV head, 128-row query tile).  The B_s block
//     queries of the g = Hq/Hkv query heads that share a KV head are packed as the
//     rows of one M=128 tile (row r = i*g + j: block position i, head j of the
//     group), so QK^T and PV are M=128 tcgen05 MMAs that read each K/V tile once.
//   * A thread-block cluster of CS CTAs splits the unit's keys; each CTA streams its
//     share of 128-key K/V tiles through a 3-stage TMA ring (SWIZZLE_128B), computes
//     S = Q K^T into tensor memory, runs an online softmax (fp32, exp2 domain, lazy
//     rescale of the TMEM accumulator when the row max grows by more than 2^8),
//     writes P (bf16) back into tensor memory (three S/P buffers) and accumulates O += P V
//     with P as the TMEM A operand.  The partial results are merged by the CTAs that own the rows:
//     every CTA scales its rows and pushes them to their owners through distributed shared memory,
//     or, where a CTA owns few rows (wide clusters) and the workspace has the room, leaves them as
//     they are in its own slot there, and the owner loads and weighs them.
//   * The flat split (below) cuts the tiles of all units evenly over the CTAs instead, or deals the
//     units out; a second kernel merges the units that were cut.
//   * Units are issued longest-first so that ragged batches finish together.
//   Warp roles: warp 0 = TMA producer + TMEM allocator, warp 1 = MMA issuer,
//   warps 2..5 = softmax / epilogue (one query row per thread, TMEM lane = row).  Units of at
//   most 64 rows (a block of up to 64/g positions) use the spread layout instead: the rows fill
//   16 lanes of each TMEM sub-partition and each half-warp takes one 64-key half of a row, so
//   all four softmax warps share the exp2 work.
//
// fp32 path (CUDA cores): register-tiled online softmax, keys split over a thread-block cluster; contexts of a few
// keys: a warp per row.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "ptx_sm103.cuh"

namespace cg = cooperative_groups;

namespace bp {
namespace {

constexpr int kD = 128;       // head_dim of the tensor-core path
constexpr int kTileN = 128;   // keys per K/V tile
constexpr int kM = 128;       // query rows per tile
constexpr int kStages = 3;    // K/V ring depth
constexpr int kHalf = kTileN * 64 * 2;          // one 64-column SW128 half of a 128-row tile: 16 KB
constexpr int kQBytes = kM * kD * 2;            // 32 KB
constexpr int kKVBytes = kTileN * kD * 2;       // 32 KB for K, 32 KB for V
constexpr int kStageBytes = 2 * kKVBytes;       // 64 KB
constexpr int kDynSmem = kQBytes + kStages * kStageBytes + 1024;
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 512;
static_assert(kDynSmem >= tmem_smem_share((int)kTmemCols, 228 * 1024), "leaves no other CTA's tensor memory room");
constexpr uint32_t kColO = 384;
constexpr int kMaxOrderedSeqs = 256;  // longest-first ordering for batches up to this size
constexpr int kMaxDealtSeqs = 64;     // flat split: batches whose units may be dealt out instead of cut evenly
constexpr int kMaxCluster = 16;

struct AttnParams {
    const __nv_bfloat16* q;
    __nv_bfloat16* o;
    float* lse;
    const int32_t* cu_q;
    const int32_t* cu_kv;
    int num_seqs, num_q_heads, num_kv_heads, group, m_tiles;
    int total_q, total_kv;
    int causal;
    float scale_log2;  // softmax scale * log2(e)
    int q_tma;         // Q tile loaded by TMA (group divides 128)
    // paged KV cache: sequence s's key j lives in page block_table[s * pages_per_seq + (j >> page_shift)]
    // at row j & (page size - 1); NULL block_table = contiguous K/V rows from cu_kv[s]
    const int32_t* block_table;
    int pages_per_seq, page_shift;
    // flat split: partial (O, m, l) slots in the workspace, two per CTA, slot_rows rows each; and one
    // work entry (two int4) per CTA for the merge: (first tile, end tile, all tiles, rows) and (first
    // query row, query tile, parts) of the cut unit whose first tile the CTA holds, or first tile -1; parts > 0:
    // the unit lies in the first slots of that many CTA groups from this one on
    float* part;
    int4* work;
    int slot_rows;
    float us_whole, us_part, us_cut;  // flat split: us per key tile of whole units, of parts, with every SM streaming
    int sm_count, ahead_ok;  // flat split: may K's ring refill ahead of V's (pages of at least 32 keys)
    int early_release;  // the grid is one wave of short runs: dependents may launch as soon as every CTA has started
    unsigned int* err;
};
constexpr int kMaxSub = kTileN / 16;  // sub-boxes per K/V tile at the smallest page size (16 keys)

__device__ __forceinline__ uint32_t col_s(int st) { return (uint32_t)st * 128u; }  // TMEM column of stage st's S (then P)

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ int cdiv(int a, int b) { return (a + b - 1) / b; }

// One stretch of consecutive 128-key tiles of one work unit (sequence s, KV head h, 128-row query
// tile mt), processed by one CTA.
struct Seg {
    int s, h, mt;
    int q0, B, kv0, n;  // the sequence's first query row, block size, first key row, key count
    int jt0, nt;        // first tile of the stretch within the unit, tiles in it
    int whole;          // flat split: the stretch is the whole unit (the CTA writes the output)
    int slot;           // flat split, part of a unit: the CTA's partial slot (0 first stretch, 1 last)
    int parts;          // flat split, units dealt out: the parts the unit is cut into (0: cut evenly with the others)
};

// Flat split: key tiles of every sequence over its 128-row query tiles, counted once for all KV heads
// (a group of CTAs, one per KV head, streams the same tiles of every head at the same time); a
// sequence without block rows has none.
__device__ __forceinline__ int flat_seq_tiles(int B, int n, int G) {
    return B > 0 ? cdiv(B * G, kM) * cdiv(n, kTileN) : 0;
}

// Flat split: the prefix sums of the sequences' tile counts into pre[0..S] (S <= kMaxOrderedSeqs), by the whole CTA:
// every thread loads its own sequences' offsets (one round trip), then one warp's lanes sum 8 consecutive counts and
// scan the lane sums.
__device__ __forceinline__ void flat_prefix(const AttnParams& p, int32_t* pre, int tid) {
    constexpr int kPer = kMaxOrderedSeqs / 32;
    static_assert(kPer * 32 == kMaxOrderedSeqs, "whole lanes");
    for (int s = tid; s < p.num_seqs; s += kThreads) {
        const int B = __ldg(p.cu_q + s + 1) - __ldg(p.cu_q + s);
        const int n = __ldg(p.cu_kv + s + 1) - __ldg(p.cu_kv + s);
        pre[s + 1] = flat_seq_tiles(B, n, p.group);
    }
    __syncthreads();
    if (tid < 32) {
        int loc[kPer];
        int run = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int s = tid * kPer + k;
            if (s < p.num_seqs) run += pre[s + 1];
            loc[k] = run;
        }
        int incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (tid >= o) incl += y;
        }
        const int excl = incl - run;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int s = tid * kPer + k;
            if (s < p.num_seqs) pre[s + 1] = excl + loc[k];
        }
        if (tid == 0) pre[0] = 0;
    }
    __syncthreads();
}

// Flat split: the stretch that starts at global tile t of a CTA (KV head h) whose range ends at t_end
// (pre: the sequences' tile prefix sums; a single sequence needs none).  first: the CTA's first stretch.
__device__ __forceinline__ Seg flat_seg(const AttnParams& p, const int32_t* pre, int t, int t_end, int h, bool first) {
    Seg g;
    int s = 0;
    if (p.num_seqs > 1) {  // the last sequence whose tiles start at or before t
        int lo = 0, hi = p.num_seqs;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pre[mid] <= t) lo = mid; else hi = mid;
        }
        s = lo;
    }
    const int base = p.num_seqs > 1 ? pre[s] : 0;
    g.s = s;
    g.q0 = p.num_seqs == 1 ? 0 : __ldg(p.cu_q + s);
    g.B = p.num_seqs == 1 ? p.total_q : __ldg(p.cu_q + s + 1) - g.q0;
    g.kv0 = p.num_seqs == 1 ? 0 : __ldg(p.cu_kv + s);
    g.n = p.num_seqs == 1 ? p.total_kv : __ldg(p.cu_kv + s + 1) - g.kv0;
    const int ntu = cdiv(g.n, kTileN);
    const int local = t - base;
    g.mt = local / ntu;
    g.jt0 = local - g.mt * ntu;
    g.h = h;
    g.nt = min(ntu - g.jt0, t_end - t);
    g.whole = g.jt0 == 0 && g.nt == ntu;
    g.slot = first ? 0 : 1;
    g.parts = 0;
    return g;
}

// Flat split, units dealt out: the parts of a unit of L tiles where c groups of CTAs are free for each (the cluster
// split's rule: a merge costs about three tiles of one CTA's chain).
__device__ __forceinline__ int dealt_parts(int L, int c) { return L - cdiv(L, c) >= 3 ? min(c, L) : 1; }

// Flat split, units dealt out: the rank (longest first) of the t-th unit of CTA group grp of ng, S sequences: c = ng / S
// groups a unit, or rounds there and back over the groups.
__device__ __forceinline__ int dealt_rank(int t, int grp, int ng, int c) {
    return c >= 1 ? grp / c : t * ng + ((t & 1) ? ng - 1 - grp : grp);
}

// ... and its stretch (order: the sequences by rank).
__device__ __forceinline__ Seg dealt_seg(const AttnParams& p, const uint8_t* order, int t, int grp, int ng, int c, int h) {
    Seg g;
    g.s = order[dealt_rank(t, grp, ng, c)];
    g.q0 = __ldg(p.cu_q + g.s);
    g.B = __ldg(p.cu_q + g.s + 1) - g.q0;
    g.kv0 = __ldg(p.cu_kv + g.s);
    g.n = __ldg(p.cu_kv + g.s + 1) - g.kv0;
    g.h = h;
    g.mt = 0;
    const int L = cdiv(g.n, kTileN);
    g.parts = c >= 1 ? dealt_parts(L, c) : 1;
    const int part = c >= 1 ? grp - grp / c * c : 0;
    g.jt0 = part * L / g.parts;
    g.nt = (part + 1) * L / g.parts - g.jt0;
    g.whole = g.parts == 1;
    g.slot = 0;
    return g;
}

// PAGED: K/V rows come from pages named by p.block_table (the contiguous instantiation carries no
// paging code at all).
// SPREAD (units of at most 64 query rows, group size dividing 16): logical row r sits at TMEM lane
// (r / 16) * 32 + r % 16, so the 64 rows fill 16 lanes of each of the four TMEM sub-partitions and
// all four softmax warps (and their SMSPs' exp2 units) work; the two half-warps take the two
// 64-column halves of a row (tcgen05 16x32bx2 accesses), combining row statistics by shuffle.
// FLAT: the flat split.  The key tiles of all units, in order, are cut into gridDim.x equal ranges,
// one per CTA (no clusters); a CTA works through the stretches of its range one after another with
// one pipeline (K/V ring, S/P buffers, O accumulator) and writes a unit it covers whole straight
// to the output, a partial stretch to its workspace slot for attn_combine_kernel.  FLAT == 2: where the lengths turn
// out even (the host knows only a bound and their sum), the CTAs deal the units out instead, longest first, whole
// or in equal parts.  Otherwise the cluster split: a unit per cluster, its tiles cut into CS ranges, partials merged
// through distributed shared memory or the workspace.
// AHEAD (cluster split; FLAT == 2 where every CTA has one stretch): K and V are separate rings.  K's stage is free after Q K^T, a softmax and a P V before
// V's, and refills then, V a tile behind (the order in which the stages come free); with the rings joined both
// wait for the tile's P V and only one of the three stages is in flight.  Where the line lies:
// launch_attention_bf16.
template <bool PAGED, bool SPREAD, int FLAT, bool AHEAD>
__global__ void __launch_bounds__(kThreads, 1)
    attn_bf16_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                        const __grid_constant__ CUtensorMap vmap, const AttnParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;
    uint8_t* sKV = smem + kQBytes;  // stage s: K at s*64KB, V at s*64KB + 32KB

    // one set per ring stage; the tile's S and P have a tensor-memory buffer of the same index.  done: the
    // tile's P V is complete, so its K, V and P are read (the stage may be refilled, the buffer overwritten).
    // With two S buffers Q K^T of a tile waited for the P V two tiles before it, which the same thread had just
    // issued, and each tile took four commits; three buffers leave two commits and no such wait (25 sequences
    // of up to 10412 keys: 100.7 -> 96.5 us, the ragged 32 90.5 -> 89.1 us, 1 x 2064 keys 8.35 -> 8.23 us).
    __shared__ uint64_t bar_kv_full[kStages], bar_s_full[kStages], bar_p_full[kStages], bar_done[kStages];
    __shared__ uint64_t bar_k_full[kStages], bar_k_empty[kStages];  // AHEAD: the K ring's; bar_kv_full is the V ring's then
    __shared__ uint64_t bar_o_done, bar_drain, bar_q_full, bar_q_empty;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int unit_seq_sh;
    // cluster split: the sequences' key offsets (longest-first order); flat split: their tile prefix sums
    __shared__ int32_t seq_sh[kMaxOrderedSeqs + 1];
    __shared__ uint8_t order_sh[FLAT == 2 ? kMaxDealtSeqs : 1];  // units dealt out: the sequences, longest first

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        if (p.q_tma) prefetch_tensormap(&qmap);
        prefetch_tensormap(&kmap);
        prefetch_tensormap(&vmap);
    }
    if (p.early_release) griddep_launch_dependents();
    if (p.num_seqs > 1) griddep_wait();  // the sequence offsets are read from global memory
    const int G = p.group;
    const uint32_t CS = FLAT ? 1u : cluster_size();
    const uint32_t crank = FLAT ? 0u : cluster_rank();

    // ---- work assignment.  Flat split: global tiles [t_lo, t_hi).  Cluster split: one stretch, `one`.
    int t_lo = 0, t_hi = 0, T = 0;
    bool dealt = false;
    bool ahead = AHEAD && !FLAT;  // (flat split: where every CTA has one stretch)
    Seg one{};
    const int ngroups = FLAT ? gridDim.x / p.num_kv_heads : 1, grp = FLAT ? blockIdx.x / p.num_kv_heads : 0;
    const int free_groups = FLAT == 2 ? ngroups / p.num_seqs : 0;  // groups of CTAs per unit, if at least one
    if (FLAT) {
        if (p.num_seqs > 1) {
            flat_prefix(p, seq_sh, tid);
            T = seq_sh[p.num_seqs];
        } else {
            T = flat_seq_tiles(p.total_q, p.total_kv, G);
        }
        // CTAs come in groups of one per KV head; group j has tiles [t_lo, t_hi) of every head
        t_lo = (int)((long long)grp * T / ngroups);
        t_hi = (int)((long long)(grp + 1) * T / ngroups);
        // Lengths the host could only bound: even cuts, or the units dealt out -- by the host's estimates, on the
        // lengths as they are.  Every CTA decides the same.  (16 x 2016 keys in a cache of 8192: 37.0 us cut evenly,
        // 29.7 dealt out, 26.9 in clusters.)
        const int S = p.num_seqs;
        if constexpr (FLAT == 2) {  // (1 < S <= kMaxDealtSeqs, one query tile)
            if (tid == 0) unit_seq_sh = 0;
            if (tid < S) {
                const int len = seq_sh[tid + 1] - seq_sh[tid];
                int rank = 0;
                for (int u = 0; u < S; ++u) {
                    const int lu = seq_sh[u + 1] - seq_sh[u];
                    rank += (lu > len) || (lu == len && u < tid);
                }
                order_sh[rank] = (uint8_t)tid;
            }
            __syncthreads();
            const auto tiles_of = [&](int rank) { return seq_sh[order_sh[rank] + 1] - seq_sh[order_sh[rank]]; };
            const int rounds = cdiv(S, ngroups), longest = tiles_of(0);
            int chain;  // key tiles of the busiest CTA
            if (free_groups >= 1) {
                chain = cdiv(longest, dealt_parts(longest, free_groups));
            } else {
                for (int g = tid; g < ngroups; g += kThreads) {
                    int sum = 0;
                    for (int t = 0; t < rounds; ++t) {
                        const int rank = dealt_rank(t, g, ngroups, 0);
                        if (rank < S) sum += tiles_of(rank);
                    }
                    atomicMax(&unit_seq_sh, sum);
                }
                __syncthreads();
                chain = unit_seq_sh;
            }
            const float even = p.us_cut * (float)T / (float)ngroups;
            const float est_cut = even + 10.f + fminf(4.2f * (1.f + (float)S / (float)ngroups), 11.f);
            const float est_dealt = free_groups >= 1 && chain < longest
                                        ? fmaxf(p.us_part * (float)chain, even) + 10.5f
                                        : fmaxf(p.us_whole * (float)chain, even) + 9.5f + 4.f * (float)(rounds - 1);
            dealt = est_dealt < est_cut;
            if (dealt) {
                const int parts = free_groups >= 1 ? dealt_parts(longest, free_groups) : 0;
                ahead = AHEAD && p.ahead_ok && parts >= 1 && parts <= 5 && chain >= 6 &&
                        S * parts * p.num_kv_heads * 10 <= 9 * p.sm_count;
                t_lo = 0;
                t_hi = 0;
                if (free_groups >= 1) {
                    const int rank = grp / free_groups, part = grp - rank * free_groups;
                    t_hi = rank < S && tiles_of(rank) > 0 && part < dealt_parts(tiles_of(rank), free_groups) ? 1 : 0;
                } else {
                    while (t_hi < rounds && dealt_rank(t_hi, grp, ngroups, 0) < S &&
                           tiles_of(dealt_rank(t_hi, grp, ngroups, 0)) > 0)
                        ++t_hi;
                }
            }
        }
    } else {
        const int unit_rank = blockIdx.x / CS;
        const int units_per_seq = p.num_kv_heads * p.m_tiles;
        const int seq_rank = unit_rank / units_per_seq;
        one.h = (unit_rank / p.m_tiles) % p.num_kv_heads;
        one.mt = unit_rank % p.m_tiles;
        // which sequence: the seq_rank-th longest (ties by index) for small batches
        int s;
        if (p.num_seqs == 1) {
            s = 0;
        } else if (p.num_seqs <= kMaxOrderedSeqs) {
            for (int t = tid; t <= p.num_seqs; t += kThreads) seq_sh[t] = p.cu_kv[t];
            __syncthreads();
            for (int t = tid; t < p.num_seqs; t += kThreads) {
                const int len = seq_sh[t + 1] - seq_sh[t];
                int rank = 0;
                for (int u = 0; u < p.num_seqs; ++u) {
                    const int lu = seq_sh[u + 1] - seq_sh[u];
                    rank += (lu > len) || (lu == len && u < t);
                }
                if (rank == seq_rank) unit_seq_sh = t;
            }
            __syncthreads();
            s = unit_seq_sh;
        } else {
            s = seq_rank;
        }
        one.s = s;
        // a single sequence starts at offset 0 (cu_*[0] = 0) and spans the whole tensors: no loads
        one.q0 = p.num_seqs == 1 ? 0 : __ldg(p.cu_q + s);
        one.B = p.num_seqs == 1 ? p.total_q : __ldg(p.cu_q + s + 1) - one.q0;
        one.kv0 = p.num_seqs == 1 ? 0 : __ldg(p.cu_kv + s);
        one.n = p.num_seqs == 1 ? p.total_kv : __ldg(p.cu_kv + s + 1) - one.kv0;
        if (one.B * G - one.mt * kM <= 0) {  // uniform across the cluster: every CTA decodes the same unit
            griddep_wait();  // this grid must not complete before the one it depends on
            return;
        }
        const int tiles = cdiv(one.n, kTileN);
        one.jt0 = (int)((long long)crank * tiles / CS);
        one.nt = (int)((long long)(crank + 1) * tiles / CS) - one.jt0;
        one.whole = 0;
        one.slot = 0;
        one.parts = 0;
    }
    // The stretches of this CTA, in order: `first` is the CTA's first one; t advances past each.
    auto seg_at = [&](int t, bool first) -> Seg {
        if (!FLAT) return one;
        const int h = (int)(blockIdx.x % p.num_kv_heads);
        return FLAT == 2 && dealt ? dealt_seg(p, order_sh, t, grp, ngroups, free_groups, h)
                                  : flat_seg(p, seq_sh, t, t_hi, h, first);
    };
    const int t_begin = FLAT ? t_lo : 0;
    const int t_end = FLAT ? t_hi : 1;
    auto seg_len = [&](const Seg& g) { return FLAT && !(FLAT == 2 && dealt) ? g.nt : 1; };

    // ---- Q tile -> shared memory, SWIZZLE_128B K-major (two 64-column halves).  With a TMA map the
    // 128/G block positions x G heads box lands exactly as rows r = i*G + j; otherwise (cluster split
    // only) plain loads.
    if (!FLAT && !p.q_tma) {
        griddep_wait();
        const int row0 = one.mt * kM, m_valid = min(kM, one.B * G - row0);
        for (int idx = tid; idx < kM * 16; idx += kThreads) {
            const int r = idx >> 4, ch = idx & 15;
            uint4 val = make_uint4(0, 0, 0, 0);
            if (r < m_valid) {
                const int lr = row0 + r;
                const int i = lr / G, j = lr % G;
                val = *reinterpret_cast<const uint4*>(p.q + ((size_t)(one.q0 + i) * p.num_q_heads + one.h * G + j) *
                                                      kD + ch * 8);
            }
            const int half = ch >> 3, c8 = ch & 7;
            *reinterpret_cast<uint4*>(sQ + half * kHalf + r * 128 + ((c8 ^ (r & 7)) << 4)) = val;
        }
        fence_proxy_async_smem();
    }
    // paged cache: the pool rows of a tile's sub-boxes (sub_rows keys each); keys past the end of the
    // sequence read the rows of its last page (finite values the mask then drops)
    constexpr bool paged = PAGED;
    const int sub_rows = paged ? min(kTileN, 1 << p.page_shift) : kTileN;
    const int nsub = kTileN / sub_rows;
    auto tile_rows = [&](const Seg& g, int jl, int (&row)[kMaxSub]) {
        if (!paged) return;
        const int32_t* bt = p.block_table + (size_t)g.s * p.pages_per_seq;
        const int last_page = max(0, (g.n - 1) >> p.page_shift);
        const int key0 = (g.jt0 + jl) * kTileN;
#pragma unroll
        for (int sb = 0; sb < kMaxSub; ++sb)
            if (sb < nsub) {
                const int key = key0 + sb * sub_rows;
                const int pi = min(key >> p.page_shift, last_page);
                row[sb] = __ldg(bt + pi) * (1 << p.page_shift) + (key & ((1 << p.page_shift) - 1));
            }
    };
    // the K rows (or the V rows) of tile jl of stretch g -> stage J % kStages of the ring (J counts the CTA's
    // tiles; producer thread only)
    auto load_rows = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* bar, const Seg& g, int jl,
                         const int (&row)[kMaxSub]) {
        if (!paged) {
            const int key = g.kv0 + (g.jt0 + jl) * kTileN;
            tma_load_3d(dst, map, bar, 0, g.h, key);
            tma_load_3d(dst + kHalf, map, bar, 64, g.h, key);
        } else {
#pragma unroll
            for (int sb = 0; sb < kMaxSub; ++sb) {  // sub-box sb lands at row sb * sub_rows of the tile
                if (sb < nsub) {
                    const int off = sb * sub_rows * 128;
                    tma_load_3d(dst + off, map, bar, 0, g.h, row[sb]);
                    tma_load_3d(dst + kHalf + off, map, bar, 64, g.h, row[sb]);
                }
            }
        }
    };
    auto issue_k = [&](int J, const Seg& g, int jl, const int (&row)[kMaxSub]) {
        const int st = J % kStages;
        uint64_t* bar = ahead ? &bar_k_full[st] : &bar_kv_full[st];
        mbar_arrive_expect_tx(bar, ahead ? kKVBytes : kStageBytes);  // not ahead: V's bytes too
        load_rows(sKV + st * kStageBytes, &kmap, bar, g, jl, row);
    };
    auto issue_v = [&](int J, const Seg& g, int jl, const int (&row)[kMaxSub]) {
        const int st = J % kStages;
        if (ahead) mbar_arrive_expect_tx(&bar_kv_full[st], kKVBytes);
        load_rows(sKV + st * kStageBytes + kKVBytes, &vmap, &bar_kv_full[st], g, jl, row);
    };
    // the Q tile of stretch g (producer thread only)
    auto issue_q = [&](const Seg& g) {
        const int row0 = g.mt * kM;
        if (SPREAD) {  // four boxes of 16 rows, at shared-memory rows 0, 32, 64, 96
            mbar_arrive_expect_tx(&bar_q_full, kQBytes / 2);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                const int qrow = g.q0 + (row0 + 16 * qq) / G;
                tma_load_3d(sQ + qq * 32 * 128, &qmap, &bar_q_full, 0, g.h * G, qrow);
                tma_load_3d(sQ + kHalf + qq * 32 * 128, &qmap, &bar_q_full, 64, g.h * G, qrow);
            }
        } else {
            mbar_arrive_expect_tx(&bar_q_full, kQBytes);
            const int qrow = g.q0 + row0 / G;
            tma_load_3d(sQ, &qmap, &bar_q_full, 0, g.h * G, qrow);
            tma_load_3d(sQ + kHalf, &qmap, &bar_q_full, 64, g.h * G, qrow);
        }
    };
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&bar_kv_full[i], 1);
            mbar_init(&bar_s_full[i], 1);
            mbar_init(&bar_p_full[i], 128);
            mbar_init(&bar_done[i], 1);
            if (AHEAD) {
                mbar_init(&bar_k_full[i], 1);
                mbar_init(&bar_k_empty[i], 1);
            }
        }
        mbar_init(&bar_o_done, 1);
        mbar_init(&bar_drain, 1);
        mbar_init(&bar_q_full, 1);
        mbar_init(&bar_q_empty, 1);
        fence_mbar_init();
    }
    if (warp == 1) {  // tensor memory is allocated (and released) by warp 1, in parallel
        tmem_alloc(&tmem_base_sh, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;
    // inputs may be produced by the previous kernel on the stream: wait for it before any global access
    griddep_wait();
    // the merge's first cluster barrier joins the softmax warps' row statistics; these two warps have nothing
    // to publish there and must not hold it up
    if (!FLAT && CS > 1 && warp < 2) cluster_arrive_relaxed();

    if (warp == 0) {
        // ================= TMA producer: the Q tile of each stretch, the K/V tiles through the ring
        if (lane == 0) {
            int J = 0, nq = 0;
            bool ok = true;
            int jv = 0, rows_v[kMaxSub];  // AHEAD: tiles whose V is issued, the pool rows of the next one
            for (int t = t_begin; t < t_end && ok;) {
                const Seg g = seg_at(t, t == t_begin);
                t += seg_len(g);
                if (g.nt == 0) continue;
                for (int jl = 0; jl < g.nt; ++jl, ++J) {
                    int rows[kMaxSub];
                    tile_rows(g, jl, rows);  // page lookups in flight while the stage drains
                    if (J >= kStages && !mbar_wait(ahead ? &bar_k_empty[J % kStages] : &bar_done[J % kStages],
                                                   ((J / kStages) - 1) & 1, kWaitBudget)) {
                        ok = false;
                        break;
                    }
                    issue_k(J, g, jl, rows);
                    if (ahead) {  // one stretch: tile J - 1's V, once its stage is free
                        if (J > 0) {
                            if (jv >= kStages &&
                                !mbar_wait(&bar_done[jv % kStages], ((jv / kStages) - 1) & 1, kWaitBudget)) {
                                ++J;
                                ok = false;
                                break;
                            }
                            issue_v(jv, g, jv, rows_v);
                            ++jv;
                        }
                        if (paged) {
#pragma unroll
                            for (int sb = 0; sb < kMaxSub; ++sb) rows_v[sb] = rows[sb];
                        }
                    } else {
                        issue_v(J, g, jl, rows);
                    }
                    if (jl == 0 && p.q_tma) {
                        // the stretch's Q, once the MMAs of the previous stretch no longer read the buffer
                        if (nq > 0 && !mbar_wait(&bar_q_empty, (nq - 1) & 1, kWaitBudget)) {
                            ++J;
                            ok = false;
                            break;
                        }
                        issue_q(g);
                        ++nq;
                    }
                }
                if (ahead && ok) {  // the last tile's V
                    ok = jv < kStages || mbar_wait(&bar_done[jv % kStages], ((jv / kStages) - 1) & 1, kWaitBudget);
                    if (ok) {
                        issue_v(jv, g, jv, rows_v);
                        ++jv;
                    }
                }
            }
            if (!ok) raise_error(p.err, kErrTimeout);
            // no copy may still be in flight when the CTA leaves
            const int nv = ahead ? jv : J;
            for (int j = max(0, nv - kStages); j < nv; ++j)
                if (!mbar_wait(&bar_kv_full[j % kStages], (j / kStages) & 1, kDrainBudget)) raise_error(p.err, kErrTimeout);
            if (ahead)
                for (int j = max(0, J - kStages); j < J; ++j)
                    if (!mbar_wait(&bar_k_full[j % kStages], (j / kStages) & 1, kDrainBudget)) raise_error(p.err, kErrTimeout);
            if (nq > 0 && !mbar_wait(&bar_q_full, (nq - 1) & 1, kDrainBudget)) raise_error(p.err, kErrTimeout);
        }
    } else if (warp == 1) {
        // ================= MMA issuer
        if (lane == 0) {
            const uint32_t id_s = idesc_bf16_f32(kM, kTileN, false, false);
            const uint32_t id_o = idesc_bf16_f32(kM, kD, false, true);
            const uint32_t q_addr = smem_addr(sQ);
            int J = 0, nq = 0;
            bool ok = true;
            auto issue_pv = [&](int Jx, bool first) {
                const int st = Jx % kStages;
                if (ahead && !mbar_wait(&bar_kv_full[st], (Jx / kStages) & 1, kWaitBudget)) return false;
                if (!mbar_wait(&bar_p_full[st], (Jx / kStages) & 1, kWaitBudget)) return false;
                tc_fence_after();
                const uint32_t v_addr = smem_addr(sKV + st * kStageBytes + kKVBytes);
#pragma unroll
                for (int kk = 0; kk < kTileN / 16; ++kk) {
                    const uint64_t bdesc = smem_desc(v_addr + kk * 2048, kHalf, 1024, kSwizzle128B);
                    umma_ts(tmem + kColO, tmem + col_s(st) + kk * 8, bdesc, id_o, (!first || kk > 0) ? 1u : 0u);
                }
                umma_commit(&bar_done[st]);
                return true;
            };
            for (int t = t_begin; t < t_end && ok;) {
                const Seg g = seg_at(t, t == t_begin);
                t += seg_len(g);
                if (g.nt == 0) continue;
                if (p.q_tma && !mbar_wait(&bar_q_full, nq & 1, kWaitBudget)) {
                    ok = false;
                    break;
                }
                for (int jl = 0; jl < g.nt; ++jl, ++J) {
                    // (the stage was refilled after the P V of tile J - kStages, so its S buffer is free too)
                    const int st = J % kStages;
                    if (!mbar_wait(ahead ? &bar_k_full[st] : &bar_kv_full[st], (J / kStages) & 1, kWaitBudget)) { ok = false; break; }
                    if (ahead && J >= kStages && !mbar_wait(&bar_done[st], ((J / kStages) - 1) & 1, kWaitBudget)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t k_addr = smem_addr(sKV + st * kStageBytes);
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk) {
                        const uint32_t off = (kk >> 2) * kHalf + (kk & 3) * 32;
                        const uint64_t adesc = smem_desc(q_addr + off, 16, 1024, kSwizzle128B);
                        const uint64_t bdesc = smem_desc(k_addr + off, 16, 1024, kSwizzle128B);
                        umma_ss(tmem + col_s(st), adesc, bdesc, id_s, kk > 0 ? 1u : 0u);
                    }
                    umma_commit(&bar_s_full[st]);
                    if (ahead) umma_commit(&bar_k_empty[st]);
                    if (jl == g.nt - 1) umma_commit(&bar_q_empty);  // the last read of this stretch's Q
                    if (jl >= 1 && !issue_pv(J - 1, jl == 1)) { ++J; ok = false; break; }
                }
                if (!ok) break;
                if (!issue_pv(J - 1, g.nt == 1)) { ok = false; break; }
                umma_commit(&bar_o_done);
                ++nq;
            }
            if (!ok) raise_error(p.err, kErrTimeout);
            if (J > 0) {
                // no MMA may still be writing tensor memory when it is released (a barrier of its own: a second
                // phase of bar_o_done completing right behind the first could pass a softmax warp that has not
                // yet looked at the first, which would then wait until its budget expired)
                umma_commit(&bar_drain);
                if (!mbar_wait(&bar_drain, 0, kDrainBudget)) raise_error(p.err, kErrTimeout);
            }
        }
    }

    // ================= softmax / epilogue warps (2..5).  Dense: row r = TMEM lane quad*32 + lane, all
    // columns.  SPREAD: row r = quad*16 + lane%16 at TMEM lane quad*32 + lane%16, columns of half lane/16.
    constexpr int kCols = SPREAD ? kTileN / 2 : kTileN;  // S / P columns (keys) per thread
    constexpr int kOCols = SPREAD ? kD / 2 : kD;         // O columns per thread
    const int quad = warp & 3;
    const int half = SPREAD ? (lane >> 4) : 0;
    const int r = SPREAD ? quad * 16 + (lane & 15) : quad * 32 + lane;
    const bool is_softmax = warp >= 2;
    const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
    const float kLn2 = 0.6931471805599453f;
    float m_run = -INFINITY, l_run = 0.f;  // SPREAD: l_run is this half's share of the row sum
    float o_acc[kOCols];
    bool failed = false;
    bool row_active = false;  // the cluster split's merge below needs the (one) stretch's values
    int m_valid = 0;
    // merge of the cluster split: the CTA's (m, l) per row, in the last K stage (every Q K^T is complete before
    // it is written)
    float2* row_ml = reinterpret_cast<float2*>(sKV + (kStages - 1) * kStageBytes);

    // normalised output row r of stretch g (and its log-sum-exp)
    auto write_row = [&](const Seg& g) {
        const int lr = g.mt * kM + r;
        const int i = lr / G, jh = lr % G;
        const size_t orow = (size_t)(g.q0 + i) * p.num_q_heads + g.h * G + jh;
        const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
        __nv_bfloat16* dst = p.o + orow * kD + half * kOCols;
#pragma unroll
        for (int c = 0; c < kOCols / 8; ++c) {
            uint4 w;
            w.x = pack_bf16x2(o_acc[c * 8 + 0] * inv, o_acc[c * 8 + 1] * inv);
            w.y = pack_bf16x2(o_acc[c * 8 + 2] * inv, o_acc[c * 8 + 3] * inv);
            w.z = pack_bf16x2(o_acc[c * 8 + 4] * inv, o_acc[c * 8 + 5] * inv);
            w.w = pack_bf16x2(o_acc[c * 8 + 6] * inv, o_acc[c * 8 + 7] * inv);
            *reinterpret_cast<uint4*>(dst + c * 8) = w;
        }
        if (p.lse && half == 0) p.lse[orow] = (m_run + __log2f(l_run)) * kLn2;
    };

    if (is_softmax) {
        int J = 0, nq = 0;
        int4 entry = make_int4(-1, 0, 0, 0), entry2 = make_int4(0, 0, 0, 0);  // flat split: the merge's work entry
        for (int t = t_begin; t < t_end && !failed;) {
            const Seg g = seg_at(t, t == t_begin);
            if (FLAT && !g.whole && g.jt0 == 0) {  // a cut unit that starts here
                entry = make_int4(t, t + cdiv(g.n, kTileN), T, min(min(kM, g.B * G - g.mt * kM), p.slot_rows));
                entry2 = make_int4(g.q0, g.mt, g.parts, 0);
            }
            t += seg_len(g);
            const int row0 = g.mt * kM;
            m_valid = min(kM, g.B * G - row0);
            row_active = r < m_valid;
            const bool warp_active = (SPREAD ? quad * 16 : quad * 32) < m_valid;
            const int L = g.n - g.B;
            const int limit = row_active ? (p.causal ? L + (row0 + r) / G + 1 : g.n) : 0;
            m_run = -INFINITY;
            l_run = 0.f;
            for (int jl = 0; jl < g.nt; ++jl, ++J) {
                const int st = J % kStages;
                if (!__all_sync(0xffffffffu, mbar_wait(&bar_s_full[st], (J / kStages) & 1, kWaitBudget))) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                if (warp_active) {
                    const int nvalid = limit - (g.jt0 + jl) * kTileN;
                    // the raw scores: every load in flight before the one wait; only the unit's last tiles hold
                    // keys some row does not see
                    uint32_t x[kCols / 32][32];
#pragma unroll
                    for (int c = 0; c < kCols / 32; ++c) {
                        if (SPREAD) tmem_ld16x2_32<kTileN / 2>(tmem + lane_base + col_s(st) + c * 32, x[c]);
                        else tmem_ld32(tmem + lane_base + col_s(st) + c * 32, x[c]);
                    }
                    tmem_ld_wait();
                    if (!__all_sync(0xffffffffu, nvalid >= kTileN)) {
#pragma unroll
                        for (int c = 0; c < kCols / 32; ++c)
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (half * (kTileN / 2) + c * 32 + e >= nvalid) x[c][e] = 0xff800000u;  // -inf
                    }
                    // row maximum in four independent chains: one warp runs on each scheduler, so a single chain
                    // would pay an instruction's latency per key.  With the unmasked tiles' compares gone, the
                    // chains split and the weights formed as packed pairs, 36 layers' step went from 423.4 to
                    // 407.8 us, the ragged 32 from 95.5 to 91.9 us, 16 x 4112 keys from 51.4 to 49.6 us.
                    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int c = 0; c < kCols / 32; ++c)
#pragma unroll
                        for (int e = 0; e < 32; e += 2)
                            mx[(e >> 1) & 3] = fmaxf(mx[(e >> 1) & 3],
                                                     fmaxf(__uint_as_float(x[c][e]), __uint_as_float(x[c][e + 1])));
                    float mt_ = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                    if (SPREAD) mt_ = fmaxf(mt_, __shfl_xor_sync(0xffffffffu, mt_, 16));
                    mt_ *= p.scale_log2;  // the scale is positive: the scaled maximum
                    const float m_new = fmaxf(m_run, mt_);
                    const bool need = m_new > m_run + 8.f;
                    const float alpha = need ? fast_exp2(m_run - m_new) : 1.f;
                    // rescale the TMEM accumulator of rows whose max grew (warp-uniform TMEM access)
                    if (__any_sync(0xffffffffu, need && jl > 0 && m_run != -INFINITY)) {
                        if (!__all_sync(0xffffffffu,
                                        mbar_wait(&bar_done[(J - 1) % kStages], ((J - 1) / kStages) & 1, kWaitBudget))) {
                            failed = true;
                        } else {
                            tc_fence_after();
#pragma unroll
                            for (int c = 0; c < kOCols / 32; ++c) {
                                uint32_t v[32];
                                if (SPREAD) tmem_ld16x2_32<kD / 2>(tmem + lane_base + kColO + c * 32, v);
                                else tmem_ld32(tmem + lane_base + kColO + c * 32, v);
                                tmem_ld_wait();
                                if (SPREAD) {
#pragma unroll
                                    for (int e = 0; e < 32; ++e)
                                        v[e] = __float_as_uint(__uint_as_float(v[e]) * alpha);
                                    tmem_st16x2_32<kD / 2>(tmem + lane_base + kColO + c * 32, v);
                                } else {
                                    uint32_t w0[16], w1[16];
#pragma unroll
                                    for (int e = 0; e < 16; ++e) {
                                        w0[e] = __float_as_uint(__uint_as_float(v[e]) * alpha);
                                        w1[e] = __float_as_uint(__uint_as_float(v[16 + e]) * alpha);
                                    }
                                    tmem_st16(tmem + lane_base + kColO + c * 32, w0);
                                    tmem_st16(tmem + lane_base + kColO + c * 32 + 16, w1);
                                }
                            }
                        }
                    }
                    if (need) {
                        l_run *= alpha;
                        m_run = m_new;
                    }
                    // weights 2^(scale * s - m) as packed pairs (one fused multiply-add each; a row that has
                    // seen no key yet has every score at -inf and gets zeros), summed in four chains
                    const float negm = m_run == -INFINITY ? 0.f : -m_run;
                    const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2), negm2 = pack_f32x2(negm, negm);
                    uint64_t sum2[2] = {0ull, 0ull};  // (+0, +0) pairs
                    auto weights = [&](uint32_t xa, uint32_t xb, int chain) -> uint32_t {
                        float a, b;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(xa), __uint_as_float(xb)), scale2, negm2), a, b);
                        a = fast_exp2(a);
                        b = fast_exp2(b);
                        sum2[chain] = add_f32x2(sum2[chain], pack_f32x2(a, b));
                        return pack_bf16x2(a, b);
                    };
                    if (SPREAD) {  // this half's 64 keys -> 32 packed P columns (the other half 32 further)
                        uint32_t pk[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) pk[e] = weights(x[e / 16][2 * e % 32], x[e / 16][2 * e % 32 + 1], e & 1);
                        tmem_st16x2_32<kTileN / 4>(tmem + lane_base + col_s(st), pk);
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t pk[16];
#pragma unroll
                            for (int e = 0; e < 16; ++e) pk[e] = weights(x[c % (kCols / 32)][2 * e], x[c % (kCols / 32)][2 * e + 1], e & 1);
                            tmem_st16(tmem + lane_base + col_s(st) + c * 16, pk);
                        }
                    }
                    float s0, s1, s2, s3;
                    unpack_f32x2(sum2[0], s0, s1);
                    unpack_f32x2(sum2[1], s2, s3);
                    const float lsum = (s0 + s1) + (s2 + s3);
                    l_run += lsum;
                    tmem_st_wait();
                }
                tc_fence_before();
                mbar_arrive(&bar_p_full[st]);
                if (failed) break;
            }
            if (SPREAD) l_run += __shfl_xor_sync(0xffffffffu, l_run, 16);  // the whole row's sum
            if (!FLAT && CS > 1 && !p.part) {  // the rows' (m, l) for the merge, while the last P V runs
                if (half == 0) row_ml[r] = make_float2(m_run, l_run);
                __syncwarp();
                cluster_arrive_release();
            }
            // the stretch's accumulator
            if (g.nt > 0 && !failed && !__all_sync(0xffffffffu, mbar_wait(&bar_o_done, nq & 1, kWaitBudget)))
                failed = true;
            failed = __any_sync(0xffffffffu, failed);
            tc_fence_after();
            if (warp_active && g.nt > 0 && !failed) {
#pragma unroll
                for (int c = 0; c < kOCols / 32; ++c) {
                    uint32_t v[32];
                    if (SPREAD) tmem_ld16x2_32<kD / 2>(tmem + lane_base + kColO + c * 32, v);
                    else tmem_ld32(tmem + lane_base + kColO + c * 32, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) o_acc[c * 32 + e] = __uint_as_float(v[e]);
                }
            } else {
#pragma unroll
                for (int e = 0; e < kOCols; ++e) o_acc[e] = 0.f;
                if (g.nt == 0 || failed) {
                    m_run = -INFINITY;
                    l_run = 0.f;
                }
            }
            if (g.nt > 0) ++nq;
            const bool partial = FLAT ? !g.whole : CS > 1 && p.part != nullptr;  // goes to a workspace slot
            if (partial && m_valid > p.slot_rows) {  // a block longer than max_q_len: rows past the slot are dropped
                if (r == 0 && warp == 2) raise_error(p.err, kErrDeviceArg);
                row_active = row_active && r < p.slot_rows;
            }
            if (FLAT && g.whole) {
                if (!failed && row_active) write_row(g);
            } else if (partial && row_active) {  // the partial (O, m, l) of this stretch's rows, for the merge
                float* slot = p.part + (size_t)(FLAT ? 2 * blockIdx.x + g.slot : blockIdx.x) * p.slot_rows * (kD + 2);
                float* orow = slot + (size_t)r * kD + half * kOCols;
#pragma unroll
                for (int c = 0; c < kOCols / 8; ++c) st_global_f32x8(orow + c * 8, &o_acc[c * 8]);
                if (half == 0)
                    *reinterpret_cast<float2*>(slot + (size_t)p.slot_rows * kD + 2 * r) = make_float2(m_run, l_run);
            }
        }
        if (failed) raise_error(p.err, kErrTimeout);
        if (FLAT && tid == 64) {
            p.work[2 * blockIdx.x] = entry;
            p.work[2 * blockIdx.x + 1] = entry2;
        }
    }

    if (!FLAT) {
        if (CS == 1) {
            if (row_active) write_row(one);
        } else if (p.part) {
            // ---- merge of the CS partial (m, l, O) triples through the workspace slots, i.e. through L2: every CTA
            // has written its own; behind one cluster barrier each CTA loads the rows it owns of all of them, a
            // warp per row: lane c the 16-byte chunk c of every partial and, c below the cluster size, partial c's
            // (m, l), whose weights go round the warp by shuffles.  SM to SM a partial crosses at about 14 bytes a
            // clock, through L2 several times faster: 1 x 2064 keys 8.18 -> 7.92 us in clusters of 9 and 8.31 -> 7.70
            // in clusters of 11, 1 x 4112 9.24 -> 8.66 us.  With more than two rows a warp (clusters of 2 to 4) the
            // rounds of loads cost more than the remote stores below (8 x 915 keys 16.4 against 12.8 us).
            __syncwarp();
            if (is_softmax) cluster_arrive_release();
            cluster_wait();
            m_valid = min(min(kM, one.B * G - one.mt * kM), p.slot_rows);
            const int row0 = one.mt * kM;
            const int per = (m_valid + (int)CS - 1) / (int)CS;
            const int rbeg = (int)crank * per;
            const int nmy = max(0, min(m_valid, rbeg + per) - rbeg);
            const size_t slot_floats = (size_t)p.slot_rows * (kD + 2);
            const float* first = p.part + (size_t)(blockIdx.x - crank) * slot_floats;  // the cluster's first slot
            // two rows a warp at most (launch_attention_bf16), their loads in flight together
            constexpr int kRowsPerWarp = 2;
            float4 v[kRowsPerWarp][kMaxCluster];
            float2 ml[kRowsPerWarp];
#pragma unroll
            for (int k = 0; k < kRowsPerWarp; ++k) {
                const int j = warp + k * (kThreads / 32), row = rbeg + j;
                ml[k] = make_float2(-INFINITY, 0.f);
                if (j < nmy) {
#pragma unroll
                    for (int pr = 0; pr < kMaxCluster; ++pr)
                        if (pr < (int)CS)
                            v[k][pr] = __ldcg(reinterpret_cast<const float4*>(first + pr * slot_floats + (size_t)row * kD) + lane);
                    if (lane < (int)CS)
                        ml[k] = __ldcg(reinterpret_cast<const float2*>(first + lane * slot_floats + (size_t)p.slot_rows * kD + 2 * row));
                }
            }
#pragma unroll
            for (int k = 0; k < kRowsPerWarp; ++k) {
                const int j = warp + k * (kThreads / 32);
                if (j >= nmy) break;
                float M = ml[k].x;
#pragma unroll
                for (int o = kMaxCluster / 2; o >= 1; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                M = __shfl_sync(0xffffffffu, M, 0);
                const float w = ml[k].x == -INFINITY ? 0.f : fast_exp2(ml[k].x - M);
                float L = w * ml[k].y;
#pragma unroll
                for (int o = kMaxCluster / 2; o >= 1; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
                L = __shfl_sync(0xffffffffu, L, 0);
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int pr = 0; pr < kMaxCluster; ++pr) {
                    if (pr < (int)CS) {
                        const float wp = __shfl_sync(0xffffffffu, w, pr);
                        acc.x += wp * v[k][pr].x;
                        acc.y += wp * v[k][pr].y;
                        acc.z += wp * v[k][pr].z;
                        acc.w += wp * v[k][pr].w;
                    }
                }
                const float inv = L > 0.f ? 1.f / L : 0.f;
                const int lr = row0 + rbeg + j;
                const size_t orow = (size_t)(one.q0 + lr / G) * p.num_q_heads + one.h * G + lr % G;
                uint2 w2;
                w2.x = pack_bf16x2(acc.x * inv, acc.y * inv);
                w2.y = pack_bf16x2(acc.z * inv, acc.w * inv);
                *reinterpret_cast<uint2*>(p.o + orow * kD + lane * 4) = w2;
                if (p.lse && lane == 0) p.lse[orow] = (M + __log2f(L)) * kLn2;
            }
        } else {
            // ---- merge of the CS partial (m, l, O) triples through distributed shared memory.  Row r of the
            // unit belongs to CTA r / per.  Behind the first cluster barrier (arrived at when the last weights
            // were written, so it completes while the last P V runs) a thread reads its row's (m, l) of every
            // CTA, scales its partial O by 2^(m - M) / L and stores it straight into the owner's slot for this
            // CTA; behind the second the owner adds its slots, in CTA order, from its own shared memory.  Nothing
            // reads a peer's memory after that, so CTAs leave on their own.  The slots lie where the owner's Q
            // and K tiles were: every CTA's Q K^T is complete at the first barrier.  What bounds it: the partials
            // cross between SMs at about 14 bytes a clock (32 KB a CTA in 2400 cycles; whole rows per store,
            // staged through shared memory, were no faster).  Against pulling the partials row by row behind one
            // barrier and leaving behind another: 8 x 915 keys 14.1 -> 12.8 us, 8 ragged 13.4 -> 11.8 us, 4 x 8208
            // 28.9 -> 28.1 us, 1 x 2064 the same (8.2 us).
            m_valid = min(kM, one.B * G - one.mt * kM);
            const int row0 = one.mt * kM;
            const int per = (m_valid + (int)CS - 1) / (int)CS;
            // slot j, 512 bytes: the Q buffer and K stage 0 are adjacent (128 slots), then K stage 1
            static_assert(kStages >= 3 && kQBytes + kKVBytes == 128 * kD * 4 && kMaxCluster * kD * 4 <= kKVBytes,
                          "slots of at most kM + kMaxCluster - 1 rows");
            auto slot = [&](int j) {
                return j < 128 ? sQ + j * (kD * 4) : sKV + kStageBytes + (j - 128) * (kD * 4);
            };
            __syncwarp();
            cluster_wait();
            if (is_softmax && row_active) {
                float2 ml[kMaxCluster];
                const uint32_t ml_addr = smem_addr(row_ml + r);
#pragma unroll
                for (int pr = 0; pr < kMaxCluster; ++pr) {  // every load in flight together
                    ml[pr] = make_float2(-INFINITY, 0.f);
                    if (pr < (int)CS) ml[pr] = ld_cluster_f32x2(mapa(ml_addr, (uint32_t)pr));
                }
                float M = -INFINITY, L = 0.f;
#pragma unroll
                for (int pr = 0; pr < kMaxCluster; ++pr) M = fmaxf(M, ml[pr].x);
#pragma unroll
                for (int pr = 0; pr < kMaxCluster; ++pr)
                    if (ml[pr].x != -INFINITY) L += fast_exp2(ml[pr].x - M) * ml[pr].y;
                const float w = m_run != -INFINITY && L > 0.f ? fast_exp2(m_run - M) * (1.f / L) : 0.f;
                const int owner = r / per;
                const uint32_t dst = mapa(smem_addr(slot((int)crank * per + r - owner * per)), (uint32_t)owner);
#pragma unroll
                for (int c = 0; c < kOCols / 4; ++c)  // 16-byte chunks swizzled by row: rows 512 bytes apart
                    st_cluster_f32x4(dst + (((half * (kOCols / 4) + c) ^ (r & 31)) << 4), o_acc[c * 4] * w,
                                     o_acc[c * 4 + 1] * w, o_acc[c * 4 + 2] * w, o_acc[c * 4 + 3] * w);
                if (p.lse && half == 0 && owner == (int)crank) {
                    const int lr = row0 + r;
                    p.lse[(size_t)(one.q0 + lr / G) * p.num_q_heads + one.h * G + lr % G] = (M + __log2f(L)) * kLn2;
                }
            }
            __syncwarp();
            cluster_sync_all();
            const int rbeg = (int)crank * per;
            const int nmy = max(0, min(m_valid, rbeg + per) - rbeg);
            for (int j = warp; j < nmy; j += kThreads / 32) {  // a warp per owned row, a 16-byte chunk per lane
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                const int ch = (lane ^ ((rbeg + j) & 31)) << 4;
#pragma unroll 4
                for (int pr = 0; pr < (int)CS; ++pr) {
                    const float4 v = *reinterpret_cast<const float4*>(slot(pr * per + j) + ch);
                    acc.x += v.x;
                    acc.y += v.y;
                    acc.z += v.z;
                    acc.w += v.w;
                }
                const int lr = row0 + rbeg + j;
                const size_t orow = (size_t)(one.q0 + lr / G) * p.num_q_heads + one.h * G + lr % G;
                uint2 w2;
                w2.x = pack_bf16x2(acc.x, acc.y);
                w2.y = pack_bf16x2(acc.z, acc.w);
                *reinterpret_cast<uint2*>(p.o + orow * kD + lane * 4) = w2;
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
    // A grid of one wave of short runs lets its dependents launch from its start (their prologues overlap it:
    // batch-1 calls back to back, 9.25 against 9.87 us each); otherwise they launch once every CTA is here or has
    // left.  Released at the start, a grid of two waves followed by the acceptance's statistics (thousands
    // of CTAs, chained by programmatic launch) made a step of the ragged batch take 720-820 us instead of
    // 195, and the flat split's step took 206.8 us instead of 200.3.
    if (!p.early_release) griddep_launch_dependents();
}

// Flat split, second kernel: the units whose tiles were cut between CTA groups.  The CTA of the main
// kernel that holds a cut unit's first tile names it in its work entry.  Thread (row, 16-byte chunk) merges the partial
// (O, m, l) of the unit's CTAs in order -- O = sum_j 2^(m_j - M) O_j / sum_j 2^(m_j - M) l_j, M the
// largest m_j, as a running merge over batches of kCombBatch partials whose loads are all in flight --
// and writes the bf16 output chunk (and the row's log-sum-exp).
constexpr int kCombRows = 8;
constexpr int kCombThreads = kCombRows * kD / 4;  // 256: one 16-byte chunk of a row each
constexpr int kCombBatch = 8;

// Rows [r * kCombRows, (r + 1) * kCombRows) of the cut unit of work entry (wk, wk2) of CTA c; gstart: the CTA groups'
// ranges, group j has [gstart[j], gstart[j + 1]) (not read for a unit dealt out).
__device__ __forceinline__ void combine_rows(const AttnParams& p, const int32_t* gstart, int ngroups, const int4& wk,
                                             const int4& wk2, int c, int r) {
    const int tid = threadIdx.x, G = p.group;
    const int U0 = wk.x, U1 = wk.y, rows = wk.w, q0 = wk2.x, mt = wk2.y;
    const int parts = wk2.z;  // dealt out: the first slots of this many groups
    const int h = c % p.num_kv_heads;
    int lo = c / p.num_kv_heads, hi = ngroups;
    // the group whose range holds the unit's last tile: the last j with gstart[j] <= U1 - 1
    while (parts == 0 && hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (gstart[mid] <= U1 - 1) lo = mid; else hi = mid;
    }
    const int j0 = c / p.num_kv_heads, j1 = parts > 0 ? j0 + parts - 1 : lo;
    const int rl = r * kCombRows + tid / (kD / 4);  // the row within the unit
    const int c4 = tid % (kD / 4);                  // its 16-byte chunk
    if (rl >= rows) return;
    const size_t slot_floats = (size_t)p.slot_rows * (kD + 2);
    const size_t ml_off = (size_t)p.slot_rows * kD + 2 * rl;
    float M = -INFINITY, Lsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int jb = j0; jb <= j1; jb += kCombBatch) {
        float2 ml[kCombBatch];
        float4 v[kCombBatch];
#pragma unroll
        for (int k = 0; k < kCombBatch; ++k) {
            const int j = jb + k;
            ml[k] = make_float2(-INFINITY, 0.f);
            v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j <= j1 && (parts > 0 || gstart[j] < gstart[j + 1])) {
                // CTA (group j, head h): its first stretch (slot 0) unless its range began before the unit
                const float* sp = p.part + (size_t)(2 * (j * p.num_kv_heads + h) +
                                                    (parts > 0 || gstart[j] >= U0 ? 0 : 1)) * slot_floats;
                ml[k] = __ldcg(reinterpret_cast<const float2*>(sp + ml_off));
                v[k] = __ldcg(reinterpret_cast<const float4*>(sp + (size_t)rl * kD + c4 * 4));
            }
        }
#pragma unroll
        for (int k = 0; k < kCombBatch; ++k) {
            if (ml[k].x == -INFINITY) continue;  // nothing (or no visible key) in this partial
            if (ml[k].x > M) {
                const float sc = M == -INFINITY ? 0.f : fast_exp2(M - ml[k].x);
                Lsum *= sc;
                acc.x *= sc;
                acc.y *= sc;
                acc.z *= sc;
                acc.w *= sc;
                M = ml[k].x;
            }
            const float w = fast_exp2(ml[k].x - M);
            Lsum += w * ml[k].y;
            acc.x += w * v[k].x;
            acc.y += w * v[k].y;
            acc.z += w * v[k].z;
            acc.w += w * v[k].w;
        }
    }
    const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
    const int lr = mt * kM + rl;
    const size_t orow = (size_t)(q0 + lr / G) * p.num_q_heads + h * G + lr % G;
    uint2 w2;
    w2.x = pack_bf16x2(acc.x * inv, acc.y * inv);
    w2.y = pack_bf16x2(acc.z * inv, acc.w * inv);
    *reinterpret_cast<uint2*>(p.o + orow * kD + c4 * 4) = w2;
    if (p.lse && c4 == 0) p.lse[orow] = (M + __log2f(Lsum)) * 0.6931471805599453f;
}

// LIST = false: CTA (c, r) takes work entry c and its piece r.  LIST = true, behind the kernel that may have dealt the
// units out so that few or none were cut: three CTAs an SM list the cut units and take their pieces in turn.  (A CTA
// for every piece there could be takes 2.6 us where nothing was cut, the list 1.5; where most units were cut both take
// the same, and with one unit per head the list 0.5 us more.)
constexpr int kCombPerSm = 3;
static_assert(kCombThreads >= kAttnFlatMaxGrid, "a thread per work entry");
template <bool LIST>
__global__ void __launch_bounds__(kCombThreads, kCombPerSm) attn_combine_kernel(const AttnParams p, int grid_main) {
    __shared__ int32_t gstart[kAttnFlatMaxGrid + 1];
    griddep_launch_dependents();
    griddep_wait();  // the partials and work entries of the main kernel
    const int tid = threadIdx.x, ngroups = grid_main / p.num_kv_heads;
    const int chunks = (p.slot_rows + kCombRows - 1) / kCombRows;
    auto ranges = [&](int T) {
        for (int j = tid; j <= ngroups; j += kCombThreads) gstart[j] = (int)((long long)j * T / ngroups);
        __syncthreads();
    };
    if constexpr (!LIST) {
        const int c = blockIdx.x / chunks, r = blockIdx.x - c * chunks;
        const int4 wk = __ldcg(p.work + 2 * c), wk2 = __ldcg(p.work + 2 * c + 1);
        if (wk.x < 0 || r * kCombRows >= wk.w) return;  // CTA c holds no cut unit's first tile, or it has no such rows
        ranges(wk.z);
        combine_rows(p, gstart, ngroups, wk, wk2, c, r);
    } else {
        __shared__ int4 unit[kAttnFlatMaxGrid], unit2[kAttnFlatMaxGrid];  // the cut units' entries; their CTA in .w
        __shared__ int cuts[kCombThreads / 32];
        int4 mine = make_int4(-1, 0, 0, 0), mine2 = mine;
        if (tid < grid_main) {
            mine = __ldcg(p.work + 2 * tid);
            mine2 = __ldcg(p.work + 2 * tid + 1);
        }
        const unsigned ball = __ballot_sync(0xffffffffu, mine.x >= 0);
        if ((tid & 31) == 0) cuts[tid >> 5] = __popc(ball);
        __syncthreads();
        int n = 0, at = __popc(ball & ((1u << (tid & 31)) - 1u));
#pragma unroll
        for (int w = 0; w < kCombThreads / 32; ++w) {
            if (w < (tid >> 5)) at += cuts[w];
            n += cuts[w];
        }
        if (n == 0) return;
        if (mine.x >= 0) {
            unit[at] = mine;
            unit2[at] = make_int4(mine2.x, mine2.y, mine2.z, tid);
        }
        __syncthreads();
        if (unit2[0].z == 0) ranges(unit[0].z);  // cut evenly: every entry names the same number of tiles
        for (int piece = blockIdx.x; piece < n * chunks; piece += gridDim.x) {
            const int4 wk2 = unit2[piece / chunks];
            combine_rows(p, gstart, ngroups, unit[piece / chunks], wk2, wk2.w, piece % chunks);
        }
    }
}

// --------------------------------------------------------------------------- fp32 path
// Unit = (sequence, KV head, tile of kFR of the block's query rows x the head group's heads).  A cluster of
// CS CTAs splits the unit's keys into runs of 64-key chunks; a CTA streams its chunks' K and V rows through
// two shared-memory stages (16-byte cp.async, zero-filled past the sequence and past D) and runs the online
// softmax on register tiles: a thread owns 2 rows x 4 keys of the scores and 2 rows x DP / 16 columns of the
// output, the 16 threads of a row pair sit in one half-warp, so the row statistics are shuffles and the
// weights cross through shared memory without a CTA barrier.  The CS partial (m, l, O) are merged through
// distributed shared memory.  Everything is fp32 (FFMA and expf).
// What bounds it: these shapes hold a few MB, so latency: the number of chunks in a CTA's chain and the one
// merge.  Within a chunk, the 10 shared-memory wavefronts a warp needs for its 32 FFMAs.  The kernel it
// replaces (a warp per output row, a key per lane, each lane walking its key row alone) read 32 rows per load
// instruction and put the whole context into one warp's chain: 4 sequences x 1008 keys x 8 positions, 4 / 2
// heads of 64, took 322.7 us a call and takes 10.2 us here; the error against 64-bit sums went from 6.3e-7
// to 3.3e-7 (shorter chains).
constexpr int kF32MaxD = 128;
constexpr int kFR = 32;         // query rows per tile
constexpr int kFK = 64;         // keys per chunk
constexpr int kFThreads = 256;  // 16 row pairs x 16 key / column groups
constexpr int kFPadP = kFK + 4;

struct F32Params {
    const float* q;
    const float* k;
    const float* v;
    float* o;
    float* lse;
    const int32_t* cu_q;
    const int32_t* cu_kv;
    int hq, hkv, D, m_tiles, causal;
    float scale;
};

template <int DP>
constexpr size_t f32_smem_bytes() {
    return sizeof(float) * ((size_t)kFR * (DP + 4) + 2 * (size_t)kFK * (DP + 4) + 2 * (size_t)kFK * DP +
                            (size_t)kFR * kFPadP + 2 * kFR);
}

// ROWS rows of D floats, row_stride apart, into shared memory rows of DP floats, ld apart; rows from `valid`
// on and columns from D on become zero.
template <int ROWS, int DP, bool VEC>
__device__ __forceinline__ void f32_load_rows(float* dst, int ld, const float* src, size_t row_stride, int valid,
                                              int D, int tid) {
    if (VEC) {
        for (int idx = tid; idx < ROWS * (DP / 4); idx += kFThreads) {
            const int r = idx / (DP / 4), c = 4 * (idx % (DP / 4));
            const bool ok = r < valid && c < D;
            cp_async16(dst + r * ld + c, ok ? src + r * row_stride + c : src, ok);
        }
    } else {
        for (int idx = tid; idx < ROWS * DP; idx += kFThreads) {
            const int r = idx / DP, c = idx % DP;
            dst[r * ld + c] = r < valid && c < D ? __ldg(src + r * row_stride + c) : 0.f;
        }
    }
}

template <int DP, bool VEC>
__global__ void __launch_bounds__(kFThreads) attn_f32_kernel(const F32Params p) {
    extern __shared__ float4 f32_smem[];
    float* sQ = reinterpret_cast<float*>(f32_smem);  // [kFR][DP + 4]
    float* sK = sQ + kFR * (DP + 4);                 // [2][kFK][DP + 4]
    float* sV = sK + 2 * kFK * (DP + 4);             // [2][kFK][DP]
    float* sP = sV + 2 * kFK * DP;                   // [kFR][kFPadP] weights of the current chunk
    float2* sML = reinterpret_cast<float2*>(sP + kFR * kFPadP);  // [kFR] the CTA's (m, l)
    constexpr int kLdK = DP + 4;  // 16-byte reads of 8 consecutive keys fall on distinct banks
    constexpr int kCols = DP / 64;  // 16-byte column groups per thread

    griddep_launch_dependents();
    griddep_wait();
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = (int)cluster_size(), crank = (int)cluster_rank();
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int unit = blockIdx.x / CS;
    const int G = p.hq / p.hkv, D = p.D;
    const int mt = unit % p.m_tiles, kvh = (unit / p.m_tiles) % p.hkv, s = unit / (p.m_tiles * p.hkv);
    const int q0 = __ldg(p.cu_q + s), B = __ldg(p.cu_q + s + 1) - q0;
    const int kv0 = __ldg(p.cu_kv + s), n = __ldg(p.cu_kv + s + 1) - kv0;
    const int L = n - B, rows = B * G;
    const size_t kvstride = (size_t)p.hkv * D;
    const float* kbase = p.k + ((size_t)kv0 * p.hkv + kvh) * D;
    const float* vbase = p.v + ((size_t)kv0 * p.hkv + kvh) * D;

    // (one pass, unless a block is longer than max_q_len; the bounds are the same in every CTA of the cluster)
    for (int row0 = mt * kFR; row0 < rows; row0 += p.m_tiles * kFR) {
        const int nr = min(kFR, rows - row0);
        const int visible = p.causal ? L + (row0 + nr - 1) / G + 1 : n;  // keys the tile's last row sees
        const int chunks = cdiv(visible, kFK);
        const int c0 = (int)((long long)crank * chunks / CS), c1 = (int)((long long)(crank + 1) * chunks / CS);
        auto load_chunk = [&](int c, int st) {
            const int key0 = c * kFK, valid = min(kFK, n - key0);
            f32_load_rows<kFK, DP, VEC>(sK + st * kFK * kLdK, kLdK, kbase + key0 * kvstride, kvstride, valid, D, tid);
            f32_load_rows<kFK, DP, VEC>(sV + st * kFK * DP, DP, vbase + key0 * kvstride, kvstride, valid, D, tid);
            cp_async_commit();
        };
        // row r of the tile: block position (row0 + r) / G, head (row0 + r) % G of the group
        auto row_offset = [&](int r) {
            const int lr = row0 + r;
            return ((size_t)(q0 + lr / G) * p.hq + kvh * G + lr % G) * D;
        };
        if (VEC) {
            for (int idx = tid; idx < kFR * (DP / 4); idx += kFThreads) {
                const int r = idx / (DP / 4), c = 4 * (idx % (DP / 4));
                const bool ok = r < nr && c < D;
                cp_async16(sQ + r * kLdK + c, ok ? p.q + row_offset(r) + c : p.q, ok);
            }
        } else {
            for (int idx = tid; idx < kFR * DP; idx += kFThreads) {
                const int r = idx / DP, c = idx % DP;
                sQ[r * kLdK + c] = r < nr && c < D ? __ldg(p.q + row_offset(r) + c) : 0.f;
            }
        }
        if (c0 < c1) load_chunk(c0, 0);

        int limit[2];  // keys rows 2 ty and 2 ty + 1 see (0 past the tile)
        float m[2], l[2], acc[2][4 * kCols];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int r = 2 * ty + a;
            limit[a] = r < nr ? (p.causal ? L + (row0 + r) / G + 1 : n) : 0;
            m[a] = -INFINITY;
            l[a] = 0.f;
#pragma unroll
            for (int e = 0; e < 4 * kCols; ++e) acc[a][e] = 0.f;
        }
        for (int c = c0; c < c1; ++c) {
            const int st = (c - c0) & 1;
            if (c + 1 < c1) {
                load_chunk(c + 1, st ^ 1);
                cp_async_wait_group<1>();
            } else {
                cp_async_wait_group<0>();
            }
            __syncthreads();
            if (4 * (tid >> 5) < nr) {  // a warp of padding rows only leaves shared memory to the others
                const float* kk = sK + st * kFK * kLdK;
                const float* vv = sV + st * kFK * DP;
                float x[2][4];
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int j = 0; j < 4; ++j) x[a][j] = 0.f;
#pragma unroll 4
                for (int d = 0; d < DP; d += 4) {
                    const float4 qa = *reinterpret_cast<const float4*>(sQ + (2 * ty) * kLdK + d);
                    const float4 qb = *reinterpret_cast<const float4*>(sQ + (2 * ty + 1) * kLdK + d);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 kv = *reinterpret_cast<const float4*>(kk + (tx + 16 * j) * kLdK + d);
                        x[0][j] = fmaf(qa.w, kv.w, fmaf(qa.z, kv.z, fmaf(qa.y, kv.y, fmaf(qa.x, kv.x, x[0][j]))));
                        x[1][j] = fmaf(qb.w, kv.w, fmaf(qb.z, kv.z, fmaf(qb.y, kv.y, fmaf(qb.x, kv.x, x[1][j]))));
                    }
                }
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    float mx = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        x[a][j] = c * kFK + tx + 16 * j < limit[a] ? x[a][j] * p.scale : -INFINITY;
                        mx = fmaxf(mx, x[a][j]);
                    }
#pragma unroll
                    for (int o = 8; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    const float mn = fmaxf(m[a], mx);
                    const bool any = mn != -INFINITY;  // some key of this CTA is visible to the row so far
                    const float alpha = m[a] == -INFINITY ? 0.f : expf(m[a] - mn);
                    float sum = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float w = any ? expf(x[a][j] - mn) : 0.f;
                        sum += w;
                        sP[(2 * ty + a) * kFPadP + tx + 16 * j] = w;
                    }
                    l[a] = l[a] * alpha + sum;  // this thread's keys; joined over the row below
#pragma unroll
                    for (int e = 0; e < 4 * kCols; ++e) acc[a][e] *= alpha;
                    m[a] = mn;
                }
                __syncwarp();  // a row pair's weights are written and read by one half-warp
#pragma unroll 2
                for (int k4 = 0; k4 < kFK; k4 += 4) {
                    const float4 pa = *reinterpret_cast<const float4*>(sP + (2 * ty) * kFPadP + k4);
                    const float4 pb = *reinterpret_cast<const float4*>(sP + (2 * ty + 1) * kFPadP + k4);
                    const float wa[4] = {pa.x, pa.y, pa.z, pa.w}, wb[4] = {pb.x, pb.y, pb.z, pb.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int cc = 0; cc < kCols; ++cc) {
                            const float4 z = *reinterpret_cast<const float4*>(vv + (k4 + e) * DP + 64 * cc + 4 * tx);
                            acc[0][4 * cc] = fmaf(wa[e], z.x, acc[0][4 * cc]);
                            acc[0][4 * cc + 1] = fmaf(wa[e], z.y, acc[0][4 * cc + 1]);
                            acc[0][4 * cc + 2] = fmaf(wa[e], z.z, acc[0][4 * cc + 2]);
                            acc[0][4 * cc + 3] = fmaf(wa[e], z.w, acc[0][4 * cc + 3]);
                            acc[1][4 * cc] = fmaf(wb[e], z.x, acc[1][4 * cc]);
                            acc[1][4 * cc + 1] = fmaf(wb[e], z.y, acc[1][4 * cc + 1]);
                            acc[1][4 * cc + 2] = fmaf(wb[e], z.z, acc[1][4 * cc + 2]);
                            acc[1][4 * cc + 3] = fmaf(wb[e], z.w, acc[1][4 * cc + 3]);
                        }
                }
            }
            __syncthreads();  // the stage and the weights are free
        }
        if (c0 >= c1) {  // no chunk: the query rows' copies still have to land before the memory is used again
            cp_async_wait_group<0>();
            __syncthreads();
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1) l[a] += __shfl_xor_sync(0xffffffffu, l[a], o);

        // four output columns of a row: any D and any alignment of o
        auto store = [&](int r, int col, float4 val) {
            float* dst = p.o + row_offset(r) + col;
            if (VEC && col < D) {
                *reinterpret_cast<float4*>(dst) = val;
            } else if (!VEC) {
                if (col < D) dst[0] = val.x;
                if (col + 1 < D) dst[1] = val.y;
                if (col + 2 < D) dst[2] = val.z;
                if (col + 3 < D) dst[3] = val.w;
            }
        };
        if (CS == 1) {
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int r = 2 * ty + a;
                if (r >= nr) continue;
#pragma unroll
                for (int cc = 0; cc < kCols; ++cc)
                    store(r, 64 * cc + 4 * tx,
                          make_float4(acc[a][4 * cc] / l[a], acc[a][4 * cc + 1] / l[a], acc[a][4 * cc + 2] / l[a],
                                      acc[a][4 * cc + 3] / l[a]));
                if (p.lse && tx == 0) p.lse[row_offset(r) / D] = m[a] + logf(l[a]);
            }
            continue;
        }
        // ---- merge of the cluster's partials: each CTA leaves its own in the first K stage and (m, l) beside
        // it; the tile's 16-byte output chunks are dealt out over the cluster's threads
        float* opart = sK;  // [kFR][DP]
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int r = 2 * ty + a;
#pragma unroll
            for (int cc = 0; cc < kCols; ++cc)
                *reinterpret_cast<float4*>(opart + r * DP + 64 * cc + 4 * tx) =
                    make_float4(acc[a][4 * cc], acc[a][4 * cc + 1], acc[a][4 * cc + 2], acc[a][4 * cc + 3]);
            if (tx == 0) sML[r] = make_float2(m[a], l[a]);
        }
        cluster.sync();
        for (int item = crank * kFThreads + tid; item < nr * (DP / 4); item += CS * kFThreads) {
            const int r = item / (DP / 4), col = 4 * (item % (DP / 4));
            float2 ml[kMaxCluster];
            float4 z[kMaxCluster];
#pragma unroll
            for (int pr = 0; pr < kMaxCluster; ++pr) {  // every peer's loads in flight together
                ml[pr] = make_float2(-INFINITY, 0.f);
                z[pr] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (pr < CS) {
                    ml[pr] = *cluster.map_shared_rank(sML + r, pr);
                    z[pr] = *cluster.map_shared_rank(reinterpret_cast<const float4*>(opart + r * DP + col), pr);
                }
            }
            float M = -INFINITY, sum = 0.f;
#pragma unroll
            for (int pr = 0; pr < kMaxCluster; ++pr) M = fmaxf(M, ml[pr].x);
            float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int pr = 0; pr < kMaxCluster; ++pr) {
                const float w = ml[pr].x == -INFINITY ? 0.f : expf(ml[pr].x - M);
                sum = fmaf(w, ml[pr].y, sum);
                out.x = fmaf(w, z[pr].x, out.x);
                out.y = fmaf(w, z[pr].y, out.y);
                out.z = fmaf(w, z[pr].z, out.z);
                out.w = fmaf(w, z[pr].w, out.w);
            }
            store(r, col, make_float4(out.x / sum, out.y / sum, out.z / sum, out.w / sum));
            if (p.lse && col == 0) p.lse[row_offset(r) / D] = M + logf(sum);
        }
        cluster.sync();  // no CTA reuses or leaves its shared memory while a peer may still read it
    }
}

// Contexts of a few keys: one warp per (query row, query head), online softmax over the row's visible keys in chunks
// of 32 (lane = key), lane d-slices of the output.  Its chain grows with the keys, but it needs no shared memory to
// speak of: thousands of short rows run at once where the tiled kernel takes one wave of two CTAs an SM after
// another (8 heads of 64: 256 sequences of 5 keys 8.6 against 31.3 us, of 17 keys 20.1 and 31.4, of 41 48.4 and 32.0;
// one of 5 keys and heads of 32 3.4 and 4.3).
__global__ void __launch_bounds__(128) attn_f32_row_kernel(const float* __restrict__ q, const float* __restrict__ k,
                                                            const float* __restrict__ v, float* __restrict__ o,
                                                            float* __restrict__ lse, const int32_t* __restrict__ cu_q,
                                                            const int32_t* __restrict__ cu_kv, int num_seqs,
                                                            int total_q, int hq, int hkv, int D, int causal,
                                                            float scale) {
    __shared__ float qs[4][kF32MaxD];
    griddep_launch_dependents();
    griddep_wait();
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * 4 + wib;
    if (row >= (long long)total_q * hq) return;
    const int t = (int)(row / hq), h = (int)(row % hq);
    const int g = hq / hkv, kvh = h / g;
    int lo = 0, hi = num_seqs;  // sequence containing query t: cu_q[s] <= t < cu_q[s+1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cu_q[mid] <= t) lo = mid; else hi = mid;
    }
    const int s = lo;
    const int B = cu_q[s + 1] - cu_q[s];
    const int i = t - cu_q[s];
    const int kv0 = cu_kv[s];
    const int n = cu_kv[s + 1] - kv0;
    const int L = n - B;
    const int nk = causal ? L + i + 1 : n;
    for (int d = lane; d < D; d += 32) qs[wib][d] = q[((size_t)t * hq + h) * D + d];
    __syncwarp();
    float m = -INFINITY, l = 0.f;
    float acc[kF32MaxD / 32];
#pragma unroll
    for (int e = 0; e < kF32MaxD / 32; ++e) acc[e] = 0.f;
    for (int j0 = 0; j0 < nk; j0 += 32) {
        const int j = j0 + lane;
        float sc = -INFINITY;
        if (j < nk) {
            const float* kr = k + ((size_t)(kv0 + j) * hkv + kvh) * D;
            float dot = 0.f;
            for (int d = 0; d < D; ++d) dot = fmaf(qs[wib][d], kr[d], dot);
            sc = dot * scale;
        }
        float cm = sc;
        for (int off = 16; off; off >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, off));
        const float m_new = fmaxf(m, cm);
        const float alpha = (m == -INFINITY) ? 0.f : expf(m - m_new);
        const float pj = (j < nk) ? expf(sc - m_new) : 0.f;
        float ps = pj;
        for (int off = 16; off; off >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, off);
        l = l * alpha + ps;
#pragma unroll
        for (int e = 0; e < kF32MaxD / 32; ++e) acc[e] *= alpha;
        const int cnt = min(32, nk - j0);
        for (int jj = 0; jj < cnt; ++jj) {
            const float pjj = __shfl_sync(0xffffffffu, pj, jj);
            const float* vr = v + ((size_t)(kv0 + j0 + jj) * hkv + kvh) * D;
#pragma unroll
            for (int e = 0; e < kF32MaxD / 32; ++e) {
                const int d = lane + e * 32;
                if (d < D) acc[e] = fmaf(pjj, vr[d], acc[e]);
            }
        }
        m = m_new;
    }
#pragma unroll
    for (int e = 0; e < kF32MaxD / 32; ++e) {
        const int d = lane + e * 32;
        if (d < D) o[((size_t)t * hq + h) * D + d] = acc[e] / l;
    }
    if (lse && lane == 0) lse[(size_t)t * hq + h] = m + logf(l);
}

}  // namespace

namespace {
// Rows of one partial slot of the flat split: a unit's query rows (at most one 128-row tile), rounded
// up to 16 so that every slot starts on a 16-byte boundary.
int flat_slot_rows(int max_q_len, int group) {
    const long long rows = (long long)max_q_len * group;
    return (int)((std::min<long long>(kM, rows) + 15) / 16 * 16);
}
}  // namespace

size_t attention_flat_scratch_bytes(int max_q_len, int group) {
    if (max_q_len < 1 || group < 1) return 0;
    return (size_t)2 * kAttnFlatMaxGrid * flat_slot_rows(max_q_len, group) * (kD + 2) * sizeof(float) +
           (size_t)2 * kAttnFlatMaxGrid * sizeof(int4);
}

namespace {
// The instantiations: [variant][spread][paged], variants cluster split, cluster split AHEAD, flat split, flat split or
// dealt out.
using AttnKernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, AttnParams);
const AttnKernel kAttnKernels[16] = {
    attn_bf16_tc_kernel<false, false, 0, false>, attn_bf16_tc_kernel<true, false, 0, false>,
    attn_bf16_tc_kernel<false, true, 0, false>,  attn_bf16_tc_kernel<true, true, 0, false>,
    attn_bf16_tc_kernel<false, false, 0, true>,  attn_bf16_tc_kernel<true, false, 0, true>,
    attn_bf16_tc_kernel<false, true, 0, true>,   attn_bf16_tc_kernel<true, true, 0, true>,
    attn_bf16_tc_kernel<false, false, 1, false>, attn_bf16_tc_kernel<true, false, 1, false>,
    attn_bf16_tc_kernel<false, true, 1, false>,  attn_bf16_tc_kernel<true, true, 1, false>,
    attn_bf16_tc_kernel<false, false, 2, true>,  attn_bf16_tc_kernel<true, false, 2, true>,
    attn_bf16_tc_kernel<false, true, 2, true>,   attn_bf16_tc_kernel<true, true, 2, true>};
}  // namespace

int launch_attention_bf16(const AttentionArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.head_dim != kD) return BP_ERR_UNSUPPORTED;
    const int G = a.num_q_heads / a.num_kv_heads;
    const int m_tiles = (a.max_q_len * G + kM - 1) / kM;
    const long long units = (long long)a.num_seqs * a.num_kv_heads * m_tiles;
    if (units == 0 || a.total_q == 0) return BP_OK;

    CUtensorMap qmap, kmap, vmap;
    // Q: box of (64 columns) x (G heads) x (128/G block positions) = the packed 128-row tile; for units
    // of at most 64 rows (spread layout) four boxes of 16 rows (16/G block positions) instead
    const bool q_tma = (kM % G == 0);
    const bool spread = q_tma && 16 % G == 0 && (long long)a.max_q_len * G <= 64;
    if (q_tma) {
        const cuuint64_t qdims[3] = {(cuuint64_t)kD, (cuuint64_t)a.num_q_heads, (cuuint64_t)a.total_q};
        const cuuint64_t qstrides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)a.num_q_heads * kD * 2};
        const cuuint32_t qbox[3] = {64, (cuuint32_t)G, (cuuint32_t)((spread ? 16 : kM) / G)};
        const int rq = encode_tensor_map(&qmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(a.q), qdims,
                                         qstrides, qbox, CU_TENSOR_MAP_SWIZZLE_128B);
        if (rq != BP_OK) return rq;
    }
    // K/V: contiguous rows, or the page pool with boxes of one page (at most one 128-key tile)
    const bool paged = a.block_table != nullptr;
    const cuuint64_t kv_rows = paged ? (cuuint64_t)a.num_pages * a.page_size : (cuuint64_t)a.total_kv;
    const cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)a.num_kv_heads, kv_rows};
    const cuuint64_t strides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)a.num_kv_heads * kD * 2};
    const cuuint32_t box[3] = {64, 1, (cuuint32_t)(paged && a.page_size < kTileN ? a.page_size : kTileN)};
    int rc = encode_tensor_map(&kmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(a.k), dims, strides,
                               box, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != BP_OK) return rc;
    rc = encode_tensor_map(&vmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(a.v), dims, strides, box,
                           CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != BP_OK) return rc;

    AttnParams p;
    p.q = static_cast<const __nv_bfloat16*>(a.q);
    p.o = static_cast<__nv_bfloat16*>(a.o);
    p.lse = a.lse;
    p.cu_q = a.cu_q;
    p.cu_kv = a.cu_kv;
    p.num_seqs = a.num_seqs;
    p.total_q = a.total_q;
    p.total_kv = a.total_kv;
    p.num_q_heads = a.num_q_heads;
    p.num_kv_heads = a.num_kv_heads;
    p.group = G;
    p.m_tiles = m_tiles;
    p.causal = a.mask == BP_MASK_CAUSAL_BLOCK;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    p.q_tma = q_tma ? 1 : 0;
    p.block_table = a.block_table;
    p.pages_per_seq = paged ? a.pages_per_seq : 0;
    p.page_shift = 0;
    while (paged && (1 << p.page_shift) < a.page_size) ++p.page_shift;
    p.part = nullptr;
    p.work = nullptr;
    p.slot_rows = flat_slot_rows(a.max_q_len, G);
    p.early_release = 0;
    p.err = a.err_word;
    if (!q_tma) qmap = kmap;  // unused by the kernel

    // once per device (under a lock: calls may come from several host threads): opt in to the
    // shared-memory size and non-portable clusters, and record how many clusters of each size (1..16)
    // the GPU can keep resident at once (queried outside any graph capture; the answer reflects how
    // the SMs are grouped into GPCs)
    static std::mutex cfg_mu;
    static bool configured[64] = {};
    static int max_active_dev[64][kMaxCluster + 1];
    if (dev.device < 0 || dev.device >= 64) return BP_ERR_UNSUPPORTED;
    int max_active[kMaxCluster + 1];
    std::unique_lock<std::mutex> cfg_lock(cfg_mu);
    if (!configured[dev.device]) {
        for (AttnKernel kern : kAttnKernels)
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared) != cudaSuccess)
                return BP_ERR_CUDA;
        for (int cs = 1; cs <= kMaxCluster; ++cs) {
            cudaLaunchConfig_t probe = {};
            cudaLaunchAttribute pa[1];
            probe.gridDim = dim3(cs, 1, 1);
            probe.blockDim = dim3(kThreads, 1, 1);
            probe.dynamicSmemBytes = kDynSmem;
            pa[0].id = cudaLaunchAttributeClusterDimension;
            pa[0].val.clusterDim.x = cs;
            pa[0].val.clusterDim.y = 1;
            pa[0].val.clusterDim.z = 1;
            probe.attrs = pa;
            probe.numAttrs = 1;
            int n_clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&n_clusters, kAttnKernels[0], &probe) !=
                cudaSuccess) {
                cudaGetLastError();
                n_clusters = 0;
            }
            max_active_dev[dev.device][cs] = n_clusters;
        }
        configured[dev.device] = true;
    }
    for (int c = 0; c <= kMaxCluster; ++c) max_active[c] = max_active_dev[dev.device][c];
    cfg_lock.unlock();

    const int max_tiles = (std::min(a.max_kv_len, a.total_kv) + kTileN - 1) / kTileN;  // of the longest, at most
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kDynSmem;
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;

    // cluster split: a split of each unit's keys for which every unit's cluster is resident in the same
    // wave (a unit left for a second wave would double the time).  The tiles of the longest unit per CTA
    // set the time: minimise them; among equal counts take the smallest cluster whose merge needs the
    // fewest passes (a pass merges up to 6 owned rows per CTA, one a warp: 1 x 2064 keys in 2 tiles a CTA
    // take 7.70 us in clusters of 11, 7.92 us in clusters of 9).  A cluster's barriers and merge cost
    // about three tiles of one CTA's chain (batch 1, Qwen3-4B heads: 2 tiles 5.0 us alone against
    // 7.0-7.4 us in clusters; 5 tiles 7.2 us in clusters of 5), so a split that saves fewer than three
    // tiles stays whole
    const int m_rows = std::min(kM, a.max_q_len * G);
    int cs = 1, best = max_tiles, best_pass = 0;
    for (int c = 2; c <= kMaxCluster; ++c) {
        if (c > max_tiles || units > max_active[c] || units * c > dev.sm_count) continue;
        const int per = (max_tiles + c - 1) / c;
        const int passes = ((m_rows + c - 1) / c + kThreads / 32 - 1) / (kThreads / 32);
        if (per < best || (per == best && cs > 1 && passes < best_pass)) {
            best = per;
            cs = c;
            best_pass = passes;
        }
    }
    if (cs > 1 && max_tiles - best < 3) cs = 1;

    // AHEAD: a CTA's bandwidth is what it keeps in flight; where SMs are idle and each CTA streams a long run,
    // refilling K's stages early took 8 x 32784 keys (128 CTAs of 129 tiles) from 163.9 to 153.6 us, 16 x 4112 (128
    // of 33) from 48.8 to 46.5, 3 x 8208 (clusters of 5, 13 tiles a CTA) from 25.7 to 24.7.  With nearly every SM
    // streaming, HBM is the bound and the freer order of requests costs more than it hides (144 CTAs: 18 x 16400
    // keys 178.3 without, 187.8 with; pages of 64 94.8 and 94.0); it loses too in wide clusters (1 x 65552: 54.5
    // and 55.3), on short runs (4 tiles: 13.2 and 13.4) and with 16-key pages (8 x 32784: 246 and 260).
    const auto ahead_for = [&](int c) {
        const long long ctas = units * c;
        return (paged ? a.page_size >= 32 && ctas < dev.sm_count : ctas * 10 <= 9LL * dev.sm_count) && c <= 5 &&
               max_tiles >= 12 * c;
    };

    // flat split: the tiles of every sequence's query tiles cut evenly over groups of CTAs, one CTA per KV
    // head and per SM (at most kAttnFlatMaxGrid in all, and no more groups than one head has tiles); units
    // cut between groups are merged by a second kernel.  It needs the Q tile by TMA, the sequences'
    // offsets in shared memory and the workspace's partial slots and work entries.  BP_ATTENTION_SPLIT=flat or
    // =cluster overrides the choice, =cluster:N also the cluster size, =dealt lets the kernel choose between cuts and
    // dealing (for tests and measurements).
    const long long tiles_bound = (long long)a.num_seqs * m_tiles * max_tiles;
    const int ngroups = (int)std::min<long long>(std::min(dev.sm_count, kAttnFlatMaxGrid) / a.num_kv_heads,
                                                 tiles_bound);
    const int flat_grid = ngroups * a.num_kv_heads;
    const bool flat_ok = q_tma && a.num_seqs <= kMaxOrderedSeqs && a.scratch != nullptr &&
                         a.scratch_bytes >= attention_flat_scratch_bytes(a.max_q_len, G) && ngroups >= 1;
    const long long cluster_ctas = units * cs;
    const double avg_tiles = (double)a.num_kv_heads * m_tiles * ((double)a.total_kv / kTileN + 0.5 * a.num_seqs) /
                             dev.sm_count;
    // Estimates (us) of both splits, fitted to 100 shapes timed in both (1-128 sequences of 200-160K keys) and checked
    // against 260 more (1 to 32 KV heads, blocks of 1 to 64, pages of 16 to 64).
    // us per key tile of a CTA: AHEAD, clusters of up to 5, wider clusters, flat (all SMs together then)
    const double big[4] = {1.10, 1.32, 1.41, 1.39}, p32[4] = {1.26, 1.37, 1.62, 1.45};
    const double p16[4] = {1.83, 1.83, 2.42, 1.70};
    const bool page16 = paged && a.page_size < 32;
    const double* us = page16 ? p16 : paged && a.page_size < 64 ? p32 : big;
    // A sequence's query tiles read the same K and V, which its units of one wave share in L2 (16 x 4112 keys, blocks
    // of 40 -- two tiles: clusters 79.2, flat 103.5 us; 12: 77.9 and 70.9).
    const bool shared = m_tiles > 1;
    // flat: the second kernel merges eight partials a round, and with few KV heads a unit is cut over many groups (16 / 2
    // heads, 1 x 16016 keys, 76 parts: 21.8 us, in clusters 15.4)
    const double cut_parts = (double)ngroups / ((double)a.num_seqs * m_tiles);
    const double est_flat =
        (shared ? 1.2 : 1.0) * us[3] * avg_tiles + 10.0 +
        std::min(4.2 * (1.0 + (double)a.num_seqs / std::max(ngroups, 1)), 11.0) +
        0.7 * std::max(0.0, std::ceil(cut_parts / 8.0) - 3.0);
    // clusters, the longest unit of `longest` key tiles; mixed: how far the others fall short of it
    double mixed = 0.0;
    const auto est_cluster_for = [&](int longest) {
        if (cluster_ctas <= dev.sm_count) {
            // One wave.  Flat for 1 x 65552 keys (50.5 against 54.5 us), 7 x 32784 (145 against 151), 10 x 16400 (110
            // against 146); clusters for 8 x 32784 (153.6 against 163), 16 x 16400 (152 against 168), 5 x 8208 (34.4
            // against 38.4).  Wide clusters stream as fast as HBM lets so many CTAs, down to a CTA's own chain (16 / 2
            // heads, 1 x 16016 keys: 32 CTAs of 8 tiles, 15.4 us); with small pages the chain alone counts.
            const double wide = us == big ? std::max(0.68, (double)cluster_ctas / 128.0) * us[2] : us[2];
            mixed = 0.0;
            return (ahead_for(cs) ? us[0] : cs <= 5 ? us[1] : wide) * ((longest + cs - 1) / cs) +
                   (cs == 1 ? 7.0 : cs <= 5 ? 10.0 : 8.0);
        }
        // Several waves of whole units, longest first.  With lengths spread evenly between 2 mean - longest and longest,
        // the units of the last wave (at most `last` tiles) land on the shortest of the wave before, which pairs up
        // to 2 last.  The tiles then stream at HBM's rate where every SM has a unit and faster where some have
        // none.  20 x 8208 keys: 114.6 flat against 158.6 us; 39 x 4112 113.9 against 136.9; 32 x 4112 98.2 against
        // 95.1; 20 x 528 23.7 against 19.2.  Batches of mixed lengths pack better than that and cut worse.
        const int waves = (int)((units + dev.sm_count - 1) / dev.sm_count);
        const double mean = std::min(avg_tiles * dev.sm_count / units, (double)longest);
        const double least = std::max(2.0 * mean - longest, 0.0);
        const double last = least + (longest - least) * (units - (waves - 1.0) * dev.sm_count) / units;
        const double chain = std::max((double)longest, (waves - 2.0) * longest + 2.0 * last);
        mixed = 1.0 - mean / longest;
        return (shared ? us[0] * chain : (0.86 * chain + 0.48 * avg_tiles) * us[0] / big[0]) +
               (shared ? 6.0 : 5.0 + 5.0 * units / dev.sm_count) - 8.0 * mixed;
    };
    // The longest sequence may have max_kv_len keys, or under a loose bound (a captured loop's cache capacity) all of
    // them total_kv / num_seqs.  Flat where it is the faster split either way.  Where only the bound says so, the
    // kernel looks at the lengths and, if they are even, deals the units out as clusters would have them, about 3 us
    // slower (the second launch): worth the risk where the even lengths take 20 us in clusters, or 25 if the bound is
    // so far above the mean that it is more likely loose.  us dealt or cut by the kernel / in clusters / always cut:
    // 12 x 4016 keys, bound 8192, 43.9 / 40.9 / 44.5; 16 x 2016, bound 8192, 29.7 / 26.9 / 36.2; 16 x 1016 20.0 / 17.1 /
    // 26.4; 10 of 512 to 8192 keys 41.6 / 75.3 / 40.8.  And flat by the simple rule: many waves (57 x 528 keys 33.1
    // against 39.6 us; blocks of 40, 64 x 1040 102.8 against 106.0, pages of 16, 40 x 1540 118.3 against 144.2), and
    // where clusters leave SMs idle on long runs, unless they are clearly the faster.
    const long long mean_kv = ((long long)a.total_kv + a.num_seqs - 1) / a.num_seqs;
    const int even_tiles = std::min(max_tiles, (int)((mean_kv + kTileN - 1) / kTileN));
    const bool many = cluster_ctas >= (shared && !page16 ? 5LL : 3LL) * dev.sm_count;
    const bool simple = (cluster_ctas * 10 <= 9LL * dev.sm_count && tiles_bound >= 64LL * ngroups) ||
                        cluster_ctas >= 3LL * dev.sm_count;
    const double est_even = est_cluster_for(even_tiles), flat_even = est_flat + 6.0 * mixed;
    const double est_cluster = est_cluster_for(max_tiles), flat_bound = est_flat + 6.0 * mixed;
    const bool deals = m_tiles == 1 && a.num_seqs > 1 && a.num_seqs <= kMaxDealtSeqs;
    const double risk = cluster_ctas > dev.sm_count || max_tiles <= 2.4 * even_tiles ? 20.0 : 25.0;
    bool flat = flat_ok && (many || (flat_bound < est_cluster
                                         ? simple || flat_even < est_even || (deals && est_even >= risk)
                                         : simple && est_cluster > 0.97 * flat_bound));
    // (where cutting evenly is the faster either way the kernel is spared the choice: 10 x 16400 keys 110.3 us, 111.9
    // with it)
    bool deal = deals && flat_even >= est_even;
    p.sm_count = dev.sm_count;
    p.ahead_ok = !page16;
    p.us_whole = (float)us[0];
    p.us_part = (float)us[1];
    p.us_cut = (float)us[3];
    if (const char* force = getenv("BP_ATTENTION_SPLIT")) {
        if (strcmp(force, "flat") == 0) {
            flat = flat_ok;
            deal = false;
        } else if (strcmp(force, "dealt") == 0) {  // flat with the choice left to the kernel
            flat = flat_ok;
            deal = deals;
        } else if (strncmp(force, "cluster", 7) == 0) {
            flat = false;
            // cluster:N forces clusters of N CTAs when every unit's cluster is then resident in one wave
            const int c = force[7] == ':' ? atoi(force + 8) : 0;
            if (c >= 2 && c <= kMaxCluster && units <= max_active[c] && units * c <= dev.sm_count) cs = c;
        }
    }
    cudaError_t e;
    if (flat) {
        p.part = static_cast<float*>(a.scratch);
        p.work = reinterpret_cast<int4*>(p.part + (size_t)2 * kAttnFlatMaxGrid * p.slot_rows * (kD + 2));
        cfg.gridDim = dim3((unsigned)flat_grid, 1, 1);
        cfg.attrs = &attr[1];
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, kAttnKernels[(deal ? 12 : 8) + 2 * spread + paged], qmap, kmap, vmap, p);
        if (e != cudaSuccess) return BP_ERR_CUDA;
        if (a.max_kv_len <= kTileN) return BP_OK;  // every unit is one tile: none is cut between CTAs
        cudaLaunchConfig_t cc = {};
        const int pieces = flat_grid * ((p.slot_rows + kCombRows - 1) / kCombRows);
        cc.gridDim = dim3((unsigned)(deal ? std::min(pieces, kCombPerSm * dev.sm_count) : pieces), 1, 1);
        cc.blockDim = dim3(kCombThreads, 1, 1);
        cc.stream = stream;
        cc.attrs = &attr[1];
        cc.numAttrs = 1;
        e = cudaLaunchKernelEx(&cc, deal ? attn_combine_kernel<true> : attn_combine_kernel<false>, p, flat_grid);
        return e == cudaSuccess ? BP_OK : BP_ERR_CUDA;
    }

    cfg.gridDim = dim3((unsigned)(units * cs), 1, 1);
    // a cluster's partials meet in the workspace where it has the flat split's slots and the rows a CTA owns are
    // at most two a warp, else in shared memory
    if (cs > 1 && (p.slot_rows + cs - 1) / cs <= 2 * kThreads / 32 && units * cs <= 2 * kAttnFlatMaxGrid &&
        a.scratch != nullptr &&
        a.scratch_bytes >= attention_flat_scratch_bytes(a.max_q_len, G))
        p.part = static_cast<float*>(a.scratch);
    // one wave of short runs: dependents start their prologues at once.  Behind a long run an early acceptance waits
    // on the SMs for nothing and its thousands of CTAs start worse for it: 8 x 32784 keys (129 tiles a CTA) with
    // the T = 1 acceptance took 194.2 us a step released at the start and 189.7 at the end; alone, 33 tiles a CTA
    // take 44.8 us either way, 17 tiles 28.0 and 28.4
    p.early_release = units <= max_active[cs] && units * cs <= dev.sm_count && even_tiles < 24 * cs;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kAttnKernels[4 * ahead_for(cs) + 2 * spread + paged], qmap, kmap, vmap, p);
    if (e != cudaSuccess) return BP_ERR_CUDA;
    return BP_OK;
}

namespace {
// One instantiation of the fp32 kernel: its shared-memory opt-in and how many clusters of each size the
// device holds at once, found once per device (from any host thread).
template <int DP, bool VEC>
int run_attention_f32(const F32Params& p, int units, int chunks, const DeviceInfo& dev, cudaStream_t stream) {
    static std::mutex mu;
    static bool configured[64] = {};
    static int max_active[64][kMaxCluster + 1];
    constexpr size_t smem = f32_smem_bytes<DP>();
    auto kern = attn_f32_kernel<DP, VEC>;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.blockDim = dim3(kFThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (dev.device < 0 || dev.device >= 64) return BP_ERR_UNSUPPORTED;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!configured[dev.device]) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                return BP_ERR_CUDA;
            for (int c = 1; c <= kMaxCluster; ++c) {
                cfg.gridDim = dim3((unsigned)c, 1, 1);
                attr[0].val.clusterDim.x = (unsigned)c;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
                    cudaGetLastError();
                    n = 0;
                }
                max_active[dev.device][c] = n;
            }
            configured[dev.device] = true;
        }
    }
    // the widest split of the keys (a chunk per CTA at least) whose clusters are all resident at once
    int cs = 1;
    for (int c = 2; c <= kMaxCluster && c <= chunks; ++c)
        if (units <= max_active[dev.device][c] && (long long)units * c <= dev.sm_count) cs = c;
    cfg.gridDim = dim3((unsigned)(units * cs), 1, 1);
    cfg.stream = stream;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, p) == cudaSuccess ? BP_OK : BP_ERR_CUDA;
}
}  // namespace

int launch_attention_f32(const AttentionArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.head_dim > kF32MaxD) return BP_ERR_UNSUPPORTED;
    if (a.total_q == 0) return BP_OK;
    const int G = a.num_q_heads / a.num_kv_heads;
    F32Params p;
    p.q = static_cast<const float*>(a.q);
    p.k = static_cast<const float*>(a.k);
    p.v = static_cast<const float*>(a.v);
    p.o = static_cast<float*>(a.o);
    p.lse = a.lse;
    p.cu_q = a.cu_q;
    p.cu_kv = a.cu_kv;
    p.hq = a.num_q_heads;
    p.hkv = a.num_kv_heads;
    p.D = a.head_dim;
    p.m_tiles = (int)std::max<long long>(1, ((long long)a.max_q_len * G + kFR - 1) / kFR);
    p.causal = a.mask == BP_MASK_CAUSAL_BLOCK;
    p.scale = a.scale;
    const long long units = (long long)a.num_seqs * a.num_kv_heads * p.m_tiles;
    const int chunks = (a.max_kv_len + kFK - 1) / kFK;
    // Up to one chunk of keys: a warp per row where that is faster, by estimates (us) fitted to 360 shapes timed both
    // ways (1-256 sequences of 5-258 keys, blocks of 1-8, head_dim 32-128): a row's chain and the keys all rows read,
    // against waves of tiles.
    if (chunks <= 1) {
        const double n = std::min(a.max_kv_len, a.total_kv), D = a.head_dim, rows = (double)a.total_q * a.num_q_heads;
        const long long at_once = (a.head_dim <= 64 ? 2LL : 1LL) * dev.sm_count, waves = (units + at_once - 1) / at_once;
        const double filled = std::min((long long)kFR, (long long)a.max_q_len * G) / (double)kFR;
        const double est_rows = 2.0 + (0.19 + 0.002 * D) * n + 4.2e-6 * rows * n * D;
        const double est_tiles =
            waves * (a.head_dim <= 64 ? (waves == 1 ? 4.5 : 4.85) + 1.9 * filled : 5.3 + 3.9 * filled);
        if (est_rows < est_tiles) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[1];
            cfg.gridDim = dim3((unsigned)(((long long)a.total_q * a.num_q_heads + 3) / 4), 1, 1);
            cfg.blockDim = dim3(128, 1, 1);
            cfg.stream = stream;
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, attn_f32_row_kernel, p.q, p.k, p.v, p.o, p.lse, p.cu_q, p.cu_kv, a.num_seqs,
                                      a.total_q, p.hq, p.hkv, p.D, p.causal, p.scale) == cudaSuccess
                       ? BP_OK
                       : BP_ERR_CUDA;
        }
    }
    if (units > INT32_MAX) return BP_ERR_UNSUPPORTED;
    const auto aligned16 = [](const void* x) { return (reinterpret_cast<uintptr_t>(x) & 15) == 0; };
    const bool vec = a.head_dim % 4 == 0 && aligned16(a.q) && aligned16(a.k) && aligned16(a.v) && aligned16(a.o);
    if (a.head_dim <= 64)
        return vec ? run_attention_f32<64, true>(p, (int)units, chunks, dev, stream)
                   : run_attention_f32<64, false>(p, (int)units, chunks, dev, stream);
    return vec ? run_attention_f32<128, true>(p, (int)units, chunks, dev, stream)
               : run_attention_f32<128, false>(p, (int)units, chunks, dev, stream);
}

// --------------------------------------------------------------------------- paged KV append
// Writes each sequence's new K/V rows (its block) into their slots of the paged cache: new row
// i of sequence s is key L_s + i, with L_s = (cu_kv[s+1] - cu_kv[s]) - (cu_new[s+1] - cu_new[s]).
// One warp per (new row, KV head): 16-byte copies of the K row and of the V row.  In a decoding loop this runs
// once a layer between two attentions and is a chain of round trips to L2, not a copy: so the warp's first 32
// copies are loaded ahead of their place, up to 32 sequences' offsets are read in one round instead of a binary
// search, and a single sequence's page is picked from block-table entries loaded with the offsets.
__global__ void __launch_bounds__(256) kv_append_kernel(uint8_t* __restrict__ kc, uint8_t* __restrict__ vc,
                                                        const uint8_t* __restrict__ kn,
                                                        const uint8_t* __restrict__ vn,
                                                        const int32_t* __restrict__ cu_new,
                                                        const int32_t* __restrict__ cu_kv,
                                                        const int32_t* __restrict__ bt, int pages_per_seq,
                                                        int page_shift, int num_seqs, int total_new, int hkv,
                                                        int row_bytes) {
    griddep_launch_dependents();
    griddep_wait();
    const int warp = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (warp >= total_new * hkv) return;
    const int t = warp / hkv, hh = warp % hkv;
    // copy `item`: 16 bytes of the K row, then of the V row
    const int n16 = row_bytes / 16;
    const size_t src = ((size_t)t * hkv + hh) * row_bytes;
    auto from = [&](int item) {
        return reinterpret_cast<const uint4*>(item < n16 ? kn + src + (size_t)item * 16 : vn + src + (size_t)(item - n16) * 16);
    };
    uint4 first = make_uint4(0u, 0u, 0u, 0u);
    if (lane < 2 * n16) first = *from(lane);
    int s = 0, pos, page0 = 0, page1 = 0;
    const bool one = num_seqs == 1;
    if (one) {
        if (lane < pages_per_seq) page0 = __ldg(bt + lane);
        if (lane + 32 < pages_per_seq) page1 = __ldg(bt + lane + 32);
        pos = __ldg(cu_kv + 1) - __ldg(cu_kv) - __ldg(cu_new + 1) + t;
    } else if (num_seqs <= 32) {  // the sequences after the first that start at or before row t, counted
        const int begin = lane < num_seqs ? __ldg(cu_new + lane) : 0, end = lane < num_seqs ? __ldg(cu_new + lane + 1) : 0;
        const int len = lane < num_seqs ? __ldg(cu_kv + lane + 1) - __ldg(cu_kv + lane) : 0;
        s = __popc(__ballot_sync(0xffffffffu, lane > 0 && lane < num_seqs && begin <= t));
        pos = __shfl_sync(0xffffffffu, len - (end - begin) - begin, s) + t;
    } else {
        int lo = 0, hi = num_seqs;  // largest s with cu_new[s] <= t
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(cu_new + mid) <= t) lo = mid; else hi = mid;
        }
        s = lo;
        const int nb = __ldg(cu_new + s + 1) - __ldg(cu_new + s);
        const int len = __ldg(cu_kv + s + 1) - __ldg(cu_kv + s);
        pos = len - nb + (t - __ldg(cu_new + s));
    }
    const int pi = pos >> page_shift;
    long long page;
    if (one && pi < 64) page = __shfl_sync(0xffffffffu, pi < 32 ? page0 : page1, pi & 31);
    else page = __ldg(bt + (size_t)s * pages_per_seq + pi);
    const long long slot = (page << page_shift) + (pos & ((1 << page_shift) - 1));
    const size_t dst = ((size_t)slot * hkv + hh) * row_bytes;
    auto to = [&](int item) {
        return reinterpret_cast<uint4*>(item < n16 ? kc + dst + (size_t)item * 16 : vc + dst + (size_t)(item - n16) * 16);
    };
    if (lane < 2 * n16) *to(lane) = first;
    for (int item = lane + 32; item < 2 * n16; item += 32) *to(item) = *from(item);
}

int launch_kv_append(const KvAppendArgs& a, cudaStream_t stream) {
    if (a.total_new == 0) return BP_OK;
    int shift = 0;
    while ((1 << shift) < a.page_size) ++shift;
    const long long warps = (long long)a.total_new * a.num_kv_heads;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)((warps + 7) / 8), 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kv_append_kernel, static_cast<uint8_t*>(a.k_cache), static_cast<uint8_t*>(a.v_cache),
                              static_cast<const uint8_t*>(a.k_new), static_cast<const uint8_t*>(a.v_new), a.cu_new,
                              a.cu_kv, a.block_table, a.pages_per_seq, shift, a.num_seqs, a.total_new,
                              a.num_kv_heads, a.row_bytes) == cudaSuccess
               ? BP_OK
               : BP_ERR_CUDA;
}

}  // namespace bp
