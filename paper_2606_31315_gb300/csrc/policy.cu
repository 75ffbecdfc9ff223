// Block-size policy head (Sections 2.3-2.4 of the BlockPilot paper): once per request,
//   h = max(0, W1 x + b1),  o = W2 h + b2,  block size = candidates[argmax o].
//
// bf16 weights -- tensor cores (sm_103a).  Inputs of up to 8 atoms per CTA, one launch (policy_tc_kernel):
//   * W1 [hidden x d_in] is cut into 128-row tiles; a thread-block cluster of KS CTAs splits one
//     tile's d_in into 64-column swizzle atoms.  Each CTA brings its W1 atoms in with TMA
//     (SWIZZLE_128B), gathers the requests' pooled rows x (row_index) into the matching
//     K-major layout, and four threads issue M=128 x N=requests tcgen05 MMAs (bf16 in, fp32
//     accumulated in tensor memory): W1 is read from HBM exactly once for up to 64 requests.
//   * The KS partial tiles are summed through distributed shared memory; each CTA takes a
//     share of the rows, adds b1 and applies ReLU, and folds its rows of h straight into the
//     output layer (W2 columns of those rows), so h never goes to global memory.
//   * The cluster's output-layer partials go to the workspace; the last tile to finish (an
//     atomic ticket, no waiting) adds them in tile order with b2 and takes the argmax (lowest
//     index on ties).  Every sum runs in a fixed order: the result is deterministic.
// Wider inputs stream W1 and x through a TMA ring: in the same kernel with one issuing thread, or, where a CTA's share
// is long (policy_flat_kernel), with the atoms of all tiles cut evenly over the SMs.  Pooled rows that row_index picks
// are first gathered into contiguous rows; without row_index the features are read in place.
// fp32 weights -- CUDA cores: register-tiled products with d_in split over a cluster, then (one CTA per
// request) the output layer and the argmax.
// bf16 shapes outside the tensor-core limits -- CUDA cores: a kernel that streams W1 once for a group of up
// to 32 requests (rows staged in shared memory, a warp per hidden row, bias and ReLU fused into the store of
// h), then the same output layer.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <limits.h>

#include <mutex>

#include "common.cuh"
#include "ptx_sm103.cuh"
#include "softmax_math.cuh"

namespace cg = cooperative_groups;

namespace bp {
namespace {

constexpr int kGroup = 32;       // requests per pass over W1
constexpr int kThreads1 = 256;   // 8 warps
constexpr int kRowsPerWarp = 2;
constexpr int kSmemBudget = 160 * 1024;

template <typename T>
struct Vec8;  // 8 consecutive elements as fp32
template <>
struct Vec8<__nv_bfloat16> {
    __device__ __forceinline__ static void load(const __nv_bfloat16* p, float (&f)[8]) {
        const uint4 u = *reinterpret_cast<const uint4*>(p);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};
template <typename T>
__global__ void __launch_bounds__(kThreads1) policy_hidden_kernel(const T* __restrict__ feats, int64_t row_stride,
                                                                  const int32_t* __restrict__ row_index, int n0,
                                                                  int ng, int d_in, const T* __restrict__ w1,
                                                                  const float* __restrict__ b1, int hidden,
                                                                  float* __restrict__ hbuf) {
    extern __shared__ uint8_t smem_raw[];
    T* xs = reinterpret_cast<T*>(smem_raw);  // [ng][d_in]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    griddep_launch_dependents();
    griddep_wait();
    // stage the pooled rows of this request group (16-byte copies)
    const int per_row = d_in * (int)sizeof(T) / 16;
    for (int idx = tid; idx < ng * per_row; idx += kThreads1) {
        const int n = idx / per_row, c = idx % per_row;
        const long long row = row_index ? (long long)row_index[n0 + n] : (long long)(n0 + n);
        reinterpret_cast<uint4*>(xs + (size_t)n * d_in)[c] =
            reinterpret_cast<const uint4*>(feats + row * row_stride)[c];
    }
    __syncthreads();
    const int row_base = (blockIdx.x * (kThreads1 / 32) + warp) * kRowsPerWarp;
    for (int rr = 0; rr < kRowsPerWarp; ++rr) {
        const int j = row_base + rr;
        if (j >= hidden) break;
        float acc[kGroup];
#pragma unroll
        for (int n = 0; n < kGroup; ++n) acc[n] = 0.f;
        const T* wr = w1 + (size_t)j * d_in;
        for (int d = lane * 8; d < d_in; d += 256) {
            float w8[8];
            Vec8<T>::load(wr + d, w8);
#pragma unroll
            for (int n = 0; n < kGroup; ++n) {
                if (n < ng) {
                    float x8[8];
                    Vec8<T>::load(xs + (size_t)n * d_in + d, x8);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[n] = fmaf(w8[e], x8[e], acc[n]);
                }
            }
        }
        float mine = 0.f;
#pragma unroll
        for (int n = 0; n < kGroup; ++n) {
            float v = acc[n];
#pragma unroll
            for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == n) mine = v;
        }
        if (lane < ng) hbuf[(size_t)(n0 + lane) * hidden + j] = fmaxf(0.f, mine + b1[j]);
    }
}

// Output layer and argmax of one request per CTA.  Every thread takes the hidden units 256 apart for up to kOutC
// candidates at a time, kOutUnroll units' loads in flight: what bounds it is the number of round trips to L2.  (fp32,
// 1 x 64 -> 3262 -> 9: 23.2 us a call with a warp per candidate and hidden / 128 rounds, 16.3 with the block on one
// candidate after the other, 8.2 here.)  Dependents launch behind the wait: released at the start, calls back to back
// took 92 us instead of 58 at 32 x 16000 -> 512 and 145 instead of 101 at 64.
constexpr int kOutC = 16, kOutUnroll = 4;
template <typename T>
__global__ void __launch_bounds__(256) policy_out_kernel(const float* __restrict__ hbuf, int hidden,
                                                         const T* __restrict__ w2, const float* __restrict__ b2,
                                                         int num_cand, const int32_t* __restrict__ candidates,
                                                         float* __restrict__ logits_out,
                                                         int32_t* __restrict__ block_size_out) {
    __shared__ float red[8][kOutC], logits[64];
    const int n = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    griddep_wait();
    griddep_launch_dependents();  // (before its wait, a next call's hidden layer settles on the SMs this one's runs on)
    const float* h = hbuf + (size_t)n * hidden;
    for (int c0 = 0; c0 < num_cand; c0 += kOutC) {
        const int nc = min(kOutC, num_cand - c0);
        const T* w = w2 + (size_t)c0 * hidden;
        float acc[kOutC];
#pragma unroll
        for (int c = 0; c < kOutC; ++c) acc[c] = 0.f;
        for (int j0 = tid; j0 < hidden; j0 += 256 * kOutUnroll) {
            float hv[kOutUnroll], wv[kOutUnroll][kOutC];
#pragma unroll
            for (int u = 0; u < kOutUnroll; ++u) {
                const int j = j0 + 256 * u;
                hv[u] = j < hidden ? h[j] : 0.f;
#pragma unroll
                for (int c = 0; c < kOutC; ++c)
                    wv[u][c] = c < nc && j < hidden ? static_cast<float>(w[(size_t)c * hidden + j]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < kOutUnroll; ++u)
#pragma unroll
                for (int c = 0; c < kOutC; ++c) acc[c] = fmaf(wv[u][c], hv[u], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < kOutC; ++c) {
            if (c < nc) {
#pragma unroll
                for (int o = 16; o; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
                if (lane == 0) red[warp][c] = acc[c];
            }
        }
        __syncthreads();
        if (tid < nc) {
            float sum = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) sum += red[k][tid];
            logits[c0 + tid] = sum + b2[c0 + tid];
        }
        __syncthreads();
    }
    if (tid == 0) {
        int best = 0;
        for (int c = 1; c < num_cand; ++c)
            if (logits[c] > logits[best]) best = c;
        block_size_out[n] = candidates[best];
    }
    if (logits_out)
        for (int c = tid; c < num_cand; c += 256) logits_out[(size_t)n * num_cand + c] = logits[c];
}

// ---------------------------------------------------------------- hidden layer, fp32 weights
// A cluster of up to 8 CTAs takes a tile of 64 hidden rows x 32 requests and splits d_in; a CTA streams its
// 32-column chunks of W1 and of the pooled rows through a 4-stage cp.async ring and keeps 4 x 2 outputs per thread
// (fp32 FFMA, in order along its columns).  The partial tiles are summed in rank order through distributed shared
// memory, with b1 and ReLU.  What bounds it: for a few requests the stream of W1, for many the shared-memory reads
// of the products (11 wavefronts a warp for 32 FFMAs).  A warp per hidden row, its requests' rows read whole from
// shared memory for every row of W1, took 8 wavefronts for 8 FFMAs on part of the SMs: with the output layer 20 x
// 4000 -> 1024 went from 81.4 to 23.1 us, 1 x 1024 -> 256 from 13.0 to 7.2, 128 x 8192 -> 3072 from 3350 to 518.
constexpr int kPfRows = 64, kPfReqs = 32, kPfK = 32, kPfStages = 4, kPfMaxKS = 8;
constexpr int kPfLd = kPfK + 4;  // 16-byte reads of 8 consecutive rows fall on distinct banks
constexpr int kPfStageFloats = (kPfRows + kPfReqs) * kPfLd;
constexpr size_t kPfSmem = sizeof(float) * kPfStages * kPfStageFloats;

__global__ void __launch_bounds__(256) policy_f32_hidden_kernel(const float* __restrict__ feats, int64_t row_stride,
                                                                const int32_t* __restrict__ row_index, int num_reqs,
                                                                int d_in, const float* __restrict__ w1,
                                                                const float* __restrict__ b1, int hidden, int g0,
                                                                float* __restrict__ hbuf) {
    extern __shared__ float4 pf_smem[];
    float* ring = reinterpret_cast<float*>(pf_smem);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;  // rows tx + 16 i, requests 2 ty and 2 ty + 1
    griddep_launch_dependents();
    griddep_wait();
    cg::cluster_group cluster = cg::this_cluster();
    const int KS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int j0 = (blockIdx.x / KS) * kPfRows, n0 = (g0 + (int)blockIdx.y) * kPfReqs;
    const int nr = min(kPfRows, hidden - j0), ng = min(kPfReqs, num_reqs - n0);
    const int chunks = (d_in + kPfK - 1) / kPfK;
    const int c0 = (int)((long long)rank * chunks / KS), nc = (int)((long long)(rank + 1) * chunks / KS) - c0;
    // copies of a chunk: thread t's 16 bytes (t % 8) of W1 rows t / 8 and t / 8 + 32 and of request t / 8
    const int lr = tid >> 3, lk = 4 * (tid & 7);
    const bool va = lr < nr, vb = lr + 32 < nr, vx = lr < ng;
    const float* wa = w1 + (size_t)(j0 + (va ? lr : 0)) * d_in;
    const float* wb = w1 + (size_t)(j0 + (vb ? lr + 32 : 0)) * d_in;
    const float* xr = feats + (vx ? (row_index ? (long long)row_index[n0 + lr] : (long long)(n0 + lr)) : 0ll) * row_stride;
    auto load = [&](int c) {
        if (c < nc) {
            const int k = (c0 + c) * kPfK + lk;
            const bool in = k < d_in;
            float* st = ring + (c % kPfStages) * kPfStageFloats + lr * kPfLd + lk;
            cp_async16(st, wa + (in ? k : 0), in && va);
            cp_async16(st + 32 * kPfLd, wb + (in ? k : 0), in && vb);
            cp_async16(st + kPfRows * kPfLd, xr + (in ? k : 0), in && vx);
        }
        cp_async_commit();
    };
    for (int c = 0; c < kPfStages - 1; ++c) load(c);
    float acc[4][2] = {};
    const bool active = 4 * (tid >> 5) < ng;  // the warp's four requests
    for (int c = 0; c < nc; ++c) {
        cp_async_wait_group<kPfStages - 2>();
        __syncthreads();  // chunk c has landed everywhere, and everyone is done with chunk c - 1
        load(c + kPfStages - 1);
        if (active) {
            const float* w = ring + (c % kPfStages) * kPfStageFloats + tx * kPfLd;
            const float* x = ring + (c % kPfStages) * kPfStageFloats + (kPfRows + 2 * ty) * kPfLd;
#pragma unroll
            for (int k = 0; k < kPfK; k += 4) {
                const float4 xa = *reinterpret_cast<const float4*>(x + k);
                const float4 xb = *reinterpret_cast<const float4*>(x + kPfLd + k);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = *reinterpret_cast<const float4*>(w + 16 * i * kPfLd + k);
                    acc[i][0] = fmaf(v.w, xa.w, fmaf(v.z, xa.z, fmaf(v.y, xa.y, fmaf(v.x, xa.x, acc[i][0]))));
                    acc[i][1] = fmaf(v.w, xb.w, fmaf(v.z, xb.z, fmaf(v.y, xb.y, fmaf(v.x, xb.x, acc[i][1]))));
                }
            }
        }
    }
    cp_async_wait_group<0>();
    __syncthreads();
    // the partial tile [request][row], then each CTA its share of the rows
    float* part = ring;
    constexpr int kLdP = kPfRows + 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        part[(2 * ty) * kLdP + tx + 16 * i] = acc[i][0];
        part[(2 * ty + 1) * kLdP + tx + 16 * i] = acc[i][1];
    }
    cluster.sync();
    const int per = (kPfRows + KS - 1) / KS, r0 = rank * per, rows = min(nr, r0 + per) - r0;
    for (int item = tid; item < rows * ng; item += 256) {
        const int r = r0 + item % rows, n = item / rows;
        float v[kPfMaxKS];
#pragma unroll
        for (int q = 0; q < kPfMaxKS; ++q) v[q] = q < KS ? *cluster.map_shared_rank(part + n * kLdP + r, q) : 0.f;
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < kPfMaxKS; ++q) sum += v[q];
        hbuf[(size_t)(n0 + n) * hidden + j0 + r] = fmaxf(0.f, sum + b1[j0 + r]);
    }
    cluster.sync();  // no CTA leaves while a peer may still read its shared memory
}

// ---------------------------------------------------------------- tensor-core path (bf16)
constexpr int kTcM = 128;          // hidden rows per tile: the MMA M
constexpr int kTcMaxN = 64;        // requests per group: the MMA N (padded to a multiple of 16)
constexpr int kTcAtom = 64;        // d_in columns per 128-byte swizzle atom
constexpr int kTcAtomBytes = kTcM * kTcAtom * 2;  // 16 KB of W1 per atom
constexpr int kTcMaxAtoms = 8;     // atoms per CTA when all of them are loaded at once
constexpr int kTcStages = 5;       // ring depth at most, when the atoms of a CTA are streamed (large d_in)
constexpr int kTcMaxKS = 9;        // CTAs per cluster (non-portable above 8)
constexpr int kTcThreads = 128;    // thread t = tile row t = TMEM lane t
constexpr int kTcIssuers = kTcThreads / 32;  // one-shot: warps that issue MMAs, each into its own accumulator
constexpr int kTcMaxSmem = 200 * 1024;

struct PolicyTcParams {
    const __nv_bfloat16* feats;
    int64_t row_stride;
    const int32_t* row_index;
    int num_reqs, d_in, hidden, num_cand;
    int atoms_total, atoms_per_cta, tiles, npad;
    int w_bytes, x_bytes, h_bytes, op_bytes;  // dynamic shared-memory regions
    uint32_t tmem_cols;
    int gathered;  // streamed: the gather kernel came before (it releases this one behind its own wait)
    const float* b1;
    const __nv_bfloat16* w2;
    const float* b2;
    const int32_t* candidates;
    float* logits_out;
    int32_t* block_size_out;
    float* part;    // [groups][tiles][kTcMaxN][num_cand] output-layer partials of each tile
    int* counters;  // [groups] tickets, zero between calls
    unsigned int* err;
};

__device__ __forceinline__ int atomic_add_acq_rel_gpu(int* addr, int v) {
    int old;
    asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], %2;" : "=r"(old) : "l"(addr), "r"(v) : "memory");
    return old;
}

// Gathers the pooled rows of every request group into a contiguous [groups*64][d_in] buffer (rows
// past the last request zero), so that the streamed path can load x with TMA like W1.  (Without a row index
// the feature rows are loaded where they are and nothing is gathered.)  It releases the streamed kernel behind
// its own wait, when every earlier kernel is complete, so that one may load what this one does not write.
__global__ void __launch_bounds__(256) policy_gather_kernel(const __nv_bfloat16* __restrict__ feats,
                                                            int64_t row_stride, const int32_t* __restrict__ row_index,
                                                            int num_reqs, int d_in, int groups, int npad,
                                                            __nv_bfloat16* __restrict__ xg) {
    griddep_wait();
    griddep_launch_dependents();
    const int chunks = d_in / 8;
    const long long total = (long long)groups * npad * chunks;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(idx % chunks);
        const long long gn = idx / chunks;
        const int n = (int)(gn % npad), g = (int)(gn / npad);
        const int req = g * kTcMaxN + n;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (req < num_reqs) {
            const long long row = row_index ? (long long)row_index[req] : (long long)req;
            v = *reinterpret_cast<const uint4*>(feats + row * row_stride + c * 8);
        }
        *reinterpret_cast<uint4*>(xg + (size_t)req * d_in + c * 8) = v;
    }
}

// RING = false: every W1 and x atom of the CTA is loaded at once (x gathered by the CTA itself).
// RING = true: the atoms stream through a ring of S stages of one atom (W1 and the gathered x by TMA),
// for any d_in; thread 0 produces, thread 32 issues the MMAs.  S is compile-time: the producer and the
// issuer are single threads on the critical path of every stage (with S and the atoms per stage as
// runtime values the same ring ran 127.0 instead of 116.8 us at 32 requests x 151936 -> 2048; two
// atoms per stage at half the depth, 256-byte row fetches, measured 127.4 us).
template <bool RING, int S>
__global__ void __launch_bounds__(kTcThreads) policy_tc_kernel(const __grid_constant__ CUtensorMap w1map,
                                                              const __grid_constant__ CUtensorMap xmap,
                                                              const PolicyTcParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sW = base;                                         // W1 atoms, later the partial tile
    uint8_t* sX = base + p.w_bytes;                             // x atoms
    float* hs = reinterpret_cast<float*>(sX + p.x_bytes);       // h of the owned rows [rows][npad]
    float* op = reinterpret_cast<float*>(sX + p.x_bytes + p.h_bytes);  // output-layer partial [n][c]
    float* w2s = op + p.op_bytes / 4;  // W2 columns of the owned rows [c][row]
    __shared__ float b1s[kTcM], b2s[64];
    __shared__ int cands[64];
    __shared__ uint64_t bar_w[kTcMaxAtoms], bar_mma;  // one-shot: an atom's landing; ring: full stages
    __shared__ uint64_t bar_empty[kTcStages];
    __shared__ uint32_t tmem_sh;
    __shared__ int last_sh;

    cg::cluster_group cluster = cg::this_cluster();
    const int KS = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5;
    const int tile = blockIdx.x / KS, g = blockIdx.y;
    const int m0 = tile * kTcM, n0 = g * kTcMaxN;
    const int ng = min(kTcMaxN, p.num_reqs - n0);
    const int npad = p.npad;
    const int a0 = rank * p.atoms_per_cta;
    const int na = max(0, min(p.atoms_total, a0 + p.atoms_per_cta) - a0);
    const int C = p.num_cand;
    const int rpr = (kTcM + KS - 1) / KS;  // rows of the tile owned by each CTA after the split-K sum
    const int rb = rank * rpr;
    const int nr = max(0, min(kTcM, rb + rpr) - rb);

    cluster_arrive_relaxed();  // peers must be running before any distributed shared memory access
    if (tid == 0) {
        prefetch_tensormap(&w1map);
        if (RING) prefetch_tensormap(&xmap);
        const int nb = RING ? S : na;
        for (int a = 0; a < nb; ++a) mbar_init(&bar_w[a], 1);
        if (RING)
            for (int st = 0; st < S; ++st) mbar_init(&bar_empty[st], 1);
        mbar_init(&bar_mma, RING ? 1 : max(1, min(na, kTcIssuers)));  // one commit per issuer
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_sh, p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // The one-shot kernel lets its dependents launch at once; the streamed one, which fills the SMs for longer,
    // once its stream has ended: clusters of a next call placed into what is left of the SMs share some of them
    // while others idle (32 x 151936, calls back to back: 122.3 us released here).
    if (!RING) griddep_launch_dependents();
    const uint32_t tmem = tmem_sh;
    // inputs may come from the previous kernel on the stream; behind the gather kernel only x does
    const bool early = RING && p.gathered && tid < 32;
    if (!early) griddep_wait();
    if (RING) {
        static_assert(!RING || (S >= 2 && S <= kTcStages && S <= kTcMaxAtoms), "ring depth");
        const uint32_t stage_bytes = (uint32_t)(kTcAtomBytes + npad * 128);
        if (tid == 0) {  // producer: W1 and x atoms through the ring
            const int first = min(S, na);
            for (int i = 0; i < first; ++i) {
                mbar_arrive_expect_tx(&bar_w[i], stage_bytes);
                tma_load_2d(sW + i * kTcAtomBytes, &w1map, &bar_w[i], (a0 + i) * kTcAtom, m0);
            }
            if (early) griddep_wait();  // the gathered x
            for (int i = 0; i < first; ++i) tma_load_2d(sX + i * npad * 128, &xmap, &bar_w[i], (a0 + i) * kTcAtom, n0);
            int j = first;
            for (; j < na; ++j) {
                const int st = j % S;
                if (!mbar_wait(&bar_empty[st], ((j / S) - 1) & 1, kWaitBudget)) {
                    raise_error(p.err, kErrTimeout);
                    break;
                }
                mbar_arrive_expect_tx(&bar_w[st], stage_bytes);
                tma_load_2d(sW + st * kTcAtomBytes, &w1map, &bar_w[st], (a0 + j) * kTcAtom, m0);
                tma_load_2d(sX + st * npad * 128, &xmap, &bar_w[st], (a0 + j) * kTcAtom, n0);
            }
            if (j < na)  // wound down early: the copies still in flight land before the CTA moves on
                for (int jj = max(0, j - S); jj < j; ++jj) mbar_wait(&bar_w[jj % S], (jj / S) & 1, kDrainBudget);
        } else if (tid == 32) {  // MMA issuer
            if (na > 0) {
                const uint32_t idesc = idesc_bf16_f32(kTcM, npad, false, false);
                bool ok = true;
                for (int j = 0; j < na; ++j) {
                    const int st = j % S;
                    if (!mbar_wait(&bar_w[st], (j / S) & 1, kWaitBudget)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t wa = smem_addr(sW + st * kTcAtomBytes), xa = smem_addr(sX + st * npad * 128);
#pragma unroll
                    for (int kk = 0; kk < kTcAtom / 16; ++kk)
                        umma_ss(tmem, smem_desc(wa + kk * 32, 16, 1024, kSwizzle128B),
                                smem_desc(xa + kk * 32, 16, 1024, kSwizzle128B), idesc, (j | kk) ? 1u : 0u);
                    umma_commit(&bar_empty[st]);  // the stage is free once these MMAs have read it
                }
                if (!ok) raise_error(p.err, kErrTimeout);
                umma_commit(&bar_mma);
            }
        } else if (warp >= 2) {  // the small operands of the epilogue, while the ring runs
            const int t = tid - 64;
            for (int i = t; i < C * nr; i += kTcThreads - 64) {
                const int c = i / nr, rr = i % nr;
                const int j = m0 + rb + rr;
                w2s[c * rpr + rr] = j < p.hidden ? __bfloat162float(p.w2[(size_t)c * p.hidden + j]) : 0.f;
            }
            for (int rr = t; rr < nr; rr += kTcThreads - 64) b1s[rr] = m0 + rb + rr < p.hidden ? p.b1[m0 + rb + rr] : 0.f;
            if (rank == 0)
                for (int c = t; c < C; c += kTcThreads - 64) {
                    b2s[c] = p.b2[c];
                    cands[c] = p.candidates[c];
                }
        }
        __syncthreads();  // the epilogue operands
    } else {
        // x of the group, K-major SWIZZLE_128B: atom a holds rows n of 128 bytes, 16-byte chunk c of
        // row n stored at chunk c ^ (n & 7); rows past the group and columns past d_in are zero.
        // Asynchronous 16-byte copies: every copy of a thread is in flight at once.  Thread t copies chunk
        // t % 8 of rows t / 8, t / 8 + 16, ...: its rows' indexes load at once and the addresses step by
        // constants (with a division per copy and the indexes through shared memory the copies took 3300
        // cycles to issue, 20% of a call at 32 x 2560).
        const int xc = tid & 7, xn = tid >> 3;
        constexpr int kRows = kTcMaxN / (kTcThreads / 8);  // rows per thread at most
        long long xrow[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int n = xn + 16 * i;
            xrow[i] = n < ng ? (p.row_index ? (long long)p.row_index[n0 + n] : (long long)(n0 + n)) : -1;
        }
        if (tid == 0)
            for (int a = 0; a < na; ++a) {
                mbar_arrive_expect_tx(&bar_w[a], kTcAtomBytes);
                tma_load_2d(sW + a * kTcAtomBytes, &w1map, &bar_w[a], (a0 + a) * kTcAtom, m0);
            }
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int n = xn + 16 * i;
            if (n >= npad) break;
            const __nv_bfloat16* src = p.feats + (xrow[i] < 0 ? 0 : xrow[i] * p.row_stride);
            uint8_t* dst = sX + n * 128 + ((xc ^ (n & 7)) << 4);
            int k = a0 * kTcAtom + xc * 8;
            for (int a = 0; a < na; ++a, k += kTcAtom, dst += npad * 128) {
                const bool valid = xrow[i] >= 0 && k < p.d_in;
                cp_async16(dst, src + (valid ? k : 0), valid);
            }
        }
        cp_async_wait_all();
        fence_proxy_async_smem();  // the MMAs read x through the async proxy
        __syncthreads();
        // A thread of each warp issues the MMAs of atoms warp, warp + 4, ... into the warp's own accumulator: at
        // N = 32 an MMA runs in a few tens of cycles but takes one thread about 120 to issue, so one issuer
        // needed 2400 cycles for 5 atoms.  The four accumulators are added when they are read.
        if ((tid & 31) == 0) {
            const uint32_t idesc = idesc_bf16_f32(kTcM, npad, false, false);
            const uint32_t acc = tmem + (uint32_t)(warp * npad);
            bool ok = true;
            for (int a = warp; a < na && ok; a += kTcIssuers) {
                if (!mbar_wait(&bar_w[a], 0, kWaitBudget)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t wa = smem_addr(sW + a * kTcAtomBytes), xa = smem_addr(sX + a * npad * 128);
#pragma unroll
                for (int kk = 0; kk < kTcAtom / 16; ++kk)
                    umma_ss(acc, smem_desc(wa + kk * 32, 16, 1024, kSwizzle128B),
                            smem_desc(xa + kk * 32, 16, 1024, kSwizzle128B), idesc, (a - warp) | kk ? 1u : 0u);
            }
            if (!ok) {  // the warp's W1 atoms land before the CTA moves on
                raise_error(p.err, kErrTimeout);
                for (int a = warp; a < na; a += kTcIssuers) mbar_wait(&bar_w[a], 0, kDrainBudget);
            }
            if (warp < na) umma_commit(&bar_mma);
        }
        __syncwarp();
        // the small operands of the epilogue, read while the MMAs run
        for (int i = tid; i < C * nr; i += kTcThreads) {
            const int c = i / nr, rr = i % nr;
            const int j = m0 + rb + rr;
            w2s[c * rpr + rr] = j < p.hidden ? __bfloat162float(p.w2[(size_t)c * p.hidden + j]) : 0.f;
        }
        for (int rr = tid; rr < nr; rr += kTcThreads) b1s[rr] = m0 + rb + rr < p.hidden ? p.b1[m0 + rb + rr] : 0.f;
        if (rank == 0)
            for (int c = tid; c < C; c += kTcThreads) {
                b2s[c] = p.b2[c];
                cands[c] = p.candidates[c];
            }
    }
    if (RING && na > 0 && !mbar_wait(&bar_mma, 0, kDrainBudget)) raise_error(p.err, kErrTimeout);
    if (RING) griddep_launch_dependents();
    // ---- this CTA's partial tile row (thread = row = TMEM lane)
    float d[kTcMaxN];
#pragma unroll
    for (int e = 0; e < kTcMaxN; ++e) d[e] = 0.f;
    if (na > 0) {
        if (!mbar_wait(&bar_mma, 0, kDrainBudget)) raise_error(p.err, kErrTimeout);
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < kTcMaxN; c0 += 16) {
            if (c0 < npad) {  // uniform: npad is the same in every thread
                constexpr int kAcc = RING ? 1 : kTcIssuers;  // accumulators, npad columns apart
                uint32_t v[kAcc][16];
#pragma unroll
                for (int w = 0; w < kAcc; ++w)
                    if (w < na) tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(w * npad + c0), v[w]);
                tmem_ld_wait();
#pragma unroll
                for (int w = 0; w < kAcc; ++w)
                    if (w < na) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) d[c0 + e] += __uint_as_float(v[w][e]);
                    }
            }
        }
    }
    // the W1 atoms are consumed: the partial tile takes their place, rows npad + 4 floats apart
    // (an odd number of 16-byte chunks, so the row writes of 8 consecutive threads do not collide)
    float* pd = reinterpret_cast<float*>(sW);
    const int ldp = npad + 4;
#pragma unroll
    for (int c = 0; c < kTcMaxN / 4; ++c)
        if (4 * c < npad)
            *reinterpret_cast<float4*>(pd + tid * ldp + 4 * c) = make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]);
    cluster_wait();  // every peer is running
    cluster_sync_all();  // partial tiles complete and visible
    // ---- owned rows: sum of the KS partials, + b1, ReLU
    for (int item = tid; item < nr * (npad / 4); item += kTcThreads) {
        const int rr = item / (npad / 4), c4 = item % (npad / 4);
        const int row = rb + rr;
        const float4* src = reinterpret_cast<const float4*>(pd + row * ldp + 4 * c4);
        float4 v[kTcMaxKS];  // every remote load in flight at once, then summed in rank order
#pragma unroll
        for (int pr = 0; pr < kTcMaxKS; ++pr)
            v[pr] = pr < KS ? *cluster.map_shared_rank(src, pr) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int pr = 0; pr < kTcMaxKS; ++pr) {
            acc.x += v[pr].x;
            acc.y += v[pr].y;
            acc.z += v[pr].z;
            acc.w += v[pr].w;
        }
        const int j = m0 + row;
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < p.hidden) {
            const float bj = b1s[rr];
            h = make_float4(fmaxf(0.f, acc.x + bj), fmaxf(0.f, acc.y + bj), fmaxf(0.f, acc.z + bj),
                            fmaxf(0.f, acc.w + bj));
        }
        *reinterpret_cast<float4*>(hs + rr * npad + 4 * c4) = h;
    }
    __syncthreads();
    // ---- the owned rows' share of the output layer: op[n][c] = sum_j W2[c][j] h[j][n]
    for (int item = tid; item < ng * C; item += kTcThreads) {
        const int n = item / C, c = item % C;
        const float* w2r = w2s + c * rpr;
        float acc = 0.f;
        for (int rr = 0; rr < nr; ++rr) acc = fmaf(w2r[rr], hs[rr * npad + n], acc);  // zero past hidden
        op[item] = acc;
    }
    cluster_sync_all();  // every CTA's share visible to rank 0
    if (rank == 0) {
        float* dst = p.part + ((size_t)g * p.tiles + tile) * (kTcMaxN * C);
        for (int item = tid; item < ng * C; item += kTcThreads) {
            float v[kTcMaxKS];
#pragma unroll
            for (int pr = 0; pr < kTcMaxKS; ++pr) v[pr] = pr < KS ? *cluster.map_shared_rank(op + item, pr) : 0.f;
            float sum = 0.f;
#pragma unroll
            for (int pr = 0; pr < kTcMaxKS; ++pr) sum += v[pr];
            dst[item] = sum;
        }
        // the CTA barrier orders every thread's partial before thread 0's release (cumulative); its
        // acquire makes the other tiles' partials visible to this CTA once it holds the last ticket
        __syncthreads();
        if (tid == 0) last_sh = atomic_add_acq_rel_gpu(p.counters + g, 1) == p.tiles - 1;
        __syncthreads();
        if (last_sh) {
            // every tile has published: logits in tile order, then the argmax per request
            float* logits = hs;  // this CTA's h is no longer needed (ng * C <= npad * rpr floats)
            const float* base = p.part + (size_t)g * p.tiles * (kTcMaxN * C);
            constexpr int kItems = 3;  // items per thread per round: 48 loads in flight
            for (int i0 = 0; i0 < ng * C; i0 += kItems * kTcThreads) {
                for (int t0 = 0; t0 < p.tiles; t0 += 16) {
                    float v[kItems][16];
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        const int item = i0 + tid + k * kTcThreads;
#pragma unroll
                        for (int u = 0; u < 16; ++u)
                            v[k][u] = item < ng * C && t0 + u < p.tiles
                                          ? __ldcg(base + (size_t)(t0 + u) * (kTcMaxN * C) + item) : 0.f;
                    }
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        const int item = i0 + tid + k * kTcThreads;
                        if (item < ng * C) {
                            float sum = t0 == 0 ? b2s[item % C] : logits[item];
#pragma unroll
                            for (int u = 0; u < 16; ++u) sum += v[k][u];  // tile order
                            logits[item] = sum;
                        }
                    }
                }
            }
            if (p.logits_out)  // the same items as above: each thread reads back its own sums
                for (int item = tid; item < ng * C; item += kTcThreads)
                    p.logits_out[(size_t)n0 * C + item] = logits[item];
            __syncthreads();
            for (int n = tid; n < ng; n += kTcThreads) {
                int best = 0;
                for (int c = 1; c < C; ++c)
                    if (logits[n * C + c] > logits[n * C + best]) best = c;
                p.block_size_out[n0 + n] = cands[best];
            }
            if (tid == 0) p.counters[g] = 0;  // ready for the next call
        }
    }
    cluster_sync_all();  // no CTA leaves while a peer may still read its shared memory
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, p.tmem_cols);
}

// ---------------------------------------------------------------- streamed W1, split flat over the SMs
// For d_in too wide to hold a CTA's share of W1 at once.  The 64-column atoms of every (request group, 128-row
// tile of W1) form one list, cut into equal runs, one per CTA and one CTA per SM (no clusters: 16 clusters of 9
// CTAs never fill 152 SMs, and where they land decides how many share one).  A CTA streams its run through one
// TMA ring; a run that ends or begins inside a tile leaves a partial tile, so every run's part of a tile goes to a
// workspace slot, and the CTA that completes a tile (an atomic ticket, no waiting) adds the tile's parts in run
// order, applies b1, ReLU and its columns of W2; the one that completes the last tile adds the tiles' shares of
// the output layer in tile order and takes the argmax.  Every sum runs in a fixed order.
// What bounds it: HBM, W1 read once (32 x 151936 -> 2048: 632 MB in 108 to 111 us, 5.8 TB/s, about 8 us of it the tail's
// two tickets and sums).  An MMA at N <= 64 costs one thread more to issue than to run, so two warps take the
// stages in turn, each with an accumulator of its own.
constexpr int kFlStages = 8;        // 16 KB of W1 and up to 8 KB of x each
constexpr int kFlThreads = 224;     // warp 0 TMA, warps 1 and 6 MMA, warps 2-5 epilogue (thread = tile row)
constexpr int kFlMaxGrid = 192;
constexpr int kFlC = 16;            // candidates per round of the output layer's reduction

struct PolicyFlatParams {
    PolicyTcParams tc;
    int groups, runs_total;   // request groups; atoms of the whole list
    float4* slots;            // [grid + tiles * groups][npad / 4][128] partial tiles
    int* tile_tickets;        // [groups * tiles], zero between calls
    uint32_t cols;
};

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__global__ void __launch_bounds__(kFlThreads, 1) policy_flat_kernel(const __grid_constant__ CUtensorMap w1map,
                                                                   const __grid_constant__ CUtensorMap xmap,
                                                                   const PolicyFlatParams f) {
    constexpr int S = kFlStages;
    const PolicyTcParams& p = f.tc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[S], empty[S], acc_full[2], acc_empty[2], mma_done;
    __shared__ uint32_t tmem_sh;
    __shared__ int last_sh, ok_sh[4];
    __shared__ float red[4][kFlC][kTcMaxN];  // the warps' sums of one round; the final logits
    __shared__ float w2_sh[kFlC][kTcM];      // a round's columns of W2 (each thread its own row's)

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int npad = p.npad, A = p.atoms_total, C = p.num_cand;
    const int stage_bytes = kTcAtomBytes + npad * 128;
    const int grid = (int)gridDim.x, cta = (int)blockIdx.x;
    const int lo = (int)((long long)cta * f.runs_total / grid), hi = (int)((long long)(cta + 1) * f.runs_total / grid);
    if (tid == 0) {
        prefetch_tensormap(&w1map);
        prefetch_tensormap(&xmap);
        for (int st = 0; st < S; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 2);
            mbar_init(&acc_empty[b], 4);
        }
        mbar_init(&mma_done, 2);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(&tmem_sh, f.cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    griddep_launch_dependents();
    const uint32_t tmem = tmem_sh;
    // inputs may come from the previous kernel on the stream; behind the gather kernel only x does
    const bool early = p.gathered && warp == 0;
    if (!early) griddep_wait();

    if (warp == 0) {
        if (lane == 0) {
            auto issue_w = [&](int J, int i) {
                mbar_arrive_expect_tx(&full[J % S], (uint32_t)stage_bytes);
                tma_load_2d(base + (J % S) * stage_bytes, &w1map, &full[J % S], (i % A) * kTcAtom, (i / A) % p.tiles * kTcM);
            };
            auto issue_x = [&](int J, int i) {
                tma_load_2d(base + (J % S) * stage_bytes + kTcAtomBytes, &xmap, &full[J % S], (i % A) * kTcAtom,
                            i / A / p.tiles * kTcMaxN);
            };
            const int first = min(S, hi - lo);
            for (int J = 0; J < first; ++J) issue_w(J, lo + J);
            if (early) griddep_wait();  // the gathered x
            for (int J = 0; J < first; ++J) issue_x(J, lo + J);
            int issued = first;
            for (int i = lo + first; i < hi; ++i) {
                const int J = i - lo;
                if (!mbar_wait(&empty[J % S], ((J / S) - 1) & 1, kWaitBudget)) {
                    raise_error(p.err, kErrTimeout);
                    break;
                }
                issue_w(J, i);
                issue_x(J, i);
                issued = J + 1;
            }
            if (issued < hi - lo)  // wound down early: the copies still in flight land before the CTA leaves
                for (int J = max(0, issued - S); J < issued; ++J) mbar_wait(&full[J % S], (J / S) & 1, kDrainBudget);
        }
    } else if (warp == 1 || warp == 6) {
        // ---- MMA issuers: stage J goes to issuer J % 2; part sg of a tile accumulates into buffer sg % 2
        if (lane == 0) {
            const int me = warp == 1 ? 0 : 1;
            const uint32_t idesc = idesc_bf16_f32(kTcM, npad, false, false);
            bool ok = true;
            int sg = 0;
            for (int i = lo; i < hi && ok; ++sg) {
                const int end = min(hi, (i / A + 1) * A), b = sg & 1;
                if (sg >= 2 && !mbar_wait(&acc_empty[b], ((sg >> 1) - 1) & 1, kWaitBudget)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)((2 * b + me) * npad);
                uint32_t add = 0u;
                for (int J = i - lo + (((i - lo) & 1) != me); J < end - lo; J += 2) {
                    if (!mbar_wait(&full[J % S], (J / S) & 1, kWaitBudget)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t wa = smem_addr(base + (J % S) * stage_bytes), xa = wa + kTcAtomBytes;
#pragma unroll
                    for (int kk = 0; kk < kTcAtom / 16; ++kk) {
                        umma_ss(acc, smem_desc(wa + kk * 32, 16, 1024, kSwizzle128B),
                                smem_desc(xa + kk * 32, 16, 1024, kSwizzle128B), idesc, add);
                        add = 1u;
                    }
                    umma_commit(&empty[J % S]);  // the stage is free once these MMAs have read it
                }
                if (ok) umma_commit(&acc_full[b]);
                i = end;
            }
            if (!ok) raise_error(p.err, kErrTimeout);
            umma_commit(&mma_done);  // every MMA issued is complete before tensor memory is released
            mbar_wait(&mma_done, 0, kDrainBudget);
        }
    } else {
        // ---- epilogue: thread = tile row = tensor-memory lane (quad * 32 + lane)
        const int quad = warp & 3, row = quad * 32 + lane, et = tid - 64;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
        int sg = 0;
        for (int i = lo; i < hi; ++sg) {
            const int gt = i / A, end = min(hi, (gt + 1) * A), b = sg & 1, natoms = end - i;
            const bool two = natoms > 1;            // both issuers have atoms of this part
            const int only = (i - lo) & 1;          // the one that has, otherwise
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (sg >> 1) & 1, kWaitBudget));
            if (lane == 0) ok_sh[quad] = ok;
            epi_sync();  // the four warps go on or leave together
            if (!(ok_sh[0] && ok_sh[1] && ok_sh[2] && ok_sh[3])) {
                if (et == 0) raise_error(p.err, kErrTimeout);
                break;
            }
            tc_fence_after();
            float4* slot = f.slots + (size_t)(cta + gt) * (npad / 4) * kTcM;
#pragma unroll 1
            for (int c0 = 0; c0 < npad; c0 += 16) {
                uint32_t v0[16], v1[16];
                tmem_ld16(tq + (uint32_t)((2 * b + (two ? 0 : only)) * npad + c0), v0);
                if (two) tmem_ld16(tq + (uint32_t)((2 * b + 1) * npad + c0), v1);
                tmem_ld_wait();
                float x[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = __uint_as_float(v0[e]) + (two ? __uint_as_float(v1[e]) : 0.f);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    slot[(c0 / 4 + e) * kTcM + row] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
            // the parts of this tile: runs j0 .. j1 (run j begins at j * runs_total / grid)
            const long long T = f.runs_total;
            const int j0 = (int)((((long long)gt * A + 1) * grid - 1) / T), j1 = (int)(((long long)(gt + 1) * A * grid - 1) / T);
            epi_sync();  // every thread's part before thread 0's release (cumulative)
            if (et == 0) last_sh = atomic_add_acq_rel_gpu(f.tile_tickets + gt, 1) == j1 - j0;
            epi_sync();
            i = end;
            if (!last_sh) continue;
            // ---- the tile is complete: its parts in run order, + b1, ReLU, its columns of W2
            if (et == 0) f.tile_tickets[gt] = 0;  // ready for the next call
            const int g = gt / p.tiles, tile = gt - g * p.tiles, j = tile * kTcM + row;
            const int ng = min(kTcMaxN, p.num_reqs - g * kTcMaxN);
            const float bias = j < p.hidden ? p.b1[j] : 0.f;
            auto load_w2 = [&](int c0) {  // every load in flight before the first is used
                float w[kFlC];
#pragma unroll
                for (int c = 0; c < kFlC; ++c)
                    w[c] = c0 + c < C && j < p.hidden ? __bfloat162float(p.w2[(size_t)(c0 + c) * p.hidden + j]) : 0.f;
#pragma unroll
                for (int c = 0; c < kFlC; ++c) w2_sh[c][row] = w[c];
            };
            if (C <= kFlC) load_w2(0);
            float* dst = p.part + ((size_t)g * p.tiles + tile) * (kTcMaxN * C);
#pragma unroll 1
            for (int h0 = 0; h0 < npad; h0 += 32) {  // 32 requests at a time
                float h[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) h[e] = 0.f;
                for (int q = j0; q <= j1; q += 4) {  // four parts' loads in flight
                    float4 z[4][8];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            z[u][e] = q + u <= j1 && h0 + 4 * e < npad
                                          ? __ldcg(f.slots + ((size_t)(q + u + gt) * (npad / 4) + h0 / 4 + e) * kTcM + row)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            h[4 * e] += z[u][e].x;
                            h[4 * e + 1] += z[u][e].y;
                            h[4 * e + 2] += z[u][e].z;
                            h[4 * e + 3] += z[u][e].w;
                        }
                }
#pragma unroll
                for (int e = 0; e < 32; ++e) h[e] = j < p.hidden ? fmaxf(0.f, h[e] + bias) : 0.f;
                for (int c0 = 0; c0 < C; c0 += kFlC) {
                    const int nc = min(kFlC, C - c0);
                    if (C > kFlC) load_w2(c0);
#pragma unroll 1
                    for (int c = 0; c < nc; ++c) {  // lane n: the sum over the warp's 32 rows for request h0 + n
                        const float w = w2_sh[c][row];
                        float v[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = h[e] * w;
                        red[quad][c][lane] = reduce_scatter32(v, lane);
                    }
                    epi_sync();
                    for (int k = et; k < nc * 32; k += 128) {
                        const int c = k >> 5, n = h0 + (k & 31);
                        if (n < ng)
                            dst[n * C + c0 + c] = (red[0][c][k & 31] + red[1][c][k & 31]) + (red[2][c][k & 31] + red[3][c][k & 31]);
                    }
                    epi_sync();
                }
            }
            if (et == 0) last_sh = atomic_add_acq_rel_gpu(p.counters + g, 1) == p.tiles - 1;
            epi_sync();
            if (!last_sh) continue;
            // ---- every tile of the group: logits in tile order, then the argmax per request
            if (et == 0) p.counters[g] = 0;  // ready for the next call
            float* logits = &red[0][0][0];   // ng * C <= 64 * 64 floats
            const float* from = p.part + (size_t)g * p.tiles * (kTcMaxN * C);
            for (int k = et; k < ng * C; k += 128) {
                float sum = p.b2[k % C];
                for (int t0 = 0; t0 < p.tiles; t0 += 16) {
                    float v[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u)
                        v[u] = t0 + u < p.tiles ? __ldcg(from + (size_t)(t0 + u) * (kTcMaxN * C) + k) : 0.f;
#pragma unroll
                    for (int u = 0; u < 16; ++u) sum += v[u];
                }
                logits[k] = sum;
                if (p.logits_out) p.logits_out[(size_t)g * kTcMaxN * C + k] = sum;
            }
            epi_sync();
            for (int n = et; n < ng; n += 128) {
                int best = 0;
                for (int c = 1; c < C; ++c)
                    if (logits[n * C + c] > logits[n * C + best]) best = c;
                p.block_size_out[g * kTcMaxN + n] = p.candidates[best];
            }
            epi_sync();
        }
    }
    // ---- release tensor memory
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, f.cols);
}

// Scratch of the tensor-core path: partials and tickets (after the CUDA-core path's h buffer).
size_t tc_part_bytes(int num_reqs, int hidden, int num_cand) {
    const size_t groups = ((size_t)num_reqs + kTcMaxN - 1) / kTcMaxN;
    const size_t tiles = ((size_t)hidden + kTcM - 1) / kTcM;
    return align_up(sizeof(float) * groups * tiles * kTcMaxN * (size_t)num_cand, 256) +
           align_up(sizeof(int) * groups, 256);
}
// The gathered x of the streamed path: [groups * 64][d_in] bf16.
size_t tc_x_bytes(int num_reqs, int d_in) {
    const size_t groups = ((size_t)num_reqs + kTcMaxN - 1) / kTcMaxN;
    return align_up(groups * kTcMaxN * (size_t)d_in * 2, 256);
}

// The flat split's region: its slots and its tile tickets.
size_t flat_slot_bytes(int num_reqs, int hidden) {
    const size_t groups = ((size_t)num_reqs + kTcMaxN - 1) / kTcMaxN, tiles = ((size_t)hidden + kTcM - 1) / kTcM;
    const size_t npad = ((size_t)(num_reqs < kTcMaxN ? num_reqs : kTcMaxN) + 15) / 16 * 16;
    return align_up((kFlMaxGrid + groups * tiles) * kTcM * npad * sizeof(float), 256);
}
size_t flat_bytes(int num_reqs, int hidden) {
    const size_t groups = ((size_t)num_reqs + kTcMaxN - 1) / kTcMaxN, tiles = ((size_t)hidden + kTcM - 1) / kTcM;
    return flat_slot_bytes(num_reqs, hidden) + align_up(groups * tiles * sizeof(int), 256);
}

// The instantiations: the one-shot kernel, then the rings, deepest first (the order of preference).
using TcFn = void (*)(CUtensorMap, CUtensorMap, PolicyTcParams);
struct TcKernel {
    TcFn fn;
    int stages;
};
constexpr int kTcRings = 4;
const TcKernel kTcKernels[1 + kTcRings] = {{policy_tc_kernel<false, 1>, 0}, {policy_tc_kernel<true, 5>, 5},
                                           {policy_tc_kernel<true, 4>, 4}, {policy_tc_kernel<true, 3>, 3},
                                           {policy_tc_kernel<true, 2>, 2}};

// Opt-in shared memory and non-portable cluster sizes, once per device.
int configure_tc(int device) {
    static std::mutex mu;
    static bool configured[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (device >= 0 && device < 64 && configured[device]) return BP_OK;
    for (const TcKernel k : kTcKernels)
        if (cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem) != cudaSuccess ||
            cudaFuncSetAttribute(k.fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return BP_ERR_CUDA;
    if (cudaFuncSetAttribute(policy_flat_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem) != cudaSuccess)
        return BP_ERR_CUDA;
    if (device >= 0 && device < 64) configured[device] = true;
    return BP_OK;
}

// Clusters of ks CTAs of an instantiation with smem bytes of dynamic shared memory each that the device holds at
// once (cached per device, instantiation, cluster size and size).  The occupancy query counts clusters at one CTA
// per SM (on this GB300 it answers 15 nine-CTA clusters at every size); clusters also share SMs when the
// shared memory lets several CTAs fit, so its count is scaled by the CTAs per SM (measured: 16 such
// clusters ran at once at two CTAs per SM, not at one).
int active_clusters(int device, int kernel, int ks, int smem) {
    struct Entry {
        int device, kernel, ks, smem, n;
    };
    static std::mutex mu;
    static Entry cache[256];
    static int used = 0, next = 0;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < used; ++i)
        if (cache[i].device == device && cache[i].kernel == kernel && cache[i].ks == ks && cache[i].smem == smem)
            return cache[i].n;
    cudaLaunchConfig_t probe = {};
    cudaLaunchAttribute pa[1];
    probe.gridDim = dim3((unsigned)ks, 1, 1);
    probe.blockDim = dim3(kTcThreads, 1, 1);
    probe.dynamicSmemBytes = (size_t)smem;
    pa[0].id = cudaLaunchAttributeClusterDimension;
    pa[0].val.clusterDim.x = (unsigned)ks;
    pa[0].val.clusterDim.y = 1;
    pa[0].val.clusterDim.z = 1;
    probe.attrs = pa;
    probe.numAttrs = 1;
    int n = 0, per_sm = 0, reserved = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kTcKernels[kernel].fn, &probe) != cudaSuccess ||
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    const int ctas_per_sm = per_sm / (smem + reserved);
    n *= ctas_per_sm > 1 ? ctas_per_sm : 1;
    cache[next] = Entry{device, kernel, ks, smem, n};  // the oldest entry makes room
    next = (next + 1) % 256;
    used = used < 256 ? used + 1 : 256;
    return n;
}

// Launches the tensor-core path; returns -1 when the shape is outside its limits.
int run_tc(const PolicyArgs& a, const DeviceInfo& dev, float* part, int* counters, __nv_bfloat16* xg, uint8_t* flat,
           cudaStream_t stream) {
    if (reinterpret_cast<uintptr_t>(a.w1) % 16 != 0 || a.num_cand > 64) return -1;
    const int atoms_total = (a.d_in + kTcAtom - 1) / kTcAtom;
    const int tiles = (a.hidden + kTcM - 1) / kTcM;
    const int groups = (a.num_reqs + kTcMaxN - 1) / kTcMaxN;
    const int npad = ((a.num_reqs < kTcMaxN ? a.num_reqs : kTcMaxN) + 15) / 16 * 16;
    // split d_in over as many CTAs as one wave of SMs holds, kTcMaxKS at most
    int ks = dev.sm_count / (tiles * groups);
    ks = ks < 1 ? 1 : ks;
    ks = ks > kTcMaxKS ? kTcMaxKS : ks;
    ks = ks > atoms_total ? atoms_total : ks;
    const bool ring = (atoms_total + ks - 1) / ks > kTcMaxAtoms;  // too many atoms to hold at once: stream them
    const int pd_bytes = kTcM * (npad + 4) * 4;
    const int lg_bytes = kTcMaxN * a.num_cand * 4;  // the last tile's logits reuse the h region
    const int op_bytes = kTcMaxN * a.num_cand * 4;
    const auto h_for = [&](int k) {  // h of the rows a CTA of k owns
        const int h = (kTcM + k - 1) / k * npad * 4;
        return h > lg_bytes ? h : lg_bytes;
    };
    const auto smem_for = [&](int slots, int k) {  // slots: atoms held at once
        const int wb = slots * kTcAtomBytes > pd_bytes ? slots * kTcAtomBytes : pd_bytes;
        return 1024 + wb + slots * npad * 128 + h_for(k) + op_bytes + a.num_cand * ((kTcM + k - 1) / k) * 4;
    };
    // Tensor memory: one accumulator of npad columns, or one per issuer.  A CTA waits for its columns while its
    // cluster peers wait for it: its shared memory keeps what meets on an SM to the columns there are (tmem_share.cuh).
    const int cols = tmem_columns(npad * (ring ? 1 : kTcIssuers));
    const auto launch_smem = [&](int slots, int k) { return (int)tmem_smem(dev, cols, (size_t)smem_for(slots, k)); };
    if (configure_tc(dev.device) != BP_OK) return BP_ERR_CUDA;
    // one-shot: the widest split whose clusters are all resident at once, while a CTA still holds its atoms (a
    // cluster left for a second wave doubles the call: 60 x 2000 -> 3000, 24 tiles, clusters of 6: 27.0 us)
    if (!ring)
        for (int k = ks; k >= 1 && (atoms_total + k - 1) / k <= kTcMaxAtoms; --k) {
            const int sm = launch_smem((atoms_total + k - 1) / k, k);
            if (sm <= kTcMaxSmem && active_clusters(dev.device, 0, k, sm) >= tiles * groups) {
                ks = k;
                break;
            }
        }
    const int per = (atoms_total + ks - 1) / ks;
    const int h_bytes = h_for(ks);
    // ring: the deepest under which every cluster of the grid is resident at once -- a cluster left for
    // a second wave streams its tile alone at a fraction of the bandwidth (measured at 64 requests x
    // 151936 -> 2048: 16 tiles of 9-CTA clusters took 200 us with the 5-stage ring at one CTA per SM);
    // if none, the deepest that fits
    int kernel = 0;  // index into kTcKernels
    // flat split: where a cluster's CTA would stream far more atoms than its share if every SM took part (clusters
    // hold at most 9 CTAs a tile).  Meeting through the workspace costs the equivalent of about 32 atoms, more the
    // more runs meet in a tile (one CTA adds them), and beyond 32 requests the sums' second round.  Fitted to 330
    // shapes timed both ways; atoms per CTA in clusters / flat, and the times in clusters / flat: 4 x 151936 -> 700:
    // 264 / 94, 82.5 / 46.5 us; 17 x 84288 -> 1280: 147 / 87, 51.2 / 47.6; 64 x 151936 -> 700: 264 / 94, 86.6 / 63.4;
    // 64 x 151936 -> 1700: 264 / 219, 96.3 / 107.8; 40 x 50304 -> 256: 88 / 10, 33.5 / 39.5; 40 x 84288 -> 2048: 147 /
    // 139, 65.4 / 71.8; 5 x 32000 -> 1280: 56 / 33, 24.7 / 26.5.
    // And for long runs in place where the clusters outnumber those that get SMs of their own: where they land then
    // decides the time (32 x 151936 -> 2048, 16 clusters of 9: 109 to 121 us, flat 111).  Behind a gather kernel
    // clusters stay the better half (40 x 151936 -> 2048 122.9 and 126.5, 32 -> 2650 144.9 and 152.1).
    const long long atoms_all = (long long)groups * tiles * atoms_total, share = atoms_all / dev.sm_count;
    const long long meet = atoms_total / (share > 0 ? share : 1);  // runs of a tile
    const bool flat_split =
        ring && flat != nullptr && atoms_all <= INT_MAX / 2 &&
        (per >= share + 32 + 3 * meet * npad / 640 + (npad > 32 ? 48 : 0) ||
         (a.row_index == nullptr && per >= 240 && tiles * groups > active_clusters(dev.device, 1, ks, kTcMaxSmem)));
    if (ring && !flat_split) {
        for (int i = 1; i <= kTcRings; ++i) {
            const int sm = launch_smem(kTcKernels[i].stages, ks);
            if (sm > kTcMaxSmem) continue;
            if (kernel == 0) kernel = i;
            if (active_clusters(dev.device, i, ks, sm) >= tiles * groups) {
                kernel = i;
                break;
            }
        }
        if (kernel == 0) return -1;
    }
    const int slots = flat_split ? kFlStages : ring ? kTcKernels[kernel].stages : per;
    const int w_bytes = slots * kTcAtomBytes > pd_bytes ? slots * kTcAtomBytes : pd_bytes;
    const int x_bytes = slots * npad * 128;
    const int flat_cols = tmem_columns(4 * npad);
    const int smem = flat_split ? (int)tmem_smem(dev, flat_cols, 1024 + kFlStages * (kTcAtomBytes + (size_t)npad * 128))
                                : launch_smem(slots, ks);
    if (smem > kTcMaxSmem) return -1;

    CUtensorMap w1map, xmap;
    const cuuint64_t dims[2] = {(cuuint64_t)a.d_in, (cuuint64_t)a.hidden};
    const cuuint64_t strides[1] = {(cuuint64_t)a.d_in * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kTcAtom, (cuuint32_t)kTcM};
    if (encode_tensor_map(&w1map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(a.w1), dims, strides, box,
                          CU_TENSOR_MAP_SWIZZLE_128B) != BP_OK)
        return -1;
    xmap = w1map;  // not read by the one-shot kernel
    const bool gather = ring && a.row_index != nullptr;
    if (ring) {  // the gathered rows, or the feature rows themselves (rows past the last request read zero)
        const cuuint64_t xdims[2] = {(cuuint64_t)a.d_in, gather ? (cuuint64_t)groups * kTcMaxN : (cuuint64_t)a.num_reqs};
        // (a single request's stride is not used and may be any, also more than a map can hold)
        const cuuint64_t xstrides[1] = {(cuuint64_t)(gather || a.num_reqs == 1 ? a.d_in : a.row_stride) * 2};
        const cuuint32_t xbox[2] = {(cuuint32_t)kTcAtom, (cuuint32_t)npad};
        if (encode_tensor_map(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, gather ? xg : const_cast<void*>(a.feats),
                              xdims, xstrides, xbox, CU_TENSOR_MAP_SWIZZLE_128B) != BP_OK)
            return -1;
    }
    PolicyTcParams p;
    p.feats = static_cast<const __nv_bfloat16*>(a.feats);
    p.row_stride = a.row_stride;
    p.row_index = a.row_index;
    p.num_reqs = a.num_reqs;
    p.d_in = a.d_in;
    p.hidden = a.hidden;
    p.num_cand = a.num_cand;
    p.atoms_total = atoms_total;
    p.atoms_per_cta = per;
    p.tiles = tiles;
    p.npad = npad;
    p.w_bytes = w_bytes;
    p.x_bytes = x_bytes;
    p.h_bytes = h_bytes;
    p.op_bytes = op_bytes;
    p.tmem_cols = (uint32_t)cols;
    p.gathered = gather;
    p.b1 = a.b1;
    p.w2 = static_cast<const __nv_bfloat16*>(a.w2);
    p.b2 = a.b2;
    p.candidates = a.candidates;
    p.logits_out = a.logits_out;
    p.block_size_out = a.block_size_out;
    p.part = part;
    p.counters = counters;
    p.err = a.err_word;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    if (gather) {
        const long long total = (long long)groups * npad * (a.d_in / 8);
        long long blocks = (total + 255) / 256;
        const long long cap = 4LL * dev.sm_count;
        cudaLaunchConfig_t gcfg = {};
        gcfg.gridDim = dim3((unsigned)(blocks < cap ? blocks : cap), 1, 1);
        gcfg.blockDim = dim3(256, 1, 1);
        gcfg.stream = stream;
        gcfg.attrs = pdl;
        gcfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&gcfg, policy_gather_kernel, p.feats, a.row_stride, a.row_index, a.num_reqs, a.d_in,
                               groups, npad, xg) != cudaSuccess)
            return BP_ERR_CUDA;
    }
    if (flat_split) {
        PolicyFlatParams f;
        f.tc = p;
        f.groups = groups;
        f.runs_total = groups * tiles * atoms_total;
        f.slots = reinterpret_cast<float4*>(flat);
        f.tile_tickets = reinterpret_cast<int*>(flat + flat_slot_bytes(a.num_reqs, a.hidden));
        f.cols = (uint32_t)flat_cols;
        int ctas = dev.sm_count < kFlMaxGrid ? dev.sm_count : kFlMaxGrid;
        ctas = ctas < f.runs_total ? ctas : f.runs_total;
        cudaLaunchConfig_t fcfg = {};
        fcfg.gridDim = dim3((unsigned)ctas, 1, 1);
        fcfg.blockDim = dim3(kFlThreads, 1, 1);
        fcfg.dynamicSmemBytes = (size_t)smem;
        fcfg.stream = stream;
        fcfg.attrs = pdl;
        fcfg.numAttrs = 1;
        return cudaLaunchKernelEx(&fcfg, policy_flat_kernel, w1map, xmap, f) == cudaSuccess ? BP_OK : BP_ERR_CUDA;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3((unsigned)(tiles * ks), (unsigned)groups, 1);
    cfg.blockDim = dim3(kTcThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl[0];
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kTcKernels[kernel].fn, w1map, xmap, p);
    return e == cudaSuccess ? BP_OK : BP_ERR_CUDA;
}

// The output layer behind a hidden layer in hbuf.
template <typename T>
int run_out(const PolicyArgs& a, const float* hbuf, cudaStream_t stream) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.num_reqs, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, policy_out_kernel<T>, hbuf, a.hidden, static_cast<const T*>(a.w2), a.b2, a.num_cand,
                              a.candidates, a.logits_out, a.block_size_out) == cudaSuccess
               ? BP_OK
               : BP_ERR_CUDA;
}

// bf16 shapes outside the tensor-core limits.
int run_bf16(const PolicyArgs& a, cudaStream_t stream) {
    using T = __nv_bfloat16;
    float* hbuf = static_cast<float*>(a.scratch);
    const int max_group = kSmemBudget / (a.d_in * (int)sizeof(T));
    if (max_group < 1) return BP_ERR_UNSUPPORTED;
    const int group = max_group < kGroup ? max_group : kGroup;
    const int rows_per_block = (kThreads1 / 32) * kRowsPerWarp;
    const unsigned blocks = (unsigned)((a.hidden + rows_per_block - 1) / rows_per_block);
    static std::mutex cfg_mu;
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BP_ERR_CUDA;
    std::lock_guard<std::mutex> cfg_lock(cfg_mu);  // once per device, from any host thread
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(policy_hidden_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget) !=
                cudaSuccess ||
            cudaFuncSetAttribute(policy_hidden_kernel<T>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            return BP_ERR_CUDA;
        configured[dev] = true;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int n0 = 0; n0 < a.num_reqs; n0 += group) {
        const int ng = a.num_reqs - n0 < group ? a.num_reqs - n0 : group;
        cfg.gridDim = dim3(blocks, 1, 1);
        cfg.blockDim = dim3(kThreads1, 1, 1);
        cfg.dynamicSmemBytes = (size_t)ng * a.d_in * sizeof(T);
        if (cudaLaunchKernelEx(&cfg, policy_hidden_kernel<T>, static_cast<const T*>(a.feats), a.row_stride,
                               a.row_index, n0, ng, a.d_in, static_cast<const T*>(a.w1), a.b1, a.hidden,
                               hbuf) != cudaSuccess)
            return BP_ERR_CUDA;
    }
    return run_out<T>(a, hbuf, stream);
}

int run_f32(const PolicyArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.d_in * (long long)sizeof(float) > kSmemBudget) return BP_ERR_UNSUPPORTED;  // the entry point's limit
    float* hbuf = static_cast<float*>(a.scratch);
    static std::mutex cfg_mu;
    static bool configured[64] = {};
    if (dev.device < 0 || dev.device >= 64) return BP_ERR_CUDA;
    {
        std::lock_guard<std::mutex> cfg_lock(cfg_mu);  // once per device, from any host thread
        if (!configured[dev.device]) {
            if (cudaFuncSetAttribute(policy_f32_hidden_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kPfSmem) != cudaSuccess)
                return BP_ERR_CUDA;
            configured[dev.device] = true;
        }
    }
    const int tiles = (a.hidden + kPfRows - 1) / kPfRows, groups = (a.num_reqs + kPfReqs - 1) / kPfReqs;
    const int chunks = (a.d_in + kPfK - 1) / kPfK;
    // d_in split so that about two CTAs reach every SM, with at least two chunks each
    const long long want = 2LL * dev.sm_count / ((long long)tiles * groups);
    int ks = (int)(want < kPfMaxKS ? want : kPfMaxKS);
    ks = ks < chunks / 2 ? ks : chunks / 2;
    ks = ks < 1 ? 1 : ks;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = kPfSmem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    for (int g0 = 0; g0 < groups; g0 += 65535) {  // the grid's y limit
        cfg.gridDim = dim3((unsigned)(tiles * ks), (unsigned)(groups - g0 < 65535 ? groups - g0 : 65535), 1);
        if (cudaLaunchKernelEx(&cfg, policy_f32_hidden_kernel, static_cast<const float*>(a.feats), a.row_stride,
                               a.row_index, a.num_reqs, a.d_in, static_cast<const float*>(a.w1), a.b1, a.hidden, g0,
                               hbuf) != cudaSuccess)
            return BP_ERR_CUDA;
    }
    return run_out<float>(a, hbuf, stream);
}

}  // namespace

size_t policy_scratch_bytes(int num_reqs, int d_in, int hidden, int num_cand, bool full) {
    return align_up(sizeof(float) * (size_t)num_reqs * hidden, 256) + tc_part_bytes(num_reqs, hidden, num_cand) +
           tc_x_bytes(num_reqs, d_in) + (full ? flat_bytes(num_reqs, hidden) : 0);
}

int launch_policy(const PolicyArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.num_reqs == 0) return BP_OK;
    if (a.wdtype == BP_BF16) {
        uint8_t* w = static_cast<uint8_t*>(a.scratch) + align_up(sizeof(float) * (size_t)a.num_reqs * a.hidden, 256);
        float* part = reinterpret_cast<float*>(w);
        const size_t groups = ((size_t)a.num_reqs + kTcMaxN - 1) / kTcMaxN;
        const size_t tiles = ((size_t)a.hidden + kTcM - 1) / kTcM;
        int* counters = reinterpret_cast<int*>(w + align_up(sizeof(float) * groups * tiles * kTcMaxN * (size_t)a.num_cand, 256));
        __nv_bfloat16* xg = reinterpret_cast<__nv_bfloat16*>(w + tc_part_bytes(a.num_reqs, a.hidden, a.num_cand));
        // the flat split's region comes last: a workspace without it streams through clusters
        uint8_t* flat = static_cast<uint8_t*>(a.scratch) + policy_scratch_bytes(a.num_reqs, a.d_in, a.hidden, a.num_cand, false);
        if (a.scratch_bytes < policy_scratch_bytes(a.num_reqs, a.d_in, a.hidden, a.num_cand, true)) flat = nullptr;
        const int rc = run_tc(a, dev, part, counters, xg, flat, stream);
        if (rc != -1) return rc;
        return run_bf16(a, stream);
    }
    return run_f32(a, dev, stream);
}

}  // namespace bp
