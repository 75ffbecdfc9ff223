// Verify epilogue for batches whose logits cannot stay on chip: the LM-head projection of the
// verified (and drafted) positions streamed through tensor memory, with every row's softmax
// statistics formed in the GEMM's epilogue, followed by the throughput acceptance.
//
// Section 2.1 / Figure 1: the target scores every drafted position in one pass and keeps the longest
// prefix the acceptance rule admits; the rule reads p = softmax(W h_t / T) and q = softmax(W h_d / T)
// over the whole vocabulary.  The resident kernel (verify_epilogue.cu) keeps a batch's whole
// [rows, V] accumulator in tensor memory, which bounds it to 64 rows: the GPU's tensor memory holds
// about 39 MB, and 248 rows of a 151,936-entry vocabulary take 151 MB in fp32.  Here:
//   1. lm_head_stream_kernel: one CTA per SM owns an equal contiguous share of the vocabulary,
//      streamed in passes of 256 entries and a last pass of what is left.  Per pass, its W rows (256 entries x 64
//      hidden columns per stage) and the states of
//      up to 256 rows stream through a TMA ring; one thread issues M=128 (state rows) x N=256 (entries)
//      x K=16 tcgen05 MMAs, one per 128-row half of the states.  Tensor-memory lane = state row, so each
//      epilogue thread owns part of one row's entries and folds their logits into a running (max, sum of
//      2^(l*log2e/T - max)) -- at T = 0 its (max, lowest index) -- with one exponential per logit and no
//      exchange between threads until the end.  At T > 0 it also writes the logits once (each warp's 32 x 16
//      half chunk staged in shared memory and sent by one TMA store): the draw at the first rejection needs a
//      whole row pair again, and no on-chip store can hold every row until the decisions are known.
//      At T = 0 nothing but the statistics leaves the chip.  Each CTA writes its slice's statistics
//      of every row.
//   2. The decisions and the draw of accept_batch.cu, whose CTAs first merge the slices' statistics of their
//      sequence's rows in a fixed order: only the draw's row pair per sequence (and the logits at the drafted
//      tokens) is read back.
// Rows beyond 256 go in groups of at most 256, one projection launch per group (W is read once per
// group).  Every wait is bounded; an expired wait sets the workspace error word and the kernel winds
// down after its own copies and MMAs have completed.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "ptx_sm103.cuh"
#include "softmax_math.cuh"

namespace bp {
namespace {

constexpr int kVsN = 256;                // vocabulary entries per pass: the MMA N
constexpr int kVsWBytes = kVsN * 128;    // W of one stage: 256 entries x 128 bytes
constexpr int kVsM = 128;                // state rows per half: the MMA M, tensor-memory lanes
constexpr int kVsAtom = 64;              // hidden columns per 128-byte swizzle atom
constexpr int kVsHBytes = kVsM * 128;    // states of one stage and half: 128 rows x 128 bytes
// Warps 0-15 epilogue, 16 TMA producer, 17 MMA issuer.  Sixteen epilogue warps with 2 KB of staging each hide one
// another's waits for tensor memory and for the stores' reads a little better than eight with 4 KB (hidden 2560,
// 151,936 entries, T = 1: 248 rows 183.1 -> 181.4 us, 62 rows 145.1 -> 143.8).
constexpr int kVsThreads = 576;
constexpr int kVsEpiWarps = 16;
constexpr int kVsProducer = 16, kVsIssuer = 17;

// MT halves of 128 state rows.  Tensor memory (512 columns) holds two passes' accumulators with one
// half -- the epilogue of one pass overlaps the MMAs of the next -- or one pass with two.  (Passes of
// 128 entries would let two halves double-buffer too, but the MMAs' operand reads and the ring's
// fills then ask more of shared memory per entry than it serves: measured slower.)  Stages
// of W and states together: 4 x 48 KB with one half, 3 x 64 KB with two; then the store staging.
__host__ __device__ constexpr int vs_stages(int MT) { return MT == 2 ? 3 : 4; }
// Per epilogue warp: half a chunk of logits (32 rows x 16) where they are written, and at the end its rows' statistics.
__host__ __device__ constexpr int vs_warp_bytes(bool write) { return write ? 32 * 64 : 32 * (int)sizeof(float2); }
template <int MT, bool WRITE>
constexpr size_t vs_smem_bytes() {
    return 1024 + (size_t)vs_stages(MT) * (kVsWBytes + MT * kVsHBytes) + kVsEpiWarps * vs_warp_bytes(WRITE);
}

struct VsParams {
    int vocab, atoms;
    int slice, tail;                // CTA c: entries from c * slice on; entries of a slice's last pass (multiples of 8)
    int nt, nt8, nd;                // the group's target rows, nt rounded up to 8, its drafter rows
    int ht0, hd0;                   // first target / drafter state of the group (TMA row coordinates)
    int row_t0, row_d0;             // their stacked rows (target rows first, then the drafter's)
    float c2;                       // log2(e) / T (0 at T = 0)
    float* logits;                  // [rows][ld] fp32, or null
    int ld;                         // floats from one logits row to the next
    int vec;                        // logits rows start 16-byte aligned
    int tma_store;                  // the group's rows are contiguous stacked rows: chunks go out by TMA
    int grows;                      // stacked rows of the group
    int w_first;                    // W is loaded to leave L2 first
    float2* part;                   // [rows][nslices] slice statistics
    int nslices;
    unsigned int* err;
};

// Named barrier among `count` threads (a multiple of 32) of the CTA.
__device__ __forceinline__ void named_barrier_sync(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Stacked row of row `srow` of the group's state tile (-1: a padding row).
__device__ __forceinline__ int stacked_row(const VsParams& p, int srow) {
    if (srow < p.nt) return p.row_t0 + srow;
    return srow >= p.nt8 && srow < p.nt8 + p.nd ? p.row_d0 + (srow - p.nt8) : -1;
}

// The 32 logits of one chunk of columns folded into a row's running statistics; n valid entries.
// Four interleaved partial results shorten the dependency chains; they merge in a fixed order.
template <bool GREEDY>
__device__ __forceinline__ void fold_chunk(const uint32_t (&r)[32], int n, int v0, float c2, float& a0, float& a1) {
    if (GREEDY) {
        float bv[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        int bi[4] = {INT_MAX, INT_MAX, INT_MAX, INT_MAX};
#pragma unroll
        for (int e = 0; e < 32; ++e) {  // increasing entries per partial: strict > keeps the lowest index
            const float l = __uint_as_float(r[e]);
            if (e < n && l > bv[e & 3]) {
                bv[e & 3] = l;
                bi[e & 3] = v0 + e;
            }
        }
        int ai = __float_as_int(a1);
#pragma unroll
        for (int k = 0; k < 4; ++k) amax_merge(a0, ai, bv[k], bi[k]);
        a1 = __int_as_float(ai);
    } else {
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 32; ++e)
            if (e < n) mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(r[e]));
        const float lm = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        const float mn = fmaxf(a0, __fmul_rn(lm, c2));
        float sm[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 32; ++e)
            if (e < n) sm[e & 3] += ex2(__fmaf_rn(__uint_as_float(r[e]), c2, -mn));
        a1 = __fmaf_rn(a1, ex2d(a0, mn), (sm[0] + sm[1]) + (sm[2] + sm[3]));
        a0 = mn;
    }
}

// Half a chunk, the warp's 32 rows x 16 entries, written to the logits.  Each lane puts its row into the
// warp's 2 KB staging buffer, 16-byte chunk i of row l at chunk i ^ ((l >> 1) & 3) -- the 64-byte swizzle of
// a TMA box of 32 rows x 16 fp32, and a layout in which neither row-wise writes nor column-wise reads
// conflict.  Where the group's rows are contiguous stacked rows (lmap: the group's rows of the logits),
// one TMA store sends the box and the warp goes on (it waits only, before the next half, until the
// copy has read the buffer); otherwise every store instruction covers whole 64-byte pieces of rows: eight rows
// per 16-byte store, two per 4-byte store where rows are not 16-byte aligned.  srow0: the state-tile
// row of lane 0; n valid entries from v0.  Warp-collective.
__device__ __forceinline__ void store_half(uint8_t* stage, const uint32_t* r, int lane, int srow0, const VsParams& p,
                                           const CUtensorMap* lmap, int v0, int n) {
    if (p.tma_store) {
        if (lane == 0) bulk_wait_group_read<0>();  // the previous half's copy has read the buffer
        __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<uint4*>(stage + lane * 64 + ((i ^ ((lane >> 1) & 3)) << 4)) =
            make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
    if (p.tma_store && n == 16) {
        fence_proxy_async_smem();  // the copy reads the buffer through the async proxy
        __syncwarp();
        if (lane == 0 && srow0 < p.grows) {  // rows past the group: clipped
            tma_store_2d(lmap, stage, v0, srow0);
            bulk_commit_group();
        }
        return;
    }
    __syncwarp();
    if (p.vec && n == 16) {
        const int c = lane & 3;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = 8 * k + (lane >> 2);
            const int row = stacked_row(p, srow0 + j);
            const float4 x = *reinterpret_cast<const float4*>(stage + j * 64 + ((c ^ ((j >> 1) & 3)) << 4));
            if (row >= 0) __stcs(reinterpret_cast<float4*>(p.logits + (size_t)row * p.ld + v0) + c, x);
        }
    } else {
        const int e = lane & 15;
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            const int j = 2 * k + (lane >> 4);
            const int row = stacked_row(p, srow0 + j);
            const float x =
                *reinterpret_cast<const float*>(stage + j * 64 + (((e >> 2) ^ ((j >> 1) & 3)) << 4) + ((e & 3) << 2));
            if (row >= 0 && e < n) __stcs(p.logits + (size_t)row * p.ld + v0 + e, x);
        }
    }
    __syncwarp();  // the buffer is free for the next half
}

template <bool GREEDY, int MT, bool WRITE>
__global__ void __launch_bounds__(kVsThreads, 1)
    lm_head_stream_kernel(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap wtail,
                          const __grid_constant__ CUtensorMap htmap, const __grid_constant__ CUtensorMap hdmap,
                          const __grid_constant__ CUtensorMap lmap, const VsParams p) {
    constexpr int STG = vs_stages(MT);
    constexpr int NB = 2 / MT;                     // accumulator buffers of MT x 256 columns
    constexpr int STAGE = kVsWBytes + MT * kVsHBytes;
    constexpr int PARTS = 4 / MT, CW = kVsN / PARTS;  // column parts of a half's epilogue; columns of a warp per pass
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sbase = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[STG], empty[STG], acc_full[NB], acc_empty[NB], mma_done;
    __shared__ uint32_t tmem_sh;

    griddep_launch_dependents();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c = (int)blockIdx.x;
    const int e0 = c * p.slice, e1 = min(p.vocab, e0 + p.slice);  // the slice's entries [e0, e1)
    const int npass = (e1 - e0 + kVsN - 1) / kVsN, tail_pass = (p.slice - 1) / kVsN;
    const int J = npass * p.atoms;  // ring stages of this CTA

    if (tid == 0) {
        prefetch_tensormap(&wmap);
        prefetch_tensormap(&wtail);
        if (p.nt) prefetch_tensormap(&htmap);
        if (p.nd) prefetch_tensormap(&hdmap);
        if (WRITE && p.tma_store) prefetch_tensormap(&lmap);
        for (int st = 0; st < STG; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        for (int b = 0; b < NB; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kVsEpiWarps);
        }
        mbar_init(&mma_done, 1);
        fence_mbar_init();
    }
    if (warp == kVsIssuer) {
        tmem_alloc(&tmem_sh, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    griddep_wait();  // the states (and the scratch the previous call's kernels read) come from earlier kernels

    if (warp == kVsProducer) {
        // ---- TMA producer: stage j = (pass j / atoms, hidden atom j % atoms): 256 W rows, the group's states
        if (lane == 0) {
            int issued = 0;
            const uint64_t pol = p.w_first ? l2_policy_evict_first() : l2_policy_normal();
            for (int j = 0; j < J; ++j) {
                const int st = j % STG;
                if (j >= STG && !mbar_wait(&empty[st], ((j / STG) - 1) & 1, kWaitBudget)) {
                    raise_error(p.err, kErrTimeout);
                    break;
                }
                const int pp = j / p.atoms, a = j - pp * p.atoms;
                uint8_t* sw = sbase + st * STAGE;
                uint8_t* sh = sw + kVsWBytes;
                // a slice's last pass has `tail` entries; the rest of its stage keeps older rows, whose columns of
                // the accumulator nobody reads
                const bool last = pp == tail_pass;
                mbar_arrive_expect_tx(&full[st], (uint32_t)(((last ? p.tail : kVsN) + p.nt + p.nd) * 128));
                tma_load_2d_hint(sw, last ? &wtail : &wmap, &full[st], a * kVsAtom, e0 + pp * kVsN, pol);
                if (p.nt) tma_load_2d(sh, &htmap, &full[st], a * kVsAtom, p.ht0);
                if (p.nd) tma_load_2d(sh + p.nt8 * 128, &hdmap, &full[st], a * kVsAtom, p.hd0);
                issued = j + 1;
            }
            if (issued < J)  // wound down early: let the copies still in flight land before exiting
                for (int j = max(0, issued - STG); j < issued; ++j)
                    mbar_wait(&full[j % STG], (j / STG) & 1, kDrainBudget);
        }
    } else if (warp == kVsIssuer) {
        // ---- MMA issuer: pass pp accumulates into buffer pp % NB; half m of the states into its own 256 columns
        if (lane == 0) {
            const uint32_t idesc_full = idesc_bf16_f32(kVsM, kVsN, false, false);
            const uint32_t idesc_tail = idesc_bf16_f32(kVsM, (p.tail + 15) / 16 * 16, false, false);
            bool ok = true;
            int j = 0;
            for (int pp = 0; pp < npass && ok; ++pp) {
                const int b = pp % NB;
                if (pp >= NB && !mbar_wait(&acc_empty[b], ((pp / NB) - 1) & 1, kWaitBudget)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t idesc = pp == tail_pass ? idesc_tail : idesc_full;
                const uint32_t dcol = tmem + (uint32_t)(b * MT * kVsN);
                for (int a = 0; a < p.atoms; ++a, ++j) {
                    const int st = j % STG;
                    if (!mbar_wait(&full[st], (j / STG) & 1, kWaitBudget)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t wa = smem_addr(sbase + st * STAGE), ha = wa + kVsWBytes;
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int kk = 0; kk < kVsAtom / 16; ++kk)
                            umma_ss(dcol + (uint32_t)(m * kVsN),
                                    smem_desc(ha + m * kVsHBytes + kk * 32, 16, 1024, kSwizzle128B),
                                    smem_desc(wa + kk * 32, 16, 1024, kSwizzle128B), idesc, (a | kk) ? 1u : 0u);
                    umma_commit(&empty[st]);  // the stage is free once these MMAs have read it
                }
                if (ok) umma_commit(&acc_full[b]);
            }
            if (!ok) raise_error(p.err, kErrTimeout);
            umma_commit(&mma_done);  // every MMA issued is complete before tensor memory is released
            mbar_wait(&mma_done, 0, kDrainBudget);
        }
    } else {
        // ---- epilogue: thread = state row (tensor-memory lane); warp w reads lane quarter w % 4 of half
        // (w / 4) % MT, and of its columns part w / (4 MT)
        const int q = warp & 3, m = (warp >> 2) % MT, part = (warp >> 2) / MT, cb = part * CW;
        const int srow0 = m * kVsM + q * 32;  // state-tile row of lane 0
        const int row = stacked_row(p, srow0 + lane);
        float a0 = -INFINITY, a1 = GREEDY ? __int_as_float(INT_MAX) : 0.f;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * kVsN + cb);
        uint8_t* stage = sbase + STG * STAGE + warp * vs_warp_bytes(WRITE);
        bool ok = true;
        for (int pp = 0; pp < npass; ++pp) {
            const int b = pp % NB;
            ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (pp / NB) & 1, kWaitBudget));
            if (!ok) break;
            tc_fence_after();
            const int vb = e0 + pp * kVsN + cb;  // entry of the warp's first column
#pragma unroll 1
            for (int c0 = 0; c0 < CW; c0 += 32) {
                const int v0 = vb + c0, n = min(32, e1 - v0);
                if (n <= 0) break;
                uint32_t r[32];
                tmem_ld32(tq + (uint32_t)(b * MT * kVsN + c0), r);
                tmem_ld_wait();
                if (WRITE) store_half(stage, r, lane, srow0, p, &lmap, v0, min(n, 16));
                if (row >= 0) fold_chunk<GREEDY>(r, n, v0, p.c2, a0, a1);
                if (WRITE && n > 16) store_half(stage, r + 16, lane, srow0, p, &lmap, v0 + 16, n - 16);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
        if (WRITE && p.tma_store && lane == 0) bulk_wait_group<0>();  // this warp's logits are written
        if (!ok && lane == 0) raise_error(p.err, kErrTimeout);
        // the column parts of a row, merged in entry order
        __syncwarp();
        reinterpret_cast<float2*>(stage)[lane] = make_float2(a0, a1);
        named_barrier_sync(1, kVsEpiWarps * 32);
        if (part == 0 && row >= 0) {
#pragma unroll
            for (int k = 1; k < PARTS; ++k) {
                const float2 o = reinterpret_cast<const float2*>(stage + k * 4 * MT * vs_warp_bytes(WRITE))[lane];
                if (GREEDY) {
                    int bi = __float_as_int(a1);
                    amax_merge(a0, bi, o.x, __float_as_int(o.y));
                    a1 = __int_as_float(bi);
                } else {
                    lse_merge(a0, a1, o.x, o.y);
                }
            }
            p.part[(size_t)row * p.nslices + c] = make_float2(a0, a1);
        }
    }

    // ---- release tensor memory
    tc_fence_before();
    __syncthreads();
    if (warp == kVsIssuer) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

template <bool GREEDY, int MT, bool WRITE>
int vs_launch(const CUtensorMap& wmap, const CUtensorMap& wtail, const CUtensorMap& htmap, const CUtensorMap& hdmap,
              const CUtensorMap& lmap, const VsParams& p, int grid, const DeviceInfo& dev, cudaStream_t stream) {
    static std::mutex cfg_mu;  // per instantiation (a template's own statics)
    static int configured[64] = {};
    const size_t smem = tmem_smem(dev, kTmemColumns, vs_smem_bytes<MT, WRITE>());
    if (dev.device >= 0 && dev.device < 64) {
        std::lock_guard<std::mutex> cfg_lock(cfg_mu);  // once per device, from any host thread
        if (!configured[dev.device]) {
            if (cudaFuncSetAttribute(lm_head_stream_kernel<GREEDY, MT, WRITE>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
                return BP_ERR_CUDA;
            configured[dev.device] = 1;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kVsThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // the set-up overlaps the previous kernel
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, lm_head_stream_kernel<GREEDY, MT, WRITE>, wmap, wtail, htmap, hdmap, lmap, p) ==
                   cudaSuccess
               ? BP_OK
               : BP_ERR_CUDA;
}

template <bool GREEDY>
int vs_dispatch(int mt, bool write, const CUtensorMap& wmap, const CUtensorMap& wtail, const CUtensorMap& htmap,
                const CUtensorMap& hdmap, const CUtensorMap& lmap, const VsParams& p, int grid, const DeviceInfo& dev,
                cudaStream_t stream) {
    if (mt == 2)
        return write ? vs_launch<GREEDY, 2, true>(wmap, wtail, htmap, hdmap, lmap, p, grid, dev, stream)
                     : vs_launch<GREEDY, 2, false>(wmap, wtail, htmap, hdmap, lmap, p, grid, dev, stream);
    return write ? vs_launch<GREEDY, 1, true>(wmap, wtail, htmap, hdmap, lmap, p, grid, dev, stream)
                 : vs_launch<GREEDY, 1, false>(wmap, wtail, htmap, hdmap, lmap, p, grid, dev, stream);
}

int encode_rows(CUtensorMap* map, const void* base, int hidden, int rows, int box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)hidden, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)hidden * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kVsAtom, (cuuint32_t)box_rows};
    return encode_tensor_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                             CU_TENSOR_MAP_SWIZZLE_128B);
}

}  // namespace

// Entries per CTA: equal shares of the vocabulary, in eights (the swizzle's rows).  Runs of whole passes left SMs idle
// at the end: of 151,936 entries 138 CTAs had 4 passes and 14 had 3 (8 x 16 rows, hidden 2560, T = 0: 122.2 -> 116.5
// us), of 50,257 entries 45 had 2 and 107 had 1 (8 x 31 rows, T = 1: 82.4 -> 77.0 us).  Shares are a pass at least
// where that gives three quarters of the SMs one -- every CTA reads all states, so more CTAs cost L2 traffic (8 x 31
// rows, T = 1, 32,000 entries: 125 CTAs 50.2, 152 CTAs 50.9 us; 28,000: 110 CTAs 47.7, 152 CTAs 45.5) -- and go down
// to 64 entries below that (8,192: 32 CTAs 39.3, 128 CTAs 30.7 us).
static int verify_stream_slice(int vocab, int sm_count) {
    const int sms = min(sm_count, kMaxSlices), passes = (vocab + kVsN - 1) / kVsN;
    const int ctas = min(sms, 4 * passes > 3 * sms ? passes : (vocab + 63) / 64);
    return ctas < 1 ? 0 : (int)(((long long)vocab + ctas * 8 - 1) / (ctas * 8) * 8);
}
int verify_stream_grid(int vocab, int sm_count) {
    const int slice = verify_stream_slice(vocab, sm_count);
    return slice < 1 ? 0 : (vocab + slice - 1) / slice;
}

// When W is loaded to leave L2 first.  Without logits to write, in the last group of rows, which reads W for the last
// time (64 rows, 128,256 x 1024: 46.8 us with, 47.8 without; 320 rows, 100,352 x 1024 in two groups: 78.3 in both, 75.9
// in the last, 79.7 in none).  With logits, where a CTA has one or two passes: the group's logits wait in L2 for their
// way to memory (120 rows, 40,000 x 1536: 39.7 and 43.2; 620 rows, 50,257 x 2560 192.8 and 200.4); with more passes the
// write-back keeps up and the hint costs second reads of W (120 rows, 151,936 x 896: 71.3 and 67.5; 128,256 x 1024 68.2
// and 65.3; 100,352 x 1024 53.5 and 53.2), but for two halves of rows on a head several times their logits (248 rows,
// 151,936 x 2560: 184.3 and 186.1).  And not where W and the logits stay in L2 from call to call (120 rows, 32,000
// x 1024: 24.2 and 19.6; 40,000 x 896 29.2 and 25.4).  Timed over 260 shapes of 48 to 1240 rows.
static bool w_leaves_first(bool write, bool last_group, int rows, int slice, long long w_bytes, long long logits_bytes) {
    if (!write) return last_group;
    return w_bytes + logits_bytes > (95LL << 20) &&
           (slice <= 2 * kVsN || (rows > kVsM && w_bytes >= 4 * logits_bytes));
}

int launch_verify_stream(const VerifyEpilogueArgs& a, const VerifyStreamScratch& s, const DeviceInfo& dev,
                         cudaStream_t stream) {
    const bool greedy = a.temperature == 0.f;
    const int rows_t = a.total_draft + a.num_seqs;
    const int rows = rows_t + (greedy ? 0 : a.total_draft);
    float* logits = a.logits_out ? a.logits_out : (greedy ? nullptr : s.logits);
    const bool write = logits != nullptr;
    const int grid = verify_stream_grid(a.vocab, dev.sm_count);
    if (grid < 1 || a.hidden % kVsAtom != 0) return BP_ERR_UNSUPPORTED;

    CUtensorMap wmap, wtail, htmap, hdmap, lmap;
    VsParams p;
    p.vocab = a.vocab;
    p.atoms = a.hidden / kVsAtom;
    p.slice = verify_stream_slice(a.vocab, dev.sm_count);
    p.tail = p.slice - (p.slice - 1) / kVsN * kVsN;
    if (encode_rows(&wmap, a.lm_head, a.hidden, a.vocab, kVsN) != BP_OK ||
        encode_rows(&wtail, a.lm_head, a.hidden, a.vocab, p.tail) != BP_OK)
        return BP_ERR_CUDA;
    p.c2 = greedy ? 0.f : 1.4426950408889634f / a.temperature;
    p.logits = logits;
    // the path's own rows are padded to 16-byte boundaries where the workspace has the room (8 x 31 rows of a
    // 50257-entry vocabulary: 115 -> 86 us); the caller's logits_out has rows of exactly the vocabulary
    const int ld = a.logits_out ? a.vocab : s.ld;
    p.ld = ld;
    p.vec = write && ld % 4 == 0 && reinterpret_cast<uintptr_t>(logits) % 16 == 0;
    p.part = s.part;
    p.nslices = grid;
    p.err = a.err_word;
    // groups of at most 256 stacked rows; a group that holds both kinds keeps its drafter rows at an
    // 8-row boundary of the state tile (the 1024-byte swizzle atom), so it may hold a few rows less
    for (int r0 = 0; r0 < rows;) {
        int r1 = min(rows, r0 + 2 * kVsM);
        if (r0 < rows_t && r1 > rows_t) {
            const int nt = rows_t - r0, nt8 = (nt + 7) & ~7;
            if (nt8 + (r1 - rows_t) > 2 * kVsM) r1 -= nt8 - nt;
        }
        p.nt = max(0, min(r1, rows_t) - r0);
        p.nt8 = (p.nt + 7) & ~7;
        p.nd = max(0, r1 - max(r0, rows_t));
        p.ht0 = r0;
        p.row_t0 = r0;
        p.hd0 = max(r0, rows_t) - rows_t;
        p.row_d0 = max(r0, rows_t);
        if (p.nt && encode_rows(&htmap, a.h_target, a.hidden, rows_t, p.nt) != BP_OK) return BP_ERR_CUDA;
        if (p.nd && encode_rows(&hdmap, a.h_draft, a.hidden, a.total_draft, p.nd) != BP_OK) return BP_ERR_CUDA;
        const int mt = p.nt8 + p.nd > kVsM ? 2 : 1;
        // TMA stores where state-tile row i is stacked row r0 + i for every row the group holds
        p.tma_store = p.vec && (p.nt % 8 == 0 || p.nd == 0);
        p.grows = r1 - r0;
        p.w_first = w_leaves_first(write, r1 >= rows, r1 - r0, p.slice, (long long)a.vocab * a.hidden * 2,
                                   (long long)(r1 - r0) * ld * 4);
        if (p.tma_store) {
            const cuuint64_t dims[2] = {(cuuint64_t)a.vocab, (cuuint64_t)(r1 - r0)};
            const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
            const cuuint32_t box[2] = {16, 32};
            if (encode_tensor_map(&lmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, logits + (size_t)r0 * ld, dims,
                                  strides, box, CU_TENSOR_MAP_SWIZZLE_64B) != BP_OK)
                return BP_ERR_CUDA;
        }
        const CUtensorMap& ht = p.nt ? htmap : wmap;  // an unused map slot holds any valid map
        const CUtensorMap& hd = p.nd ? hdmap : wmap;
        const CUtensorMap& lm = p.tma_store ? lmap : wmap;
        const int rc = greedy ? vs_dispatch<true>(mt, write, wmap, wtail, ht, hd, lm, p, grid, dev, stream)
                              : vs_dispatch<false>(mt, write, wmap, wtail, ht, hd, lm, p, grid, dev, stream);
        if (rc != BP_OK) return rc;
        r0 = r1;
    }

    AcceptArgs aa;
    aa.target = logits;
    aa.draft = logits ? logits + (size_t)rows_t * ld : nullptr;
    aa.tokens = a.tokens;
    aa.cu_draft = a.cu_draft;
    aa.num_seqs = a.num_seqs;
    aa.total_draft = a.total_draft;
    aa.vocab = a.vocab;
    aa.temperature = a.temperature;
    aa.u_accept = a.u_accept;
    aa.u_sample = a.u_sample;
    aa.n_accepted = a.n_accepted;
    aa.out_tokens = a.out_tokens;
    aa.accept_prob = a.accept_prob;
    aa.scratch = nullptr;
    aa.err_word = a.err_word;
    return launch_accept_slices(aa, ld, s.part, grid, dev.sm_count, s.tickets, s.draw, stream);
}

}  // namespace bp
