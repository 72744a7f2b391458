// logits.cu -- Alg. 1's v' = m (.) v and the decode of given masks (sm_103a):
// masked argmax / log-sum-exp / log-probabilities and Gumbel-max draws, and
// the allocation-free entry point.
//
// logits_kernel   one CTA per row, or a cluster of up to 8 that share out the
//                 row's mask words while the rows alone leave SMs idle; the
//                 slices' results are merged through the cluster's shared
//                 memory, and every CTA then writes its slice's
//                 log-probabilities (decode.cuh).
// logits_gather_kernel  one CTA per row for batches of more rows than SMs:
//                 a compacted gather of the allowed logits.
// logprobs_kernel the log-probabilities alone, given the rows' log-sum-exp.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>

#include "decode.cuh"
#include "domino_internal.h"

namespace domino {
namespace {

constexpr int kLogitsSegment = 4096;     // mask words in shared memory at a time (33 KB a CTA in all)
constexpr int kLogitsMaxDevices = 64;

// Where row r's mask words are: row r of `base` ([batch][W]), or, for the
// table-driven step, row states[r] of a precomputed [Q][W] state table.  An
// out-of-range state reads as an all-zero row (nothing allowed) and sets the
// error word.
struct MaskRows {
    const uint32_t* base;       // nullptr (and no row_state): every token allowed
    const int32_t* row_state;   // nullptr: base is [batch][W]
    int32_t Q;
    uint32_t* err;
    __device__ __forceinline__ bool all() const { return base == nullptr; }
    __device__ __forceinline__ const uint32_t* row(int r, int W, bool report) const {
        if (all()) return nullptr;
        if (!row_state) return base + (size_t)r * W;
        const int32_t q = __ldg(row_state + r);
        if (q < 0 || q >= Q) {
            if (report) atomicOr(err, DOMINO_DEVERR_BAD_STATE);
            return nullptr;
        }
        return base + (size_t)q * W;
    }
    // word j of a row given by row(); all-allowed rows read as all ones
    __device__ __forceinline__ uint32_t word(const uint32_t* mrow, int j) const {
        return all() ? 0xFFFFFFFFu : (mrow ? __ldg(mrow + j) : 0u);
    }
};

struct LogitsArgs {
    const void* logits;
    int64_t stride;
    MaskRows mask;
    int32_t V, W, batch;
    int32_t slices, slice_words;   // CTAs per row, mask words of each (a multiple of 4)
    int32_t segment;               // mask words held at a time (a multiple of 4)
    int32_t* argmax;
    float* lse;
    float* logprobs;
    SampleArgs sample;
};

// Words [w0, w0 + n) of a row's mask into shared memory, a zero word on either
// side and no bits past V.  Every thread of the CTA calls it; ends with a
// barrier.
__device__ __forceinline__ void stage_mask(uint32_t* s_mask, const MaskRows& mask, const uint32_t* mrow, int w0, int n,
                                           int V, int tid) {
    if (mrow && (reinterpret_cast<uintptr_t>(mrow + w0) & 15) == 0 && (n & 3) == 0) {
#pragma unroll 2
        for (int j = tid; j < n / 4; j += kDecodeThreads)
            reinterpret_cast<uint4*>(s_mask)[j] = __ldg(reinterpret_cast<const uint4*>(mrow + w0) + j);
    } else {
#pragma unroll 4
        for (int j = tid; j < n; j += kDecodeThreads)
            s_mask[j] = mask.all() ? 0xFFFFFFFFu : mrow ? __ldg(mrow + w0 + j) : 0u;
    }
    if (tid == 0) s_mask[-1] = s_mask[n] = 0u;
    __syncthreads();
    const int left = V - 32 * (w0 + n - 1);   // tokens of the last word
    if (left < 32) {
        if (tid == 0) s_mask[n - 1] &= (1u << left) - 1u;
        __syncthreads();
    }
}

// the mask words with a zero word on either side, then the lists
__host__ __device__ inline int logits_mask_smem(int segment) { return 32 + segment * 4; }
__host__ __device__ inline int logits_smem(int segment) { return logits_mask_smem(segment) + kDecodeListBytes; }

template <bool BF16, int FOLD>
__global__ void __launch_bounds__(kDecodeThreads, 2)
    logits_kernel(const __grid_constant__ LogitsArgs a, const RowList list) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ DecodeShared sh;
    __shared__ uint4 s_keep[BF16 && FOLD != kFoldSample ? kDecodeKeep : 1];
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + 16);   // a zero word on either side
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint16_t* s_list = reinterpret_cast<uint16_t*>(smem + logits_mask_smem(a.segment)) + warp * kDecodeList;
    const int r = blockIdx.x / a.slices, slice = blockIdx.x - r * a.slices;
    if (BF16 && FOLD != kFoldSample) fill_keep(s_keep, tid);
    pdl_wait();
    pdl_trigger();
    if (r >= list.rows(a.batch)) return;   // the whole cluster
    const int w0 = slice * a.slice_words, w1 = min(a.W, w0 + a.slice_words);
    const uint32_t* mrow = a.mask.row(r, a.W, tid == 0 && slice == 0);
    const int orow = list.row(r);   // the batch row: logits, outputs and the sampling counter
    Decoder<BF16, FOLD> d;
    d.init(a.logits, a.stride, orow, a.V, a.logprobs != nullptr, a.sample, s_keep, lane);
    for (int j = w0; j < w1; j += a.segment) {
        const int n = min(a.segment, w1 - j);
        if (j > w0) __syncthreads();   // the segment before has been read
        stage_mask(s_mask, a.mask, mrow, j, n, a.V, tid);
        d.slice(s_mask, 32 * j, min(32 * n, a.V - 32 * j), s_list, warp);
    }
    d.finish();
    float m = d.m, s = d.s;
    int idx = d.idx;
    decode_combine(sh, m, idx, s, a.slices, lane, warp);
    const float lse = FOLD == kFoldLse ? log_sum_exp(m, s) : 0.0f;
    if (tid == 0 && slice == 0) {
        a.argmax[orow] = m == -INFINITY ? -1 : idx;
        if (FOLD == kFoldLse && a.lse) a.lse[orow] = lse;
    }
    if constexpr (FOLD == kFoldLse) {
        if (a.logprobs) {
            for (int j = w0; j < w1; j += a.segment) {
                const int n = min(a.segment, w1 - j);
                if (w1 - w0 > a.segment) {   // more than one: staged again
                    __syncthreads();
                    stage_mask(s_mask, a.mask, mrow, j, n, a.V, tid);
                }
                write_logprobs<BF16>(d.lrow, a.V, s_mask, 32 * j, min(32 * n, a.V - 32 * j), lse,
                                     a.logprobs + (size_t)orow * a.V, tid);
            }
        }
    }
    if (a.slices > 1) cluster_wait();
}

// The log-probabilities alone, slice_words mask words per CTA, read in place:
// a pass of loads per thread and no barrier (staged through shared memory in
// clusters' slices it took 3.0 us instead of 2.3 at 64000 tokens, batch 24).
template <bool BF16>
__global__ void __launch_bounds__(kDecodeThreads, 2)
    logprobs_kernel(const __grid_constant__ LogitsArgs a) {
    const int r = blockIdx.x / a.slices, w0 = (blockIdx.x - r * a.slices) * a.slice_words;
    pdl_wait();
    pdl_trigger();
    write_logprobs<BF16>(reinterpret_cast<const char*>(a.logits) + (size_t)r * (size_t)a.stride * (BF16 ? 2 : 4), a.V,
                         a.mask.row(r, a.W, false) + w0, 32 * w0, min(32 * a.slice_words, a.V - 32 * w0),
                         __ldg(a.lse + r), a.logprobs + (size_t)r * a.V, threadIdx.x);
}

// Gumbel variate of token t of row r: g_t = -ln(-ln(u_t)), u_t = (2k + 1) / 2^24,
// k = (word t % 4 of Philox on (t / 4, r, offset)) >> 9.  `blk` / `rnd` cache
// the last Philox block.
__device__ __forceinline__ float gumbel(const SampleArgs& a, int r, int t, int& blk, uint4& rnd) {
    if ((t >> 2) != blk) {
        blk = t >> 2;
        rnd = philox10(make_uint4((uint32_t)blk, (uint32_t)r, a.off0, a.off1), a.key0, a.key1);
    }
    const uint32_t w = (t & 2) ? ((t & 1) ? rnd.w : rnd.z) : ((t & 1) ? rnd.y : rnd.x);
    const float u = __fmul_rn(__uint2float_rn(2u * (w >> 9) + 1u), 0x1p-24f);
    return -ln_rn(-ln_rn(u));
}

// ---- the greedy / log-sum-exp pass over bf16 rows: a compacted gather -----
// One CTA per row, its warps (up to 16) on consecutive segments of the row's
// mask words, each segment cut into spans of 32 x kGatherSpan words (lane l
// holds words l*kGatherSpan ... +kGatherSpan-1 of the span).  Each lane finds
// its words' 16-byte logit vectors that hold an allowed token (a 32-bit map,
// one bit per vector), a warp scan places the lanes' lists one after the
// other in token order, and the warp then loads the listed vectors
// kGatherRound per lane at once (entry k goes to lane k % 32, so each lane
// still sees its tokens in increasing order) and folds them.  Zero words cost
// a few instructions, every load of a span is independent, and a span costs
// one memory latency whatever its density.  The warps' partials are merged in
// shared memory.  Logit lines are not kept in L1 and go first in L2: no pass
// after this one reads them.
constexpr int kGatherMaxWarps = 16;   // warps per CTA (one row); two CTAs per SM
constexpr int kGatherSpan = 8;     // mask words per lane per span (8192 tokens)
constexpr int kGatherWarpSmem = 32 * kGatherSpan * (4 + 4 * 2);   // a span's words and its list
constexpr int kGatherRound = 4;    // vectors per lane loaded together

// element e (0..7) of eight bf16 values
__device__ __forceinline__ float bf16_of(const uint4& q, int e) {
    const uint32_t h = (e & 4) ? ((e & 2) ? q.w : q.z) : ((e & 2) ? q.y : q.x);
    return (e & 1) ? bf16_hi(h) : bf16_lo(h);
}

// chunk: words per warp, a multiple of kGatherSpan.  A sampling pass draws
// row r with the counter of its batch row.
template <int FOLD>
__global__ void __launch_bounds__(kGatherMaxWarps * 32, 2)
    logits_gather_kernel(const void* __restrict__ logits, int64_t stride, const MaskRows mask, int V, int W, int B,
                         int chunk, int32_t* __restrict__ argmax, float* __restrict__ lse, const SampleArgs sa,
                         const RowList list) {
    constexpr int kSpanWords = 32 * kGatherSpan;
    extern __shared__ __align__(16) unsigned char g_smem[];   // per warp: words, then list
    __shared__ float4 s_part[kGatherMaxWarps];
    pdl_wait();
    pdl_trigger();
    const int r = blockIdx.x;
    if (r >= list.rows(B)) return;   // the whole CTA
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint32_t* sw = reinterpret_cast<uint32_t*>(g_smem + wid * kGatherWarpSmem);   // a span's mask words
    uint16_t* lst = reinterpret_cast<uint16_t*>(sw + kSpanWords);                // its vectors, in token order
    const uint64_t pol = l2_policy(false);
    const int full_vec = V / 8;   // vectors that lie wholly inside the row
    const int j0 = wid * chunk, j1 = min(W, j0 + chunk);
    const uint32_t* mrow = mask.row(r, W, threadIdx.x == 0);
    const int orow = list.row(r);
    const char* lrow = reinterpret_cast<const char*>(logits) + (size_t)orow * stride * 2;
    float m = -INFINITY, ref = sum_ref(m), s = 0.0f;
    int idx = INT_MAX;
    int blk = -1;   // Philox block cached by gumbel()
    uint4 rnd = make_uint4(0u, 0u, 0u, 0u);
    // one allowed logit x of token t (t increasing within a lane)
    auto fold1 = [&](float x, int t) {
        if constexpr (FOLD == kFoldSample) {
            const float sx = __fmul_rn(x, sa.inv_t);
            if (__fadd_rn(sx, kGumbelMax) < m) return;
            const float sc = __fadd_rn(sx, gumbel(sa, orow, t, blk, rnd));
            if (sc > m) {
                m = sc;
                idx = t;
            }
        } else if constexpr (FOLD == kFoldMax) {
            if (x > m) {
                m = x;
                idx = t;
            }
        } else {
            acc_add(m, ref, idx, s, x, t);
        }
    };
    for (int js = j0; js < j1; js += kSpanWords) {
        uint32_t w[kGatherSpan];
        const int jl = js + lane * kGatherSpan;
        if (mrow && jl + kGatherSpan <= j1 && (reinterpret_cast<uintptr_t>(mrow + jl) & 15) == 0) {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(mrow + jl));
            const uint4 b = __ldg(reinterpret_cast<const uint4*>(mrow + jl) + 1);
            w[0] = a.x, w[1] = a.y, w[2] = a.z, w[3] = a.w, w[4] = b.x, w[5] = b.y, w[6] = b.z, w[7] = b.w;
        } else {
#pragma unroll
            for (int g = 0; g < kGatherSpan; ++g) w[g] = jl + g < j1 ? mask.word(mrow, jl + g) : 0u;
        }
        uint32_t nb = 0;   // bit 4g + b: byte b of word g holds an allowed token
#pragma unroll
        for (int g = 0; g < kGatherSpan; ++g) nb |= nonzero_bytes(w[g]) << (4 * g);
        reinterpret_cast<uint4*>(sw)[2 * lane] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(sw)[2 * lane + 1] = make_uint4(w[4], w[5], w[6], w[7]);
        const int c = __popc(nb);
        int incl = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        const int T = __shfl_sync(0xffffffffu, incl, 31);
        if (T == 0) continue;   // warp-uniform
        int pos = incl - c;
        while (nb) {
            const int bit = __ffs(nb) - 1;
            nb &= nb - 1;
            lst[pos++] = (uint16_t)(lane * 4 * kGatherSpan + bit);
        }
        __syncwarp();
        const int vbase = js * 4;   // the span's first vector in the row
        // rounds of kGatherRound vectors per lane; the next round's loads are
        // issued before this round is folded
        int ent[kGatherRound];
        uint4 q[kGatherRound];
        auto load_round = [&](int k0, int(&en)[kGatherRound], uint4(&qq)[kGatherRound]) {
#pragma unroll
            for (int i = 0; i < kGatherRound; ++i) {
                const int k = k0 + i * 32 + lane;
                en[i] = k < T ? (int)lst[k] : -1;
                const int vi = vbase + en[i];
                qq[i] = (en[i] >= 0 && vi < full_vec) ? ld_once16(lrow + (size_t)vi * 16, pol)
                                                     : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        load_round(0, ent, q);
        for (int k0 = 0; k0 < T; k0 += 32 * kGatherRound) {
            int ent_n[kGatherRound];
            uint4 q_n[kGatherRound];
            const bool more = k0 + 32 * kGatherRound < T;   // warp-uniform
            if (more) load_round(k0 + 32 * kGatherRound, ent_n, q_n);
#pragma unroll
            for (int i = 0; i < kGatherRound; ++i) {
                if (ent[i] < 0) continue;
                const int vi = vbase + ent[i], t0 = vi * 8;
                uint32_t bm = (sw[ent[i] >> 2] >> (8 * (ent[i] & 3))) & 0xFFu;
                if (vi >= full_vec) {   // the row's last, partial vector: token by token
                    while (bm) {
                        const int e = __ffs(bm) - 1;
                        bm &= bm - 1;
                        if (t0 + e >= V) break;
                        fold1(logit_at<true>(lrow, t0 + e), t0 + e);
                    }
                } else if (FOLD == kFoldSample) {
                    while (bm) {
                        const int e = __ffs(bm) - 1;
                        bm &= bm - 1;
                        fold1(bf16_of(q[i], e), t0 + e);
                    }
                } else if (__popc(bm) > 2) {
                    // a dense vector: its allowed maximum (first on ties), one
                    // rescale, then its sum, all eight lanes of it predicated;
                    // earlier vectors hold lower ids, so an equal maximum keeps idx
                    float xs[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) xs[e] = ((bm >> e) & 1u) ? bf16_of(q[i], e) : -INFINITY;
                    float vm = xs[0];
                    int ve = 0;
#pragma unroll
                    for (int e = 1; e < 8; ++e)
                        if (xs[e] > vm) {
                            vm = xs[e];
                            ve = e;
                        }
                    if constexpr (FOLD == kFoldMax) {
                        if (vm > m) {
                            m = vm;
                            idx = t0 + ve;
                        }
                    } else {
                        if (vm > m) {
                            s = s == 0.0f ? 0.0f : s * exp_diff(ref, vm);
                            m = ref = vm;
                            idx = t0 + ve;
                        }
                        float acc = 0.0f;
#pragma unroll
                        for (int e = 0; e < 8; ++e) acc += ((bm >> e) & 1u) ? exp_diff(xs[e], ref) : 0.0f;
                        s += acc;
                    }
                } else {
                    while (bm) {
                        const int e = __ffs(bm) - 1;
                        bm &= bm - 1;
                        fold1(bf16_of(q[i], e), t0 + e);
                    }
                }
            }
            if (more) {
#pragma unroll
                for (int i = 0; i < kGatherRound; ++i) {
                    ent[i] = ent_n[i];
                    q[i] = q_n[i];
                }
            }
        }
        __syncwarp();   // the span buffers are rewritten by the next span
    }
    warp_merge(m, idx, s);
    if (lane == 0) s_part[wid] = make_float4(m, __int_as_float(idx), s, 0.f);
    __syncthreads();
    if (wid == 0) {
        m = -INFINITY;
        s = 0.0f;
        idx = INT_MAX;
        if (lane < nwarps) {
            const float4 p = s_part[lane];
            m = p.x;
            idx = __float_as_int(p.y);
            s = p.z;
        }
        warp_merge(m, idx, s);
        if (lane == 0) {
            argmax[orow] = m == -INFINITY ? -1 : idx;
            if (lse) lse[orow] = log_sum_exp(m, s);
        }
    }
}

// CTAs per row: doubled while every SM has at most one and a warp more than 16
// mask words, or at most two and 128 words.  Two CTAs an SM whose warps have
// fewer wait for the launch and the cluster's barriers (GB300, batch 100, V =
// 8000, 1 % allowed: one CTA a row 4.4 us, two 7.1; fp32, batch 32, V = 32000,
// half allowed: two 7.0, four 6.5, eight 8.4, a draw 12.7 / 10.2 / 12.4; V =
// 152064, batch 128, 80 %: one 15.2, two 12.9, with log-probabilities 38.2 /
// 27.7, a draw 97 / 59).
void cut_rows(LogitsArgs& a, int num_sms) {
    int s = 1;
    while (s < 8 && ((int64_t)a.batch * s * 2 <= num_sms ? a.W > 256 * s
                                                         : (int64_t)a.batch * s <= num_sms && a.W > 2048 * s))
        s *= 2;
    a.slices = s;
    a.slice_words = ((a.W + s - 1) / s + 3) / 4 * 4;
    a.segment = std::min(a.slice_words, kLogitsSegment);
}

// the gather kernels' dynamic shared memory passes the default 48 KB at 16
// warps: the limit is raised once per device and fold
template <int FOLD>
cudaError_t gather_smem_ready() {
    static bool configured[kLogitsMaxDevices] = {false};   // one array per fold
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError();
    if (dev >= kLogitsMaxDevices) dev = kLogitsMaxDevices - 1;
    std::lock_guard<std::mutex> lk(mu);
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(logits_gather_kernel<FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kGatherMaxWarps * kGatherWarpSmem);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    return cudaSuccess;
}

template <int FOLD>
cudaError_t launch_gather(const LogitsArgs& a, const RowList& list, cudaStream_t st) {
    // a warp per span of the row, at most kGatherMaxWarps (two CTAs per SM); a
    // warp's words rounded up to whole lanes
    const int nwarps = std::max(1, std::min(kGatherMaxWarps, (a.W + 32 * kGatherSpan - 1) / (32 * kGatherSpan)));
    int chunk = (a.W + nwarps - 1) / nwarps;
    chunk = (chunk + kGatherSpan - 1) / kGatherSpan * kGatherSpan;
    if (cudaError_t e = gather_smem_ready<FOLD>(); e != cudaSuccess) return e;
    return launch_pdl(logits_gather_kernel<FOLD>, dim3((unsigned)a.batch), dim3(nwarps * 32),
                      (size_t)(nwarps * kGatherWarpSmem), st, a.logits, a.stride, a.mask, a.V, a.W, a.batch, chunk,
                      a.argmax, a.lse, a.sample, list);
}

template <bool BF16, int FOLD>
cudaError_t launch_logits_t(const LogitsArgs& a, const RowList& list, cudaStream_t st) {
    return launch_cluster(logits_kernel<BF16, FOLD>, dim3((unsigned)a.batch * (unsigned)a.slices), dim3(kDecodeThreads),
                          a.slices, (size_t)logits_smem(a.segment), st, a, list);
}

template <bool BF16>
cudaError_t launch_logits_f(const LogitsArgs& a, bool sample, const RowList& list, cudaStream_t st) {
    if (sample) return launch_logits_t<BF16, kFoldSample>(a, list, st);
    return a.lse || a.logprobs ? launch_logits_t<BF16, kFoldLse>(a, list, st)
                               : launch_logits_t<BF16, kFoldMax>(a, list, st);
}

}  // namespace

cudaError_t launch_mask_logits(const LaunchEnv& env, const void* logits, int dtype, int32_t batch,
                               int64_t row_stride, int32_t V, const uint32_t* mask, int32_t* argmax, float* lse,
                               float* logprobs, cudaStream_t st, const int32_t* row_state, int32_t Q, uint32_t* err,
                               const SampleArgs* sample, const int32_t* row_ids, const int32_t* row_count) {
    LogitsArgs a{};
    a.logits = logits;
    a.stride = row_stride;
    a.mask = MaskRows{mask, row_state, Q, err};
    a.V = V;
    a.W = (V + 31) / 32;
    a.batch = batch;
    a.argmax = argmax;
    a.lse = lse;
    a.logprobs = logprobs;
    a.sample = sample ? *sample : SampleArgs{0u, 0u, 0u, 0u, 1.0f};
    cut_rows(a, env.num_sms);
    const RowList list{row_ids, row_count, 0};
    // The gather wants one CTA per row to fill the SMs, aligned bf16 rows, and
    // no second pass: there it is the faster one where masks are sparse
    // (GB300, V = 128256, 1 % allowed, batch 256: 6.0 against 8.0 us, batch
    // 1000: 22 against 29 us) and the slower one where they are dense (JSON, V =
    // 152064, batch 512: 45 against 38 us).  The host does not see the masks
    // and takes the gather for all of these batches, the unmasked argmax and
    // draws among them.  With fewer rows, or rows off 16-byte boundaries, fp32 or
    // log-probabilities, the cluster kernel: V = 152064, batch 128, 80 %
    // allowed: 12.9 us (24.6 us for the flat split over one-warp CTAs that it
    // replaced), with log-probabilities 27.7 us (40.0); batch 24, V = 50001:
    // 7.1 us (13.6); fp32, V = 32000, batch 64, with log-probabilities: 9.0 us
    // (28.9); a draw at V = 152064, batch 128, 80 %: 57.9 us (115).
    const bool aligned = reinterpret_cast<uintptr_t>(logits) % 16 == 0 && ((size_t)row_stride * 2) % 16 == 0;
    if (dtype == DOMINO_DTYPE_BF16 && aligned && batch > env.num_sms && !logprobs)
        return sample ? launch_gather<kFoldSample>(a, list, st)
                      : lse ? launch_gather<kFoldLse>(a, list, st) : launch_gather<kFoldMax>(a, list, st);
    return dtype == DOMINO_DTYPE_BF16 ? launch_logits_f<true>(a, sample != nullptr, list, st)
                                      : launch_logits_f<false>(a, sample != nullptr, list, st);
}

cudaError_t launch_logprobs_bf16(const LaunchEnv& env, const void* logits, int32_t batch, int64_t row_stride,
                                 int32_t V, const uint32_t* mask, const float* lse, float* logprobs, cudaStream_t st) {
    LogitsArgs a{};
    a.logits = logits;
    a.stride = row_stride;
    a.mask = MaskRows{mask, nullptr, 0, nullptr};
    a.V = V;
    a.W = (V + 31) / 32;
    a.batch = batch;
    a.lse = const_cast<float*>(lse);
    a.logprobs = logprobs;
    a.slice_words = 128;   // one 8-token vector per thread
    a.slices = (a.W + a.slice_words - 1) / a.slice_words;
    return launch_pdl(logprobs_kernel<true>, dim3((unsigned)batch * (unsigned)a.slices), dim3(kDecodeThreads), 0, st, a);
}

cudaError_t launch_mask_sample(const LaunchEnv& env, const void* logits, int dtype, int32_t batch,
                               int64_t row_stride, int32_t V, const uint32_t* mask, float temperature,
                               uint64_t seed, uint64_t offset, int32_t* tokens, cudaStream_t st) {
    const SampleArgs sa{(uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)offset, (uint32_t)(offset >> 32),
                        1.0f / temperature};   // one correctly rounded fp32 division
    return launch_mask_logits(env, logits, dtype, batch, row_stride, V, mask, tokens, nullptr, nullptr, st, nullptr, 0,
                              nullptr, &sa);
}

}  // namespace domino

// ---------------------------------------------------------------------------
// domino_mask_logits_noalloc: the masked argmax / log-sum-exp for callers that
// cannot allocate device memory.  The kernel needs no scratch in device
// memory; the limit on the batch is part of the entry point's contract.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocMaxRows = 512;
constexpr int kNoAllocMaxDevices = 64;

struct NoAllocDevice {
    bool ready;
    int num_sms;
};
NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];
std::mutex g_noalloc_mu;

// Once per device, with that device current.
int noalloc_setup(int dev, NoAllocDevice* out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocDevice& d = g_noalloc_dev[dev];
    if (!d.ready) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
            cudaGetLastError();
            return DOMINO_E_CUDA;
        }
        d.num_sms = sms;
        d.ready = true;
    }
    *out = d;
    return DOMINO_OK;
}

}  // namespace

extern "C" int domino_mask_logits_noalloc(const void* logits_dev, int32_t dtype, int32_t batch, int32_t n_tokens,
                                          int64_t row_stride_elems, const uint32_t* mask_dev, int32_t* argmax_dev,
                                          float* lse_dev, float* logprobs_dev, void* stream) {
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0 || batch > kNoAllocMaxRows || n_tokens < 1 || n_tokens > (1 << 24) || row_stride_elems < n_tokens)
        return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_dev || !mask_dev || !argmax_dev) return DOMINO_E_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return DOMINO_E_CUDA;
    }
    if (dev < 0 || dev >= kNoAllocMaxDevices) return DOMINO_E_UNSUPPORTED;
    NoAllocDevice d{};
    int rc = noalloc_setup(dev, &d);
    if (rc != DOMINO_OK) return rc;
    domino::LaunchEnv env{d.num_sms, 0};
    cudaError_t e = domino::launch_mask_logits(env, logits_dev, dtype, batch, row_stride_elems, n_tokens, mask_dev,
                                               argmax_dev, lse_dev, logprobs_dev, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return DOMINO_E_CUDA;
    }
    return DOMINO_OK;
}
