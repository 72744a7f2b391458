// decode.cuh -- the masked decode of one row by one CTA (or a cluster of CTAs
// that share out the row's tokens), used by the mask step that decodes its row
// at once (rows.cu) and by the decode of given masks (logits.cu): masked
// maximum, lowest-index argmax and sum of exponentials, or a Gumbel-max draw,
// over bf16 or fp32 logits at any alignment, and the log-probabilities.
//
// The row's mask words lie in shared memory.  Logits are read as 8-token
// vectors on 16-byte boundaries of the row (a row that starts off such a
// boundary shifts the vectors against the mask by `shift` tokens); vectors
// without an allowed token are never read.  A warp takes 256 mask words at a
// time, 8 per lane: a span with many vectors to read is read as it lies, else
// the vectors' numbers are listed in shared memory, in token order, and read
// four per lane together, so that a sparse row costs about one memory latency.
#pragma once
#include "walk_common.cuh"

namespace domino {
namespace {

// What a row's allowed logits are folded into.
enum Fold : int {
    kFoldLse = 0,      // max, lowest-index argmax and sum of exp (log-sum-exp)
    kFoldMax = 1,      // max and lowest-index argmax only (no lse requested)
    kFoldSample = 2,   // Gumbel-max draw
};

constexpr int kDecodeThreads = 512;   // a CTA's, where nothing else is said
constexpr int kDecodeWarps = kDecodeThreads / 32;
constexpr int kDecodeSpan = 8;          // mask words per lane looked over at a time
constexpr int kDecodeList = 384;        // of a span's 1024 vectors: more are read as they lie
constexpr int kDecodeListBytes = kDecodeWarps * kDecodeList * 2;

// Byte b of a mask as four words that keep (all ones) or drop (zero) the
// bf16 halves of a vector: kDecodeKeep entries in shared memory.
constexpr int kDecodeKeep = 256;
template <int THREADS = kDecodeThreads>
__device__ __forceinline__ void fill_keep(uint4* keep, int tid) {
    for (int b = tid; b < kDecodeKeep; b += THREADS) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[k] = ((b >> (2 * k)) & 1 ? 0xFFFFu : 0u) | ((b >> (2 * k + 1)) & 1 ? 0xFFFF0000u : 0u);
        keep[b] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// bit b of the result: byte b of x is not zero
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t x) {
    x |= x >> 4;
    x |= x >> 2;
    x |= x >> 1;
    return ((x & 0x01010101u) * 0x10204080u) >> 28;
}

// (a, b) * (c, c) + (d, d), both lanes rounded once
__device__ __forceinline__ float2 fma2(float2 a, float c, float d) {
    unsigned long long x, y, z, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(y) : "f"(c));
    asm("mov.b64 %0, {%1, %1};" : "=l"(z) : "f"(d));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long x, y, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}

// the larger of two pairs of bf16, a NaN losing to a number
__device__ __forceinline__ uint32_t max2_bf16(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint64_t l2_policy(bool keep) {
    uint64_t p;
    if (keep)
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
    else
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint4 ld_once16(const void* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;\n"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

template <bool BF16>
__device__ __forceinline__ float logit_at(const void* row, int t) {
    if constexpr (BF16) {
        const unsigned short u = __ldg(reinterpret_cast<const unsigned short*>(row) + t);
        return __uint_as_float((uint32_t)u << 16);
    } else {
        return __ldg(reinterpret_cast<const float*>(row) + t);
    }
}

// ---- sampling: Gumbel-max over the allowed logits --------------------------
// Philox4x32-10 (Salmon, Moraes, Dror and Shaw, SC'11): ten rounds of two
// 32x32 -> 64-bit products on the counter, the key advanced by the Weyl
// constants between rounds.
__device__ __forceinline__ uint4 philox10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// ln(x) for a positive normal float: x = 2^e m, m in [sqrt(1/2), sqrt(2)),
// ln x = e ln 2 + 2 atanh(z), z = (m - 1) / (m + 1), with atanh's odd power
// series up to z^11.  Every operation is an explicitly rounded fp32 intrinsic
// (no contraction), so the value is reproducible bit for bit.
__device__ __forceinline__ float ln_rn(float x) {
    const uint32_t bits = __float_as_uint(x);
    int e = (int)((bits >> 23) & 0xFFu) - 127;
    float m = __uint_as_float((bits & 0x7FFFFFu) | 0x3F800000u);
    if (m > 0x1.6a09e6p+0f) {
        m = __fmul_rn(m, 0.5f);
        e += 1;
    }
    const float z = __fdiv_rn(__fsub_rn(m, 1.0f), __fadd_rn(m, 1.0f));
    const float z2 = __fmul_rn(z, z);
    float p = 0x1.745d18p-4f;
    p = __fmaf_rn(p, z2, 0x1.c71c72p-4f);
    p = __fmaf_rn(p, z2, 0x1.24924ap-3f);
    p = __fmaf_rn(p, z2, 0x1.99999ap-3f);
    p = __fmaf_rn(p, z2, 0x1.555556p-2f);
    p = __fmaf_rn(p, z2, 1.0f);
    const float r = __fmul_rn(__fadd_rn(z, z), p);
    const float ef = __int2float_rn(e);
    return __fmaf_rn(ef, 0x1.62e43p-1f, __fmaf_rn(ef, -0x1.05c61p-29f, r));
}

// Every Gumbel variate is below this: u <= 1 - 2^-24 gives -ln(u) >= 5.96e-8
// and g <= 16.64.  A token with x / T + kGumbelMax below a score already seen
// cannot win (rounding is monotonic), so its variate is never drawn.
constexpr float kGumbelMax = 17.0f;

// A lane's fold over a row's tokens.  The sum of exponentials is kept against
// a reference that follows the maximum only when it falls more than kLag
// behind, and the maximum's vector is kept instead of its token, so that a
// vector costs no branch in the common case: the bf16 vector takes about 55
// instructions for 8 tokens (208 with the maximum's token found and the sum
// rescaled whenever some lane's maximum rose), 8 of them ex2, whose unit
// (16 a clock and SM) then bounds dense rows.
//
// A term is 2^(x log2(e) - ref) in one fused operation, so it is off by its
// own rounding only; that ref is a rounded m log2(e) is made good in finish().
// Its rounding must stay within 2^x's range: a reference below kLowRef is held
// there.  The terms of smaller logits (-1e10 or the lowest value of the type
// that ban a token) then come out as 0, which they are beside any other; where
// there is no other, and above 2^29, log_sum_exp() takes no sum.
template <bool BF16, int FOLD>
struct Decoder {
    static constexpr float kLowRef = -0x1p30f;   // half a unit in its last place is 32
    static constexpr int kWords = BF16 ? 4 : 8;   // 32-bit words of a vector
    static constexpr int kTogether = BF16 ? 4 : 2;   // vectors per lane read together
    struct Vec {
        uint32_t q[kWords];
        __device__ __forceinline__ float at(int e) const {
            if constexpr (BF16) return (e & 1) ? bf16_hi(q[e >> 1]) : bf16_lo(q[e >> 1]);
            else return __uint_as_float(q[e]);
        }
    };

    const char* lrow;        // the row's logits
    int V;
    int shift;               // tokens between the 16-byte boundary at or before the row and the row
    uint64_t pol;
    SampleArgs sa;
    uint32_t srow;           // sampling: the row's counter word
    int lane;
    const uint4* keep;       // fill_keep's table
    float m;                 // maximum (sampling: the best score)
    float ref, s;            // the sum's reference (times log2(e)) and the sum of 2^(x log2(e) - ref)
    int idx;                 // sampling: its token; else the token of element 0 of the maximum's vector
    uint32_t top[kWords];    // the maximum's vector, -inf where not allowed
    float seen;              // sampling: a score some lane of the warp has seen

    __device__ __forceinline__ void init(const void* logits, int64_t stride, int row, int V_, bool keep_l2,
                                         const SampleArgs& sample, const uint4* keep_, int lane_) {
        constexpr int esz = BF16 ? 2 : 4;
        lrow = reinterpret_cast<const char*>(logits) + (size_t)row * (size_t)stride * esz;
        V = V_;
        shift = (int)((reinterpret_cast<uintptr_t>(lrow) & 15) / esz);
        pol = l2_policy(keep_l2);
        sa = sample;
        srow = (uint32_t)row;
        lane = lane_;
        keep = keep_;
        m = seen = -INFINITY;
        ref = 0.0f;
        s = 0.0f;
        idx = INT_MAX;
#pragma unroll
        for (int k = 0; k < kWords; ++k) top[k] = BF16 ? 0xFF80FF80u : 0xFF800000u;
    }

    // the allowed tokens of vector b of a slice whose mask bytes start at
    // `bytes` (a zero byte before and after): bit e is token tok0 + 8b - shift + e
    __device__ __forceinline__ uint32_t allowed(const uint8_t* bytes, int b) const {
        if (shift == 0) return bytes[b];
        return ((uint32_t)bytes[b - 1] | ((uint32_t)bytes[b] << 8)) >> (8 - shift) & 0xFFu;
    }

    // vector b of a slice whose vectors start at `vec`
    __device__ __forceinline__ Vec load(const char* vec, int b) const {
        Vec x;
        const char* p = vec + (size_t)(unsigned)b * (kWords * 4);
        const uint4 q = ld_once16(p, pol);
        x.q[0] = q.x, x.q[1] = q.y, x.q[2] = q.z, x.q[3] = q.w;
        if constexpr (!BF16) {
            const uint4 r = ld_once16(p + 16, pol);
            x.q[4] = r.x, x.q[5] = r.y, x.q[6] = r.z, x.q[7] = r.w;
        }
        return x;
    }

    // N vectors, of which vector k's allowed tokens are bits[k] (0: none) and
    // whose element 0 is token t0[k].  Without branches between the vectors, so
    // that their latencies overlap.
    template <int N>
    __device__ __forceinline__ void fold(const Vec (&x)[N], const uint32_t (&bits)[N], const int (&t0)[N]) {
        if constexpr (FOLD == kFoldSample) {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                if (bits[k]) sample(x[k], bits[k], t0[k]);
                share();
            }
        } else {
            // the tokens not allowed as -inf, and the vectors' maxima
            uint32_t w[N][kWords];
            float vm[N];
#pragma unroll
            for (int k = 0; k < N; ++k) {
                if constexpr (BF16) {
                    const uint4 y = keep[bits[k]];
                    w[k][0] = (x[k].q[0] & y.x) | (0xFF80FF80u & ~y.x), w[k][1] = (x[k].q[1] & y.y) | (0xFF80FF80u & ~y.y);
                    w[k][2] = (x[k].q[2] & y.z) | (0xFF80FF80u & ~y.z), w[k][3] = (x[k].q[3] & y.w) | (0xFF80FF80u & ~y.w);
                    const uint32_t mm = max2_bf16(max2_bf16(w[k][0], w[k][1]), max2_bf16(w[k][2], w[k][3]));
                    vm[k] = fmaxf(bf16_lo(mm), bf16_hi(mm));
                } else {
                    float y[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        w[k][e] = (bits[k] >> e) & 1u ? x[k].q[e] : 0xFF800000u;
                        y[e] = __uint_as_float(w[k][e]);
                    }
                    vm[k] = fmaxf(fmaxf(fmaxf(y[0], y[1]), fmaxf(y[2], y[3])), fmaxf(fmaxf(y[4], y[5]), fmaxf(y[6], y[7])));
                }
            }
            if constexpr (FOLD == kFoldLse) {
                constexpr float kLag = 16.0f;   // terms of 2^16 at most: no overflow, and nothing lost in relative terms
                float most = vm[0];
#pragma unroll
                for (int k = 1; k < N; ++k) most = fmaxf(most, vm[k]);
                const float vL = most * kLog2e;
                if ((vL > ref + kLag || m == -INFINITY) && most != -INFINITY) {   // rare after the first vectors
                    s *= s == 0.0f ? 0.0f : ex2(ref - vL);
                    ref = fmaxf(vL, kLowRef);
                }
            }
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (vm[k] > m || (vm[k] == m && t0[k] < idx)) {
                    m = vm[k];
                    idx = t0[k];
#pragma unroll
                    for (int e = 0; e < kWords; ++e) top[e] = w[k][e];
                }
            if constexpr (FOLD == kFoldLse) {
                float2 acc[N];
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    acc[k] = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 z = BF16 ? make_float2(bf16_lo(w[k][e]), bf16_hi(w[k][e]))
                                              : make_float2(__uint_as_float(w[k][BF16 ? 0 : 2 * e]), __uint_as_float(w[k][BF16 ? 0 : 2 * e + 1]));
                        const float2 y = fma2(z, kLog2e, -ref);
                        acc[k] = add2(acc[k], make_float2(ex2(y.x), ex2(y.y)));   // not allowed: 2^-inf = 0
                    }
                }
#pragma unroll
                for (int k = 0; k < N; ++k) s += acc[k].x + acc[k].y;
            }
        }
    }

    // The lane's result: the maximum, its lowest token, and the sum of exp
    // against it.
    __device__ __forceinline__ void finish() {
        if constexpr (FOLD != kFoldSample) {
            if (m == -INFINITY) {   // nothing allowed, or only -inf logits
                idx = INT_MAX;
                s = 0.0f;
                return;
            }
            int e = 7;
#pragma unroll
            for (int k = 6; k >= 0; --k) {
                const float v = BF16 ? ((k & 1) ? bf16_hi(top[k >> 1]) : bf16_lo(top[k >> 1])) : __uint_as_float(top[BF16 ? 0 : k]);
                if (v == m) e = k;
            }
            idx += e;
            if constexpr (FOLD == kFoldLse) s *= s == 0.0f ? 0.0f : ex2(__fmaf_rn(-m, kLog2e, ref));
        }
    }

    // sampling: a new best score x at token t, or an equal one at a lower token
    __device__ __forceinline__ void raise(float x, int t) {
        if (x > m || (x == m && t < idx)) {
            m = x;
            idx = t;
        }
    }

    // element e of a vector, e known at run time only
    __device__ __forceinline__ static float pick(const Vec& x, int e) {
        if constexpr (BF16) {
            const uint32_t h = (e & 4) ? ((e & 2) ? x.q[3] : x.q[2]) : ((e & 2) ? x.q[1] : x.q[0]);
            return (e & 1) ? bf16_hi(h) : bf16_lo(h);
        } else {
            const uint32_t a = (e & 2) ? ((e & 1) ? x.q[3] : x.q[2]) : ((e & 1) ? x.q[1] : x.q[0]);
            const uint32_t b = (e & 2) ? ((e & 1) ? x.q[7] : x.q[6]) : ((e & 1) ? x.q[5] : x.q[4]);
            return __uint_as_float((e & 4) ? b : a);
        }
    }

    // The vector's Gumbel scores: g_t = -ln(-ln(u_t)), u_t = (2k + 1) / 2^24,
    // k = (word t % 4 of Philox on (t / 4, row, offset)) >> 9.  The exactly
    // rounded variate is taken only where an upper bound could reach the best
    // score.
    __device__ __forceinline__ void sample(const Vec& x, uint32_t bits, int t0) {
        const float floor = fmaxf(m, seen);
        uint32_t cand = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (!(__fadd_rn(__fmul_rn(x.at(e), sa.inv_t), kGumbelMax) < floor)) cand |= 1u << e;
        cand &= bits;
        if ((t0 & 3) == 0) {   // the same for every vector of a row
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if ((cand >> (4 * h)) & 15u)
                    block(x.at(4 * h), x.at(4 * h + 1), x.at(4 * h + 2), x.at(4 * h + 3), (cand >> (4 * h)) & 15u,
                          t0 + 4 * h);
        } else {
#pragma unroll 1
            for (int tb = t0 & ~3; tb < t0 + 8; tb += 4) {
                const int e = tb - t0;   // the block's first element, -3 to 7
                const uint32_t c = (e >= 0 ? cand >> e : cand << -e) & 15u;
                if (c) block(pick(x, e & 7), pick(x, (e + 1) & 7), pick(x, (e + 2) & 7), pick(x, (e + 3) & 7), c, tb);
            }
        }
    }

    // An upper bound of the variate of u, less than 0.01 above it: the
    // hardware's log2 (absolute error below 2^-21 on these ranges) for
    // u < 0.99; nearer to 1, -ln(u) >= 1 - u, which is exact.
    __device__ __forceinline__ static float gumbel_bound(float u) {
        constexpr float kSlack = 1e-3f, kLn2 = 0.6931471805599453f;
        const float a = u < 0.99f ? -kLn2 * __log2f(u) : __fsub_rn(1.0f, u);
        return __fadd_rn(-kLn2 * __log2f(a), kSlack);
    }

    // The candidates c of the Philox block of tokens tb to tb + 3.
    __device__ __forceinline__ void block(float x0, float x1, float x2, float x3, uint32_t c, int tb) {
        const uint4 r = philox10(make_uint4((uint32_t)tb >> 2, srow, sa.off0, sa.off1), sa.key0, sa.key1);
        const float best = fmaxf(m, seen);
        const float xs[4] = {__fmul_rn(x0, sa.inv_t), __fmul_rn(x1, sa.inv_t), __fmul_rn(x2, sa.inv_t),
                             __fmul_rn(x3, sa.inv_t)};
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
        if (best != -INFINITY) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float u = __fmul_rn(__uint2float_rn(2u * (w[k] >> 9) + 1u), 0x1p-24f);
                if (__fadd_rn(xs[k], gumbel_bound(u)) < best) c &= ~(1u << k);   // rounding is monotonic
            }
        }
#pragma unroll 1
        while (c) {
            const int k = __ffs((int)c) - 1;
            c &= c - 1;
            const uint32_t wk = (k & 2) ? ((k & 1) ? r.w : r.z) : ((k & 1) ? r.y : r.x);
            const float xk = (k & 2) ? ((k & 1) ? xs[3] : xs[2]) : ((k & 1) ? xs[1] : xs[0]);
            const float u = __fmul_rn(__uint2float_rn(2u * (wk >> 9) + 1u), 0x1p-24f);
            raise(__fadd_rn(xk, -ln_rn(-ln_rn(u))), tb + k);
        }
    }

    // A slice: tokens [tok0, tok0 + ntok), tok0 a multiple of 128, its mask
    // words at s_mask (a zero word before and after); `list` holds kDecodeList
    // entries of this warp.
    template <int THREADS = kDecodeThreads>
    __device__ __forceinline__ void slice(const uint32_t* s_mask, int tok0, int ntok, uint16_t* list, int warp) {
        constexpr int kWarps = THREADS / 32;
        const uint8_t* bytes = reinterpret_cast<const uint8_t*>(s_mask);
        const int base = tok0 - shift;   // vector b starts at token base + 8b, word j's vectors are 4j to 4j + 3
        const int nvec = (ntok + shift + 7) / 8;
        // the vectors inside the row; its first and last tokens outside of
        // them are taken one by one, below
        const int in0 = base < 0 ? 1 : 0, in1 = max(in0, base + 8 * nvec > V ? nvec - 1 : nvec);
        const char* vec = lrow + (int64_t)base * (BF16 ? 2 : 4);
        const int words = (nvec + 3) / 4;
        const int per = ((words + kWarps - 1) / kWarps + kDecodeSpan - 1) / kDecodeSpan * kDecodeSpan;
        const int j1 = min(words, (warp + 1) * per);
#pragma unroll 1
        for (int j0 = warp * per; j0 < j1; j0 += 32 * kDecodeSpan) {
            const int jl = j0 + lane * kDecodeSpan;
            uint32_t some = 0;   // bit 4g + k: vector k of the lane's word g holds an allowed token
            uint32_t w[kDecodeSpan];
            if (jl + kDecodeSpan <= j1) {   // the slice and the warp's words begin on 16-byte boundaries
                const uint4 p = reinterpret_cast<const uint4*>(s_mask + jl)[0], q = reinterpret_cast<const uint4*>(s_mask + jl)[1];
                w[0] = p.x, w[1] = p.y, w[2] = p.z, w[3] = p.w, w[4] = q.x, w[5] = q.y, w[6] = q.z, w[7] = q.w;
            } else {
#pragma unroll
                for (int g = 0; g < kDecodeSpan; ++g) w[g] = jl + g < j1 ? s_mask[jl + g] : 0u;
            }
            if (shift && jl < j1) {
#pragma unroll
                for (int g = kDecodeSpan - 1; g >= 0; --g)
                    w[g] = __funnelshift_rc(g ? w[g ? g - 1 : 0] : s_mask[jl - 1], w[g], 32 - shift);
            }
#pragma unroll
            for (int g = 0; g < kDecodeSpan; ++g) some |= nonzero_bytes(w[g]) << (4 * g);
            // vectors outside the row
            if (4 * jl < in0) some &= ~1u;
            const int past = in1 - 4 * jl;
            if (past < 32) some &= past <= 0 ? 0u : (1u << past) - 1u;
            const int c = __popc(some);
            int incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const int n = __shfl_sync(0xffffffffu, incl, 31);
            if (n == 0) continue;   // the whole warp
            if (n <= kDecodeList) {
                uint16_t* at = list + incl - c;
                while (some) {
                    *at++ = (uint16_t)(lane * 4 * kDecodeSpan + __ffs((int)some) - 1);
                    some &= some - 1;
                }
                __syncwarp();
#pragma unroll 1
                for (int k0 = 0; k0 < n; k0 += 32 * kTogether) {
                    int b[kTogether];
#pragma unroll
                    for (int k = 0; k < kTogether; ++k) {
                        const int i = k0 + 32 * k + lane;
                        b[k] = i < n ? 4 * j0 + (int)list[i] : -1;
                    }
                    fold_together(bytes, vec, base, b);
                }
                __syncwarp();
            } else {
                const int b1 = min(in1, 4 * min(j1, j0 + 32 * kDecodeSpan));
#pragma unroll 1
                for (int b0 = max(in0, 4 * j0); b0 < b1; b0 += 32 * kTogether) {
                    int b[kTogether];
#pragma unroll
                    for (int k = 0; k < kTogether; ++k) b[k] = b0 + 32 * k + lane < b1 ? b0 + 32 * k + lane : -1;
                    fold_together(bytes, vec, base, b);
                }
            }
        }
        // a lane per token of vectors 0 and nvec - 1, by the warps that hold their words
        if (lane < 16 && nvec > 0) {
            const int b = lane < 8 ? 0 : nvec - 1, e = lane & 7, t0 = base + 8 * b;
            const bool outside = lane < 8 ? in0 == 1 : b >= in1 && b >= in0;
            if (outside && (b >> 2) / per == warp && ((allowed(bytes, b) >> e) & 1u)) {
                Vec x;
#pragma unroll
                for (int k = 0; k < kWords; ++k) x.q[k] = 0u;
                const uint32_t u = __float_as_uint(logit_at<BF16>(lrow, t0 + e));
                x.q[0] = BF16 ? u >> 16 : u;   // as element 0 of a vector that starts at the token
                if constexpr (FOLD == kFoldSample) {
                    sample(x, 1u, t0 + e);   // (fold's sampling form is the whole warp's)
                } else {
                    const Vec xs[1] = {x};
                    const uint32_t one[1] = {1u};
                    const int at[1] = {t0 + e};
                    fold<1>(xs, one, at);
                }
            }
        }
    }

    // Vectors b[k] (-1: none), read together.
    __device__ __forceinline__ void fold_together(const uint8_t* bytes, const char* vec, int base,
                                                  const int (&b)[kTogether]) {
        Vec x[kTogether];
        uint32_t by[kTogether];
        int t0[kTogether];
#pragma unroll
        for (int k = 0; k < kTogether; ++k) {
            by[k] = b[k] >= 0 ? allowed(bytes, b[k]) : 0u;
            t0[k] = base + 8 * b[k];
#pragma unroll
            for (int e = 0; e < kWords; ++e) x[k].q[e] = 0u;
            if (by[k]) x[k] = load(vec, b[k]);
        }
        fold<kTogether>(x, by, t0);
    }

    // sampling: the warp's best score so far bounds what a lane has to draw
    __device__ __forceinline__ void share() {
        if constexpr (FOLD == kFoldSample) {
            // floats as integers in the same order
            const int f = __float_as_int(m);
            const int top = __reduce_max_sync(0xffffffffu, f < 0 ? f ^ 0x7FFFFFFF : f);
            seen = __int_as_float(top < 0 ? top ^ 0x7FFFFFFF : top);
        }
    }
};

// ---- one result per row ------------------------------------------------------
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

// *p of CTA `rank` of the cluster (p: this CTA's shared memory)
__device__ __forceinline__ float4 ld_cluster(const float4* p, int rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(r)
                 : "memory");
    return v;
}

struct DecodeShared {
    float4 part[kDecodeWarps];
    float4 cta, row;
};

// The row's (max, argmax, sum) over all lanes of the CTA and all `slices` CTAs
// of its cluster, the same in every thread.  Every thread calls it; with more
// than one slice, cluster_wait() has to follow before the CTA ends.
template <int THREADS = kDecodeThreads>
__device__ __forceinline__ void decode_combine(DecodeShared& sh, float& m, int& idx, float& s, int slices, int lane,
                                               int warp) {
    warp_merge(m, idx, s);
    if (lane == 0) sh.part[warp] = make_float4(m, __int_as_float(idx), s, 0.f);
    __syncthreads();
    if (warp == 0) {
        float4 p = lane < THREADS / 32 ? sh.part[lane] : make_float4(-INFINITY, __int_as_float(INT_MAX), 0.f, 0.f);
        m = p.x;
        idx = __float_as_int(p.y);
        s = p.z;
        warp_merge(m, idx, s);
        if (lane == 0) sh.cta = make_float4(m, __int_as_float(idx), s, 0.f);
    }
    if (slices > 1) {
        cluster_arrive();
        cluster_wait();
        if (warp == 0) {
            float4 p = lane < slices ? ld_cluster(&sh.cta, lane) : make_float4(-INFINITY, __int_as_float(INT_MAX), 0.f, 0.f);
            m = p.x;
            idx = __float_as_int(p.y);
            s = p.z;
            warp_merge(m, idx, s);
            if (lane == 0) sh.row = make_float4(m, __int_as_float(idx), s, 0.f);
        }
        cluster_arrive();   // the others' results have been read
        __syncthreads();
        const float4 p = sh.row;
        m = p.x;
        idx = __float_as_int(p.y);
        s = p.z;
    } else {
        __syncthreads();
        const float4 p = sh.cta;
        m = p.x;
        idx = __float_as_int(p.y);
        s = p.z;
    }
}

// Log-probabilities of a slice's tokens (tok0 a multiple of 128): logit - lse
// where allowed, -inf elsewhere.  Rows on 32-byte boundaries of the output and
// 16-byte boundaries of the logits: a thread takes 8 tokens (one 32-byte
// store); rows of V % 4 == 0: 4 tokens; else one.
template <bool BF16, int THREADS = kDecodeThreads>
__device__ __forceinline__ void write_logprobs(const char* lrow, int V, const uint32_t* s_mask, int tok0, int ntok,
                                               float lse, float* orow, int tid) {
    const uint8_t* bytes = reinterpret_cast<const uint8_t*>(s_mask);
    if ((V & 7) == 0 && (reinterpret_cast<uintptr_t>(orow) & 31) == 0 && (reinterpret_cast<uintptr_t>(lrow) & 15) == 0) {
#pragma unroll 2
        for (int b = tid; b < ntok / 8; b += THREADS) {
            const uint32_t bits = bytes[b];
            const char* p = lrow + (size_t)(tok0 + 8 * b) * (BF16 ? 2 : 4);
            float o[8];
            if constexpr (BF16) {
                const uint4 a = __ldcs(reinterpret_cast<const uint4*>(p));
                const uint32_t q[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) o[e] = (e & 1) ? bf16_hi(q[e >> 1]) : bf16_lo(q[e >> 1]);
            } else {
                const float4 a = __ldcs(reinterpret_cast<const float4*>(p)), c = __ldcs(reinterpret_cast<const float4*>(p) + 1);
                o[0] = a.x, o[1] = a.y, o[2] = a.z, o[3] = a.w, o[4] = c.x, o[5] = c.y, o[6] = c.z, o[7] = c.w;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) o[e] = ((bits >> e) & 1u) ? o[e] - lse : -INFINITY;
            asm volatile("st.global.cs.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(orow + tok0 + 8 * b), "f"(o[0]),
                         "f"(o[1]), "f"(o[2]), "f"(o[3]), "f"(o[4]), "f"(o[5]), "f"(o[6]), "f"(o[7])
                         : "memory");
        }
    } else if ((V & 3) == 0 && (reinterpret_cast<uintptr_t>(orow) & 15) == 0) {
        for (int b = tid; b < ntok / 4; b += THREADS) {
            const uint32_t bits = bytes[b >> 1] >> (4 * (b & 1));
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                o[e] = ((bits >> e) & 1u) ? logit_at<BF16>(lrow, tok0 + 4 * b + e) - lse : -INFINITY;
            __stcs(reinterpret_cast<float4*>(orow + tok0) + b, make_float4(o[0], o[1], o[2], o[3]));
        }
    } else {
#pragma unroll 4
        for (int b = tid; b < ntok; b += THREADS)
            orow[tok0 + b] = ((bytes[b >> 3] >> (b & 7)) & 1u) ? logit_at<BF16>(lrow, tok0 + b) - lse : -INFINITY;
    }
}

}  // namespace
}  // namespace domino
