// rows.cu -- C.mask() with one CTA per row (sm_103a).
//
// The mask of a row is the set of tokens whose class string can be walked
// from the row's configuration without reaching the dead state (Alg. 1's
// mask at lookahead k = infinity, Sec. 3.5; EOS iff the state accepts with an
// empty stack).  row_kernel expands, for one row, only the live part of the
// prefix tree of the class strings (the subterminal tree of Sec. 3.3 / Alg. 2
// over byte classes): the children of a live node that stay alive are the
// intersection of the node's child classes with its state's live classes, so
// a prefix that dies is never visited at all.
//
// Work is a pool of (node, state[, stack]) items in shared memory.  In a
// round every thread takes one item from the pool's top, reads the node's and
// the state's 32-byte record together (both L2-resident, one round trip),
// leaves the node's tokens to be set and adds the live children.  The mask is
// built in shared memory and written once; with next states the row is filled
// first and the allowed tokens' states are stored over it.
//
// What bounds it: latency.  A round is one L2 round trip (about 650 cycles)
// plus about 1100 cycles of dependent shared-memory, shuffle and barrier
// steps, whatever its width; a row of the 5000-state random DFA over 128256
// tokens takes 8 to 11 rounds for its 1000 live nodes.  One CTA per row keeps
// these rounds free of any grid-wide step, and neither the tree nor the
// transition table is staged.  Measured (GB300, that workload, back to back):
// batch 256 15.7 us (35.8 us for the walk it replaced, whose CTAs each staged
// a share of the tree and walked every row in it), batch 1000 49.1 us (94.1),
// batch 32 13.5 us (19.0); the 20000-state table 2.62 ms (3.25 ms).
//
// A row with more live nodes at a time than the pool holds is walked token by
// token instead (every_token), which bounds what a dense state costs: 500
// states with 16 of 32 classes live, V = 128256, one row 26 us, 28 classes live
// 51 us.  Small batches and automata most of whose rows are like that are the
// per-token walk's from the start (row_cost, use_rows, decode_rows in host.cpp).
// With more than 64 classes the children's entries are read instead of masks
// (add_wide).
//
// States that loop on most classes (string bodies) allow nearly every token.
// For the widest such loop sets the host keeps the tokens that stay inside
// the set as a bitmap, copied into the row's mask, and a second tree over the
// other tokens' remainders after their longest prefix inside the set, so that
// such a row costs a copy and a short walk.  A subtree entered in such a state
// is a filtered range of its tokens plus the edges that leave the set (see
// RowTree).
//
// The whole decode step in one kernel (launch_row_decode): the row's mask is
// still in shared memory when its logits are folded (decode.cuh), the cluster
// merges its slices' results, and the row is advanced by its token.  Measured
// against the separate kernels before it: 5000 states, V = 128256, batch 256
// 22.5 us (45.9 us in four launches), batch 1000 74.5 us (127); JSON, V =
// 152064, batch 128 35.5 us (86.1 us in two launches), with log-probabilities
// 47.5 us (105), batch 512 76.7 us (304).
//
// Batches with fewer rows than SMs give each row a cluster of CTAs that share
// out the row's mask words; each walks the row itself (the walk is latency,
// not work) and keeps the tokens of its words.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>

#include "decode.cuh"
#include "domino_internal.h"
#include "walk_common.cuh"

namespace domino {
namespace {

constexpr int kRowSlots = 4096;       // slots of the pool's items (run)
constexpr int kRowFan = 8;            // threads per item while there are few
constexpr int kRowSmall = 512;        // ranges of 2 to kRowSmallTokens tokens left to the whole CTA
constexpr int kRowSmallTokens = 64;
constexpr int kRowBig = 128;          // longer ranges
constexpr int kRowNextHalf = 49152;   // tokens up to which rows of next states take half the threads
constexpr int kRowSpawn = 2048;       // exits taken at a time
constexpr int kRowExits = 512;        // loop subtrees whose exits are still to be walked
constexpr int kWideAtOnce = 8;        // children of a wide node read together
constexpr int kRowLoopMin = 4;        // fewest tokens of a subtree taken as a loop subtree
constexpr int kRowMaxDevices = 64;
static_assert(kRowBig <= kRowThreads / 2 && kRowExits <= kRowThreads, "one entry per thread in the prefix sums");
static_assert(kRowSlots - kRowPool >= kRowThreads && kRowSpawn <= kRowPool, "the next round's items fit");
static_assert(kRowThreads == kDecodeThreads && kRowSlots * 8 >= kDecodeListBytes, "the decode's lists lie in the pool");

enum RowOut : int {
    kRowMask = 0,    // the mask
    kRowNext = 1,    // the mask (optional) and the next states
    kRowBf16 = 2,    // the mask, the greedy decode of bf16 logits and the update
    kRowF32 = 3,     // the same for fp32 logits
};

// How child and live classes are held: a 32-bit mask (K <= 32), a 64-bit
// mask (K <= 64), or, for more classes, child classes listed one byte each
// and transitions read from the dense table.
enum RowClasses : int { kRow32 = 0, kRow64 = 1, kRowWide = 2 };

struct RowArgs {
    const int32_t* states;
    const uint64_t* stacks;
    int32_t batch;
    int32_t row_is_state;
    int32_t slices;         // CTAs per row (a cluster)
    int32_t slice_words;    // mask words per CTA (a multiple of 4)
    uint32_t* mask;
    int32_t* next;
    // the decode (kRowBf16, kRowF32)
    const void* logits;
    int64_t stride;
    int32_t ahead;          // logits in device memory: pulled into L2 as the tokens are set
    int32_t* argmax;
    float* lse;
    float* logprobs;
    int32_t* states_out;    // the update, or nullptr
    uint64_t* stacks_out;
};

// Shared-memory layout (byte offsets).  The mask slice has a zero word on
// either side.
struct RowLayout {
    int mask, items, bits, range, exits, pre, keep, dec, total;
};

__host__ __device__ inline RowLayout row_layout(int slice_words, bool stack, bool loops, bool decode) {
    RowLayout L{};
    int o = 16;
    L.mask = o;   o += align16(slice_words * 4) + 16;
    L.items = o;  o += align16(kRowSlots * 8);
    L.bits = o;   o += stack ? align16(kRowSlots * 4) : 0;
    L.range = o;  o += (kRowSmall + kRowBig) * 16;
    L.exits = o;  o += loops ? kRowExits * 16 : 0;
    L.pre = o;    o += align16((kRowThreads + 1) * 4);
    L.keep = o;   o += decode ? kDecodeKeep * 16 : 0;
    L.dec = o;    o += decode ? (int)sizeof(DecodeShared) : 0;
    L.total = align16(o);
    return L;
}

struct RowShared {
    int4 st[3];      // by round: {items added, the pool is full, lists half full, 0}
    uint4 rc;        // the row's configuration (read_row)
    int back;        // exits walked (spawn_exits)
    int nrange[2], nexit;
    int wsum[kRowThreads / 32];
};

__device__ __forceinline__ int warp_scan_incl(int x, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    return x;
}

__device__ __forceinline__ int popc(uint32_t m) { return __popc(m); }
__device__ __forceinline__ int popc(unsigned long long m) { return __popcll(m); }

// the entry k of the prefix sums pre[0..n] (pre[0] = 0) with pre[k] <= f < pre[k + 1]
__device__ __forceinline__ int find_range(const int* pre, int n, int f) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] <= f) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The state a token's class string ends in, walked from (s, bits, depth) over
// the automaton's own table; 0 when it dies, and for EOS and empty tokens.
template <bool STACK>
__device__ __forceinline__ uint32_t token_end(const StepView& v, const RowTree& t, int32_t tk, uint32_t s, uint32_t& bits,
                                              uint32_t& depth) {
    const uint8_t* rec = t.trec + 32 * (size_t)tk;   // {length (255: or more), classes}
    int len = (int)__ldg(rec);
    const uint8_t* tail = v.tail;
    const uint8_t* head = rec + 1;
    if (len > 31) {   // the arena's record
        const int p = __ldg(v.pos_of + tk);
        len = (int)(__ldg(v.info + p) >> 16);
        head = reinterpret_cast<const uint8_t*>(v.head + 2 * (size_t)p);
        if (len > kInlineBytes) tail += __ldg(v.tail_off + p);
    }
    using E = typename std::conditional<STACK, uint32_t, uint16_t>::type;
    Tab<E, kDenseGlobal> tab;
    tab.dense = reinterpret_cast<const E*>(STACK ? (const void*)v.t32 : (const void*)v.t16);
    tab.K = (uint32_t)v.K;
    debug_bounds(tab, v);
    return len > 0 ? walk<STACK, 0>(tab, v.ret, (uint32_t)v.max_depth, s, bits, depth, head, len, tail) : 0u;
}

// The CTA's part of a row by walking each of its tokens from the row's
// configuration rc, kAtOnce words of 32 tokens per warp at a time: for rows
// with so many live nodes that the pool fills (a state that lets most classes
// through without looping).  Bound by the latency of the table reads, hence
// several tokens of a thread in flight; a warp's 32 tokens are a mask word, so
// whole words are stored.  Not inlined: its registers would spill beside the
// decode's (JSON, V = 152064, batch 512, with log-probabilities 152 against
// 142 us).
template <bool STACK, int OUT>
__device__ __noinline__ void every_token(const StepView& v, const RowTree& t, const uint4& rc, uint32_t* s_mask, int nw,
                                         int tok0, int ntok, int32_t* nrow, const char* ahead) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    using E = typename std::conditional<STACK, uint32_t, uint16_t>::type;
    constexpr int kAtOnce = STACK ? 2 : 4;
    const E* table = reinterpret_cast<const E*>(STACK ? (const void*)v.t32 : (const void*)v.t16);
    for (int w = warp * kAtOnce; w < nw; w += (int)(blockDim.x >> 5) * kAtOnce) {
        uint4 rec[kAtOnce];   // {length, the first 15 classes}, shifted by a byte per step
        uint32_t s[kAtOnce], bits[kAtOnce], depth[kAtOnce];
        int len[kAtOnce];
#pragma unroll
        for (int q = 0; q < kAtOnce; ++q) {
            const int x = (w + q) * 32 + lane;
            rec[q] = x < ntok ? __ldg(reinterpret_cast<const uint4*>(t.trec + 32 * (size_t)(tok0 + x)))
                              : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int q = 0; q < kAtOnce; ++q) {
            len[q] = (int)(rec[q].x & 0xFFu);   // EOS and empty tokens: 0
            s[q] = len[q] ? rc.x : 0u;
            bits[q] = rc.y;
            depth[q] = rc.z;
        }
        for (int i = 0; i < 15; ++i) {
            bool more = false;
#pragma unroll
            for (int q = 0; q < kAtOnce; ++q) {
                rec[q].x = __funnelshift_r(rec[q].x, rec[q].y, 8);
                rec[q].y = __funnelshift_r(rec[q].y, rec[q].z, 8);
                rec[q].z = __funnelshift_r(rec[q].z, rec[q].w, 8);
                rec[q].w >>= 8;
            }
            uint32_t e[kAtOnce];
#pragma unroll
            for (int q = 0; q < kAtOnce; ++q)
                e[q] = s[q] != 0u && i < len[q] ? (uint32_t)__ldg(table + (size_t)s[q] * v.K + (rec[q].x & 0xFFu)) : 0u;
#pragma unroll
            for (int q = 0; q < kAtOnce; ++q) {
                if (s[q] != 0u && i < len[q]) {
                    s[q] = e[q];
                    if constexpr (STACK) s[q] = pda_apply(e[q], bits[q], depth[q], (uint32_t)v.max_depth, v.ret);
                }
                more |= s[q] != 0u && i + 1 < len[q];
            }
            if (!__any_sync(0xffffffffu, more)) break;
        }
#pragma unroll
        for (int q = 0; q < kAtOnce; ++q) {
            const int x = (w + q) * 32 + lane, tk = tok0 + x;
            if (s[q] != 0u && len[q] > 15) {   // longer: from its start
                bits[q] = rc.y;
                depth[q] = rc.z;
                s[q] = token_end<STACK>(v, t, tk, rc.x, bits[q], depth[q]);
            }
            const unsigned word = __ballot_sync(0xffffffffu, s[q] != 0u);
            if (w + q >= nw) continue;
            if (lane == 0) s_mask[w + q] = word;
            if constexpr (OUT == kRowBf16 || OUT == kRowF32) {
                if (ahead && s[q] != 0u)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(ahead + (size_t)tk * (OUT == kRowBf16 ? 2 : 4)));
            }
            if constexpr (OUT == kRowNext) {
                if (nrow && x < ntok) nrow[tk] = (int32_t)s[q];
            }
        }
    }
}

// One row's walk.
template <bool STACK, int CLS, int OUT, int THREADS>
struct RowWalk {
    static constexpr int kExits = kRowExits < THREADS ? kRowExits : THREADS;   // one per thread in the prefix sums
    static constexpr bool WIDE = CLS == kRowWide;
    using Mask = typename std::conditional<CLS == kRow32, uint32_t, unsigned long long>::type;

    const StepView& v;
    const RowTree& t;
    uint32_t* s_mask;
    uint2* s_item;       // {node, state | depth << 16}
    uint32_t* s_bits;    // the items' stack symbols
    // token ranges: {first token, tokens, state, 0 or the filter: depth | (loop set + 1) << 8}
    uint4* s_range;      // kRowSmall short ones, then kRowBig longer ones
    uint4* s_exit;       // {first exit | depth << 24, exits, state | stack depth << 16, stack symbols}
    int* s_pre;
    RowShared& sh;
    int32_t* nrow;       // the row's next states
    const char* ahead;   // the row's logits in device memory, or nullptr
    int tok0, ntok;      // this CTA's token ids
    int tid, lane, warp;

    struct Item {
        uint32_t node, s, depth, bits;   // s == 0: none
    };

    // Tokens allowed with state s: n of the preorder list from lo on, the
    // first of which is `first`.
    struct Tokens {
        uint32_t lo, n, first, s;
    };
    // An item's expansion: its live children and its tokens.
    struct Node {
        Mask m, live, kids;   // live children, the state's live classes, the node's child classes
        uint32_t first_child;
        int c;                // WIDE: children
        Tokens em;
    };

    __device__ __forceinline__ void emit(int tk, uint32_t s) const {
        const int x = tk - tok0;
        if ((unsigned)x >= (unsigned)ntok) return;
        atomicOr(&s_mask[x >> 5], 1u << (x & 31));
        if constexpr (OUT == kRowBf16 || OUT == kRowF32) {   // its logit is read after the walk
            if (ahead) asm volatile("prefetch.global.L2 [%0];" ::"l"(ahead + (size_t)tk * (OUT == kRowBf16 ? 2 : 4)));
        }
        if constexpr (OUT == kRowNext) {
            if (nrow) nrow[tk] = (int32_t)s;
        }
    }

    // a node's tokens: one is set here, a range is left to the whole CTA (a
    // thread would wait for its token ids)
    __device__ __forceinline__ void emit(const Tokens& x, int4* st) const {
        if (x.n == 0u) return;
        if (x.n == 1u) {
            emit((int)x.first, x.s);
        } else if (!later(make_uint4(x.lo, x.n, x.s, 0u), st)) {
#pragma unroll 1
            for (uint32_t j = 0; j < x.n; ++j) emit(__ldg(t.dtok + x.lo + j), x.s);
        }
    }

    // leaves a token range to the whole CTA; false: its list is full
    __device__ __forceinline__ bool later(const uint4& range, int4* st) const {
        const bool small = range.y <= (uint32_t)kRowSmallTokens;
        const int which = small ? 0 : 1, i = atomicAdd(&sh.nrange[which], 1), cap = small ? kRowSmall : kRowBig;
        if (i >= cap / 2) st->z = 1;
        if (i >= cap) return false;
        s_range[which * kRowSmall + i] = range;
        return true;
    }

    // the entry of a class in state s, given its rank among the state's live classes
    __device__ __forceinline__ uint32_t target(uint32_t s, int rank) const {
        const unsigned char* r = reinterpret_cast<const unsigned char*>(t.srec) + (size_t)s * t.srec_stride + 16;
        if constexpr (STACK) return __ldg(reinterpret_cast<const uint32_t*>(r) + rank);
        else return __ldg(reinterpret_cast<const uint16_t*>(r) + rank);
    }
    __device__ __forceinline__ uint4 state_header(uint32_t s) const {
        return __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(t.srec) +
                                                    (size_t)s * t.srec_stride));
    }
    __device__ __forceinline__ uint32_t dense(uint32_t s, uint32_t c) const {
        if constexpr (STACK) return __ldg(v.t32 + (size_t)s * v.K + c);
        else return __ldg(v.t16 + (size_t)s * v.K + c);
    }
    __device__ __forceinline__ static Mask mask_of(uint32_t lo, uint32_t hi) {
        if constexpr (CLS == kRow32) return lo;
        else return ((unsigned long long)hi << 32) | lo;
    }

    // entry e taken with the stack (depth, bits): the child item (s == 0 when refused)
    __device__ __forceinline__ Item step(uint32_t child, uint32_t e, uint32_t depth, uint32_t bits) const {
        Item it{child, e, depth, bits};
        if constexpr (STACK) it.s = pda_apply(e, it.bits, it.depth, (uint32_t)v.max_depth, t.ret);
        return it;
    }

    __device__ __forceinline__ void put(int slot, const Item& it) const {
        s_item[slot] = make_uint2(it.node, it.s | (it.depth << 16));
        if constexpr (STACK) s_bits[slot] = it.bits;
    }
    __device__ __forceinline__ Item get(int slot) const {
        const uint2 x = s_item[slot];
        return Item{x.x, x.y & 0xFFFFu, x.y >> 16, STACK ? s_bits[slot] : 0u};
    }

    // The item's node record and state record, read together.  lead: this
    // thread answers for the item (and may add it to the loop subtrees).
    // before: the tokens of the thread's last item, set meanwhile.
    __device__ __forceinline__ Node read(const Item& it, bool lead, const Tokens& before, int4* st) const {
        Node x{};
        uint4 A = make_uint4(0u, 0u, 0u, 0u), B = A, h = A;
        if (it.s != 0u) {
#ifdef DOMINO_DEBUG
            if (it.node >= (uint32_t)t.n_nodes || it.s >= (uint32_t)v.Q) atomicOr(v.err, DOMINO_DEVERR_INTERNAL);
#endif
            A = __ldg(t.node + 2 * (size_t)it.node);
            B = __ldg(t.node + 2 * (size_t)it.node + 1);
            if constexpr (!WIDE) h = state_header(it.s);
        }
        emit(before, st);   // while the records are on their way
        if (it.s == 0u) return x;
        x.first_child = A.z & 0xFFFFFFu;
        x.em.lo = B.x;
        x.em.first = A.w;
        x.em.s = it.s;
        x.em.n = A.z >> 24;   // the tokens that end here
        if constexpr (WIDE) {
            x.c = (int)A.x;   // dead children too
            if (x.c == 0) x.em.n = B.y - B.x;
            else if (x.em.n == 255u) x.em.n = __ldg(&t.node[2 * (size_t)x.first_child + 1].x) - B.x;
        } else {
            x.live = mask_of(h.x, h.y);
            x.kids = mask_of(A.x, A.y);
            const Mask keep = mask_of(h.z, CLS == kRow32 ? 0u : h.w & 0x7FFFFFFFu);
            if ((mask_of(B.z, B.w) & ~keep) == 0) {
                x.em.n = B.y - B.x;   // every class below keeps the state: the subtree is allowed with it
            } else {
                x.m = x.kids & x.live;
                if (x.em.n == 255u) x.em.n = __ldg(&t.node[2 * (size_t)x.first_child + 1].x) - B.x;
                if ((h.w >> 31) && t.n_loops > 0 && lead && B.y - B.x > (uint32_t)kRowLoopMin && (x.kids & keep) != 0 &&
                    loop_subtree(it, B.x + x.em.n, B.y, st))
                    x.m = 0;
            }
        }
        return x;
    }

    // Places in the pool for c items of every thread of the warp: the slot of
    // the thread's first, or -1 when the pool is full.  `base` items stay in
    // the pool and the next round's item j lies in slot lo + j.  some: the
    // threads with c > 0 (not 0).
    __device__ __forceinline__ int places(int c, unsigned some, int base, int lo, int4* st) const {
        int at, tot;
        if (!__any_sync(0xffffffffu, c > 1)) {
            at = __popc(some & ((1u << lane) - 1u));
            tot = __popc(some);
        } else {
            const int incl = warp_scan_incl(c, lane);
            at = incl - c;
            tot = __shfl_sync(0xffffffffu, incl, 31);
        }
        int first = 0;
        if (lane == 0) first = base + atomicAdd(&st->x, tot);
        first = __shfl_sync(0xffffffffu, first, 0);
        if (first + tot > kRowPool) {
            st->y = 1;
            return -1;
        }
        return lo + first + at;
    }

    // WIDE: adds the item's live children, kWideAtOnce of them at a time, whose
    // classes and then entries are read together; kRowFan threads share an item
    // when split.  A wide node has up to 256 children of which few live in any
    // one state: with every child placed (and dropped a round later) rows of 1000
    // live nodes filled the pool.  GB300, 500 states, V = 128256, batch 256, masks,
    // us: 100 classes, 20 live 168 -> 27, 256 classes, 40 live 156 -> 26.
    __device__ __forceinline__ void add_wide(const Item& it, const Node& x, bool split, int base, int lo,
                                             int4* st) const {
        const int by = split ? kRowFan : 1;
        for (int k0 = split ? tid & (kRowFan - 1) : 0; __any_sync(0xffffffffu, k0 < x.c); k0 += kWideAtOnce * by) {
            uint32_t e[kWideAtOnce];
#pragma unroll
            for (int q = 0; q < kWideAtOnce; ++q)
                e[q] = k0 + q * by < x.c ? (uint32_t)__ldg(t.ncls + x.first_child + (uint32_t)(k0 + q * by)) : 0u;
            int c = 0;
#pragma unroll
            for (int q = 0; q < kWideAtOnce; ++q) {
                e[q] = k0 + q * by < x.c ? dense(it.s, e[q]) : 0u;
                c += e[q] != 0u;
            }
            const unsigned some = __ballot_sync(0xffffffffu, c > 0);
            if (!some) continue;
            int at = places(c, some, base, lo, st);
            if (at < 0) return;
#pragma unroll
            for (int q = 0; q < kWideAtOnce; ++q)
                if (e[q]) put(at++, step(x.first_child + (uint32_t)(k0 + q * by), e[q], it.depth, it.bits));
        }
    }

    // Expands the pool's n items until none are left.  In a round every
    // thread takes one item from the pool's top (kRowFan threads share one
    // while there are few) and adds its live children.  A round that takes all
    // items puts them behind those, so that no warp waits for the others to have
    // read theirs; only when the items lie past the spare slots, or some stay,
    // do they take the place of those read.  In two halves of 2048 slots, taken
    // in turn, rows with levels of 2000 live nodes were full and walked twice
    // (GB300, 500 states, V = 128256, batch 256, masks, us: 48 classes, 16 live
    // 192 -> 36, 64 classes, 20 live 189 -> 35, 32 classes, 14 live 225 -> 56;
    // 5000 states 15.8 -> 15.6, JSON, V = 152064, batch 128 23.9 -> 24.0).
    // false: the pool was full (every_token() takes the row).
    __device__ __forceinline__ bool run(int n) const {
        int lo = 0;   // the items lie in slots lo to lo + n - 1
        Tokens before{0u, 0u, 0u, 0u};
        for (int r = 0;; r = r == 2 ? 0 : r + 1) {
            int4* st = &sh.st[r];
            if (n == 0) {
                n = spawn_exits();   // the same for every thread of the CTA
                if (n == 0) break;
                lo = 0;
            }
            const int take = min(n, THREADS);
            const int base = n - take;
            const bool fan = take * kRowFan <= THREADS;
            const int i = fan ? tid / kRowFan : tid;
            bool lead = !fan || (tid & (kRowFan - 1)) == 0;   // this thread answers for its item
            Item it{0u, 0u, 0u, 0u};
            if (i < take) it = get(lo + base + i);
            if (tid == 0) sh.st[r == 2 ? 0 : r + 1] = make_int4(0, 0, 0, 0);   // read by all two rounds ago
            if (base > 0 || lo + take > kRowSlots - kRowPool) {
                __syncthreads();   // the items are read before others take their place
                if (base == 0) lo = 0;
            } else {
                lo += take;
            }
            if ((fan ? (tid & ~31) / kRowFan : tid & ~31) < take) {   // warps with an item
              for (bool split = fan;;) {
                Node x = read(it, lead, before, st);
                if constexpr (WIDE) {
                    add_wide(it, x, split, base, lo, st);
                } else {
                    // this thread's share of the children
                    Mask m = x.m;
                    if (split) {
                        if (t.n_loops > 0) m = shfl_lead(m);   // the lead may have taken the subtree whole
                        constexpr int kWidth = (int)sizeof(Mask) * 8 / kRowFan;   // classes per thread
                        m &= (((Mask)1 << kWidth) - 1) << (kWidth * (tid & (kRowFan - 1)));
                    }
                    const int c = popc(m);
                    const unsigned some = __ballot_sync(0xffffffffu, c > 0);
                    // thin tails: while no warp has left work in the pool and
                    // this one's items have at most one child each, its
                    // threads go on with the children themselves
                    if (some && !__any_sync(0xffffffffu, c > 1) &&
                        __popc(some) <= __popc(__ballot_sync(0xffffffffu, lead && it.s != 0u)) &&
                        !__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&st->x) != 0)) {
                        before = x.em;
                        if (!lead) before.n = 0u;
                        if (c) {
                            const Mask below = m - 1;   // one bit
                            it = step(x.first_child + (uint32_t)popc(x.kids & below), target(it.s, popc(x.live & below)),
                                      it.depth, it.bits);
                        } else {
                            it.s = 0u;
                        }
                        split = false;
                        lead = true;
                        continue;
                    }
                    // places for the children, warp by warp
                    if (some) {
                        int at = places(c, some, base, lo, st);
                        for (m = at < 0 ? 0 : m; m; m &= m - 1) {
                            const Mask below = (m & (~m + 1)) - 1;
                            put(at++, step(x.first_child + (uint32_t)popc(x.kids & below),
                                           target(it.s, popc(x.live & below)), it.depth, it.bits));
                        }
                    }
                }
                before = x.em;
                if (!lead) before.n = 0u;
                break;
              }
            }
            __syncthreads();   // the next round's items are in place
            const int4 q = *st;
            if (q.y) return false;
            n = base + q.x;
            if (q.z) ranges();
        }
        emit(before, &sh.st[0]);
        return true;
    }

    __device__ __forceinline__ uint32_t shfl_lead(uint32_t m) const {
        return __shfl_sync(0xffffffffu, m, lane & ~(kRowFan - 1));
    }
    __device__ __forceinline__ unsigned long long shfl_lead(unsigned long long m) const {
        return ((unsigned long long)shfl_lead((uint32_t)(m >> 32)) << 32) | shfl_lead((uint32_t)m);
    }

    // A node entered in a looping state (RowTree).  The tokens [lo, hi) below
    // it whose remainder stays inside the loop set are a filtered range, the
    // others are reached through the edges that first leave the set; both are
    // left to the whole CTA.  false: not taken.
    __device__ __forceinline__ bool loop_subtree(const Item& it, uint32_t lo, uint32_t hi, int4* st) const {
        const uint32_t set = __ldg(t.loop_of + it.s);
        const uint2 x = __ldg(t.xrange + (size_t)set * t.n_nodes + it.node);   // {first exit below | depth << 24, end}
        const uint32_t d = x.x >> 24, n_exit = x.y - (x.x & 0xFFFFFFu);
        if (d == 255u) return false;   // deeper than a byte holds
        int j = 0;
        if (n_exit) {
            j = atomicAdd(&sh.nexit, 1);
            if (j >= kExits) return false;
            s_exit[j] = make_uint4(x.x, 0u, it.s | (it.depth << 16), it.bits);
        }
        if (!later(make_uint4(lo, hi - lo, it.s, d | ((set + 1u) << 8)), st)) return false;   // (an empty entry stays behind)
        if (n_exit) s_exit[j].y = n_exit;
        return true;
    }

    // Exclusive prefix sums of x over threads 0..n-1 into s_pre[0..n]; the total.
    __device__ __forceinline__ int prefix(int n, int x) const {
        int incl = warp_scan_incl(tid < n ? x : 0, lane);
        if (lane == 31) sh.wsum[warp] = incl;
        __syncthreads();
        for (int k = 0; k < warp; ++k) incl += sh.wsum[k];
        if (tid < n) s_pre[tid + 1] = incl;
        if (tid == 0) s_pre[0] = 0;
        __syncthreads();
        return s_pre[n];
    }

    // The loop subtrees' exits become the pool's items, in its first slots
    // (the pool is empty before).  Returns their number, 0 when none are left.
    __device__ __forceinline__ int spawn_exits() const {
        if (t.n_loops == 0) return 0;
        for (;;) {
            const int nx = min(*reinterpret_cast<volatile int*>(&sh.nexit), kExits);
            if (nx == 0) return 0;
            if (tid == 0) sh.back = 0;
            const int total = prefix(nx, tid < nx ? (int)s_exit[tid].y : 0);
            // as many as fit this time, the last entries first (the list is a
            // stack); an entry taken in part is cut back
            const int f0 = max(0, total - kRowSpawn);
            for (int b = f0 + warp * 32; b < total; b += THREADS) {
                const int f = b + lane;
                Item x{0u, 0u, 0u, 0u};
                if (f < total) {
                    const int k = find_range(s_pre, nx, f);
                    const uint4 e = s_exit[k];
                    const uint2 q = __ldg(t.exits + (e.x & 0xFFFFFFu) + (uint32_t)(f - s_pre[k]));
                    if ((q.y >> 8) <= e.x >> 24) {   // no edge before it leaves the set
                        const uint32_t s = e.z & 0xFFFFu;
                        const uint4 h = state_header(s);
                        const Mask live = mask_of(h.x, h.y), bit = (Mask)1 << (q.y & 0xFFu);
                        if (live & bit) x = step(q.x, target(s, popc(live & (bit - 1))), e.z >> 16, e.w);
                    }
                }
                const unsigned ok = __ballot_sync(0xffffffffu, x.s != 0u);
                int first = 0;
                if (lane == 0 && ok) first = atomicAdd(&sh.back, __popc(ok));
                first = __shfl_sync(0xffffffffu, first, 0);
                if (x.s != 0u) put(first + __popc(ok & ((1u << lane) - 1u)), x);
            }
            __syncthreads();   // the items are in place, the list has been read
            if (tid == 0) {
                int left = 0;
                if (f0 > 0) {
                    left = find_range(s_pre, nx, f0);
                    const int part = f0 - s_pre[left];
                    if (part > 0) {
                        s_exit[left].y = (uint32_t)part;
                        left++;
                    }
                }
                sh.nexit = left;
            }
            const int n = *reinterpret_cast<volatile int*>(&sh.back);
            __syncthreads();
            if (n > 0) return n;
        }
    }

    // Sets the token ranges left by the rounds and empties their lists.
    // Every thread calls it, after a barrier that follows the last round.
    __device__ __forceinline__ void ranges() const {
        const int ns = min(*reinterpret_cast<volatile int*>(&sh.nrange[0]), kRowSmall);
        const int nb = min(*reinterpret_cast<volatile int*>(&sh.nrange[1]), kRowBig);
        constexpr int kUnroll = STACK ? 8 : 4;   // 8 spill beside a DFA's folded decode: +0.8 us at 128256x256
        // short ones: four threads each
        for (int i = tid / 4; i < ns; i += THREADS / 4) {
            const uint4 x = s_range[i];
            for (uint32_t j = tid & 3; j < x.y; j += 4 * kUnroll) {
                int tk[kUnroll];
                uint32_t out[kUnroll];   // the filter's byte: greater than the range's depth drops the token
                const int32_t* p = t.dtok + x.x + j;
                const uint8_t* k = t.keeps + (x.w ? (size_t)((x.w >> 8) - 1u) * t.n_dtok + x.x + j : 0);
#pragma unroll
                for (int q = 0; q < kUnroll; ++q) {
                    tk[q] = j + 4 * q < x.y ? __ldg(p + 4 * q) : -1;
                    out[q] = x.w && j + 4 * q < x.y ? __ldg(k + 4 * q) : 0u;
                }
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (tk[q] >= 0 && out[q] <= (x.w & 0xFFu)) emit(tk[q], x.z);
            }
        }
        if (nb > 0) {   // long ones: the CTA over all of them
            const int total = prefix(nb, tid < nb ? (int)s_range[kRowSmall + tid].y : 0);
            // a warp takes 256 tokens in a row: they lie in a few ranges
            for (int f0 = warp * 32 * kUnroll; f0 < total; f0 += THREADS * kUnroll) {
                int tk[kUnroll];
                uint32_t st[kUnroll], out[kUnroll];
                int k = find_range(s_pre, nb, f0), end = s_pre[k + 1];
                uint4 b = s_range[kRowSmall + k];
                uint32_t at = b.x - (uint32_t)s_pre[k];   // the list's index of token f is at + f
#pragma unroll
                for (int q = 0; q < kUnroll; ++q) {
                    const int f = f0 + 32 * q + lane;
                    tk[q] = -1;
                    st[q] = out[q] = 0u;
                    if (f < total) {
                        while (f >= end) {
                            ++k;
                            b = s_range[kRowSmall + k];
                            at = b.x - (uint32_t)end;
                            end = s_pre[k + 1];
                        }
                        const uint32_t i = at + (uint32_t)f;
                        tk[q] = __ldg(t.dtok + i);
                        st[q] = b.z | (b.w << 16);   // the state and the filter's depth
                        if (b.w) out[q] = __ldg(t.keeps + (size_t)((b.w >> 8) - 1u) * t.n_dtok + i);
                    }
                }
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (tk[q] >= 0 && out[q] <= ((st[q] >> 16) & 0xFFu)) emit(tk[q], st[q] & 0xFFFFu);
            }
        }
        __syncthreads();   // the lists have been read
        if (tid == 0) sh.nrange[0] = sh.nrange[1] = 0;
        __syncthreads();
    }
};

// C.update() of a row in configuration rc (read_row) by its token tk, or by
// -1: as advance_row, with the token's classes in one record.
template <bool STACK>
__device__ __forceinline__ void update(const StepView& v, const RowTree& t, const uint4& rc, int32_t tk, int b,
                                       int32_t* states_out, uint64_t* stacks_out) {
    uint32_t s = 0, bits = 0, depth = 0;
    if (tk < 0 || tk == v.eos_id) {
        s = (uint32_t)v.start;   // the sequence ended; the next one starts from init
    } else if (rc.w & 1u) {
        bits = rc.y;
        depth = rc.z;
        s = token_end<STACK>(v, t, tk, rc.x, bits, depth);
        if (s == 0) bits = depth = 0;
    }
    states_out[b] = (int32_t)s;
    if (stacks_out) stacks_out[b] = ((uint64_t)depth << 32) | bits;
}

template <bool STACK, int CLS, int OUT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
    row_kernel(const __grid_constant__ StepView v, const __grid_constant__ RowTree t,
               const __grid_constant__ RowArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RowShared sh;
    const RowLayout L = row_layout(a.slice_words, STACK, t.n_loops > 0, OUT == kRowBf16 || OUT == kRowF32);
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + L.mask);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = blockIdx.x / a.slices, slice = blockIdx.x - row * a.slices;
    const int w0 = slice * a.slice_words, nw = max(0, min(a.slice_words, v.W - w0));
    const int tok0 = w0 * 32, ntok = max(0, min(nw * 32, v.V - tok0));
    for (int j = tid; j < a.slice_words / 4; j += THREADS)
        reinterpret_cast<uint4*>(s_mask)[j] = make_uint4(0u, 0u, 0u, 0u);
    constexpr bool kDecode = OUT == kRowBf16 || OUT == kRowF32;
    if constexpr (OUT == kRowBf16) fill_keep<THREADS>(reinterpret_cast<uint4*>(smem + L.keep), tid);
    if (tid == 0) {
        s_mask[-1] = s_mask[a.slice_words] = 0u;
        sh.nrange[0] = sh.nrange[1] = sh.nexit = 0;
        sh.st[0] = make_int4(0, 0, 0, 0);
    }
    pdl_wait();
    pdl_trigger();
    // The row's configuration (invalid ones set the error word, once per row),
    // in shared memory: one in pinned host memory crosses the host link once
    // per CTA, not once per warp (128256 tokens, batch 16, states read there:
    // 33.2 -> 21.4 us), and no registers are held for it during the walk.
    if (tid == 0) {
        const uint32_t q = (uint32_t)row;
        sh.rc = a.row_is_state
                    ? make_uint4(q, 0u, 0u, 1u | (((__ldg(v.accept_bits + (q >> 5)) >> (q & 31u)) & 1u) ? 2u : 0u))
                    : read_row_rw(v, a.states, a.stacks, row, slice == 0);
    }
    __syncthreads();
    const uint4 rc = sh.rc;
    // the state the walk starts from, and its loop set
    uint32_t s0 = (rc.w & 1u) ? rc.x : 0u, root = 0u;
    if (t.start) {
        const uint2 w = __ldg(t.start + s0);
        s0 = w.x;
        if (w.y != 0xFFFFFFFFu) {   // the tokens that stay inside the set, then the walk of the others
            const uint32_t* loop = t.loopbits + (size_t)w.y * v.W + w0;
            for (int j = tid; j < nw; j += THREADS) s_mask[j] = __ldg(loop + j);
            root = (uint32_t)t.loop_root[w.y];
        }
    }
    int32_t* nrow = nullptr;
    if constexpr (OUT == kRowNext) {
        // the row's next states are 0 before the walk stores its tokens'
        nrow = a.next ? a.next + (size_t)row * v.V : nullptr;
        if (nrow) {
            if ((v.V & 3) == 0 && (reinterpret_cast<uintptr_t>(a.next) & 15) == 0) {
                int4* dst = reinterpret_cast<int4*>(nrow + tok0);
                for (int j = tid; j < ntok / 4; j += THREADS) dst[j] = make_int4(0, 0, 0, 0);
            } else {
                for (int j = tid; j < ntok; j += THREADS) nrow[tok0 + j] = 0;
            }
        }
    }
    const char* ahead = nullptr;
    if constexpr (kDecode)
        if (a.ahead)
            ahead = reinterpret_cast<const char*>(a.logits) +
                    (size_t)row * (size_t)a.stride * (OUT == kRowBf16 ? 2 : 4);
    const RowWalk<STACK, CLS, OUT, THREADS> wk{v, t, s_mask, reinterpret_cast<uint2*>(smem + L.items),
                                      reinterpret_cast<uint32_t*>(smem + L.bits),
                                      reinterpret_cast<uint4*>(smem + L.range),
                                      reinterpret_cast<uint4*>(smem + L.exits), reinterpret_cast<int*>(smem + L.pre), sh,
                                      nrow, ahead, tok0, ntok, tid, lane, warp};
    if (tid == 0) wk.put(0, {root, s0, rc.z, rc.y});
    __syncthreads();   // the mask (and the next states) are filled
    if (wk.run(s0 != 0u ? 1 : 0)) {
        __syncthreads();
        wk.ranges();
    } else {
        every_token<STACK, OUT>(v, t, sh.rc, s_mask, nw, tok0, ntok, nrow, ahead);
        __syncthreads();   // whole words were stored
    }
    if (tid == 0 && v.eos_id >= 0 && (static_cast<volatile uint32_t&>(sh.rc.w) & 2u))
        wk.emit(v.eos_id, static_cast<volatile uint32_t&>(sh.rc.x));   // EOS keeps the state
    __syncthreads();
    if (a.mask) {
        uint32_t* mrow = a.mask + (size_t)row * v.W + w0;
        if ((v.W & 3) == 0 && (reinterpret_cast<uintptr_t>(a.mask) & 15) == 0) {
            for (int j = tid; j < nw / 4; j += THREADS)
                reinterpret_cast<uint4*>(mrow)[j] = reinterpret_cast<const uint4*>(s_mask)[j];
        } else {
            for (int j = tid; j < nw; j += THREADS) mrow[j] = s_mask[j];
        }
    }
    if constexpr (kDecode) {
        DecodeShared& dsh = *reinterpret_cast<DecodeShared*>(smem + L.dec);
        Decoder<OUT == kRowBf16, kFoldLse> d;
        d.init(a.logits, a.stride, row, v.V, a.logprobs != nullptr, SampleArgs{},
               reinterpret_cast<const uint4*>(smem + L.keep), lane);
        d.template slice<THREADS>(s_mask, tok0, ntok, reinterpret_cast<uint16_t*>(smem + L.items) + warp * kDecodeList, warp);
        d.finish();
        float m = d.m, sum = d.s;
        int idx = d.idx;
        decode_combine<THREADS>(dsh, m, idx, sum, a.slices, lane, warp);
        const float lse = log_sum_exp(m, sum);
        if (a.logprobs)
            write_logprobs<OUT == kRowBf16, THREADS>(d.lrow, v.V, s_mask, tok0, ntok, lse, a.logprobs + (size_t)row * v.V, tid);
        if (slice == 0 && tid == 0) {
            const int32_t tk = m == -INFINITY ? -1 : idx;
            a.argmax[row] = tk;
            if (a.lse) a.lse[row] = lse;
            // every CTA of the row has read its configuration (the outputs may alias it)
            if (a.states_out) update<STACK>(v, t, sh.rc, tk, row, a.states_out, a.stacks_out);
        }
        if (a.slices > 1) cluster_wait();
    }
}

// Raises a kernel's dynamic shared-memory limit on the current device once
// per size (one array of configured sizes per kernel instance).
template <typename K>
cudaError_t rows_allow_smem(K kern, int bytes, int* configured, std::mutex& mu) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (bytes <= 40 * 1024) return cudaSuccess;   // with the static part within the default 48 KiB
    std::lock_guard<std::mutex> lk(mu);
    if (dev < kRowMaxDevices && configured[dev] >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && dev < kRowMaxDevices) configured[dev] = bytes;
    return e;
}

template <bool STACK, int CLS, int OUT, int THREADS>
cudaError_t launch_row_d(const StepView& v, const RowTree& t, const LaunchEnv& env, RowArgs a, cudaStream_t st) {
    // CTAs per row: enough to give every SM one (two where a row is decoded
    // and has two: JSON, V = 152064, batch 128 54.6 -> 45.7 us), and enough for
    // the row's words to fit
    int s = 1;
    while (s < kRowMaxSlices &&
           ((int64_t)a.batch * s * 2 <= (s == 1 && a.logits ? 2 : 1) * env.num_sms || (v.W + s - 1) / s > kRowSliceWords))
        s *= 2;
    a.slices = s;
    a.slice_words = ((v.W + s - 1) / s + 3) / 4 * 4;
    const RowLayout L = row_layout(a.slice_words, STACK, t.n_loops > 0, OUT == kRowBf16 || OUT == kRowF32);
    if (L.total > env.max_smem_optin) return cudaErrorInvalidConfiguration;
    auto kern = row_kernel<STACK, CLS, OUT, THREADS>;
    static int configured[kRowMaxDevices] = {0};
    static std::mutex mu;
    cudaError_t e = rows_allow_smem(kern, L.total, configured, mu);
    if (e != cudaSuccess) return e;
    return launch_cluster(kern, dim3((unsigned)a.batch * (unsigned)s), dim3(THREADS), s, (size_t)L.total, st, v, t, a);
}

template <bool STACK, int CLS, int OUT>
cudaError_t launch_row_t(const StepView& v, const RowTree& t, const LaunchEnv& env, const RowArgs& a, cudaStream_t st) {
    // More rows than run at once with 2 CTAs an SM (one CTA a row): CTAs of
    // half the threads, of which up to 4 fit, take more rows a wave, each wave
    // being 1.1 to 1.3 times as long.  GB300, us, 512 / 256 threads: 5000 states,
    // V = 128256, steps of 310 rows 37.2 / 28.7, 500 rows 42.8 / 47.6 (two waves
    // either way), 1000 rows 78.8 / 74.6; V = 32000, 1000 rows 61.4 / 39.9;
    // 256 rows of 128256 23.1 / 28.5.  The log-probabilities want the threads:
    // 310 rows 91.6 / 76.9, 620 rows (three waves, two) 144 / 152.  So do long
    // rows of next states: tables, V = 32000 194 / 162, V = 64000 302 / 314.
    // 100 classes, 20 live, V = 32000, masks of 400 rows 29.7 / 22.5, 1000 rows
    // 58.5 / 39.6.
    // With a stack the rounds are longer: JSON, V = 152064, 512 rows 78.6 / 98.1.
    if constexpr (!STACK) {
        const RowLayout L = row_layout((v.W + 3) / 4 * 4, STACK, t.n_loops > 0, OUT == kRowBf16 || OUT == kRowF32);
        const int64_t fit = std::min(4, (env.max_smem_optin + 1024) / (L.total + 1024 + (int)sizeof(RowShared)));
        if (fit > 2 && a.batch > 2 * env.num_sms && (OUT != kRowNext || v.V <= kRowNextHalf)) {
            const int64_t full = (a.batch - 1) / (2 * env.num_sms) + 1, half = (a.batch - 1) / (fit * env.num_sms) + 1;
            if (a.logprobs ? 2 * half <= full : 5 * half < 4 * full)
                return launch_row_d<STACK, CLS, OUT, kRowThreads / 2>(v, t, env, a, st);
        }
    }
    return launch_row_d<STACK, CLS, OUT, kRowThreads>(v, t, env, a, st);
}

template <bool STACK, int CLS>
cudaError_t launch_row_o(const StepView& v, const RowTree& t, const LaunchEnv& env, const RowArgs& a, int dtype,
                         cudaStream_t st) {
    if (a.logits)
        return dtype == DOMINO_DTYPE_BF16 ? launch_row_t<STACK, CLS, kRowBf16>(v, t, env, a, st)
                                          : launch_row_t<STACK, CLS, kRowF32>(v, t, env, a, st);
    return a.next ? launch_row_t<STACK, CLS, kRowNext>(v, t, env, a, st)
                  : launch_row_t<STACK, CLS, kRowMask>(v, t, env, a, st);
}

cudaError_t launch_row(const StepView& v, const RowTree& t, const LaunchEnv& env, bool stack, const RowArgs& a,
                       int dtype, cudaStream_t st) {
    if (a.batch <= 0) return cudaSuccess;
    if (v.K <= 32)
        return stack ? launch_row_o<true, kRow32>(v, t, env, a, dtype, st)
                     : launch_row_o<false, kRow32>(v, t, env, a, dtype, st);
    if (v.K <= 64)
        return stack ? launch_row_o<true, kRow64>(v, t, env, a, dtype, st)
                     : launch_row_o<false, kRow64>(v, t, env, a, dtype, st);
    return stack ? launch_row_o<true, kRowWide>(v, t, env, a, dtype, st)
                 : launch_row_o<false, kRowWide>(v, t, env, a, dtype, st);
}

}  // namespace

cudaError_t launch_row_step(const StepView& v, const RowTree& t, const LaunchEnv& env, bool stack,
                            const int32_t* states, const uint64_t* stacks, int32_t batch, bool row_is_state,
                            uint32_t* mask, int32_t* next, cudaStream_t st) {
    RowArgs a{};
    a.states = states;
    a.stacks = stacks;
    a.batch = batch;
    a.row_is_state = row_is_state ? 1 : 0;
    a.mask = mask;
    a.next = next;
    return launch_row(v, t, env, stack, a, 0, st);
}

cudaError_t launch_row_decode(const StepView& v, const RowTree& t, const LaunchEnv& env, bool stack,
                              const int32_t* states, const uint64_t* stacks, int32_t batch, const void* logits,
                              int dtype, int64_t row_stride, bool on_device, uint32_t* mask, int32_t* argmax,
                              float* lse, float* logprobs, int32_t* states_out, uint64_t* stacks_out, cudaStream_t st) {
    RowArgs a{};
    a.states = states;
    a.stacks = stacks;
    a.batch = batch;
    a.mask = mask;
    a.logits = logits;
    a.stride = row_stride;
    a.ahead = on_device ? 1 : 0;
    a.argmax = argmax;
    a.lse = lse;
    a.logprobs = logprobs;
    a.states_out = states_out;
    a.stacks_out = stacks_out;
    return launch_row(v, t, env, stack, a, dtype, st);
}

int row_smem_bytes(int32_t n_words, bool stack, bool loops) {
    return row_layout(std::min(n_words, kRowSliceWords) + 4, stack, loops, true).total;
}

}  // namespace domino
