// host.cpp -- the C ABI of libdomino.so: handle lifetime, loaders (validation,
// dead-state canonicalisation, byte-class compression, vocabulary arena) and
// argument checks in front of the kernels in kernels.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <numeric>
#include <unordered_map>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "domino.h"
#include "domino_internal.h"

using namespace domino;

namespace {

struct DevBuf {
    void* p = nullptr;
    size_t n = 0;
};

}  // namespace

struct domino_ctx {
    int device = -1;
    LaunchEnv env{0, 0};

    // ---- vocabulary (host copy, kept so the arena can be rebuilt per automaton)
    bool vocab_loaded = false;
    int32_t V = 0, W = 0, eos_id = -1, max_len = 0;
    std::vector<uint8_t> tok_bytes;
    std::vector<int64_t> tok_off;

    // ---- automaton (preprocessed)
    bool auto_loaded = false;
    int32_t Q = 0, K = 0, start = 0, max_depth = 0, n_rules = 0;
    bool stack = false;
    uint8_t byte_class[256] = {0};
    std::vector<uint16_t> t16;
    std::vector<uint32_t> t32;
    std::vector<uint16_t> ret;
    std::vector<uint32_t> accept_bits;
    std::vector<uint64_t> self_mask;   // [Q]: classes that keep the state (no stack action); empty if unused
    int32_t sp_nnz = 0;       // live entries of the sparse table (0: no sparse image)
    int32_t sp_words = 0;     // uint32 words per state in the sparse row info (2 or 4)
    int64_t dense_ret_off = 0, sp_tgt_off = 0, sp_ret_off = 0;

    // ---- device copies
    DevBuf d_head, d_info, d_tail_off, d_tail, d_pos_of, d_cls_start, d_eos_slot;
    DevBuf d_dense, d_sparse, d_accept, d_self, d_tok_cls;
    DevBuf d_err, d_fpart;
    std::vector<DevBuf> fpart_old;   // outgrown ones: recorded graphs may still name them
    bool arena_ready = false;
    // prefix tree of the class strings (domino_get_prefix_tree)
    std::vector<uint4> t_node;
    std::vector<int32_t> t_dtok;
    std::vector<uint4> t_upper;      // {node, path offset, path length, 0}
    std::vector<uint8_t> t_upath;
    std::vector<uint2> t_unit;       // {root node, parent upper index}
    int32_t t_nodes = 0;
    bool trie_built = false;
    // the trees row_kernel walks (see RowTree)
    DevBuf d_rnode, d_rncls, d_rdtok, d_srec, d_srec_next, d_rret, d_rstart, d_loop_of, d_loopbits, d_keeps, d_xrange,
        d_exits, d_trec;
    RowTree rows{}, rows_next{};     // for masks; for next states
    bool rows_ready = false;
    bool rows_dense = false;         // most rows' walks are too large for it (row_cost)
    int64_t rows_visits = 0;         // nodes a row's walk visits
    // which walk the mask step takes: -1 chosen from the automaton (see
    // use_tree), 1 the prefix tree, 0 every token on its own (DOMINO_WALK=tree
    // or =token in the environment when the handle is created)
    int walk_pref = -1;
    int32_t n_windows = 0;
    // staging for domino_decode_step_host
    // s_io packs the step's small inputs and outputs (see io_layout) so that
    // each direction takes one copy through the pinned staging buffer h_io
    DevBuf s_logits, s_mask, s_io;
    void* h_io = nullptr;
    void* h_io_dev = nullptr;   // h_io as the device addresses it
    size_t h_io_n = 0;
    // opportunistic masking: proposals, the fallback row list and its length
    DevBuf o_prop, o_rows, o_count;
    // domino_decode_step_host: a copy stream and the events that hand each
    // chunk of rows from the copies to the kernels
    cudaStream_t cp_stream = nullptr;
    cudaEvent_t ev_cfg = nullptr;
    cudaEvent_t ev_chunk[8] = {};
    cudaEvent_t ev_t[4] = {};       // the chunked copy's start and end (2, 3)
    // host wall time of each path for pinned bf16 logits, a moving average
    // over settled calls: [0] the chunked copy, [1] the in-place read (0: not
    // yet seen)
    double t_wall_ms[2] = {0.0, 0.0};
    // Recorded host-buffer steps: a call whose buffers, sizes and path match an
    // earlier one replays that call's CUDA graph instead of issuing each copy
    // and launch again.  Cleared when an automaton or vocabulary is loaded.
    struct HostGraph {
        const void* key[16];
        cudaGraphExec_t exec;
        uint64_t used;
    };
    std::vector<HostGraph> host_graphs;
    uint64_t host_calls = 0;
};

namespace {

StepView make_view(domino_ctx* h);
int cuda_status(cudaError_t e);

struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    explicit DeviceGuard(int dev) {
        if (dev < 0) return;
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) {
            changed = cudaSetDevice(dev) == cudaSuccess;
        }
    }
    ~DeviceGuard() {
        if (changed) cudaSetDevice(prev);
    }
};

void dev_free(DevBuf& b) {
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.n = 0;
}

int64_t dev_bytes(const domino_ctx* h) {
    const DevBuf* all[] = {&h->d_head, &h->d_info, &h->d_tail_off, &h->d_tail, &h->d_pos_of, &h->d_cls_start,
                           &h->d_eos_slot, &h->d_dense, &h->d_sparse, &h->d_accept, &h->d_self, &h->d_tok_cls, &h->d_err, &h->d_fpart, &h->s_logits, &h->s_mask, &h->s_io,
                           &h->o_prop, &h->o_rows, &h->o_count, &h->d_rnode, &h->d_rncls, &h->d_rdtok, &h->d_srec,
                           &h->d_srec_next, &h->d_rret, &h->d_rstart, &h->d_loop_of, &h->d_loopbits, &h->d_keeps,
                           &h->d_xrange, &h->d_exits, &h->d_trec};
    int64_t n = 0;
    for (auto* b : all) n += (int64_t)b->n;
    for (const DevBuf& b : h->fpart_old) n += (int64_t)b.n;
    return n;
}

// (Re)allocates b to hold n bytes and uploads src (when non-null).
int dev_upload(DevBuf& b, const void* src, size_t n) {
    size_t want = ((n ? n : 16) + 15) / 16 * 16;   // vector staging reads whole 16-byte words
    if (b.n < want) {
        dev_free(b);
        if (cudaMalloc(&b.p, want) != cudaSuccess) {
            cudaGetLastError();
            b.p = nullptr;
            return DOMINO_E_OOM;
        }
        b.n = want;
    }
    if (src && n && cudaMemcpy(b.p, src, n, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        return DOMINO_E_CUDA;
    }
    return DOMINO_OK;
}

int dev_reserve(DevBuf& b, size_t n) { return dev_upload(b, nullptr, n); }

// The fused decode's partials, n bytes or more.  An outgrown buffer is kept
// until the handle is destroyed: a graph that a caller recorded at a smaller
// batch goes on using it.  Sizes at least double, so the outgrown ones take
// no more than the buffer itself.
int grow_fpart(domino_ctx* h, size_t n) {
    if (h->d_fpart.n >= n) return DOMINO_OK;
    DevBuf b;
    if (int rc = dev_reserve(b, std::max(n, 2 * h->d_fpart.n))) return rc;
    if (h->d_fpart.p) h->fpart_old.push_back(h->d_fpart);
    h->d_fpart = b;
    return DOMINO_OK;
}

bool is_host_only(const domino_ctx* h) { return h->device < 0; }

void clear_host_graphs(domino_ctx* h) {
    for (auto& g : h->host_graphs) cudaGraphExecDestroy(g.exec);
    h->host_graphs.clear();
    h->t_wall_ms[0] = h->t_wall_ms[1] = 0.0;   // the paths are timed afresh
}

// The prefix tree of the tokens' class strings, built from the
// tokens sorted by class string: a token shares with its predecessor the
// nodes of their longest common prefix and opens new nodes for the rest, so
// nodes come out in preorder.  EOS and empty tokens are not in the tree (the
// kernel sets EOS from the row's acceptance; other empty tokens are never
// allowed).  Host arrays only: domino_get_prefix_tree copies them, and
// make_row_image takes the tokens' order for the trees the kernel walks.
void build_trie_host(domino_ctx* h) {
    h->trie_built = false;
    h->t_node.clear();
    h->t_dtok.clear();
    h->t_upper.clear();
    h->t_upath.clear();
    h->t_unit.clear();
    if (!h->vocab_loaded || !h->auto_loaded) return;
    std::vector<uint8_t> cls(h->tok_bytes.size());
    for (size_t i = 0; i < cls.size(); i++) cls[i] = h->byte_class[h->tok_bytes[i]];
    std::vector<int32_t> order;
    order.reserve((size_t)h->V);
    for (int32_t t = 0; t < h->V; t++)
        if (t != h->eos_id && h->tok_off[t + 1] > h->tok_off[t]) order.push_back(t);
    auto str = [&](int32_t t) { return cls.data() + h->tok_off[t]; };
    auto len = [&](int32_t t) { return (size_t)(h->tok_off[t + 1] - h->tok_off[t]); };
    std::sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
        const size_t la = len(a), lb = len(b);
        const int c = std::memcmp(str(a), str(b), std::min(la, lb));
        if (c != 0) return c < 0;
        if (la != lb) return la < lb;
        return a < b;
    });
    std::vector<uint32_t> skip, tok_lo, n_end, tok_hi;
    std::vector<uint8_t> ncls;
    std::vector<int32_t> dtok;
    dtok.reserve(order.size());
    std::vector<uint32_t> path;   // open nodes, root first
    auto open_node = [&](uint8_t c) {
        path.push_back((uint32_t)skip.size());
        skip.push_back(0);
        tok_lo.push_back((uint32_t)dtok.size());
        n_end.push_back(0);
        tok_hi.push_back(0);
        ncls.push_back(c);
    };
    auto close_node = [&]() {
        const uint32_t n = path.back();
        path.pop_back();
        skip[n] = (uint32_t)skip.size();
        tok_hi[n] = (uint32_t)dtok.size();
    };
    open_node(0);   // root
    const uint8_t* prev = nullptr;
    size_t prev_len = 0;
    for (int32_t t : order) {
        const uint8_t* s = str(t);
        const size_t L = len(t);
        size_t l = 0;
        while (prev && l < std::min(L, prev_len) && prev[l] == s[l]) l++;
        while (path.size() > l + 1) close_node();
        for (size_t d = l; d < L; d++) open_node(s[d]);
        if (skip.size() > (size_t)kTrieMaxNodes) return;   // too large: the per-token walk is used
        n_end[path.back()]++;
        dtok.push_back(t);
        prev = s;
        prev_len = L;
    }
    while (!path.empty()) close_node();
    const uint32_t N = (uint32_t)skip.size();
    // parents, branching heights and the classes below each node (children
    // have larger ids than their parent: one reverse pass)
    std::vector<uint32_t> parent(N, 0), bh(N, 0);
    std::vector<uint64_t> sub(N, 0);
    const bool subs = h->K <= 64;
    for (uint32_t n = N; n-- > 0;) {
        uint32_t m = 0, k = 0;
        for (uint32_t c = n + 1; c < skip[n]; c = skip[c]) {
            k++;
            parent[c] = n;
            m = std::max(m, bh[c]);
            if (subs) sub[n] |= (1ull << ncls[c]) | sub[c];
        }
        bh[n] = m + (k >= 2 ? 1u : 0u);
    }
    // upper nodes (an ancestor of an upper node is upper: subtree size and
    // branching height only grow towards the root), their paths, and the
    // units: the subtrees hanging off upper nodes
    std::vector<int32_t> uidx(N, -1);
    std::vector<uint4> upper;
    std::vector<uint8_t> upath;
    std::vector<uint2> unit;
    for (uint32_t n = 0; n < N;) {
        const bool up = n == 0 || skip[n] - n > (uint32_t)kTrieTile || bh[n] > (uint32_t)kTrieBranch;
        if (up) {
            uidx[n] = (int32_t)upper.size();
            const uint32_t off = (uint32_t)upath.size();
            uint32_t plen = 0;
            if (n != 0) {
                const uint4 pu = upper[(size_t)uidx[parent[n]]];
                upath.insert(upath.end(), upath.begin() + pu.y, upath.begin() + pu.y + pu.z);
                upath.push_back(ncls[n]);
                plen = pu.z + 1;
            }
            upper.push_back(make_uint4(n, off, plen, 0u));
            n++;
        } else {
            unit.push_back(make_uint2(n, (uint32_t)uidx[parent[n]]));
            n = skip[n];
        }
    }
    std::vector<uint4> node((size_t)N * 2);
    for (uint32_t n = 0; n < N; n++) {
        node[2 * (size_t)n] = make_uint4(skip[n] | ((uint32_t)ncls[n] << 24), tok_lo[n], n_end[n], tok_hi[n]);
        node[2 * (size_t)n + 1] = make_uint4((uint32_t)sub[n], (uint32_t)(sub[n] >> 32), 0u, 0u);
    }
    h->t_node.swap(node);
    h->t_dtok.swap(dtok);
    h->t_upper.swap(upper);
    h->t_upath.swap(upath);
    h->t_unit.swap(unit);
    h->t_nodes = (int32_t)N;
    h->trie_built = true;
}

// The host side of RowTree while it is built.
struct RowStr {
    const uint8_t* p;   // a token's (remaining) classes
    uint32_t len;
    int32_t token;
};
bool row_str_less(const RowStr& a, const RowStr& b) {
    const int c = std::memcmp(a.p, b.p, std::min(a.len, b.len));
    if (c != 0) return c < 0;
    if (a.len != b.len) return a.len < b.len;
    return a.token < b.token;
}
struct RowBuild {
    bool wide = false;
    std::vector<uint64_t> sets;   // the loop sets
    std::vector<uint4> node;
    std::vector<uint8_t> ncls;
    std::vector<int32_t> dtok;
    std::vector<std::vector<uint8_t>> keeps;   // per loop set
    std::vector<std::vector<uint2>> xrange, exits;
};

// Appends the tree over `strs` (sorted).  Returns its root, or -1 when the
// node or exit numbers run out of their 24 bits.
int64_t add_row_tree(RowBuild& rb, const std::vector<RowStr>& strs) {
    const int64_t root = (int64_t)(rb.node.size() / 2);
    // preorder: the subtree ends and token ranges (as build_trie_host)
    std::vector<uint32_t> skip, lo, own, hi, path;
    std::vector<uint8_t> cls, depth;
    auto open_node = [&](uint8_t c) {
        depth.push_back((uint8_t)std::min<size_t>(path.size(), 255));
        path.push_back((uint32_t)skip.size());
        skip.push_back(0);
        lo.push_back((uint32_t)rb.dtok.size());
        own.push_back(0);
        hi.push_back(0);
        cls.push_back(c);
    };
    auto close_node = [&]() {
        const uint32_t n = path.back();
        path.pop_back();
        skip[n] = (uint32_t)skip.size();
        hi[n] = (uint32_t)rb.dtok.size();
    };
    open_node(0);
    const RowStr* prev = nullptr;
    for (const RowStr& s : strs) {
        uint32_t l = 0;
        while (prev && l < std::min(s.len, prev->len) && prev->p[l] == s.p[l]) l++;
        while (path.size() > (size_t)l + 1) close_node();
        for (uint32_t d = l; d < s.len; d++) open_node(s.p[d]);
        if ((int64_t)skip.size() + root > (int64_t)kTrieMaxNodes) return -1;
        own[path.back()]++;
        rb.dtok.push_back(s.token);
        for (size_t i = 0; i < rb.sets.size(); i++) {
            uint32_t k = s.len;
            while (k > 0 && ((rb.sets[i] >> s.p[k - 1]) & 1ull)) k--;
            rb.keeps[i].push_back((uint8_t)std::min<uint32_t>(k, 255));
        }
        prev = &s;
    }
    while (!path.empty()) close_node();
    const uint32_t N = (uint32_t)skip.size();
    std::vector<uint64_t> sub(N, 0);
    for (uint32_t n = N; n-- > 0;) {
        for (uint32_t c = n + 1; !rb.wide && c < skip[n]; c = skip[c]) sub[n] |= (1ull << cls[c]) | sub[c];
    }
    // breadth first: order[i] is the preorder number of node root + i
    std::vector<uint32_t> order(1, 0), at(N, 0);
    order.reserve(N);
    rb.node.resize((size_t)(root + N) * 2);
    rb.ncls.resize((size_t)(root + N));
    for (size_t i = 0; i < order.size(); i++) {
        const uint32_t n = order[i];
        const uint32_t first = (uint32_t)(root + (int64_t)order.size());
        uint64_t kids = 0;
        for (uint32_t c = n + 1; c < skip[n]; c = skip[c]) {
            order.push_back(c);
            kids = rb.wide ? kids + 1 : kids | (1ull << cls[c]);
        }
        at[n] = (uint32_t)(root + (int64_t)i);
        rb.ncls[(size_t)root + i] = cls[n];
        const uint32_t first_tok = lo[n] < hi[n] ? (uint32_t)rb.dtok[lo[n]] : 0u;
        rb.node[2 * ((size_t)root + i)] = make_uint4((uint32_t)kids, (uint32_t)(kids >> 32),
                                                     first | (std::min<uint32_t>(own[n], 255u) << 24), first_tok);
        rb.node[2 * ((size_t)root + i) + 1] =
            make_uint4(lo[n], hi[n], (uint32_t)sub[n], (uint32_t)(sub[n] >> 32));
    }
    // the edges that leave each loop set, in preorder
    for (size_t i = 0; i < rb.sets.size(); i++) {
        std::vector<uint2>& ex = rb.exits[i];
        std::vector<uint2>& xr = rb.xrange[i];
        xr.resize((size_t)(root + N));
        std::vector<uint32_t> first(N + 1, 0);   // exits before each preorder number
        std::vector<uint8_t> above(N, 0);        // depth of the nearest exit on the path to the node, itself included
        for (uint32_t n = 0; n < N; n++) {
            first[n] = (uint32_t)ex.size();
            const bool out = n != 0 && !((rb.sets[i] >> cls[n]) & 1ull);
            if (out) ex.push_back(make_uint2(at[n], (uint32_t)cls[n] | ((uint32_t)above[n] << 8)));
            if (out) above[n] = depth[n];
            for (uint32_t c = n + 1; c < skip[n]; c = skip[c]) above[c] = above[n];
        }
        first[N] = (uint32_t)ex.size();
        if (ex.size() >= (size_t)(1u << 24)) return -1;
        for (uint32_t n = 0; n < N; n++)
            xr[at[n]] = make_uint2(first[n + 1] | ((uint32_t)depth[n] << 24), first[skip[n]]);
    }
    return root;
}

// A transition entry with its target states renamed: push and plain entries
// hold the target, a pop's triple is renamed state by state.
struct RowEntries {
    std::vector<uint32_t> e;      // [states][K]
    std::vector<uint16_t> ret;    // pop targets, four per triple
    int32_t Q = 0;
};

// The states of the loaded automaton that allow the same tokens whatever the
// stack, merged: `id` names each state's class (0: the dead state).  Two
// states of a class have entries of the same kind and symbol whose targets
// are in the same classes (acceptance only matters to EOS, which is decided
// from the row's own state).  Partition refinement; without a fixed point
// after kMergeRounds rounds (long chains) nothing is merged.
RowEntries merge_states(const domino_ctx* h, std::vector<int32_t>& id) {
    constexpr int kMergeRounds = 64;
    const int32_t Q = h->Q, K = h->K;
    auto entry = [&](int64_t q, int k) -> uint32_t {
        return h->stack ? h->t32[(size_t)(q * K + k)] : h->t16[(size_t)(q * K + k)];
    };
    // an entry's identity under the current classes
    auto seen = [&](const std::vector<int32_t>& c, uint32_t e) -> uint64_t {
        if (!h->stack) return (uint64_t)c[(size_t)e];
        const uint32_t kind = (e >> kKindShift) & 3u;
        const uint64_t head = ((uint64_t)kind << 1 | ((e >> kSymShift) & 1u)) << 48;
        if (kind != 2) return head | (uint64_t)c[(size_t)(e & 0xFFFFu)];
        const uint16_t* r = h->ret.data() + (size_t)(e >> kRetShift) * 4;
        return head | (uint64_t)c[r[0]] << 32 | (uint64_t)c[r[1]] << 16 | (uint64_t)c[r[2]];
    };
    id.assign((size_t)Q, 1);
    id[0] = 0;
    int32_t n = Q > 1 ? 2 : 1;
    bool fixed = Q <= 1;
    for (int round = 0; round < kMergeRounds && !fixed; round++) {
        std::vector<int32_t> next((size_t)Q, 0);
        std::unordered_map<uint64_t, int32_t> at;
        int32_t m = 1;
        for (int64_t q = 1; q < Q; q++) {
            uint64_t hash = 1469598103934665603ull ^ (uint64_t)id[(size_t)q];
            for (int k = 0; k < K; k++) {
                hash = (hash ^ seen(id, entry(q, k))) * 0x9E3779B97F4A7C15ull;
                hash ^= hash >> 29;
            }
            const auto r = at.emplace(hash, m);
            if (r.second) m++;
            next[(size_t)q] = r.first->second;
        }
        fixed = m == n;
        n = m;
        id.swap(next);
    }
    std::vector<int64_t> first((size_t)n, -1);
    for (int64_t q = 0; q < Q; q++)
        if (first[(size_t)id[(size_t)q]] < 0) first[(size_t)id[(size_t)q]] = q;
    for (int64_t q = 1; q < Q && fixed; q++) {   // exact, whatever the hashes did
        const int64_t f = first[(size_t)id[(size_t)q]];
        for (int k = 0; k < K && fixed; k++) fixed = seen(id, entry(q, k)) == seen(id, entry(f, k));
    }
    if (!fixed) {
        std::iota(id.begin(), id.end(), 0);
        first.resize((size_t)Q);
        std::iota(first.begin(), first.end(), 0);
        n = Q;
    }
    RowEntries r;
    r.Q = n;
    r.ret = h->ret;
    for (size_t i = 0; i < r.ret.size(); i++)
        if (i % 4 != 3) r.ret[i] = (uint16_t)id[r.ret[i]];
    r.e.resize((size_t)n * (size_t)K);
    for (int32_t c = 0; c < n; c++)
        for (int k = 0; k < K; k++) {
            const uint32_t e = entry(first[(size_t)c], k);
            const bool pop = h->stack && ((e >> kKindShift) & 3u) == 2u;
            r.e[(size_t)c * K + k] = pop ? e : (e & ~0xFFFFu) | (uint32_t)id[(size_t)(e & 0xFFFFu)];
        }
    return r;
}

// Per state its live classes and the classes that keep it, then its live
// entries, padded to whole 32-byte sectors (RowTree).  flag[q]: the state has
// a loop set.
std::vector<uint8_t> state_records(const RowEntries& r, int K, bool stack, const std::vector<uint32_t>& loop,
                                   int32_t* stride_out) {
    const size_t esz = stack ? 4 : 2;
    size_t most = 0;
    for (int64_t q = 0; q < r.Q; q++) {
        size_t n = 0;
        for (int k = 0; k < K; k++) n += r.e[(size_t)(q * K + k)] != 0;
        most = std::max(most, n);
    }
    const size_t stride = (16 + most * esz + 31) / 32 * 32;
    std::vector<uint8_t> out((size_t)r.Q * stride, 0);
    for (int64_t q = 0; q < r.Q; q++) {
        uint8_t* p = out.data() + (size_t)q * stride;
        uint64_t live = 0, self = 0;
        size_t n = 0;
        for (int k = 0; k < K; k++) {
            const uint32_t e = r.e[(size_t)(q * K + k)];
            if (!e) continue;
            live |= 1ull << k;
            if (e == (uint32_t)q) self |= 1ull << k;   // next state q, no push or pop
            const uint16_t e16 = (uint16_t)e;
            std::memcpy(p + 16 + n * esz, stack ? (const void*)&e : (const void*)&e16, esz);
            n++;
        }
        if (!loop.empty() && loop[(size_t)q] != 0xFFFFFFFFu) self |= 1ull << 63;
        std::memcpy(p, &live, 8);
        std::memcpy(p + 8, &self, 8);
    }
    *stride_out = (int32_t)stride;
    return out;
}

// What row_kernel's walk of a row costs, from an even sample of the states,
// walked on the host as the kernel does: rounds of kRowThreads items from the
// pool's top, their live children in their place.  visits: the nodes a row
// visits (the median).  dense: more than an eighth of the rows visit more than
// kDenseNodes or have more items at a time than the pool holds (those are walked
// twice), so that the per-token walk is the better one.  Subtrees below a state
// that loops on their classes are left out, and so are the classes of a wide
// loop: those are not walked node by node.
constexpr int64_t kDenseNodes = 8192;
constexpr int kDenseSample = 256;
struct RowCost {
    int64_t visits = 0;
    bool dense = false;
};
RowCost row_cost(const domino_ctx* h, const RowBuild& rb, const RowEntries& merged, const std::vector<uint64_t>& self) {
    const int64_t K = h->K, n_states = rb.wide ? h->Q : merged.Q;
    const int n = (int)std::min<int64_t>(kDenseSample, n_states - 1);
    int over = 0;
    std::vector<int64_t> visits((size_t)n, 0);
    std::vector<std::pair<uint32_t, uint32_t>> pool, taken;   // (node, state)
    for (int i = 0; i < n; i++) {
        int64_t& v = visits[(size_t)i];
        bool full = false;
        pool.assign(1, {0u, (uint32_t)(1 + (n_states - 1) * i / n)});
        while (!pool.empty() && !full && v <= kDenseNodes) {
            const size_t stay = pool.size() - std::min<size_t>(pool.size(), kRowThreads);
            taken.assign(pool.begin() + (ptrdiff_t)stay, pool.end());
            pool.resize(stay);
            for (const auto& [node, q] : taken) {
                v++;
                const uint4 a = rb.node[2 * (size_t)node], b = rb.node[2 * (size_t)node + 1];
                const uint64_t keep = rb.wide ? 0 : self[q], below = ((uint64_t)b.w << 32) | b.z;
                if (!rb.wide && (below & ~keep) == 0) continue;
                const bool loop = 4 * __builtin_popcountll(keep) >= K;
                const uint32_t first = a.z & 0xFFFFFFu;
                const int kids = rb.wide ? (int)a.x : __builtin_popcountll(((uint64_t)a.y << 32) | a.x);
                for (int k = 0; k < kids; k++) {
                    const uint32_t c = rb.ncls[(size_t)first + (size_t)k];
                    if (loop && ((keep >> c) & 1ull)) continue;
                    const size_t at = (size_t)(q * K + c);
                    const uint32_t e = !rb.wide ? merged.e[at] : h->stack ? h->t32[at] : h->t16[at];
                    const uint32_t to = h->stack && ((e >> kKindShift) & 3u) == 2u ? 0u : e & 0xFFFFu;   // not past a pop
                    if (to) pool.push_back({first + (uint32_t)k, to});
                }
            }
            full = pool.size() > (size_t)kRowPool;
        }
        over += full || v > kDenseNodes;
    }
    RowCost r;
    r.dense = 8 * over > n;
    if (n > 0) {
        std::nth_element(visits.begin(), visits.begin() + n / 2, visits.end());
        r.visits = visits[(size_t)(n / 2)];
    }
    return r;
}

// RowTree's arrays on the host.
struct RowImage {
    RowBuild rb;                     // the trees
    std::vector<int64_t> roots;      // per loop set its tree
    std::vector<uint32_t> loopbits;
    std::vector<uint8_t> keeps, srec, srec_next, trec;
    std::vector<uint2> xrange, exits, start;
    std::vector<uint32_t> loop_of;
    std::vector<uint16_t> ret;       // the merged states' pop targets
    int32_t stride = 0, stride_next = 0;
    RowCost cost;
};

// The trees, state records and loop sets of RowTree; false when the vocabulary
// or its tree is too large (the per-token walk is used).
bool make_row_image(const domino_ctx* h, RowImage& im) {
    if (!h->trie_built || h->W > kRowMaxSlices * kRowSliceWords) return false;
    const int smem = h->env.max_smem_optin > 0 ? h->env.max_smem_optin : 232448;
    const bool wide = h->K > 64;
    const int32_t Q = h->Q, K = h->K;
    std::vector<uint8_t> cls(h->tok_bytes.size());
    for (size_t i = 0; i < cls.size(); i++) cls[i] = h->byte_class[h->tok_bytes[i]];
    std::vector<RowStr> strs;
    strs.reserve(h->t_dtok.size());
    for (int32_t t : h->t_dtok)   // sorted by class string already
        strs.push_back({cls.data() + h->tok_off[t], (uint32_t)(h->tok_off[t + 1] - h->tok_off[t]), t});
    std::vector<int32_t> id;
    RowEntries merged;
    std::vector<uint64_t> sets, self;   // the loop sets; per merged state the classes that keep it
    if (!wide) {
        merged = merge_states(h, id);
        self.assign((size_t)merged.Q, 0);
        for (int64_t q = 1; q < merged.Q; q++)
            for (int k = 0; k < K; k++)
                if (merged.e[(size_t)(q * K + k)] == (uint32_t)q) self[(size_t)q] |= 1ull << k;
    }
    // the loop sets worth a tree: at least a quarter of the classes (the rule
    // of self_mask), those of most states first
    if (!wide && K <= 63) {
        std::vector<std::pair<uint64_t, int32_t>> all;   // (set, states)
        std::unordered_map<uint64_t, size_t> at;
        for (int32_t q = 1; q < Q; q++) {
            const uint64_t m = self[(size_t)id[(size_t)q]];
            if (4 * __builtin_popcountll(m) < K) continue;
            const auto r = at.emplace(m, all.size());
            if (r.second) all.emplace_back(m, 0);
            all[r.first->second].second++;
        }
        std::stable_sort(all.begin(), all.end(), [](const auto& a, const auto& b) { return a.second > b.second; });
        for (size_t i = 0; i < all.size() && i < (size_t)kRowLoopSets; i++) sets.push_back(all[i].first);
    }
    RowBuild& rb = im.rb;
    std::vector<int64_t>& roots = im.roots;
    std::vector<uint32_t>& loopbits = im.loopbits;
    for (bool ok = false; !ok;) {   // once more without loop sets when they make the trees too large
        rb = RowBuild();
        rb.wide = wide;
        rb.sets = sets;
        rb.keeps.resize(sets.size());
        rb.xrange.resize(sets.size());
        rb.exits.resize(sets.size());
        roots.clear();
        loopbits.clear();
        ok = add_row_tree(rb, strs) == 0;
        for (size_t i = 0; ok && i < sets.size(); i++) {
            std::vector<uint32_t> bits((size_t)h->W, 0);
            std::vector<RowStr> rest;
            for (const RowStr& s : strs) {
                uint32_t l = 0;
                while (l < s.len && ((sets[i] >> s.p[l]) & 1ull)) l++;
                if (l == s.len) bits[(size_t)(s.token >> 5)] |= 1u << (s.token & 31);
                else rest.push_back({s.p + l, s.len - l, s.token});
            }
            std::sort(rest.begin(), rest.end(), row_str_less);
            roots.push_back(add_row_tree(rb, rest));
            ok = roots.back() >= 0;
            loopbits.insert(loopbits.end(), bits.begin(), bits.end());
        }
        size_t n_exits = 0;
        for (auto& e : rb.exits) n_exits += e.size();
        ok = ok && n_exits < (size_t)(1u << 24) &&
             row_smem_bytes(h->W, h->stack, !sets.empty()) <= smem - 1024;
        if (!ok && sets.empty()) return false;
        if (!ok) sets.clear();
    }
    const size_t n_sets = sets.size();
    for (size_t i = 0; i < n_sets; i++) {
        const uint32_t base = (uint32_t)im.exits.size();
        im.keeps.insert(im.keeps.end(), rb.keeps[i].begin(), rb.keeps[i].end());
        for (uint2 x : rb.xrange[i]) im.xrange.push_back(make_uint2(x.x + base, x.y + base));
        im.exits.insert(im.exits.end(), rb.exits[i].begin(), rb.exits[i].end());
    }
    const bool same = wide || merged.Q == Q;   // nothing was merged: one set of records
    if (!wide) {
        im.loop_of.assign((size_t)merged.Q, 0xFFFFFFFFu);   // per merged state its loop set
        for (int32_t q = 1; q < merged.Q; q++) {
            const auto it = std::find(sets.begin(), sets.end(), self[(size_t)q]);
            if (it != sets.end()) im.loop_of[(size_t)q] = (uint32_t)(it - sets.begin());
        }
        im.srec = state_records(merged, K, h->stack, im.loop_of, &im.stride);
        if (!same || n_sets) {
            for (int32_t q = 0; q < Q; q++)   // per state {merged state, its loop set}
                im.start.push_back(make_uint2((uint32_t)id[(size_t)q], im.loop_of[(size_t)id[(size_t)q]]));
            // next states: the automaton's own, without loop sets
            RowEntries own;
            own.Q = Q;
            own.e.resize((size_t)Q * (size_t)K);
            for (size_t i = 0; i < own.e.size(); i++) own.e[i] = h->stack ? h->t32[i] : h->t16[i];
            im.srec_next = state_records(own, K, h->stack, {}, &im.stride_next);
        }
    }
    im.trec.assign((size_t)h->V * 32, 0);
    for (int32_t t = 0; t < h->V; t++) {
        const int64_t len = t == h->eos_id ? 0 : h->tok_off[t + 1] - h->tok_off[t];
        im.trec[(size_t)t * 32] = (uint8_t)std::min<int64_t>(len, 255);
        if (len > 0)
            std::memcpy(&im.trec[(size_t)t * 32 + 1], cls.data() + h->tok_off[t], (size_t)std::min<int64_t>(len, 31));
    }
    im.cost = row_cost(h, rb, merged, self);
    im.ret = std::move(merged.ret);
    return true;
}

// The row walk's arrays on the device.
int build_rows(domino_ctx* h) {
    h->rows_ready = false;
    RowImage im;
    if (!make_row_image(h, im)) return DOMINO_OK;
    int rc;
    auto up = [&](DevBuf& b, const void* p, size_t n) { return dev_upload(b, n ? p : nullptr, std::max<size_t>(16, n)); };
    if ((rc = up(h->d_rnode, im.rb.node.data(), im.rb.node.size() * sizeof(uint4)))) return rc;
    if ((rc = up(h->d_rncls, im.rb.ncls.data(), im.rb.ncls.size()))) return rc;
    if ((rc = up(h->d_rdtok, im.rb.dtok.data(), im.rb.dtok.size() * 4))) return rc;
    if ((rc = up(h->d_srec, im.srec.data(), im.srec.size()))) return rc;
    if ((rc = up(h->d_srec_next, im.srec_next.data(), im.srec_next.size()))) return rc;
    if ((rc = up(h->d_rret, im.ret.data(), im.ret.size() * 2))) return rc;
    if ((rc = up(h->d_rstart, im.start.data(), im.start.size() * sizeof(uint2)))) return rc;
    if ((rc = up(h->d_loop_of, im.loop_of.data(), im.loop_of.size() * 4))) return rc;
    if ((rc = up(h->d_loopbits, im.loopbits.data(), im.loopbits.size() * 4))) return rc;
    if ((rc = up(h->d_keeps, im.keeps.data(), im.keeps.size()))) return rc;
    if ((rc = up(h->d_xrange, im.xrange.data(), im.xrange.size() * sizeof(uint2)))) return rc;
    if ((rc = up(h->d_exits, im.exits.data(), im.exits.size() * sizeof(uint2)))) return rc;
    if ((rc = up(h->d_trec, im.trec.data(), im.trec.size()))) return rc;
    const StepView v = make_view(h);
    RowTree t{};
    t.trec = (const uint8_t*)h->d_trec.p;
    t.node = (const uint4*)h->d_rnode.p;
    t.ncls = (const uint8_t*)h->d_rncls.p;
    t.dtok = (const int32_t*)h->d_rdtok.p;
    t.srec = (const uint4*)h->d_srec.p;
    t.ret = im.rb.wide ? v.ret : (const uint16_t*)h->d_rret.p;
    t.start = im.start.empty() ? nullptr : (const uint2*)h->d_rstart.p;
    t.loop_of = (const uint32_t*)h->d_loop_of.p;
    t.loopbits = (const uint32_t*)h->d_loopbits.p;
    t.keeps = (const uint8_t*)h->d_keeps.p;
    t.xrange = (const uint2*)h->d_xrange.p;
    t.exits = (const uint2*)h->d_exits.p;
    t.srec_stride = im.stride;
    t.n_nodes = (int32_t)(im.rb.node.size() / 2);
    t.n_dtok = (int32_t)im.rb.dtok.size();
    t.n_loops = (int32_t)im.roots.size();
    for (size_t i = 0; i < im.roots.size(); i++) t.loop_root[i] = (int32_t)im.roots[i];
    h->rows = t;
    if (!im.start.empty()) {
        t.srec = (const uint4*)h->d_srec_next.p;
        t.srec_stride = im.stride_next;
        t.ret = v.ret;
        t.start = nullptr;
        t.n_loops = 0;
    }
    h->rows_next = t;
    h->rows_dense = im.cost.dense;
    h->rows_visits = im.cost.visits;
    h->rows_ready = true;
    return DOMINO_OK;
}

// Byte-class strings of every token, the window sort and the slot arrays.
int build_arena(domino_ctx* h) {
    h->arena_ready = false;
    if (!h->vocab_loaded || !h->auto_loaded) return DOMINO_OK;
    const int32_t V = h->V;
    const int32_t nw = (V + kWin - 1) / kWin;
    const int64_t n_slots = (int64_t)nw * kWin;
    std::vector<uint8_t> cls(h->tok_bytes.size());
    for (size_t i = 0; i < cls.size(); i++) cls[i] = h->byte_class[h->tok_bytes[i]];
    auto tlen = [&](int32_t t) -> int32_t {
        return t == h->eos_id ? 0 : (int32_t)(h->tok_off[t + 1] - h->tok_off[t]);
    };
    // window order: empty tokens first, then by first class; inside a first-class
    // group longer tokens first (a warp's lanes then walk similar lengths), then
    // by class string (shared prefixes take the same transitions)
    auto less = [&](int32_t a, int32_t b) {
        int32_t la = tlen(a), lb = tlen(b);
        if ((la == 0) != (lb == 0)) return la == 0;
        if (la == 0) return a < b;
        const uint8_t* ca = cls.data() + h->tok_off[a];
        const uint8_t* cb = cls.data() + h->tok_off[b];
        if (ca[0] != cb[0]) return ca[0] < cb[0];
        if (la != lb) return la > lb;
        int c = std::memcmp(ca, cb, (size_t)la);
        if (c != 0) return c < 0;
        return a < b;
    };
    const int K = h->K;
    std::vector<uint8_t> head((size_t)n_slots * kInlineBytes, 0);
    const bool self = !h->self_mask.empty();
    std::vector<uint64_t> tok_cls(self ? (size_t)n_slots : 0, 0);   // classes of bytes 1.. of each slot
    std::vector<uint32_t> info((size_t)n_slots, 0);
    std::vector<int32_t> tail_off((size_t)n_slots, 0), pos_of((size_t)V, 0);
    std::vector<uint16_t> gstart((size_t)(K + 1), 0);
    std::vector<uint16_t> cls_start((size_t)nw * (size_t)(h->K + 1), 0);   // [window][class]: first slot
    std::vector<int16_t> eos_slot((size_t)nw, -1);
    std::vector<uint8_t> tail;
    std::vector<int32_t> ids;
    for (int32_t w = 0; w < nw; w++) {
        int32_t lo = w * kWin, hi = std::min(V, lo + kWin);
        ids.resize((size_t)(hi - lo));
        std::iota(ids.begin(), ids.end(), lo);
        std::sort(ids.begin(), ids.end(), less);
        uint16_t* gs = gstart.data();
        int c_next = 0;   // first class whose group start is still unset
        for (int32_t j = 0; j < hi - lo; j++) {
            int32_t t = ids[(size_t)j];
            int64_t p = (int64_t)lo + j;
            int32_t L = tlen(t);
            info[(size_t)p] = (uint32_t)(t - lo) | kInfoValid | ((uint32_t)L << 16);
            pos_of[(size_t)t] = (int32_t)p;
            if (t == h->eos_id) eos_slot[(size_t)w] = (int16_t)j;
            const uint8_t* c = cls.data() + h->tok_off[t];
            if (L > 0) {
                while (c_next <= c[0]) gs[c_next++] = (uint16_t)j;   // groups by first class
            }
            std::memcpy(head.data() + p * kInlineBytes, c, (size_t)std::min(L, kInlineBytes));
            if (self)
                for (int32_t i = 1; i < L; i++) tok_cls[(size_t)p] |= 1ull << c[i];
            if (L > kInlineBytes) {
                tail_off[(size_t)p] = (int32_t)tail.size();
                tail.insert(tail.end(), c + kInlineBytes, c + L);
            }
        }
        while (c_next <= K) gs[c_next++] = (uint16_t)(hi - lo);
        // the slots of first class c are [gs[c], gs[c + 1]) of the window
        std::copy(gs, gs + K + 1, cls_start.begin() + (ptrdiff_t)((size_t)w * (K + 1)));
    }
    if (tail.size() > (size_t)INT32_MAX) return DOMINO_E_UNSUPPORTED;
    int rc;
    if ((rc = dev_upload(h->d_head, head.data(), head.size()))) return rc;
    if ((rc = dev_upload(h->d_info, info.data(), info.size() * 4))) return rc;
    if ((rc = dev_upload(h->d_tail_off, tail_off.data(), tail_off.size() * 4))) return rc;
    if ((rc = dev_upload(h->d_tail, tail.data(), tail.size()))) return rc;
    if ((rc = dev_upload(h->d_pos_of, pos_of.data(), pos_of.size() * 4))) return rc;
    if ((rc = dev_upload(h->d_cls_start, cls_start.data(), cls_start.size() * 2))) return rc;
    if (self) {
        if ((rc = dev_upload(h->d_tok_cls, tok_cls.data(), tok_cls.size() * 8))) return rc;
    } else {
        dev_free(h->d_tok_cls);
    }
    if ((rc = dev_upload(h->d_eos_slot, eos_slot.data(), eos_slot.size() * 2))) return rc;
    h->n_windows = nw;
    build_trie_host(h);
    if ((rc = build_rows(h))) return rc;
    h->arena_ready = true;
    return DOMINO_OK;
}

StepView make_view(domino_ctx* h) {
    StepView v{};
    v.head = (const uint4*)h->d_head.p;
    v.info = (const uint32_t*)h->d_info.p;
    v.tail_off = (const int32_t*)h->d_tail_off.p;
    v.tail = (const uint8_t*)h->d_tail.p;
    v.pos_of = (const int32_t*)h->d_pos_of.p;
    v.cls_start = (const uint16_t*)h->d_cls_start.p;
    v.eos_slot = (const int16_t*)h->d_eos_slot.p;
    v.V = h->V;
    v.W = h->W;
    v.n_windows = h->n_windows;
    v.eos_id = h->eos_id;
    const char* dense = (const char*)h->d_dense.p;
    v.t16 = h->stack ? nullptr : (const uint16_t*)dense;
    v.t32 = h->stack ? (const uint32_t*)dense : nullptr;
    v.ret = dense ? (const uint16_t*)(dense + h->dense_ret_off) : nullptr;
    v.sp_info = (const uint32_t*)h->d_sparse.p;
    v.sp_tgt = h->d_sparse.p ? (const void*)((const char*)h->d_sparse.p + h->sp_tgt_off) : nullptr;
    v.accept_bits = (const uint32_t*)h->d_accept.p;
    v.self_mask = h->self_mask.empty() ? nullptr : (const unsigned long long*)h->d_self.p;
    v.tok_cls = h->self_mask.empty() ? nullptr : (const unsigned long long*)h->d_tok_cls.p;
    v.Q = h->Q;
    v.K = h->K;
    v.start = h->start;
    v.max_depth = h->max_depth;
    v.n_ret = (int32_t)(h->ret.size() / 4);
    v.sp_nnz = h->sp_nnz;
    v.err = (uint32_t*)h->d_err.p;
    return v;
}

// Table placement for the step kernel: dense in shared memory if it fits, else
// the sparse live-class form, else dense through L1/L2.
int choose_mode(const domino_ctx* h, const StepView& v, bool next) {
    if (h->env.max_smem_optin <= 0) return kDenseGlobal;
    const int64_t avail = (int64_t)h->env.max_smem_optin - step_fixed_smem_bytes(v, next) - 1024;
    if (table_smem_bytes(v, h->stack, kDenseSmem) <= avail) return kDenseSmem;
    if (h->sp_nnz > 0) {
        const int mode = h->sp_words == 2 ? kSparse32Smem : kSparse64Smem;
        if (table_smem_bytes(v, h->stack, mode) <= avail) return mode;
    }
    return kDenseGlobal;
}

// One tree for all rows: no state loops on many classes (or DOMINO_WALK=tree).
bool use_tree(const domino_ctx* h) {
    if (!h->rows_ready || h->walk_pref == 0) return false;
    return h->walk_pref == 1 || h->self_mask.empty();
}

// The (row, token) pairs from which row_kernel is the faster walk.  Its time
// is the latency of a row's rounds (8 to 40 us), once for every 2 * SMs rows;
// the per-token walk's grows with the pairs.  In units of 2^19 pairs: `first`
// for up to 2 * SMs rows, `more` for every further such wave.  Both hold for
// rows that visit up to kVisits nodes, and grow by kVisitUnits for every 1000
// more (us per token / row_kernel, masks, 500 states, V = 128256: 3770 visits
// (12 of 32 classes live), batch 32 23 / 33, batch 96 28 / 32, batch 128 35 / 32,
// batch 256 58 / 37; 7030 visits (14 live), batch 96 33 / 47, batch 192 49 / 53,
// batch 256 66 / 56; V = 32000, 2560 visits, batch 800 60 / 74; 100 classes, 20
// live, 1300 visits, V = 128256, batch 24 21 / 24, batch 64 26 / 23, batch 256 47
// / 27; 256 classes, 40 live, 1030 visits, batch 256 102 / 26).
constexpr int64_t kVisits = 1100;
constexpr double kVisitUnits = 8.0;
bool rows_pay(const domino_ctx* h, int64_t batch, int first, int more) {
    const int64_t at_once = 2 * std::max(1, h->env.num_sms);
    const double beyond = kVisitUnits * (double)std::max<int64_t>(0, h->rows_visits - kVisits) / 1000.0;
    return (double)(batch * h->V) >=
           (first + beyond + (double)((batch - 1) / at_once) * (more + beyond)) * (double)((int64_t)1 << 19);
}

// Whether row_kernel takes a mask step (GB300, us per-token / row_kernel).
// Without loop sets: 5000 states, V = 128256, batch 17 8.1 / 14.3, batch 25
// 19.5 / 13.3; V = 32000, batch 98 11.6 / 10.8; V = 8000, batch 620 15.8 / 15.7,
// batch 1000 16.0 / 18.2; V = 16000, batch 400 32.9 / 11.8; tables of masks, V =
// 8000, 16000 states 194 / 216 (4.6 units a wave), V = 16000, 8000 states 193 /
// 128; next states, V = 8000, batch 400 15.0 / 12.5, batch 300 11.3 / 11.9.
// With a stack, whose per-token walk is the dearer: JSON, V = 50000, batch 39
// 19.5 / 14.7, V = 128256, batch 17 16.1 / 24.2, batch 21 37.8 / 23.7.  With
// loop sets alone (200 states): V = 48000, batch 87 5.7 / 8.9, batch 174 9.5 /
// 9.2, V = 64000, batch 98 10.7 / 8.3; V = 16000, batch 400 26.2 / 8.3, V =
// 8000, batch 1000 11.1 / 15.2; their next states are the per-token walk's
// (loop sets hold masks only).
// Automata most of whose rows are too large (row_cost) are the per-token
// walk's: 500 states with 16 of 32 classes live, V = 128256, batch 256 76 / 247,
// 18 live 86 / 274, 28 live 179 / 542 (14 live, 4.3 % of the tokens: 66 / 56,
// row_kernel's).
bool use_rows(const domino_ctx* h, int64_t batch, bool next) {
    if (!h->rows_ready || h->walk_pref == 0) return false;
    if (h->walk_pref == 1) return true;
    if (h->rows_dense || (next && !h->self_mask.empty())) return false;
    if (h->stack) return rows_pay(h, batch, 4, 4);
    if (next) return rows_pay(h, batch, 6, 1);
    return h->self_mask.empty() ? rows_pay(h, batch, 6, 5) : rows_pay(h, batch, 10, 2);
}

// Whether the whole decode step is row_kernel's (one launch), against the
// per-token walk with the decode folded in (two launches; bf16 rows on 16-byte
// boundaries): 5000 states, V = 128256, batch 17 13.8 / 21.3, batch 25 26.9 /
// 19.1, V = 32000, batch 98 17.1 / 19.1, batch 163 19.5 / 18.2; JSON, V =
// 50000, batch 39 26.4 / 20.7, V = 128256, batch 17 22.6 / 30.6, batch 21 45.2
// / 31.2; 200 states, V = 32000, batch 196 15.1 / 14.0, V = 48000, batch 131
// 13.1 / 15.4, batch 262 18.4 / 14.4, V = 32000, batch 400 35.5 / 14.2, V =
// 16000, batch 500 15.0 / 19.2.  And
// against the three kernels one after the other (two launches more): fp32, 200
// states, V = 32000, batch 32 14.4 / 12.9, V = 64000, batch 4 11.9 / 12.1, batch
// 8 13.3 / 12.9; 5000 states, V = 32000, batch 22 15.9 / 15.4, V = 128256,
// batch 5 15.3 / 17.2.
bool decode_rows(const domino_ctx* h, int64_t batch, bool fusable) {
    if (!h->rows_ready || h->walk_pref == 0) return false;
    if (h->walk_pref == 1) return true;
    if (h->rows_dense) return false;
    if (!fusable) return rows_pay(h, batch, 1, 1);
    if (h->stack) return rows_pay(h, batch, 4, 4);
    return h->self_mask.empty() ? rows_pay(h, batch, 6, 5) : rows_pay(h, batch, 16, 6);
}

// Whether the decode can ride on the per-token walk, whose partials then take
// fpart_bytes().
bool can_fuse(const domino_ctx* h, const void* logits, int32_t dtype, int32_t batch, int64_t stride) {
    return dtype == DOMINO_DTYPE_BF16 && reinterpret_cast<uintptr_t>(logits) % 16 == 0 &&
           ((size_t)stride * 2) % 16 == 0 && (int64_t)batch * h->n_windows < (int64_t)INT32_MAX;   // partial slots are int
}
size_t fpart_bytes(const domino_ctx* h, int32_t batch) {
    return (size_t)batch * (size_t)h->n_windows * sizeof(float4);
}

int ready_for_compute(domino_ctx* h) {
    if (!h) return DOMINO_E_INVALID_ARG;
    if (is_host_only(h)) return DOMINO_E_NO_DEVICE;
    if (!h->vocab_loaded || !h->auto_loaded || !h->arena_ready) return DOMINO_E_NOT_LOADED;
    return DOMINO_OK;
}

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return DOMINO_OK;
    cudaGetLastError();
    return DOMINO_E_CUDA;
}

// An NVTX range named after each C ABI call that does work (a no-op unless a
// profiler is attached), so that a timeline shows the library's calls above
// the kernels they launch.
struct ApiRange {
    explicit ApiRange(const char* name) { nvtxRangePushA(name); }
    ~ApiRange() { nvtxRangePop(); }
    ApiRange(const ApiRange&) = delete;
    ApiRange& operator=(const ApiRange&) = delete;
};
#define DOMINO_API_RANGE() const ApiRange api_range_(__func__)

// The entry points below that allocate host memory are function-try-blocks: an
// exception must not pass into the C caller.  A load that ends this way leaves
// the handle refusing what needs the part that was being built (its flag is
// cleared first and set last).

}  // namespace

extern "C" {

const char* domino_status_string(int s) {
    switch (s) {
        case DOMINO_OK: return "ok";
        case DOMINO_E_INVALID_ARG: return "invalid argument";
        case DOMINO_E_NOT_LOADED: return "vocabulary or automaton not loaded";
        case DOMINO_E_UNSUPPORTED: return "unsupported request";
        case DOMINO_E_OOM: return "out of memory";
        case DOMINO_E_CUDA: return "CUDA runtime error";
        case DOMINO_E_NO_DEVICE: return "host-only handle has no device";
        default: return "unknown status";
    }
}

int domino_create(domino_t* out, int32_t cuda_device) {
    if (!out) return DOMINO_E_INVALID_ARG;
    *out = nullptr;
    domino_ctx* h = new (std::nothrow) domino_ctx();
    if (!h) return DOMINO_E_OOM;
    h->device = cuda_device < 0 ? -1 : cuda_device;
    if (const char* w = std::getenv("DOMINO_WALK")) {
        if (std::strcmp(w, "token") == 0) h->walk_pref = 0;
        if (std::strcmp(w, "tree") == 0) h->walk_pref = 1;
    }
    if (h->device >= 0) {
        int n = 0;
        if (cudaGetDeviceCount(&n) != cudaSuccess || cuda_device >= n) {
            cudaGetLastError();
            delete h;
            return cuda_device >= n && n > 0 ? DOMINO_E_INVALID_ARG : DOMINO_E_CUDA;
        }
        if (cudaSetDevice(h->device) != cudaSuccess) {
            cudaGetLastError();
            delete h;
            return DOMINO_E_CUDA;
        }
        cudaDeviceGetAttribute(&h->env.num_sms, cudaDevAttrMultiProcessorCount, h->device);
        cudaDeviceGetAttribute(&h->env.max_smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
        int rc = dev_reserve(h->d_err, 16);
        if (!rc && cudaMemset(h->d_err.p, 0, 16) != cudaSuccess) {
            cudaGetLastError();
            rc = DOMINO_E_CUDA;
        }
        if (rc) {
            domino_destroy(h);
            return rc;
        }
    }
    *out = h;
    return DOMINO_OK;
}

int domino_destroy(domino_t h) {
    if (!h) return DOMINO_OK;
    if (h->device >= 0) {
        DeviceGuard g(h->device);
        cudaDeviceSynchronize();
        DevBuf* all[] = {&h->d_head, &h->d_info, &h->d_tail_off, &h->d_tail, &h->d_pos_of, &h->d_cls_start,
                         &h->d_eos_slot, &h->d_dense, &h->d_sparse, &h->d_accept, &h->d_self, &h->d_tok_cls, &h->d_err, &h->d_fpart, &h->s_logits, &h->s_mask, &h->s_io,
                         &h->o_prop, &h->o_rows, &h->o_count, &h->d_rnode, &h->d_rncls, &h->d_rdtok, &h->d_srec, &h->d_srec_next, &h->d_rret,
                         &h->d_rstart, &h->d_loop_of, &h->d_loopbits, &h->d_keeps, &h->d_xrange, &h->d_exits,
                         &h->d_trec};
        for (auto* b : all) dev_free(*b);
        for (DevBuf& b : h->fpart_old) dev_free(b);
        for (cudaEvent_t& e : h->ev_chunk)
            if (e) cudaEventDestroy(e);
        for (cudaEvent_t& e : h->ev_t)
            if (e) cudaEventDestroy(e);
        if (h->ev_cfg) cudaEventDestroy(h->ev_cfg);
        if (h->cp_stream) cudaStreamDestroy(h->cp_stream);
        if (h->h_io) cudaFreeHost(h->h_io);
        clear_host_graphs(h);
        cudaGetLastError();
    }
    delete h;
    return DOMINO_OK;
}

int domino_load_vocab(domino_t h, const uint8_t* bytes, const int64_t* offsets, int32_t n_tokens,
                      int32_t eos_id) try {
    DOMINO_API_RANGE();
    if (h) clear_host_graphs(h);
    if (!h || !offsets || n_tokens < 1 || n_tokens > (1 << 24)) return DOMINO_E_INVALID_ARG;
    if (eos_id < -1 || eos_id >= n_tokens || offsets[0] != 0) return DOMINO_E_INVALID_ARG;
    int32_t max_len = 0;
    for (int32_t t = 0; t < n_tokens; t++) {
        int64_t L = offsets[t + 1] - offsets[t];
        if (L < 0 || L > 65535) return DOMINO_E_INVALID_ARG;
        if (t != eos_id) max_len = std::max<int32_t>(max_len, (int32_t)L);
    }
    if (offsets[n_tokens] > 0 && !bytes) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    h->vocab_loaded = false;
    h->arena_ready = false;
    h->tok_off.assign(offsets, offsets + n_tokens + 1);
    if (bytes && offsets[n_tokens] > 0)
        h->tok_bytes.assign(bytes, bytes + offsets[n_tokens]);
    else
        h->tok_bytes.clear();
    h->V = n_tokens;
    h->W = (n_tokens + 31) / 32;
    h->eos_id = eos_id;
    h->max_len = max_len;
    h->vocab_loaded = true;
    if (is_host_only(h)) {
        build_trie_host(h);
        return DOMINO_OK;
    }
    return build_arena(h);
} catch (...) {   // std::bad_alloc
    return DOMINO_E_OOM;
}

int domino_load_automaton(domino_t h, const int32_t* delta, int32_t n_states, const uint8_t* live,
                          const uint8_t* accepting, int32_t start_state, const domino_stack_rule* rules,
                          int32_t n_rules, int32_t max_depth) try {
    DOMINO_API_RANGE();
    if (!h || !delta || !live || n_states < 1 || n_states > DOMINO_MAX_STATES) return DOMINO_E_INVALID_ARG;
    if (start_state < 0 || start_state >= n_states || max_depth < 0 || max_depth > DOMINO_MAX_DEPTH)
        return DOMINO_E_INVALID_ARG;
    if (n_rules < 0 || (n_rules > 0 && !rules)) return DOMINO_E_INVALID_ARG;
    const int64_t Q = n_states;
    for (int64_t i = 0; i < Q * 256; i++)
        if (delta[i] < 0 || delta[i] >= n_states) return DOMINO_E_INVALID_ARG;
    if (live[0]) return DOMINO_E_INVALID_ARG;
    for (int c = 0; c < 256; c++)
        if (delta[c] != 0) return DOMINO_E_INVALID_ARG;          // state 0 absorbing
    for (int64_t q = 0; q < Q; q++)
        if (accepting && accepting[q] && !live[q]) return DOMINO_E_INVALID_ARG;
    // rules: one per (state, byte); index -1 = none
    std::vector<int32_t> rule_at((size_t)(Q * 256), -1);
    for (int32_t r = 0; r < n_rules; r++) {
        const domino_stack_rule& R = rules[r];
        if (R.state <= 0 || R.state >= n_states || R.pad != 0 || R.sym > 1 ||
            (R.kind != DOMINO_RULE_PUSH && R.kind != DOMINO_RULE_POP))
            return DOMINO_E_INVALID_ARG;
        if (R.kind == DOMINO_RULE_POP) {
            for (int32_t t : {R.next_if_empty, R.next_if_top0, R.next_if_top1})
                if (t < 0 || t >= n_states) return DOMINO_E_INVALID_ARG;
        }
        int32_t& slot = rule_at[(size_t)R.state * 256 + R.byte];
        if (slot != -1) return DOMINO_E_INVALID_ARG;
        slot = r;
    }
    // closure: a non-live state only reaches non-live states (makes early exit exact)
    for (int64_t q = 0; q < Q; q++) {
        if (live[q]) continue;
        for (int c = 0; c < 256; c++) {
            int32_t r = rule_at[(size_t)q * 256 + c];
            if (r >= 0 && rules[r].kind == DOMINO_RULE_POP) {
                if (live[rules[r].next_if_empty] || live[rules[r].next_if_top0] || live[rules[r].next_if_top1])
                    return DOMINO_E_INVALID_ARG;
            } else if (live[delta[q * 256 + c]]) {
                return DOMINO_E_INVALID_ARG;
            }
        }
    }
    auto canon = [&](int32_t t) -> uint32_t { return live[t] ? (uint32_t)t : 0u; };
    // full entry for every (q, byte): dead-canonicalised, pop targets as deduplicated triples
    const bool stack = n_rules > 0;
    std::vector<uint32_t> col((size_t)(256 * Q));   // column-major: [byte][q]
    std::vector<uint16_t> ret;
    std::unordered_map<uint64_t, uint32_t> triple_id;
    for (int64_t q = 0; q < Q; q++) {
        for (int c = 0; c < 256; c++) {
            int32_t r = rule_at[(size_t)q * 256 + c];
            uint32_t e;
            if (r < 0) {
                e = canon(delta[q * 256 + c]);
            } else if (rules[r].kind == DOMINO_RULE_PUSH) {
                e = canon(delta[q * 256 + c]) | (1u << kKindShift) | ((uint32_t)rules[r].sym << kSymShift);
            } else {
                uint64_t key = ((uint64_t)canon(rules[r].next_if_empty) << 32) |
                               ((uint64_t)canon(rules[r].next_if_top0) << 16) | canon(rules[r].next_if_top1);
                auto it = triple_id.find(key);
                uint32_t id;
                if (it == triple_id.end()) {
                    id = (uint32_t)(ret.size() / 4);
                    if (id >= kMaxRetTriples) return DOMINO_E_UNSUPPORTED;
                    triple_id.emplace(key, id);
                    ret.push_back((uint16_t)canon(rules[r].next_if_empty));
                    ret.push_back((uint16_t)canon(rules[r].next_if_top0));
                    ret.push_back((uint16_t)canon(rules[r].next_if_top1));
                    ret.push_back(0);
                } else {
                    id = it->second;
                }
                e = (2u << kKindShift) | ((uint32_t)rules[r].sym << kSymShift) | (id << kRetShift);
            }
            col[(size_t)c * Q + q] = e;
        }
    }
    // byte classes: bytes whose columns are identical for every state
    uint8_t cls[256];
    int rep[256];
    int K = 0;
    std::unordered_map<uint64_t, std::vector<int>> by_hash;
    for (int c = 0; c < 256; c++) {
        const uint32_t* cc = col.data() + (size_t)c * Q;
        uint64_t hsh = 1469598103934665603ull;
        for (int64_t q = 0; q < Q; q++) hsh = (hsh ^ cc[q]) * 1099511628211ull;
        int found = -1;
        for (int k : by_hash[hsh]) {
            if (std::memcmp(cc, col.data() + (size_t)rep[k] * Q, sizeof(uint32_t) * (size_t)Q) == 0) {
                found = k;
                break;
            }
        }
        if (found < 0) {
            found = K++;
            rep[found] = c;
            by_hash[hsh].push_back(found);
        }
        cls[c] = (uint8_t)found;
    }
    DeviceGuard g(h->device);
    clear_host_graphs(h);
    h->auto_loaded = false;
    h->arena_ready = false;
    h->Q = n_states;
    h->K = K;
    h->start = start_state;
    h->max_depth = max_depth;
    h->n_rules = n_rules;
    h->stack = stack;
    std::memcpy(h->byte_class, cls, 256);
    h->t16.clear();
    h->t32.clear();
    if (stack) {
        h->t32.resize((size_t)(Q * K));
        for (int64_t q = 0; q < Q; q++)
            for (int k = 0; k < K; k++) h->t32[(size_t)(q * K + k)] = col[(size_t)rep[k] * Q + q];
    } else {
        h->t16.resize((size_t)(Q * K));
        for (int64_t q = 0; q < Q; q++)
            for (int k = 0; k < K; k++) h->t16[(size_t)(q * K + k)] = (uint16_t)col[(size_t)rep[k] * Q + q];
    }
    h->ret = ret;
    // Self loops: class k keeps state q (with no stack action).  A token whose
    // remaining classes all keep the row's state leaves it unchanged, so the
    // walk can skip it.  Used when some state loops on at least a quarter of
    // the classes: the string, number and whitespace states of real grammars.
    h->self_mask.clear();
    if (K <= 64) {
        std::vector<uint64_t> sm((size_t)Q, 0);
        bool wide = false;
        for (int64_t q = 1; q < Q; q++) {
            for (int k = 0; k < K; k++) {
                const uint32_t e = stack ? h->t32[(size_t)(q * K + k)] : h->t16[(size_t)(q * K + k)];
                if (e == (uint32_t)q) sm[(size_t)q] |= 1ull << k;   // next state q, kind 0 (no push or pop)
            }
            wide = wide || 4 * __builtin_popcountll(sm[(size_t)q]) >= K;
        }
        if (wide) h->self_mask.swap(sm);
    }
    h->accept_bits.assign((size_t)((Q + 31) / 32), 0u);
    if (accepting)
        for (int64_t q = 0; q < Q; q++)
            if (accepting[q]) h->accept_bits[(size_t)(q / 32)] |= 1u << (q % 32);
    h->auto_loaded = true;
    // dense image: [Q][K] entries | pop targets, each part 16-byte aligned
    const size_t esz = stack ? 4 : 2;
    auto a16 = [](size_t x) { return (x + 15) / 16 * 16; };
    const size_t tab_bytes = (size_t)(Q * K) * esz;
    h->dense_ret_off = (int64_t)a16(tab_bytes);
    std::vector<uint8_t> dense_img(a16(tab_bytes) + a16(h->ret.size() * 2), 0);
    std::memcpy(dense_img.data(), stack ? (const void*)h->t32.data() : (const void*)h->t16.data(), tab_bytes);
    if (!h->ret.empty()) std::memcpy(dense_img.data() + h->dense_ret_off, h->ret.data(), h->ret.size() * 2);
    // sparse image (K <= 64): per state {live-class mask, base} | live entries | pop targets
    h->sp_nnz = 0;
    h->sp_words = 0;
    std::vector<uint8_t> sparse_img;
    if (K <= 64) {
        const int words = K <= 32 ? 2 : 4;
        std::vector<uint32_t> rinfo((size_t)(Q * words), 0);
        std::vector<uint32_t> tgt;
        for (int64_t q = 0; q < Q; q++) {
            uint64_t m = 0;
            uint32_t base = (uint32_t)tgt.size();
            for (int k = 0; k < K; k++) {
                uint32_t e = stack ? h->t32[(size_t)(q * K + k)] : h->t16[(size_t)(q * K + k)];
                if (e) {
                    m |= 1ull << k;
                    tgt.push_back(e);
                }
            }
            if (words == 2) {
                rinfo[(size_t)(q * 2)] = (uint32_t)m;
                rinfo[(size_t)(q * 2 + 1)] = base;
            } else {
                rinfo[(size_t)(q * 4)] = (uint32_t)m;
                rinfo[(size_t)(q * 4 + 1)] = (uint32_t)(m >> 32);
                rinfo[(size_t)(q * 4 + 2)] = base;
            }
        }
        if (!tgt.empty() && tgt.size() < (size_t)INT32_MAX) {
            h->sp_nnz = (int32_t)tgt.size();
            h->sp_words = words;
            h->sp_tgt_off = (int64_t)a16(rinfo.size() * 4);
            h->sp_ret_off = h->sp_tgt_off + (int64_t)a16(tgt.size() * esz);
            sparse_img.assign((size_t)h->sp_ret_off + a16(h->ret.size() * 2), 0);
            std::memcpy(sparse_img.data(), rinfo.data(), rinfo.size() * 4);
            uint8_t* tp = sparse_img.data() + h->sp_tgt_off;
            for (size_t i = 0; i < tgt.size(); i++) {
                if (stack) {
                    std::memcpy(tp + i * 4, &tgt[i], 4);
                } else {
                    uint16_t e16 = (uint16_t)tgt[i];
                    std::memcpy(tp + i * 2, &e16, 2);
                }
            }
            if (!h->ret.empty()) std::memcpy(sparse_img.data() + h->sp_ret_off, h->ret.data(), h->ret.size() * 2);
        }
    }
    if (is_host_only(h)) {
        build_trie_host(h);
        return DOMINO_OK;
    }
    int rc;
    if ((rc = dev_upload(h->d_dense, dense_img.data(), dense_img.size()))) return rc;
    if (!sparse_img.empty()) {
        if ((rc = dev_upload(h->d_sparse, sparse_img.data(), sparse_img.size()))) return rc;
    } else {
        dev_free(h->d_sparse);
    }
    if ((rc = dev_upload(h->d_accept, h->accept_bits.data(), h->accept_bits.size() * 4))) return rc;
    if (!h->self_mask.empty()) {
        if ((rc = dev_upload(h->d_self, h->self_mask.data(), h->self_mask.size() * 8))) return rc;
    } else {
        dev_free(h->d_self);
    }
    return build_arena(h);
} catch (...) {   // std::bad_alloc
    return DOMINO_E_OOM;
}

int domino_get_info(domino_t h, domino_info* out) {
    if (!h || !out) return DOMINO_E_INVALID_ARG;
    std::memset(out, 0, sizeof(*out));
    out->n_tokens = h->V;
    out->n_words = h->W;
    out->eos_id = h->eos_id;
    out->max_token_len = h->max_len;
    out->n_states = h->Q;
    out->n_classes = h->K;
    out->start_state = h->start;
    out->max_depth = h->max_depth;
    out->n_rules = h->n_rules;
    out->has_stack = h->stack ? 1 : 0;
    out->device = h->device;
    if (h->auto_loaded && h->device >= 0) {
        StepView v = make_view(h);
        out->table_in_smem = choose_mode(h, v, false) != kDenseGlobal ? 1 : 0;
    }
    out->device_bytes = dev_bytes(h);
    out->walk_tree = use_tree(h) ? 1 : 0;
    out->tree_units = h->rows_ready ? (int32_t)h->t_unit.size() : 0;
    return DOMINO_OK;
}

int domino_get_byte_classes(domino_t h, uint8_t* classes_out) {
    if (!h || !classes_out) return DOMINO_E_INVALID_ARG;
    if (!h->auto_loaded) return DOMINO_E_NOT_LOADED;
    std::memcpy(classes_out, h->byte_class, 256);
    return DOMINO_OK;
}

int domino_get_prefix_tree(domino_t h, uint32_t* nodes_out, int64_t nodes_cap, int32_t* tokens_out,
                           int64_t tokens_cap, uint32_t* upper_out, int64_t upper_cap, uint32_t* units_out,
                           int64_t units_cap, int64_t* sizes_out) {
    if (!h || !sizes_out || nodes_cap < 0 || tokens_cap < 0 || upper_cap < 0 || units_cap < 0)
        return DOMINO_E_INVALID_ARG;
    if (!h->vocab_loaded || !h->auto_loaded) return DOMINO_E_NOT_LOADED;
    if (!h->trie_built) return DOMINO_E_UNSUPPORTED;
    const int64_t nu = (int64_t)h->t_upper.size(), nn = (int64_t)h->t_unit.size();
    sizes_out[0] = h->t_nodes;
    sizes_out[1] = (int64_t)h->t_dtok.size();
    sizes_out[2] = nu;
    sizes_out[3] = nn;
    if (nodes_out)
        std::memcpy(nodes_out, h->t_node.data(), (size_t)std::min<int64_t>(nodes_cap, h->t_nodes) * 2 * sizeof(uint4));
    if (tokens_out)
        std::memcpy(tokens_out, h->t_dtok.data(), (size_t)std::min<int64_t>(tokens_cap, (int64_t)h->t_dtok.size()) * 4);
    for (int64_t i = 0; upper_out && i < std::min(upper_cap, nu); i++) {
        upper_out[2 * i] = h->t_upper[(size_t)i].x;
        upper_out[2 * i + 1] = h->t_upper[(size_t)i].z;
    }
    for (int64_t i = 0; units_out && i < std::min(units_cap, nn); i++) {
        units_out[2 * i] = h->t_unit[(size_t)i].x;
        units_out[2 * i + 1] = h->t_unit[(size_t)i].y;
    }
    return DOMINO_OK;
}

int domino_step_mask(domino_t h, const int32_t* states_dev, const uint64_t* stacks_dev, int32_t batch,
                     uint32_t* mask_dev, int32_t* next_dev, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (batch < 0 || (batch > 0 && (!states_dev || !mask_dev))) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    DeviceGuard g(h->device);
    StepView v = make_view(h);
    if (use_rows(h, batch, next_dev != nullptr)) {
        return cuda_status(launch_row_step(v, next_dev ? h->rows_next : h->rows, h->env, h->stack, states_dev,
                                           stacks_dev, batch, false, mask_dev, next_dev, (cudaStream_t)stream));
    }
    const int mode = choose_mode(h, v, next_dev != nullptr);
    return cuda_status(launch_step_mask(v, h->env, h->stack, mode, states_dev, stacks_dev, batch, false, mask_dev,
                                        next_dev, (cudaStream_t)stream));
}

int domino_precompute_table(domino_t h, int32_t* next_dev, uint32_t* mask_dev, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (!next_dev && !mask_dev) return DOMINO_E_INVALID_ARG;
    if (h->stack) return DOMINO_E_UNSUPPORTED;
    DeviceGuard g(h->device);
    StepView v = make_view(h);
    if (use_rows(h, h->Q, next_dev != nullptr)) {
        return cuda_status(launch_row_step(v, next_dev ? h->rows_next : h->rows, h->env, false, nullptr, nullptr, h->Q, true, mask_dev,
                                           next_dev, (cudaStream_t)stream));
    }
    const int mode = choose_mode(h, v, next_dev != nullptr);
    return cuda_status(launch_step_mask(v, h->env, false, mode, nullptr, nullptr, h->Q, true, mask_dev, next_dev,
                                        (cudaStream_t)stream));
}

int domino_mask_logits(domino_t h, const void* logits_dev, int32_t dtype, int32_t batch,
                       int64_t row_stride_elems, const uint32_t* mask_dev, int32_t* argmax_dev, float* lse_dev,
                       float* logprobs_dev, void* stream) {
    DOMINO_API_RANGE();
    if (!h) return DOMINO_E_INVALID_ARG;
    if (is_host_only(h)) return DOMINO_E_NO_DEVICE;
    if (!h->vocab_loaded) return DOMINO_E_NOT_LOADED;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0 || row_stride_elems < h->V) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_dev || !mask_dev || !argmax_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    return cuda_status(launch_mask_logits(h->env, logits_dev, dtype, batch, row_stride_elems, h->V, mask_dev,
                                          argmax_dev, lse_dev, logprobs_dev, (cudaStream_t)stream));
}

int domino_advance(domino_t h, const int32_t* states_dev, const uint64_t* stacks_dev, const int32_t* tokens_dev,
                   int32_t batch, int32_t* states_out, uint64_t* stacks_out, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (batch < 0) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!states_dev || !tokens_dev || !states_out || (stacks_dev && !stacks_out)) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    StepView v = make_view(h);
    const int mode = choose_mode(h, v, false);
    return cuda_status(launch_advance(v, h->stack, mode, states_dev, stacks_dev, tokens_dev, batch, states_out,
                                      stacks_out, (cudaStream_t)stream));
}

int domino_step_decode(domino_t h, const int32_t* states_dev, const uint64_t* stacks_dev, int32_t batch,
                       const void* logits_dev, int32_t dtype, int64_t row_stride_elems, uint32_t* mask_dev,
                       int32_t* argmax_dev, float* lse_dev, float* logprobs_dev, int32_t* states_out,
                       uint64_t* stacks_out, void* stream) try {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0 || row_stride_elems < h->V) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!states_dev || !logits_dev || !mask_dev || !argmax_dev || (logprobs_dev && !lse_dev) ||
        (states_out && stacks_dev && !stacks_out))
        return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    cudaStream_t st = (cudaStream_t)stream;
    const bool fusable = can_fuse(h, logits_dev, dtype, batch, row_stride_elems);
    // logits in device memory are pulled into L2 ahead of their fold;
    // host-resident logits are read only where the mask allows a token
    cudaPointerAttributes pa{};
    const bool on_device = cudaPointerGetAttributes(&pa, logits_dev) == cudaSuccess && pa.type == cudaMemoryTypeDevice;
    if (!on_device) cudaGetLastError();
    bool rows = decode_rows(h, batch, fusable);
    const size_t part_bytes = fpart_bytes(h, batch);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (!rows && fusable && h->d_fpart.n < part_bytes) {
        // growing the partials buffer synchronises the stream and reallocates,
        // neither of which a stream capture allows: the first call at a larger
        // batch must run uncaptured, or take the row kernel, which needs none
        if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return cuda_status(cudaGetLastError());
        rows = cs != cudaStreamCaptureStatusNone && on_device && use_tree(h);
    }
    if (rows) {   // the whole step in one kernel
        StepView v = make_view(h);
        return cuda_status(launch_row_decode(v, h->rows, h->env, h->stack, states_dev, stacks_dev, batch, logits_dev,
                                             dtype, row_stride_elems, on_device, mask_dev, argmax_dev, lse_dev, logprobs_dev,
                                             states_out, states_out && stacks_dev ? stacks_out : nullptr, st));
    }
    if (!fusable) {   // the kernels one after the other
        if ((rc = domino_step_mask(h, states_dev, stacks_dev, batch, mask_dev, nullptr, stream))) return rc;
        if ((rc = domino_mask_logits(h, logits_dev, dtype, batch, row_stride_elems, mask_dev, argmax_dev, lse_dev,
                                     logprobs_dev, stream)))
            return rc;
        if (!states_out) return DOMINO_OK;
        return domino_advance(h, states_dev, stacks_dev, argmax_dev, batch, states_out, stacks_dev ? stacks_out : nullptr,
                              stream);
    }
    StepView v = make_view(h);
    if (h->d_fpart.n < part_bytes) {
        if (cs != cudaStreamCaptureStatusNone) return DOMINO_E_INVALID_ARG;
        if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_status(cudaGetLastError());
        clear_host_graphs(h);   // recorded host-buffer steps name this buffer
        if ((rc = grow_fpart(h, part_bytes))) return rc;
    }
    const int mode = choose_mode(h, v, false);
    cudaError_t e = launch_step_mask(v, h->env, h->stack, mode, states_dev, stacks_dev, batch, false, mask_dev, nullptr,
                                     st, nullptr, nullptr, logits_dev, row_stride_elems, (float4*)h->d_fpart.p,
                                     on_device);
    if (e == cudaSuccess)
        e = launch_fused_combine(v, h->stack, mode, (const float4*)h->d_fpart.p, batch, h->n_windows, argmax_dev,
                                 lse_dev, states_dev, stacks_dev, states_out, stacks_dev ? stacks_out : nullptr, st);
    if (e == cudaSuccess && logprobs_dev)
        e = launch_logprobs_bf16(h->env, logits_dev, batch, row_stride_elems, h->V, mask_dev, lse_dev, logprobs_dev,
                                 st);
    return cuda_status(e);
} catch (...) {   // std::bad_alloc
    return DOMINO_E_OOM;
}

int domino_mask_sample(domino_t h, const void* logits_dev, int32_t dtype, int32_t batch, int64_t row_stride_elems,
                       const uint32_t* mask_dev, float temperature, uint64_t seed, uint64_t offset,
                       int32_t* tokens_dev, void* stream) {
    DOMINO_API_RANGE();
    if (!h) return DOMINO_E_INVALID_ARG;
    if (is_host_only(h)) return DOMINO_E_NO_DEVICE;
    if (!h->vocab_loaded) return DOMINO_E_NOT_LOADED;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (!(temperature > 0.0f) || !std::isfinite(temperature) || !std::isfinite(1.0f / temperature))
        return DOMINO_E_INVALID_ARG;
    if (batch < 0 || row_stride_elems < h->V) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_dev || !mask_dev || !tokens_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    return cuda_status(launch_mask_sample(h->env, logits_dev, dtype, batch, row_stride_elems, h->V, mask_dev,
                                          temperature, seed, offset, tokens_dev, (cudaStream_t)stream));
}

int domino_opportunistic_step(domino_t h, const void* logits_dev, int32_t dtype, int32_t batch,
                              int64_t row_stride_elems, const int32_t* states_dev, const uint64_t* stacks_dev,
                              uint32_t* mask_scratch_dev, int32_t* tokens_dev, int32_t* n_fallback_dev,
                              void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0 || row_stride_elems < h->V) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_dev || !states_dev || !mask_scratch_dev || !tokens_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    cudaStream_t st = (cudaStream_t)stream;
    if (h->o_prop.n < (size_t)batch * 4 || h->o_rows.n < (size_t)batch * 4 || h->o_count.n < 16) {
        if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_status(cudaGetLastError());
        if ((rc = dev_reserve(h->o_prop, (size_t)batch * 4))) return rc;
        if ((rc = dev_reserve(h->o_rows, (size_t)batch * 4))) return rc;
        if ((rc = dev_reserve(h->o_count, 16))) return rc;
    }
    int32_t* prop = (int32_t*)h->o_prop.p;
    int32_t* rows = (int32_t*)h->o_rows.p;
    int32_t* count = n_fallback_dev ? n_fallback_dev : (int32_t*)h->o_count.p;
    StepView v = make_view(h);
    const int mode = choose_mode(h, v, false);
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int32_t), st);
    // 1. the unmasked argmax (every token allowed)
    if (e == cudaSuccess)
        e = launch_mask_logits(h->env, logits_dev, dtype, batch, row_stride_elems, h->V, nullptr, prop, nullptr,
                               nullptr, st);
    // 2. one walk per row: keep the proposal or list the row for the fallback
    if (e == cudaSuccess)
        e = launch_propose_check(v, h->stack, mode, states_dev, stacks_dev, prop, batch, tokens_dev, rows, count, st);
    // 3. the listed rows only: their masks, then their masked argmax
    if (e == cudaSuccess)
        e = launch_step_mask(v, h->env, h->stack, mode, states_dev, stacks_dev, batch, false, mask_scratch_dev,
                             nullptr, st, rows, count);
    if (e == cudaSuccess)
        e = launch_mask_logits(h->env, logits_dev, dtype, batch, row_stride_elems, h->V, mask_scratch_dev,
                               tokens_dev, nullptr, nullptr, st, nullptr, 0, nullptr, nullptr, rows, count);
    return cuda_status(e);
}

int domino_spec_update(domino_t h, uint32_t* counts_dev, uint64_t* best_dev, uint32_t* reached_dev,
                       const int32_t* states_dev, const uint64_t* stacks_dev, const int32_t* tokens_dev,
                       int32_t batch, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (batch < 0) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!counts_dev || !best_dev || !reached_dev || !states_dev || !tokens_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    StepView v = make_view(h);
    return cuda_status(launch_spec_update(v, h->stack, states_dev, stacks_dev, tokens_dev, batch, counts_dev,
                                          (unsigned long long*)best_dev, reached_dev, (cudaStream_t)stream));
}

int domino_spec_propose(domino_t h, const uint64_t* best_dev, const uint32_t* reached_dev,
                        const int32_t* states_dev, const uint64_t* stacks_dev, int32_t batch, int32_t s,
                        int32_t min_permille, int32_t* proposals_dev, int32_t* n_prop_dev,
                        int32_t* chain_states_dev, uint64_t* chain_stacks_dev, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (batch < 0 || s < 1 || min_permille < 0 || min_permille > 1000) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!best_dev || !reached_dev || !states_dev || !proposals_dev || !n_prop_dev || !chain_states_dev)
        return DOMINO_E_INVALID_ARG;
    if (stacks_dev && !chain_stacks_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    StepView v = make_view(h);
    const int mode = choose_mode(h, v, false);
    return cuda_status(launch_spec_propose(v, h->stack, mode, states_dev, stacks_dev, batch, s, min_permille,
                                           (const unsigned long long*)best_dev, reached_dev, proposals_dev,
                                           n_prop_dev, chain_states_dev, chain_stacks_dev, (cudaStream_t)stream));
}

int domino_spec_accept(domino_t h, const int32_t* proposals_dev, const int32_t* n_prop_dev,
                       const int32_t* decoded_dev, const int32_t* chain_states_dev, const uint64_t* chain_stacks_dev,
                       int32_t batch, int32_t s, int32_t* n_accept_dev, int32_t* tokens_out_dev,
                       int32_t* states_out_dev, uint64_t* stacks_out_dev, void* stream) {
    DOMINO_API_RANGE();
    if (!h) return DOMINO_E_INVALID_ARG;
    if (is_host_only(h)) return DOMINO_E_NO_DEVICE;
    if (batch < 0 || s < 1) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!proposals_dev || !n_prop_dev || !decoded_dev || !n_accept_dev) return DOMINO_E_INVALID_ARG;
    if ((states_out_dev && !chain_states_dev) || (stacks_out_dev && !chain_stacks_dev)) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    return cuda_status(launch_spec_accept(proposals_dev, n_prop_dev, decoded_dev, chain_states_dev, chain_stacks_dev,
                                          batch, s, n_accept_dev, tokens_out_dev, states_out_dev, stacks_out_dev,
                                          (cudaStream_t)stream));
}

int domino_mask_logits_table(domino_t h, const void* logits_dev, int32_t dtype, int32_t batch,
                             int64_t row_stride_elems, const uint32_t* table_mask_dev, const int32_t* states_dev,
                             int32_t* argmax_dev, float* lse_dev, float* logprobs_dev, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (h->stack) return DOMINO_E_UNSUPPORTED;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0 || row_stride_elems < h->V) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_dev || !table_mask_dev || !states_dev || !argmax_dev) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    return cuda_status(launch_mask_logits(h->env, logits_dev, dtype, batch, row_stride_elems, h->V, table_mask_dev,
                                          argmax_dev, lse_dev, logprobs_dev, (cudaStream_t)stream, states_dev, h->Q, (uint32_t*)h->d_err.p));
}

int domino_advance_table(domino_t h, const int32_t* table_next_dev, const int32_t* states_dev,
                         const int32_t* tokens_dev, int32_t batch, int32_t* states_out, void* stream) {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (h->stack) return DOMINO_E_UNSUPPORTED;
    if (batch < 0) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!table_next_dev || !states_dev || !tokens_dev || !states_out) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    return cuda_status(launch_advance_table(table_next_dev, h->Q, h->V, h->eos_id, h->start, states_dev, tokens_dev,
                                            batch, states_out, (uint32_t*)h->d_err.p, (cudaStream_t)stream));
}

namespace {

// The host-buffer step's small inputs and outputs in one buffer (device s_io,
// pinned host h_io): [tokens | lse | states | stacks], each part on a 16-byte
// boundary.  The copy path moves states and stacks up in one copy and
// everything back in one; the in-place path's kernels read and write h_io
// directly.
struct IoLayout {
    size_t tok, lse, st, sk, in_end;
};
IoLayout io_layout(int32_t batch, bool stacks) {
    auto a16 = [](size_t x) { return (x + 15) / 16 * 16; };
    IoLayout L{};
    L.tok = 0;
    L.lse = a16(L.tok + (size_t)batch * 4);
    L.st = a16(L.lse + (size_t)batch * 4);
    L.sk = a16(L.st + (size_t)batch * 4);
    L.in_end = stacks ? L.sk + (size_t)batch * 8 : L.st + (size_t)batch * 4;
    return L;
}

// Pageable logits: the configurations and then the logits are copied in up
// to 8 chunks of rows on the copy stream; the mask step runs while they copy,
// and each chunk's masked argmax starts as soon as its rows have landed.
int copy_and_decode_chunks(domino_ctx* h, const void* logits_host, int32_t dtype, int32_t batch, bool stacks,
                           const IoLayout& L, cudaStream_t st) {
    int rc;
    void* stream = (void*)st;
    const size_t esz = dtype == DOMINO_DTYPE_BF16 ? 2 : 4;
    const size_t row_bytes = (size_t)h->V * esz;
    const size_t logit_bytes = (size_t)batch * row_bytes;
    char* io = (char*)h->s_io.p;
    int32_t* d_states = (int32_t*)(io + L.st);
    uint64_t* d_stacks = stacks ? (uint64_t*)(io + L.sk) : nullptr;
    uint32_t* d_mask = (uint32_t*)h->s_mask.p;
    int32_t* d_tok = (int32_t*)(io + L.tok);
    float* d_lse = (float*)(io + L.lse);
    const int n_chunks = (int)std::max<size_t>(1, std::min<size_t>({(size_t)8, (size_t)batch, logit_bytes >> 23}));
    cudaError_t e = cudaEventRecord(h->ev_cfg, st);   // the caller's earlier work on `stream` comes first
    if (e == cudaSuccess) e = cudaStreamWaitEvent(h->cp_stream, h->ev_cfg, 0);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(io + L.st, (char*)h->h_io + L.st, L.in_end - L.st, cudaMemcpyHostToDevice, h->cp_stream);
    if (e == cudaSuccess) e = cudaEventRecord(h->ev_cfg, h->cp_stream);
    int32_t r0s[9];   // at most 8 chunks
    for (int k = 0; k <= n_chunks; ++k) r0s[k] = (int32_t)(((int64_t)batch * k) / n_chunks);
    if (e == cudaSuccess) e = cudaEventRecord(h->ev_t[2], h->cp_stream);
    for (int k = 0; k < n_chunks && e == cudaSuccess; ++k) {
        const size_t off = (size_t)r0s[k] * row_bytes, n = (size_t)(r0s[k + 1] - r0s[k]) * row_bytes;
        e = cudaMemcpyAsync((char*)h->s_logits.p + off, (const char*)logits_host + off, n, cudaMemcpyHostToDevice,
                            h->cp_stream);
        if (e == cudaSuccess) e = cudaEventRecord(h->ev_chunk[k], h->cp_stream);
    }
    if (e == cudaSuccess) e = cudaEventRecord(h->ev_t[3], h->cp_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, h->ev_cfg, 0);
    if (e != cudaSuccess) return cuda_status(e);
    if ((rc = domino_step_mask(h, d_states, d_stacks, batch, d_mask, nullptr, stream))) return rc;
    for (int k = 0; k < n_chunks; ++k) {
        const int32_t r0 = r0s[k], rows = r0s[k + 1] - r0;
        if ((e = cudaStreamWaitEvent(st, h->ev_chunk[k], 0)) != cudaSuccess) return cuda_status(e);
        if ((rc = domino_mask_logits(h, (const char*)h->s_logits.p + (size_t)r0 * row_bytes, dtype, rows, h->V,
                                     d_mask + (size_t)r0 * h->W, d_tok + r0, d_lse + r0, nullptr, stream)))
            return rc;
    }
    // every copy-stream node rejoins `stream` (a recorded graph needs it; the
    // copies are done by now anyway)
    return cuda_status(cudaStreamWaitEvent(st, h->ev_t[3], 0));
}

// The host-buffer step's copies and launches on `st` (and the copy stream),
// without the final synchronisation.  The states and stacks are already in
// h_io; the outputs land there.
int enqueue_host_step(domino_ctx* h, const void* logits_host, void* logits_mapped, bool mapped, int32_t dtype,
                      int32_t batch, bool stacks, const IoLayout& L, cudaStream_t st) {
    int rc;
    void* stream = (void*)st;
    char* io = (char*)h->s_io.p;
    int32_t* d_states = (int32_t*)(io + L.st);
    uint64_t* d_stacks = stacks ? (uint64_t*)(io + L.sk) : nullptr;
    uint32_t* d_mask = (uint32_t*)h->s_mask.p;
    int32_t* d_tok = (int32_t*)(io + L.tok);
    float* d_lse = (float*)(io + L.lse);
    if (mapped) {
        // the mask step folds the pinned logits it allows, read in place; the
        // configurations are read from and the results written to the pinned
        // staging buffer itself (no copies: two kernels)
        char* hio = (char*)h->h_io_dev;
        int32_t* m_states = (int32_t*)(hio + L.st);
        uint64_t* m_stacks = stacks ? (uint64_t*)(hio + L.sk) : nullptr;
        return domino_step_decode(h, m_states, m_stacks, batch, logits_mapped, dtype, h->V, d_mask,
                                  (int32_t*)(hio + L.tok), (float*)(hio + L.lse), nullptr, m_states, m_stacks, stream);
    } else {
        if ((rc = copy_and_decode_chunks(h, logits_host, dtype, batch, stacks, L, st))) return rc;
        if ((rc = domino_advance(h, d_states, d_stacks, d_tok, batch, d_states, d_stacks, stream))) return rc;
    }
    return cuda_status(cudaMemcpyAsync(h->h_io, io, L.in_end, cudaMemcpyDeviceToHost, st));
}

}  // namespace

int domino_decode_step_host(domino_t h, const void* logits_host, int32_t dtype, int32_t batch,
                            int32_t* states_host, uint64_t* stacks_host, int32_t* tokens_host, float* lse_host,
                            void* stream) try {
    DOMINO_API_RANGE();
    int rc = ready_for_compute(h);
    if (rc) return rc;
    if (dtype != DOMINO_DTYPE_F32 && dtype != DOMINO_DTYPE_BF16) return DOMINO_E_INVALID_ARG;
    if (batch < 0) return DOMINO_E_INVALID_ARG;
    if (batch == 0) return DOMINO_OK;
    if (!logits_host || !states_host || !tokens_host) return DOMINO_E_INVALID_ARG;
    DeviceGuard g(h->device);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t esz = dtype == DOMINO_DTYPE_BF16 ? 2 : 4;
    const size_t row_bytes = (size_t)h->V * esz;
    const size_t logit_bytes = (size_t)batch * row_bytes;
    const bool stacks = stacks_host != nullptr;
    const IoLayout L = io_layout(batch, stacks);
    // Pinned (page-locked, mapped) bf16 logits can be read where they are: the
    // mask step folds each tile's allowed logits, so only those cross the host
    // link, while the walk runs.  Or they are copied in chunks while the mask
    // step runs and decoded as they land.  Which is faster depends on the
    // masks' density and on the link's read granularity, so it is measured:
    // each path's host wall time is averaged over settled calls (no buffer growth,
    // no recording), the faster one is used, and every 64th call takes the
    // other to keep its time current.
    const auto t_enter = std::chrono::steady_clock::now();
    cudaPointerAttributes pa{};
    const bool pinned = cudaPointerGetAttributes(&pa, logits_host) == cudaSuccess && pa.type == cudaMemoryTypeHost &&
                        pa.devicePointer != nullptr;
    if (!pinned) cudaGetLastError();
    bool mapped = pinned && dtype == DOMINO_DTYPE_BF16;
    const bool choice = mapped;
    if (choice) {
        if (h->t_wall_ms[1] == 0.0) mapped = true;
        else if (h->t_wall_ms[0] == 0.0) mapped = false;
        else mapped = (h->t_wall_ms[1] <= h->t_wall_ms[0]) != (h->host_calls % 64 == 63);
    }
    // where the in-place path folds the decode into the per-token walk, its
    // partials are grown here too, before any recording
    const bool fuse = mapped && can_fuse(h, pa.devicePointer, dtype, batch, h->V);
    const size_t part_bytes = fuse && !decode_rows(h, batch, fuse) ? fpart_bytes(h, batch) : 0;
    const bool grow = (!mapped && h->s_logits.n < logit_bytes) || h->s_io.n < L.in_end ||
                      h->s_mask.n < (size_t)batch * (size_t)h->W * 4 || h->h_io_n < L.in_end || !h->cp_stream ||
                      h->d_fpart.n < part_bytes;
    if (grow) {   // buffers may move: recorded steps that use them are dropped
        if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_status(cudaGetLastError());
        clear_host_graphs(h);
    }
    if (!mapped && (rc = dev_reserve(h->s_logits, logit_bytes))) return rc;
    if ((rc = grow_fpart(h, part_bytes))) return rc;
    if ((rc = dev_reserve(h->s_mask, (size_t)batch * (size_t)h->W * 4))) return rc;
    if ((rc = dev_reserve(h->s_io, L.in_end))) return rc;
    if (h->h_io_n < L.in_end) {
        if (h->h_io) cudaFreeHost(h->h_io);
        h->h_io = nullptr;
        h->h_io_n = 0;
        if (cudaMallocHost(&h->h_io, L.in_end) != cudaSuccess) {
            cudaGetLastError();
            h->h_io = nullptr;
            return DOMINO_E_OOM;
        }
        if (cudaHostGetDevicePointer(&h->h_io_dev, h->h_io, 0) != cudaSuccess) {
            cudaGetLastError();
            cudaFreeHost(h->h_io);
            h->h_io = h->h_io_dev = nullptr;
            return DOMINO_E_CUDA;
        }
        h->h_io_n = L.in_end;
    }
    if (!h->cp_stream) {
        cudaError_t e = cudaStreamCreateWithFlags(&h->cp_stream, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_cfg, cudaEventDisableTiming);
        for (cudaEvent_t& ev : h->ev_chunk)
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        for (cudaEvent_t& ev : h->ev_t)
            if (e == cudaSuccess) e = cudaEventCreate(&ev);
        if (e != cudaSuccess) return cuda_status(e);
    }
    std::memcpy((char*)h->h_io + L.st, states_host, (size_t)batch * 4);
    if (stacks) std::memcpy((char*)h->h_io + L.sk, stacks_host, (size_t)batch * 8);
    // The step's copies and launches, recorded once per set of buffers and
    // path on a non-default stream (the default stream cannot be captured) and
    // replayed afterwards.  The first two calls of a handle run them directly
    // (the first sets kernel attributes).
    const void* key[16] = {logits_host, (const void*)(intptr_t)batch,
                           (const void*)(intptr_t)(dtype * 4 + (mapped ? 1 : 0) + (stacks ? 2 : 0)), h->s_logits.p,
                           h->s_mask.p, h->s_io.p, h->h_io, (const void*)st, nullptr, nullptr, nullptr, nullptr,
                           nullptr, nullptr, nullptr, nullptr};
    cudaGraphExec_t exec = nullptr;
    for (auto& hg : h->host_graphs)
        if (std::equal(std::begin(key), std::end(key), std::begin(hg.key))) {
            exec = hg.exec;
            hg.used = h->host_calls;
        }
    cudaError_t e = cudaSuccess;
    const bool record = !exec && st != nullptr && h->host_calls > 1;
    if (record) {
        cudaGraph_t gr = nullptr;
        e = cudaStreamBeginCapture(st, cudaStreamCaptureModeRelaxed);
        if (e != cudaSuccess) return cuda_status(e);
        rc = enqueue_host_step(h, logits_host, pa.devicePointer, mapped, dtype, batch, stacks, L, st);
        e = cudaStreamEndCapture(st, &gr);
        if (rc || e != cudaSuccess) {
            if (gr) cudaGraphDestroy(gr);
            return rc ? rc : cuda_status(e);
        }
        e = cudaGraphInstantiate(&exec, gr, 0);
        cudaGraphDestroy(gr);
        if (e != cudaSuccess) return cuda_status(e);
        if (h->host_graphs.size() >= 8) {   // keep the 8 most recently used
            auto lru = std::min_element(h->host_graphs.begin(), h->host_graphs.end(),
                                        [](const domino_ctx::HostGraph& x, const domino_ctx::HostGraph& y) {
                                            return x.used < y.used;
                                        });
            cudaGraphExecDestroy(lru->exec);
            h->host_graphs.erase(lru);
        }
        domino_ctx::HostGraph hg{};
        std::copy(std::begin(key), std::end(key), std::begin(hg.key));
        hg.exec = exec;
        hg.used = h->host_calls;
        h->host_graphs.push_back(hg);
    }
    if (exec) {
        e = cudaGraphLaunch(exec, st);
    } else if ((rc = enqueue_host_step(h, logits_host, pa.devicePointer, mapped, dtype, batch, stacks, L, st))) {
        return rc;
    }
    h->host_calls++;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_status(e);
    const char* io = (const char*)h->h_io;
    std::memcpy(tokens_host, io + L.tok, (size_t)batch * 4);
    if (lse_host) std::memcpy(lse_host, io + L.lse, (size_t)batch * 4);
    std::memcpy(states_host, io + L.st, (size_t)batch * 4);
    if (stacks) std::memcpy(stacks_host, io + L.sk, (size_t)batch * 8);
    if (choice && !grow && !record && h->host_calls > 1) {
        // a moving average, so that one slow call (the host preempted, a
        // shared link) does not send the next 64 calls down the slower path
        const double t = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_enter).count();
        double& avg = h->t_wall_ms[mapped ? 1 : 0];
        avg = avg == 0.0 ? t : 0.75 * avg + 0.25 * t;
    }
    return DOMINO_OK;
} catch (...) {   // std::bad_alloc
    return DOMINO_E_OOM;
}


int domino_get_device_error(domino_t h, int32_t* code, void* stream) {
    if (!h || !code) return DOMINO_E_INVALID_ARG;
    *code = 0;
    if (is_host_only(h)) return DOMINO_E_NO_DEVICE;
    DeviceGuard g(h->device);
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t word = 0;
    cudaError_t e = cudaMemcpyAsync(&word, h->d_err.p, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_err.p, 0, 4, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_status(e);
    *code = (int32_t)word;
    return DOMINO_OK;
}

}  // extern "C"
