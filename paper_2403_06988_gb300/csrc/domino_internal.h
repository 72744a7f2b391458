// domino_internal.h -- shared between the host-side C ABI (host.cpp) and the
// sm_103a kernels (kernels.cu).  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "domino.h"

namespace domino {

// Vocabulary windows: original ids [w*kWin, (w+1)*kWin) form window w.  Inside
// a window the tokens are stored sorted by their byte-class strings, so tokens
// with the same first class form one contiguous group and neighbouring tokens
// share prefixes (same transitions, same early exit for a warp).  The allowed
// bits are scattered back to original ids in shared memory.
constexpr int kWin = 1024;
constexpr int kStepThreads = 1024;             // step kernel CTA size (one CTA per SM)
constexpr int kRowsPerTile = 4;                // fewest rows per tile (mask only; small batches)
constexpr int kMaxRowsPerTile = 32;            // most rows per tile (one warp ballot)
constexpr int kRowsPerTileNext = 8;            // rows per tile when next states are written
constexpr int kWalkChains = 4;                 // rows walked together by one lane (independent chains)
constexpr int kHeadBytes = 16;                 // class ids per 16-byte head block
constexpr int kInlineBytes = 32;               // class ids stored inline per token (two head blocks)
constexpr int kLogitThreads = 256;
constexpr int kAdvanceThreads = 128;

// slot info word: bits 0..9 original id within the window, bit 10 valid,
// bits 16..31 byte length (0 for EOS and empty tokens)
constexpr uint32_t kInfoValid = 1u << 10;

// Table entry of a pushdown automaton (uint32): bits 0..15 next state, bits
// 16..17 kind (0 none, 1 push, 2 pop), bit 18 symbol, bits 19..31 index of the
// pop's (empty, top0, top1) target triple.  A plain DFA uses uint16 entries.
constexpr uint32_t kKindShift = 16, kSymShift = 18, kRetShift = 19;
constexpr uint32_t kMaxRetTriples = 1u << 13;

// Where the step kernel reads transitions from.
enum TableMode : int {
    kDenseSmem = 0,    // [Q][K] entries staged in shared memory
    kSparse32Smem = 1, // per state {live-class mask, base} + packed live entries (K <= 32)
    kSparse64Smem = 2, // the same with a 64-bit class mask (K <= 64)
    kDenseGlobal = 3,  // [Q][K] entries read through L1/L2
};

struct StepView {
    // vocabulary arena (slot order)
    const uint4* head;        // [n_slots][2] class ids of bytes 0..15 and 16..31
    const uint32_t* info;     // [n_slots] original id in window | valid | length
    const int32_t* tail_off;  // [n_slots] offset of bytes 32.. in `tail`
    const uint8_t* tail;      // class ids of bytes 32.. of tokens longer than 32 bytes
    const int32_t* pos_of;    // [V] slot of original id
    // the slots of first class c in window w are [cls_start[w][c], cls_start[w][c + 1])
    const uint16_t* cls_start; // [n_windows][K + 1]
    const int16_t* eos_slot;  // [n_windows] window-local slot of EOS, -1 if not in the window
    int32_t V, W, n_windows, eos_id;
    // automaton
    const uint16_t* t16;      // [Q][K] (DFA)
    const uint32_t* t32;      // [Q][K] (pushdown)
    const uint32_t* sp_info;  // sparse rows: [Q][2] or [Q][4] uint32 words
    const void* sp_tgt;       // sparse live entries (uint16 or uint32)
    const uint16_t* ret;      // [n_ret][4]
    const uint32_t* accept_bits;
    // self loops (nullptr when not used): per state the classes that keep it,
    // per slot the classes of the token's bytes after the first
    const unsigned long long* self_mask;  // [Q]
    const unsigned long long* tok_cls;    // [n_slots]
    int32_t Q, K, start, max_depth, n_ret, sp_nnz;
    uint32_t* err;            // sticky device error word
};

// Prefix tree of the vocabulary's byte-class strings (the subterminal tree of
// Sec. 3.3, Alg. 2, over byte classes) as domino_get_prefix_tree exports it
// (RowTree below is what the kernel reads).
// Nodes are numbered in preorder (children by class), so a subtree is the
// contiguous range [n, skip) and the tokens of a subtree are a contiguous
// range of the token list: the tokens that end at n first, then those of its
// children's subtrees.
//   node[2n]     = {skip | cls << 24, tok_lo, n_end, tok_hi}
//   node[2n + 1] = {sub_lo, sub_hi, 0, 0}
// cls: the class on the edge into n; [tok_lo, tok_lo + n_end): tokens ending
// at n; [tok_lo, tok_hi): tokens of the subtree; sub: the classes on the edges
// below n (K <= 64).
// Upper nodes: the root and every node whose subtree has more than kTrieTile
// nodes or more than kTrieBranch branching levels (an ancestor of an upper
// node is upper).  Units: the subtrees hanging off upper nodes.
constexpr int kTrieTile = 64;
constexpr int kTrieBranch = 8;
constexpr int32_t kTrieMaxNodes = (1 << 24) - 1;

// The trees row_kernel walks (rows.cu).  The first (root: node 0) holds the
// class strings of all tokens (but EOS and empty ones).  The others belong to
// the loop sets: a loop set is the classes that keep some state L (with no
// stack action).  A row in L allows every token made of these classes only
// (loopbits) and stays where it is over the longest such prefix of any other
// token, so the set's tree holds the other tokens' remainders after that
// prefix.
// Nodes are numbered breadth first per tree: a node's children are
// consecutive, in class order.  Tokens are listed in preorder, so a subtree's
// are consecutive, the node's own first.
//   node[2n]     = {children's classes (64 bits; K > 64: their number, 0),
//                   first child | tokens ending here (255: or more) << 24,
//                   the subtree's first token}
//   node[2n + 1] = {subtree's tokens [x, y) in dtok, classes below (64 bits)}
// State records (K <= 64), srec_stride bytes each: {live classes, classes
// that keep the state} (64 bits each), then the live classes' entries.  Bit
// 63 of the second (K <= 63 where there are loop sets): the state has a loop
// set.  For masks the states are those of the automaton with equivalent
// states merged (start: the state a row begins in).
// Inside any tree, a node entered in L with loop set S: its subtree's tokens
// p of dtok that stay inside S from the node on are those with keeps[S][p] <=
// the node's depth; the edges below it that leave S are the entries
// xrange[S][node] of exits (preorder) whose nearest exit above (0: none) is
// no deeper than the node.
struct RowTree {
    const uint4* node;
    const uint8_t* ncls;        // [n_nodes] class on the edge into each node
    const int32_t* dtok;
    const uint4* srec;
    const uint16_t* ret;        // pop targets, [triples][4]
    const uint2* start;         // [Q]: {the record's state, its loop set or ~0}; nullptr: the state itself, no loop sets
    const uint32_t* loop_of;    // per record its loop set or ~0
    const uint32_t* loopbits;   // [loop sets][W]
    const uint8_t* keeps;       // [loop sets][n_dtok]: position after the last class outside the set (at most 255)
    const uint2* xrange;        // [loop sets][n_nodes]: {first exit below | depth << 24 (255: or more), end exit}
    const uint8_t* trec;        // [V][32]: {token length (255: or more), its first 31 classes}
    const uint2* exits;         // {node, its class | depth of the nearest exit above (at most 255) << 8}
    int32_t srec_stride, n_nodes, n_dtok, n_loops;
    int32_t loop_root[4];
};
constexpr int kRowLoopSets = 4;           // loop sets with a tree of their own
constexpr int kRowMaxSlices = 8;          // CTAs per row (one cluster)
constexpr int kRowSliceWords = 16384;     // mask words a CTA can hold
constexpr int kRowThreads = 512;          // a CTA's, or half of it (launch_row_d)
constexpr int kRowPool = 2816;            // (node, state) items a row may have at a time; a row with more is walked
                                          // token by token

struct LaunchEnv {
    int num_sms;
    int max_smem_optin;
};

// Bytes the table of `mode` occupies in shared memory (0 for kDenseGlobal).
int64_t table_smem_bytes(const StepView& v, bool stack, int mode);

// Shared-memory bytes of the step kernel other than the table.
int step_fixed_smem_bytes(const StepView& v, bool next);

// row_ids / row_count (device): only rows row_ids[i], i < *row_count <= batch,
// are walked; their masks are written to the compact rows i of `mask`.
cudaError_t launch_step_mask(const StepView& v, const LaunchEnv& env, bool stack, int mode, const int32_t* states,
                             const uint64_t* stacks, int32_t batch, bool row_is_state, uint32_t* mask,
                             int32_t* next, cudaStream_t st, const int32_t* row_ids = nullptr,
                             const int32_t* row_count = nullptr, const void* fuse_logits = nullptr,
                             int64_t fuse_stride = 0, float4* fuse_part = nullptr, bool fuse_prefetch = false);

// The mask step fused with the masked decode (bf16 logits, rows on 16-byte
// boundaries): fuse_part [batch][n_windows] receives per-window partials,
// merged into argmax / lse by launch_fused_combine, which also advances each
// row by its argmax when states_out is given (outputs may alias the inputs).
cudaError_t launch_fused_combine(const StepView& v, bool stack, int mode, const float4* part, int32_t batch,
                                 int32_t n_windows, int32_t* argmax, float* lse, const int32_t* states,
                                 const uint64_t* stacks, int32_t* states_out, uint64_t* stacks_out, cudaStream_t st);

// The mask step with one CTA (or a cluster of them) per row; arguments as
// launch_step_mask.  Any K, V <= kRowMaxSlices * kRowSliceWords * 32, and a
// tree whose row_smem_bytes fit.
cudaError_t launch_row_step(const StepView& v, const RowTree& t, const LaunchEnv& env, bool stack,
                            const int32_t* states, const uint64_t* stacks, int32_t batch, bool row_is_state,
                            uint32_t* mask, int32_t* next, cudaStream_t st);
// The mask step, the masked greedy decode and (with states_out) the update in
// one kernel; logits in device or mapped host memory, any dtype and alignment;
// outputs may alias states / stacks.
cudaError_t launch_row_decode(const StepView& v, const RowTree& t, const LaunchEnv& env, bool stack,
                              const int32_t* states, const uint64_t* stacks, int32_t batch, const void* logits,
                              int dtype, int64_t row_stride, bool on_device, uint32_t* mask, int32_t* argmax,
                              float* lse, float* logprobs, int32_t* states_out, uint64_t* stacks_out, cudaStream_t st);
// Shared-memory bytes of row_kernel at most, for a vocabulary of n_words mask words.
int row_smem_bytes(int32_t n_words, bool stack, bool loops);

// Log-probabilities only (bf16 logits, rows on 16-byte boundaries), given the
// rows' lse: logprobs[b][t] = logit - lse[b] for allowed t, -inf else.
cudaError_t launch_logprobs_bf16(const LaunchEnv& env, const void* logits, int32_t batch, int64_t row_stride,
                                 int32_t V, const uint32_t* mask, const float* lse, float* logprobs, cudaStream_t st);

// Sampling decode: Gumbel-max with Philox4x32-10 uniforms (decode.cuh).
struct SampleArgs {
    uint32_t key0, key1;     // the 64-bit seed
    uint32_t off0, off1;     // the 64-bit offset (counter words 2 and 3)
    float inv_t;             // 1 / temperature, rounded to fp32
};

// row_state (table-driven step): row r's mask is row row_state[r] of the
// [Q][W] table `mask`; out-of-range states read as empty rows and set `err`.
// sample: draw each row's token (into argmax) instead of the greedy argmax;
// lse and logprobs must then be null.  mask == nullptr (no row_state): every
// token allowed.  row_ids / row_count (device): only rows row_ids[i] for
// i < *row_count are processed, their masks being the compact rows i of
// `mask`; argmax and lse are indexed by batch row; no logprobs.
cudaError_t launch_mask_logits(const LaunchEnv& env, const void* logits, int dtype, int32_t batch,
                               int64_t row_stride, int32_t V, const uint32_t* mask, int32_t* argmax, float* lse,
                               float* logprobs, cudaStream_t st, const int32_t* row_state = nullptr, int32_t Q = 0,
                               uint32_t* err = nullptr, const SampleArgs* sample = nullptr,
                               const int32_t* row_ids = nullptr, const int32_t* row_count = nullptr);

// Fills the sampling arguments (1/T in fp32, seed and offset words).
cudaError_t launch_mask_sample(const LaunchEnv& env, const void* logits, int dtype, int32_t batch,
                               int64_t row_stride, int32_t V, const uint32_t* mask, float temperature,
                               uint64_t seed, uint64_t offset, int32_t* tokens, cudaStream_t st);

// `mode` names the table image the step kernel reads (it is L2-resident after a step).
cudaError_t launch_advance(const StepView& v, bool stack, int mode, const int32_t* states, const uint64_t* stacks,
                           const int32_t* tokens, int32_t batch, int32_t* states_out, uint64_t* stacks_out,
                           cudaStream_t st);

cudaError_t launch_advance_table(const int32_t* table_next, int32_t Q, int32_t V, int32_t eos_id, int32_t start,
                                 const int32_t* states, const int32_t* tokens, int32_t batch, int32_t* states_out,
                                 uint32_t* err, cudaStream_t st);

// Opportunistic masking: accepts row b's proposal into tokens_out[b] or
// appends b to row_ids (counter *row_count, zeroed by the caller).
cudaError_t launch_propose_check(const StepView& v, bool stack, int mode, const int32_t* states,
                                 const uint64_t* stacks, const int32_t* proposals, int32_t batch, int32_t* tokens_out,
                                 int32_t* row_ids, int32_t* row_count, cudaStream_t st);

// Count-based speculation (Sec. 3.6): count update, proposals, acceptance.
cudaError_t launch_spec_update(const StepView& v, bool stack, const int32_t* states, const uint64_t* stacks,
                               const int32_t* tokens, int32_t batch, uint32_t* counts, unsigned long long* best,
                               uint32_t* reached, cudaStream_t st);
cudaError_t launch_spec_propose(const StepView& v, bool stack, int mode, const int32_t* states,
                                const uint64_t* stacks, int32_t batch, int32_t s, int32_t min_permille,
                                const unsigned long long* best, const uint32_t* reached, int32_t* proposals,
                                int32_t* n_prop, int32_t* chain_states, uint64_t* chain_stacks, cudaStream_t st);
cudaError_t launch_spec_accept(const int32_t* proposals, const int32_t* n_prop, const int32_t* decoded,
                               const int32_t* chain_states, const uint64_t* chain_stacks, int32_t batch, int32_t s,
                               int32_t* n_accept, int32_t* tokens_out, int32_t* states_out, uint64_t* stacks_out,
                               cudaStream_t st);


}  // namespace domino
