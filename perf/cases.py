"""The calls whose speed matters to a user of this library, with inputs, the work they cannot do without and
independent 64-bit results.

A serving program keeps one handle per (grammar, vocabulary) and calls it once per decode step, so handles are made
once per process and kept; the batch's configurations, the logits and the random grammar of a table precompute come
from the seed.  Grammars, vocabularies and sizes are the repository's own workloads (`paper_2403_06988_gb300.synth`)
and sizes around them; `draw` spreads over batch 1 to 1024, vocabularies of 300 to 160000 tokens (odd ones too) and
every kind of call.

Kinds of call (`case["kind"]`):
  loop        `steps` whole decode steps (mask, greedy decode, update in place) from given configurations
  graph       the same steps captured once in a CUDA graph and replayed, as a serving engine does
  mask        one mask step, with the next states of every allowed token when `next`
  logits      the masked decode alone, over masks that another component produced
  sample      the masked draw instead of the greedy decode
  table       the state x token table of a new grammar
  table_step  a decode step driven by such a table
  opportune   opportunistic masking: check the unmasked argmax, mask only the rows it fails on
  host        one whole step from and to host memory
"""
import functools

import numpy as np
import torch

from paper_2403_06988_gb300 import Domino, synth
from paper_2403_06988_gb300 import _binding as binding

DEV = "cuda:0"


def listed():
    return [
        # one interactive sequence with a small hand-written key/value grammar, fp32 logits: latency and launches
        {"name": "loop_kv16_b1", "kind": "loop", "grammar": "kv16", "V": 1024, "B": 1, "steps": 8, "dtype": "f32",
         "logprobs": False},
        # a small server: objects over fixed keys, 32K vocabulary
        {"name": "loop_kv200_b32", "kind": "loop", "grammar": "kv200", "V": 32000, "B": 32, "steps": 4,
         "dtype": "bf16", "logprobs": False},
        # the headline workload: batch 256 and a 128K vocabulary, the decode loop replayed from a CUDA graph
        {"name": "graph_sparse5000_b256", "kind": "graph", "grammar": "sparse5000", "V": 128256, "B": 256, "steps": 4,
         "dtype": "bf16", "logprobs": False},
        # a large batch of the same, called step by step
        {"name": "loop_sparse5000_b1000", "kind": "loop", "grammar": "sparse5000", "V": 128256, "B": 1000, "steps": 2,
         "dtype": "bf16", "logprobs": False},
        # JSON with a bracket stack at batch 128, log-probabilities returned (scoring, beam search)
        {"name": "loop_json_b128_logprobs", "kind": "loop", "grammar": "json", "V": 152064, "B": 128, "steps": 2,
         "dtype": "bf16", "logprobs": True},
        # JSON at a middling batch and an odd vocabulary size: rows off 16-byte boundaries
        {"name": "loop_json_b24_odd", "kind": "loop", "grammar": "json", "V": 50001, "B": 24, "steps": 4,
         "dtype": "bf16", "logprobs": False},
        # masks and next states of a few rows (lookahead, tree search over tokens)
        {"name": "mask_next_kv200_b48", "kind": "mask", "grammar": "kv200", "V": 32003, "B": 48, "next": True},
        # offline: the whole state x token table of a large grammar
        {"name": "table_sparse20000", "kind": "table", "Q": 20000, "V": 128256},
        # masks from elsewhere applied to fp32 logits, with log-probabilities
        {"name": "logits_f32_b64", "kind": "logits", "V": 32000, "B": 64, "dtype": "f32", "permille": 300,
         "logprobs": True},
        # sampling at batch 128 from masks that allow most tokens (inside JSON strings)
        {"name": "sample_b128_dense", "kind": "sample", "V": 152064, "B": 128, "dtype": "bf16", "permille": 800},
        # opportunistic masking on JSON
        {"name": "opportune_json_b64", "kind": "opportune", "grammar": "json", "V": 152064, "B": 64, "dtype": "bf16"},
        # logits arriving in pinned host memory
        {"name": "host_sparse5000_b256", "kind": "host", "grammar": "sparse5000", "V": 128256, "B": 256,
         "dtype": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _sizes(rng, grammar):
    lo, hi = {"kv16": (300, 4096), "kv200": (4000, 64000), "json": (32000, 160000)}.get(grammar, (32000, 160000))
    V = _log(rng, lo, hi)
    V = V | 1 if rng.random() < 0.3 else V // 32 * 32 if rng.random() < 0.7 else V
    return V, _log(rng, 1, 1024 if grammar != "kv16" else 64)


def draw(rng):
    kind = rng.choice(["loop", "loop", "loop", "loop", "graph", "mask", "mask", "logits", "logits", "sample", "table",
                       "table_step", "opportune", "host"])
    grammar = rng.choice(["kv16", "kv200", "kv200", "sparse5000", "sparse5000", "sparse%d" % _log(rng, 500, 20000), "json",
                          "json"])
    V, B = _sizes(rng, grammar)
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    if kind in ("loop", "graph"):
        return {"kind": kind, "grammar": grammar, "V": V, "B": B, "steps": rng.choice([1, 2, 4, 8]) if B < 300 else 1,
                "dtype": dtype, "logprobs": rng.random() < 0.25}
    if kind == "mask":
        return {"kind": kind, "grammar": grammar, "V": V, "B": B, "next": rng.random() < 0.5}
    if kind == "logits":
        return {"kind": kind, "V": _log(rng, 1000, 160000), "B": B, "dtype": dtype, "permille": _log(rng, 2, 1000),
                "logprobs": rng.random() < 0.4}
    if kind == "sample":
        return {"kind": kind, "V": _log(rng, 1000, 160000), "B": _log(rng, 1, 256), "dtype": dtype,
                "permille": _log(rng, 2, 1000)}
    if kind == "table":
        return {"kind": kind, "Q": _log(rng, 500, 16000), "V": _log(rng, 8000, 128000)}
    if kind == "table_step":
        return {"kind": kind, "Q": _log(rng, 500, 5000), "V": _log(rng, 8000, 128000), "B": B, "dtype": dtype}
    if kind == "opportune":
        return {"kind": kind, "grammar": grammar, "V": V, "B": B, "dtype": dtype}
    return {"kind": "host", "grammar": grammar, "V": V, "B": min(B, 256), "dtype": "bf16"}


# ---------------------------------------------------------------------------
# what a program keeps: vocabularies, grammars, handles
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=16)
def _vocab(family, V):
    rng = np.random.default_rng([77, V])
    if family == "kv16":
        alpha = np.frombuffer(synth.CFG1_ALPHABET, dtype=np.uint8)
        return synth.random_vocab(rng, V, synth.CFG1_ALPHABET, lambda r, m: r.integers(1, 9, size=m).astype(np.int64),
                                  lambda r, n: alpha[r.integers(0, alpha.size, n)])
    mean, longest = {"kv200": (4.0, 16), "json": (4.0, 32)}.get(family, (4.5, 32))
    return synth.random_vocab(rng, V, bytes(range(256)), synth.geometric_lengths(mean, longest), synth._mixed_bytes)


@functools.lru_cache(maxsize=8)
def _grammar(name):
    rng = np.random.default_rng([78, sum(name.encode())])
    if name == "kv16":
        return synth.kv16_dfa()
    if name == "kv200":
        return synth.kv200_dfa(rng)[0]
    if name == "json":
        return synth.json_pda(rng)[0]
    return synth.random_sparse_dfa(rng, int(name[len("sparse"):]))


@functools.lru_cache(maxsize=4)
def _handle(grammar, V):
    d = Domino.from_parts(_grammar(grammar), _vocab(grammar.rstrip("0123456789") if "sparse" in grammar else grammar, V))
    return d


@functools.lru_cache(maxsize=2)
def _json_pool():
    """Configurations met in JSON documents: random legal walks to nesting depths 0 to 32."""
    a, rng = _grammar("json"), np.random.default_rng(79)
    return [synth.random_pda_walk(a, rng, int(rng.integers(0, a.max_depth + 1))) for _ in range(160)]


def _configs(grammar, B, rng):
    a = _grammar(grammar)
    if a.rules is None:
        states = rng.choice(np.nonzero(a.live)[0], size=B).astype(np.int32)
        return torch.from_numpy(states).to(DEV), None
    pool = _json_pool()
    pick = rng.integers(0, len(pool), size=B)
    states = np.array([pool[i][0] for i in pick], np.int32)
    stacks = np.array([synth.pack_stack(pool[i][1]) for i in pick], np.uint64)
    return torch.from_numpy(states).to(DEV), torch.from_numpy(stacks.view(np.int64)).to(DEV)


def _logits(case, gen, rows=None):
    x = torch.randn((rows or case["B"], case["V"]), generator=gen, device=DEV) * 3.0
    return x if case["dtype"] == "f32" else x.to(torch.bfloat16)


def _masks(case, gen):
    """Masks of about `permille` / 1000 allowed tokens, the share varying between rows; one row allows nothing."""
    B, V = case["B"], case["V"]
    W = (V + 31) // 32
    share = (torch.rand((B, 1), generator=gen, device=DEV) + 0.5) * (case["permille"] / 1000.0)
    bits = torch.rand((B, W * 32), generator=gen, device=DEV) < share
    bits[:, V:] = False
    if B > 8:
        bits[B // 2] = False
    w = (bits.view(B, W, 32).to(torch.int64) << torch.arange(32, device=DEV)).sum(-1)
    return torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32)


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def _steps(s):
    d, st, sk = s["d"], s["st"], s["sk"]
    st.copy_(s["st0"])
    if sk is not None:
        sk.copy_(s["sk0"])
    out = {"tokens": [], "lse": []}
    for lg in s["logits"]:
        _, tok, lse, lp = d.step_decode(st, sk, lg, want_logprobs=s["logprobs"], advance=True, out_mask=s["mask"])
        out["tokens"].append(tok)
        out["lse"].append(lse)
    out["mask"], out["states"] = s["mask"], st
    if sk is not None:
        out["stacks"] = sk
    if s["logprobs"]:
        out["logprobs"] = lp
    return out


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([80, seed])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    s = {"kind": kind}
    if kind in ("loop", "graph"):
        s["d"] = d = _handle(case["grammar"], case["V"])
        s["st0"], s["sk0"] = _configs(case["grammar"], case["B"], rng)
        s["st"], s["sk"] = s["st0"].clone(), None if s["sk0"] is None else s["sk0"].clone()
        s["logits"] = [_logits(case, gen) for _ in range(case["steps"])]
        s["mask"] = torch.empty((case["B"], d.info()["n_words"]), dtype=torch.int32, device=DEV)
        s["logprobs"] = case["logprobs"]
        if kind == "graph":
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _steps(s)
            torch.cuda.current_stream().wait_stream(side)
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                s["out"] = _steps(s)
    elif kind == "mask":
        s["d"] = _handle(case["grammar"], case["V"])
        s["st"], s["sk"] = _configs(case["grammar"], case["B"], rng)
        s["next"] = case["next"]
    elif kind in ("logits", "sample"):
        s["d"] = _handle("kv16", case["V"]) if case["V"] < 4096 else _handle("kv200", case["V"])
        s["logits"], s["mask"] = _logits(case, gen), _masks(case, gen)
        s["seed"], s["logprobs"] = seed, case.get("logprobs")
    elif kind == "table":
        s["d"] = Domino.from_parts(synth.random_sparse_dfa(rng, case["Q"]), _vocab("sparse", case["V"]))
    elif kind == "table_step":
        a = synth.random_sparse_dfa(rng, case["Q"])
        s["d"] = Domino.from_parts(a, _vocab("sparse", case["V"]))
        s["next"], s["mask"] = s["d"].precompute_table()
        s["st"] = torch.from_numpy(rng.choice(np.nonzero(a.live)[0], size=case["B"]).astype(np.int32)).to(DEV)
        s["out"] = torch.empty_like(s["st"])
        s["logits"] = _logits(case, gen)
    elif kind == "opportune":
        s["d"] = _handle(case["grammar"], case["V"])
        s["st"], s["sk"] = _configs(case["grammar"], case["B"], rng)
        s["logits"] = _logits(case, gen)
    else:
        s["d"] = _handle(case["grammar"], case["V"])
        st, sk = _configs(case["grammar"], case["B"], rng)
        s["st0"], s["sk0"] = st.cpu(), None if sk is None else sk.cpu()
        s["st"], s["sk"] = s["st0"].clone().pin_memory(), None if sk is None else s["sk0"].clone().pin_memory()
        s["logits"] = _logits(case, gen).cpu().pin_memory()
        s["tok"] = torch.empty(case["B"], dtype=torch.int32).pin_memory()
        s["lse"] = torch.empty(case["B"], dtype=torch.float32).pin_memory()
        s["stream"] = torch.cuda.Stream()
    return s


def run(s):
    kind, d = s["kind"], s["d"]
    if kind == "loop":
        return _steps(s)
    if kind == "graph":
        s["graph"].replay()
        return s["out"]
    if kind == "mask":
        mask, nxt = d.step_mask(s["st"], s["sk"], want_next=s["next"])
        return {"mask": mask, "next": nxt} if s["next"] else {"mask": mask}
    if kind == "logits":
        tok, lse, lp = d.mask_logits(s["logits"], s["mask"], want_logprobs=s["logprobs"])
        return {"tokens": tok, "lse": lse, "logprobs": lp} if s["logprobs"] else {"tokens": tok, "lse": lse}
    if kind == "sample":
        return {"tokens": d.mask_sample(s["logits"], s["mask"], 0.8, s["seed"], 1)}
    if kind == "table":
        nxt, mask = d.precompute_table()
        return {"next": nxt, "mask": mask}
    if kind == "table_step":
        tok, lse, _ = d.mask_logits_table(s["logits"], s["mask"], s["st"])
        d.advance_table(s["next"], s["st"], tok, states_out=s["out"])
        return {"tokens": tok, "lse": lse, "states": s["out"]}
    if kind == "opportune":
        tok, n = d.opportunistic_step(s["logits"], s["st"], s["sk"])
        return {"tokens": tok, "fallbacks": n}
    s["st"].copy_(s["st0"])
    if s["sk"] is not None:
        s["sk"].copy_(s["sk0"])
    binding.domino_decode_step_host(d.h, s["logits"], binding.DTYPE_BF16, s["st"].shape[0], s["st"], s["sk"], s["tok"],
                                    s["lse"], stream=s["stream"])
    out = {"tokens": s["tok"], "lse": s["lse"], "states": s["st"]}
    return out if s["sk"] is None else dict(out, stacks=s["sk"])


def work(case):
    """Each input once and each output once; two operations per (row, token) where logits are decoded."""
    kind, V = case["kind"], case["V"]
    W = (V + 31) // 32
    if kind == "table":
        return {"bytes": case["Q"] * (4 * V + 4 * W), "flops": case["Q"] * V}
    B, esz = case["B"], 4 if case.get("dtype") == "f32" else 2
    if kind == "mask":
        return {"bytes": B * (16 + 4 * W + (4 * V if case["next"] else 0)), "flops": B * V}
    per = B * (V * esz + 4 * W + 32 + (4 * V if case.get("logprobs") else 0))
    return {"bytes": per * case.get("steps", 1), "flops": 2 * B * V * case.get("steps", 1)}


def tolerance(case):
    """Masks, states and tokens are exact; the log-sum-exp and the log-probabilities are fp32 sums of fp32
    exponentials (2^x of the hardware, about 2e-7 each) over up to 160000 terms, taken in any order."""
    if case["kind"] in ("mask", "sample", "table", "opportune"):
        return "exact"
    return {"rel": 1e-6, "max": 4e-6}


# ---------------------------------------------------------------------------
# the same results in plain torch, in 64 bits
# ---------------------------------------------------------------------------
def _allowed(a, vocab, states, stacks):
    """bool [B][V] and int64 next states [B][V] (and the stacks after each token), by the definition: every token's
    bytes walked from every row's configuration."""
    V, B = vocab.n_tokens, states.shape[0]
    off = torch.from_numpy(vocab.offsets).to(DEV)
    data = torch.from_numpy(vocab.data.astype(np.int64)).to(DEV)
    delta = torch.from_numpy(a.delta.astype(np.int64)).to(DEV)
    live = torch.from_numpy(a.live.astype(np.int64)).to(DEV).bool()
    lens = off[1:] - off[:-1]
    rule = torch.full((a.n_states * 256,), -1, dtype=torch.int64, device=DEV)
    if a.rules is not None:
        r = {k: torch.from_numpy(a.rules[k].astype(np.int64)).to(DEV) for k in a.rules.dtype.names}
        rule[r["state"] * 256 + r["byte"]] = torch.arange(len(a.rules), device=DEV)
        back = torch.stack([r["next_if_empty"], r["next_if_top0"], r["next_if_top1"]], 1)
    ok = torch.zeros((B, V), dtype=torch.bool, device=DEV)
    nxt = torch.zeros((B, V), dtype=torch.int64, device=DEV)
    stk = torch.zeros((B, V), dtype=torch.int64, device=DEV) if stacks is not None else None
    tok = torch.nonzero(lens > 0).view(-1)
    for b0 in range(0, B, 64):                        # rows at a time, so that the pairs fit
        rows = torch.arange(b0, min(B, b0 + 64), device=DEV)
        row, t = rows.repeat_interleave(tok.numel()), tok.repeat(rows.numel())
        s = states[row].long()
        word = stacks[row] if stacks is not None else torch.zeros_like(row)
        bits, depth = word & 0xFFFFFFFF, word >> 32
        at = 0
        while t.numel():
            c = data[off[t] + at]
            e = delta[s, c]
            if a.rules is not None:
                q = rule[s * 256 + c]
                has = q >= 0
                q = q.clamp(min=0)
                push, pop = has & (r["kind"][q] == synth.RULE_PUSH), has & (r["kind"][q] == synth.RULE_POP)
                sym = r["sym"][q]
                bad = (push & (depth >= a.max_depth)) | (pop & ((depth == 0) | ((bits & 1) != sym)))
                nb, nd = bits >> 1, depth - 1
                e = torch.where(pop, back[q, torch.where(nd <= 0, 0, 1 + (nb & 1))], e)
                bits = torch.where(push, (bits << 1 | sym) & 0xFFFFFFFF, torch.where(pop, nb, bits))
                depth = torch.where(push, depth + 1, torch.where(pop, nd, depth))
                e = torch.where(bad, 0, e)
            at += 1
            keep = live[e]
            done = keep & (lens[t] == at)
            ok[row[done], t[done]] = True
            nxt[row[done], t[done]] = e[done]
            if stk is not None:
                stk[row[done], t[done]] = depth[done] << 32 | bits[done]
            keep &= ~done
            row, t, s, bits, depth = row[keep], t[keep], e[keep], bits[keep], depth[keep]
    if vocab.eos_id >= 0:
        acc = torch.from_numpy(a.accepting).to(DEV).bool()[states.long()]
        if stacks is not None:
            acc = acc & (stacks >> 32 == 0)
        ok[:, vocab.eos_id] = acc
    return ok, nxt, stk


def _decode(logits, ok):
    """Greedy token (lowest id on ties, -1 when nothing is allowed), log-sum-exp and log-probabilities."""
    x = logits.double().masked_fill(~ok, -torch.inf)
    best = x.max(1, keepdim=True).values
    ids = torch.arange(x.shape[1], device=DEV)
    tok = torch.where((x == best) & ok, ids, x.shape[1]).min(1).values
    lse = torch.logsumexp(x, 1)
    return torch.where(ok.any(1), tok, -1), lse, x - torch.where(torch.isfinite(lse), lse, 0.0)[:, None]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mask", "sample", "table", "opportune"):
        return None                                   # whole numbers only
    s = prepare(dict(case, kind="loop") if kind == "graph" else case, seed)
    if kind == "logits":
        V = case["V"]
        ok = (s["mask"][:, :, None] >> torch.arange(32, device=DEV) & 1).view(case["B"], -1)[:, :V].bool()
        _, lse, lp = _decode(s["logits"], ok)
        return {"tokens": None, "lse": lse, "logprobs": lp} if s["logprobs"] else {"tokens": None, "lse": lse}
    if kind == "table_step":
        a = synth.random_sparse_dfa(np.random.default_rng([80, seed]), case["Q"])
        _, lse, _ = _decode(s["logits"], _allowed(a, _vocab("sparse", case["V"]), s["st"], None)[0])
        return {"tokens": None, "lse": lse, "states": None}
    a = _grammar(case["grammar"])
    vocab = _vocab("sparse" if "sparse" in case["grammar"] else case["grammar"], case["V"])
    st = s["st0"].to(DEV).long()
    sk = None if s["sk0"] is None else s["sk0"].to(DEV)
    out = {"tokens": None, "lse": []}
    for lg in s["logits"] if kind != "host" else [s["logits"].to(DEV)]:
        ok, nxt, stk = _allowed(a, vocab, st, sk)
        tok, lse, lp = _decode(lg, ok)
        out["lse"].append(lse)
        at = tok.clamp(min=0)[:, None]
        end = (tok < 0) | (tok == vocab.eos_id)
        st = torch.where(end, a.start, nxt.gather(1, at)[:, 0])
        if sk is not None:
            sk = torch.where(end, 0, stk.gather(1, at)[:, 0])
    if kind == "host":
        out["lse"] = out["lse"][0]
    out["mask"] = out["states"] = out["stacks"] = None
    if case.get("logprobs"):
        out["logprobs"] = lp
    return out
