"""Automata and vocabularies whose rows have levels of the prefix tree with more
live nodes than row_kernel's pool holds (2816), so that the row is walked token
by token (every_token): 40 states, each of which refuses one of 40 letters that
are a class each and lead everywhere else, with brackets between them or not; or
30 states with 90 of 100 classes live.  The tokens have lengths around the parts
of the token records (15, 31, 32 classes) and beyond, most of these alive from
some state."""
import functools

import numpy as np

from paper_2403_06988_gb300 import synth

POOL = 2816
LONG = (14, 15, 16, 30, 31, 32, 33, 60)


@functools.lru_cache(maxsize=None)
def problem(kind):
    """(automaton, vocabulary) of kind "plain", "stack" or "wide"; the EOS token is number 700."""
    rng = np.random.default_rng(61)
    if kind == "wide":
        a, alphabet = synth.random_sparse_dfa(rng, 30, 100, 90), bytes(range(256))
    else:
        letters, n = bytes(range(64, 104)), 40
        b = synth._Builder()
        q = [b.state("s%d" % i, accepting=i % 2 == 0) for i in range(n)]
        for i in range(n):
            for k, c in enumerate(letters):
                if k != i:
                    b.edge(q[i], [c], q[(i + k) % n])
            if kind == "stack":
                b.push(q[i], b"(", i % 2, q[(i + 1) % n])
                b.pop(q[i], b")", i // 2 % 2, (q[(i + 7) % n], q[i], q[(i + 11) % n]))
        a = b.build(q[0], 5 if kind == "stack" else 0, "full pools")
        alphabet = letters + (b"()" if kind == "stack" else b"")
    al, toks = np.frombuffer(alphabet, np.uint8), set()
    for n in LONG:
        for _ in range(12):
            toks.add(_alive(a, rng, n))
    while len(toks) < 9000:
        toks.add(rng.choice(al, int(rng.integers(1, 6))).tobytes())
    toks = sorted(toks)
    rng.shuffle(toks)
    toks = [bytes(t) for t in toks]
    return a, synth.Vocab.from_tokens(toks[:700] + [b""] + toks[700:], eos_id=700)


def _alive(a, rng, n):
    """n bytes (no brackets) that are alive from some state."""
    s, out = int(rng.integers(1, a.n_states)), b""
    for _ in range(n):
        c = int(rng.choice([c for c in np.nonzero(a.delta[s])[0] if a.rules is None or c not in b"()"]))
        out, s = out + bytes([c]), int(a.delta[s, c])
    return out


def configurations(kind, batch, seed):
    """(states, stacks or None): row 0 in the dead state."""
    a, _ = problem(kind)
    rng = np.random.default_rng(seed)
    states = rng.integers(1, a.n_states, batch).astype(np.int32)
    states[0] = 0
    if kind != "stack":
        return states, None
    stacks = np.array([synth.pack_stack(list(rng.integers(0, 2, int(rng.integers(0, 6))))) for _ in range(batch)], np.uint64)
    stacks[0] = 0
    return states, stacks


@functools.lru_cache(maxsize=None)
def widest_level(kind, q):
    """The most class-string prefixes of one length that are alive from state q (no brackets among them)."""
    a, v = problem(kind)
    cls = np.unique(a.delta, axis=1, return_inverse=True)[1].reshape(-1)
    levels = {}
    for t in range(v.n_tokens):
        s, key = q, b""
        for c in v.data[v.offsets[t]:v.offsets[t + 1]][:4] if t != v.eos_id else b"":
            s = int(a.delta[s, c]) if a.rules is None or c not in b"()" else 0
            if s == 0:
                break
            key += bytes([cls[c]])
            levels.setdefault(len(key), set()).add(key)
    return max(len(x) for x in levels.values())
