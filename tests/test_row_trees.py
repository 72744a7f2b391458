"""The arrays that row_kernel walks (RowTree: the prefix trees, merged states,
loop sets, filters and exits that host.cpp lays out) on the CPU: the walk's
definition, restated here over those arrays, gives the oracle's masks and next
states for every state of random and hand-made automata, with and without a
bracket stack."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2403_06988_gb300 import build, synth

HERE = os.path.dirname(os.path.abspath(__file__))
NAMES = ("node", "ncls", "dtok", "roots", "loopbits", "keeps", "srec", "srec_next", "trec", "xrange", "exits", "start",
         "loop_of", "ret")
TYPES = {"ncls": np.uint8, "dtok": np.int32, "roots": np.int64, "keeps": np.uint8, "srec": np.uint8, "srec_next": np.uint8,
         "trec": np.uint8, "ret": np.uint16}
NO_SET = 0xFFFFFFFF
LOOP_MIN = 4


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("row_image") / "librow_image.so")
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    subprocess.run(["g++", "-O1", "-w", "-std=c++17", "-shared", "-fPIC", "-Wl,-z,lazy", "-I", build.INCLUDE, "-I", build.CSRC,
                    "-I", os.path.join(cuda, "include"), os.path.join(HERE, "row_image.cpp"), "-o", out,
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", "-ldl"], check=True)
    L = ctypes.CDLL(out, mode=os.RTLD_LAZY)
    L.row_image_make.restype = ctypes.c_void_p
    return L


class Image:
    """A host-only handle's RowImage as numpy arrays."""

    def __init__(self, L, a, v):
        ptr = lambda x: None if x is None else x.ctypes.data_as(ctypes.c_void_p)
        h = ctypes.c_void_p()
        assert L.domino_create(ctypes.byref(h), -1) == 0
        assert L.domino_load_vocab(h, ptr(v.data), ptr(v.offsets), v.n_tokens, v.eos_id) == 0
        delta = np.ascontiguousarray(a.delta, np.int32)
        n = 0 if a.rules is None else len(a.rules)
        assert L.domino_load_automaton(h, ptr(delta), a.n_states, ptr(a.live), ptr(a.accepting), a.start,
                                       ptr(a.rules), n, a.max_depth) == 0
        im = ctypes.c_void_p(L.row_image_make(h))
        assert im.value
        self.stack, self.max_depth = n > 0, a.max_depth

        def take(get, dtype):
            p, b = ctypes.c_void_p(), ctypes.c_int64()
            assert get(ctypes.byref(p), ctypes.byref(b)) == 0
            return np.frombuffer(ctypes.string_at(p, b.value), dtype) if b.value else np.zeros(0, dtype)
        for i, name in enumerate(NAMES):
            setattr(self, name, take(lambda p, b: L.row_image_get(im, i, p, b), TYPES.get(name, np.uint32)))
        self.node = self.node.reshape(-1, 8)
        info = (ctypes.c_int64 * 6)()
        L.row_image_info(im, info)
        self.stride, self.stride_next, self.n_loops, self.wide, self.dense, self.visits = info
        self.xrange, self.exits = self.xrange.reshape(self.n_loops or 1, -1, 2), self.exits.reshape(-1, 2)
        self.keeps = self.keeps.reshape(self.n_loops or 1, -1)
        self.loopbits = self.loopbits.reshape(self.n_loops or 1, -1)
        self.start = self.start.reshape(-1, 2)
        t, r = (ctypes.c_void_p(), ctypes.c_int64()), (ctypes.c_void_p(), ctypes.c_int64())
        assert L.row_image_table(h, ctypes.byref(t[0]), ctypes.byref(t[1]), ctypes.byref(r[0]), ctypes.byref(r[1])) == 0
        self.table = np.frombuffer(ctypes.string_at(t[0], t[1].value), np.uint32 if self.stack else np.uint16)
        self.table = self.table.reshape(a.n_states, -1).astype(np.int64)
        self.own_ret = np.frombuffer(ctypes.string_at(r[0], r[1].value), np.uint16) if r[1].value else None
        L.row_image_free(im)
        L.domino_destroy(h)
        self.records = {}

    def record(self, s, nxt):
        """(live classes, classes that keep the state, the state has a loop set, {class: entry})"""
        key = (s, nxt)
        if key not in self.records:
            src, stride = (self.srec_next, self.stride_next) if nxt and len(self.start) else (self.srec, self.stride)
            b = src[s * stride:(s + 1) * stride].tobytes()
            live, keep = int.from_bytes(b[:8], "little"), int.from_bytes(b[8:16], "little")
            entries = np.frombuffer(b[16:], np.uint32 if self.stack else np.uint16)
            on = [k for k in range(64) if live >> k & 1]
            self.records[key] = live, keep & (1 << 63) - 1, keep >> 63, {k: int(entries[i]) for i, k in enumerate(on)}
        return self.records[key]

    def step(self, e, bits, depth, ret):
        """Entry e taken with the stack: (state, bits, depth), state 0 when refused."""
        kind = e >> 16 & 3 if self.stack else 0
        if kind == 0:
            return e & 0xFFFF, bits, depth
        sym = e >> 18 & 1
        if kind == 1:
            return (0, bits, depth) if depth >= self.max_depth else (e & 0xFFFF, bits << 1 | sym, depth + 1)
        if depth == 0 or bits & 1 != sym:
            return 0, bits, depth
        bits, depth = bits >> 1, depth - 1
        return int(ret[(e >> 19) * 4 + (0 if depth == 0 else 1 + (bits & 1))]), bits, depth

    def walk(self, q, bits, depth, nxt):
        """{token: state}: the tokens allowed from state q and this stack (EOS apart)."""
        out, root, s = {}, 0, q
        ret = self.own_ret if nxt or self.wide else self.ret
        if len(self.start) and not nxt:
            s, loop = (int(x) for x in self.start[q])
            if loop != NO_SET:
                w = self.loopbits[loop]
                out.update((t, s) for t in np.nonzero(np.unpackbits(w.view(np.uint8), bitorder="little"))[0].tolist())
                root = int(self.roots[loop])
        items = [(root, s, bits, depth)] if s else []
        while items:
            n, s, bits, depth = items.pop()
            if s == 0:
                continue
            A = [int(x) for x in self.node[n]]
            first, own, lo, hi = A[2] & 0xFFFFFF, A[2] >> 24, A[4], A[5]
            below = A[6] | A[7] << 32
            if self.wide:
                kids, keep, flag, entries = None, 0, 0, None
                n_kids = A[0]
            else:
                _, keep, flag, entries = self.record(s, nxt)
                kids = A[0] | A[1] << 32
                n_kids = bin(kids).count("1")
                if below & ~keep == 0:
                    out.update((int(t), s) for t in self.dtok[lo:hi])
                    continue
            if n_kids == 0:
                own = hi - lo
            elif own == 255:
                own = int(self.node[first][4]) - lo
            out.update((int(t), s) for t in self.dtok[lo:lo + own])
            if flag and self.n_loops and not nxt and hi - lo > LOOP_MIN and kids & keep:
                S = int(self.loop_of[s])
                x0, x1 = (int(x) for x in self.xrange[S][n])
                d = x0 >> 24
                if d != 255:
                    p = np.arange(lo + own, hi)
                    out.update((int(t), s) for t in self.dtok[p[self.keeps[S][p] <= d]])
                    for k in range(x0 & 0xFFFFFF, x1):
                        node, c = int(self.exits[k][0]), int(self.exits[k][1])
                        if c >> 8 <= d and c & 0xFF in entries:
                            items.append((node, *self.step(entries[c & 0xFF], bits, depth, ret)))
                    continue
            for k in range(n_kids):
                c = int(self.ncls[first + k])
                e = int(self.table[s][c]) if self.wide else entries.get(c, 0)
                if e:
                    items.append((first + k, *self.step(e, bits, depth, ret)))
        return out


def check(L, a, v, states, stacks=None, want_next=True):
    import oracle
    im = Image(L, a, v)
    words = None if stacks is None else np.array([synth.pack_stack(k) for k in stacks], np.uint64)
    m_o, n_o, bad = oracle.Problem.from_parts(a, v).step_mask(np.asarray(states, np.int32), words, want_next=True)
    assert bad == 0
    bits_o = np.unpackbits(np.ascontiguousarray(m_o).view(np.uint8).reshape(len(states), -1), axis=1,
                           bitorder="little")[:, :v.n_tokens].astype(bool)
    if v.eos_id >= 0:
        bits_o[:, v.eos_id] = False
    for b, q in enumerate(states):
        word = 0 if words is None else int(words[b])
        got = im.walk(int(q), word & 0xFFFFFFFF, word >> 32, False)
        assert sorted(got) == np.nonzero(bits_o[b])[0].tolist(), ("mask", b, q)
        if want_next:
            got = im.walk(int(q), word & 0xFFFFFFFF, word >> 32, True)
            assert {t: int(n_o[b][t]) for t in np.nonzero(bits_o[b])[0].tolist()} == got, ("next", b, q)
    return im


def random_tokens(rng, n, alphabet, longest):
    toks, al = set(), np.frombuffer(alphabet, np.uint8)
    while len(toks) < n:
        toks.add(rng.choice(al, int(rng.integers(1, longest + 1))).tobytes())
    toks = sorted(toks)
    rng.shuffle(toks)
    toks = [bytes(t) for t in toks]
    return synth.Vocab.from_tokens(toks[:n // 3] + [b""] + toks[n // 3:], eos_id=n // 3)


@pytest.mark.parametrize("classes,live", [(5, 5), (32, 32), (33, 12), (63, 30), (64, 20), (65, 10), (200, 60), (256, 40)])
def test_random_automata(lib, classes, live):
    rng = np.random.default_rng(classes + live)
    a = synth.random_sparse_dfa(rng, 30, classes, live)
    v = random_tokens(rng, 2500, bytes(range(256)) if classes > 5 else b"abcdefgh", 4)
    im = check(lib, a, v, range(30))
    assert im.wide == (len(np.unique(a.delta, axis=1).T) > 64)


def test_kv_grammar_with_loop_sets(lib):
    rng = np.random.default_rng(3)
    a, _ = synth.kv200_dfa(rng)
    v = synth.random_vocab(rng, 4001, bytes(range(256)), synth.geometric_lengths(4.0, 16), synth._mixed_bytes)
    im = check(lib, a, v, range(0, 200, 5), want_next=False)
    assert im.n_loops > 0 and len(im.start)


def test_json_with_a_stack(lib):
    rng = np.random.default_rng(4)
    a, _ = synth.json_pda(rng)
    v = synth.random_vocab(rng, 3001, bytes(range(256)), synth.geometric_lengths(4.0, 24), synth._mixed_bytes)
    cfg = [synth.random_pda_walk(a, rng, int(rng.integers(0, 33))) for _ in range(40)]
    cfg += [(q, []) for q in range(1, 40)]
    im = check(lib, a, v, [c[0] for c in cfg], [c[1] for c in cfg])
    assert im.n_loops > 0 and (im.start[:, 0] != np.arange(len(im.start))).any()   # some states are merged


def test_states_that_differ_in_a_stack_action(lib):
    """Four states with the same targets, of which one pushes 0, one pushes 1, one neither and one pushes 0 as the first."""
    rng = np.random.default_rng(5)
    b = synth._Builder()
    top = [b.state("s%d" % i, accepting=True) for i in range(4)]
    body = b.state("body", accepting=True)
    for i, s in enumerate(top):
        if i == 2:
            b.edge(s, b"(", body)
        else:
            b.push(s, b"(", i % 3 if i < 3 else 0, body)
        b.edge(s, b"abc", top[(i + 1) % 4])
    b.edge(body, b"xyz", body)
    b.edge(body, b"a", top[0])
    b.pop(body, b")", 0, (top[1], body, top[2]))
    b.pop(body, b"]", 1, (top[2], top[0], body))
    a = b.build(top[0], 4, "kinds")
    v = random_tokens(rng, 1500, b"abcxyz()]", 5)
    states = [int(s) for s in range(1, a.n_states)] * 4
    stacks = [[], [0], [1], [0, 1], [1, 1, 0], [0, 0, 0, 0], [1, 0, 1, 1]]
    check(lib, a, v, states, [stacks[i % 7] for i in range(len(states))])


def test_equivalent_states_and_tokens_deeper_than_a_byte(lib):
    """String states copied four times (the copies lead to one another), tokens
    of up to 400 bytes that stay in the string, leave it and come back."""
    rng = np.random.default_rng(8)
    n, letters = 4, b"abcdefgh"
    delta = np.zeros((2 * n + 2, 256), np.int32)
    for k in range(n):
        s, q = 1 + k, 1 + n + k          # inside a string, after it
        for i, c in enumerate(letters):
            delta[s, c] = 1 + (k + i) % n
        delta[s, ord('"')] = 1 + n + k
        delta[q, ord('"')] = 1 + (k + 1) % n
        delta[q, ord(",")] = 2 * n + 1
    delta[2 * n + 1, ord('"')] = 1
    live = np.ones(2 * n + 2, np.uint8)
    live[0] = 0
    a = synth.Automaton(delta=delta, live=live, accepting=live.copy(), start=1, rules=None, max_depth=0, name="copies")
    toks, al = {b'"', b",", b'",', b'","', b"#"}, np.frombuffer(letters, np.uint8)
    for length in (1, 2, 3, 250, 253, 254, 255, 256, 257, 300, 400):
        base = rng.choice(al, length).tobytes()
        toks |= {base, base + b'"', base + b'","' + base[:20], b'"' + base, b'""' + base + b'"x'}
    while len(toks) < 1500:
        parts = [rng.choice(al, int(rng.integers(0, 6))).tobytes() for _ in range(int(rng.integers(1, 5)))]
        t = rng.choice([b'"', b'","', b'""', b","]).join(parts)
        if t:
            toks.add(bytes(t))
    toks = sorted(toks)
    rng.shuffle(toks)
    v = synth.Vocab.from_tokens([bytes(t) for t in toks] + [b""], eos_id=len(toks))
    im = check(lib, a, v, range(2 * n + 2))
    assert len(set(im.start[1:n + 1, 0].tolist())) == 1   # the copies are one state


def test_many_tokens_at_a_node(lib):
    """More than 254 tokens end at one node: their number is read off the first child."""
    rng = np.random.default_rng(9)
    delta = np.zeros((4, 256), np.int32)
    delta[1, 32:128] = 2
    delta[2, 32:80] = 1
    delta[2, 80:128] = 3
    delta[3, 32:128] = 3
    live = np.array([0, 1, 1, 1], np.uint8)
    a = synth.Automaton(delta=delta, live=live, accepting=live.copy(), start=1, rules=None, max_depth=0, name="two")
    check(lib, a, random_tokens(rng, 6000, bytes(range(30, 128)), 3), range(4))


def visited(a, v, q):
    """The class-string prefixes that are alive from state q: the nodes its walk visits, by definition."""
    seen = {b""}
    cols, cls = np.unique(a.delta, axis=1, return_inverse=True)
    for t in range(v.n_tokens):
        s, key = q, b""
        for c in v.data[v.offsets[t]:v.offsets[t + 1]] if t != v.eos_id else b"":
            s = int(a.delta[s, c])
            if not a.live[s]:
                break
            key += bytes([cls.reshape(-1)[c]])
            seen.add(key)
    return len(seen)


@pytest.mark.parametrize("classes,live", [(32, 6), (64, 12), (100, 30), (256, 60)])
def test_nodes_that_a_row_visits(lib, classes, live):
    """The cost by which a walk is chosen counts live nodes, not the children looked at."""
    rng = np.random.default_rng(classes)
    a = synth.random_sparse_dfa(rng, 12, classes, live)
    v = random_tokens(rng, 1200, bytes(range(256)), 3)
    im = Image(lib, a, v)
    want = sorted(visited(a, v, q) for q in range(1, 12))
    assert im.visits == want[len(want) // 2] and not im.dense


@pytest.mark.parametrize("live,dense", [(40, 0), (60, 1)])
def test_levels_that_the_pool_does_not_hold(lib, live, dense):
    """1600 and 3600 nodes alive two classes deep (below the 8192 in all that count as dense): the pool holds 2816."""
    rng = np.random.default_rng(live)
    delta = np.zeros((40, 256), np.int32)
    for q in range(1, 40):
        for c in rng.permutation(64)[:live]:
            delta[q, 4 * c:4 * c + 4] = 1 + (q + int(rng.integers(0, 38))) % 39   # never q
    alive = np.ones(40, np.uint8)
    alive[0] = 0
    a = synth.Automaton(delta=delta, live=alive, accepting=alive.copy(), start=1, rules=None, max_depth=0, name="wide levels")
    pairs = [bytes([4 * i, 4 * j]) for i in range(64) for j in range(64)]
    v = synth.Vocab.from_tokens(pairs + [b""], eos_id=len(pairs))
    im = Image(lib, a, v)
    assert im.dense == dense and (dense or im.visits == 1 + live + live * live)


def test_token_records(lib):
    """{length (255: or more), the first 31 classes} of every token; EOS and empty tokens have length 0."""
    rng = np.random.default_rng(10)
    a = synth.random_sparse_dfa(rng, 20, 16, 8)
    toks = [bytes(rng.integers(0, 256, n, dtype=np.uint8)) for n in (1, 30, 31, 32, 254, 255, 256, 700)] + [b"", b""]
    v = synth.Vocab.from_tokens(toks, eos_id=8)
    im = Image(lib, a, v)
    from paper_2403_06988_gb300 import Domino
    from paper_2403_06988_gb300 import _binding as B
    d = Domino(-1)
    d.load_automaton(a)
    cls = B.domino_get_byte_classes(d.h)
    rec = im.trec.reshape(-1, 32)
    for t, b in enumerate(toks):
        assert rec[t][0] == min(len(b), 255)
        k = min(len(b), 31)
        assert (rec[t][1:1 + k] == cls[np.frombuffer(b, np.uint8)[:k]]).all() and (rec[t][1 + k:] == 0).all()
    d.close()
