"""The walk with one CTA (or a cluster of CTAs) per row (rows.cu) against the
oracle, bit-exact, where it can go wrong: 1 to 8 CTAs per row, class counts
around the 32- and 64-bit masks and beyond, rows with more live nodes than the
pool holds (walked token by token), token ranges longer than the lists, loop sets
(bitmap, the tree of the remainders, subtrees entered in a looping state,
depths beyond a byte), equivalent states, a bracket stack.  Each case runs with
the walk forced (DOMINO_WALK=tree) and as the sizes choose it.  Output buffers
start as 0xAB bytes (tests/poison.py)."""
import functools
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2403_06988_gb300 import Domino, synth  # noqa: E402
import full_pools  # noqa: E402
import poison  # noqa: E402
from poison import assert_exact  # noqa: E402

NT = os.cpu_count() or 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_06988_gb300 import build
    build.build()


@pytest.fixture(params=["tree", None], ids=["forced", "chosen"], autouse=True)
def walk(request, monkeypatch):
    if request.param:
        monkeypatch.setenv("DOMINO_WALK", request.param)   # read when a handle is created
    else:
        monkeypatch.delenv("DOMINO_WALK", raising=False)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(a, v, states, stacks=None, want_next=False):
    import oracle
    d = Domino.from_parts(a, v, device=0)
    B = len(states)
    mask = poison.empty((B, d.info()["n_words"]), torch.int32)
    nxt = poison.empty((B, v.n_tokens), torch.int32) if want_next else None
    d.step_mask(dev(states), None if stacks is None else dev(stacks.view(np.int64)), out_mask=mask, out_next=nxt)
    m_o, n_o, bad = oracle.Problem.from_parts(a, v).step_mask(states, stacks, want_next=want_next, n_threads=NT)
    assert bad == 0
    assert_exact(mask, m_o, "mask")
    if want_next:
        assert_exact(nxt, n_o, "next")
        # the mask alone is another kernel, over merged states
        alone = poison.empty((B, d.info()["n_words"]), torch.int32)
        d.step_mask(dev(states), None if stacks is None else dev(stacks.view(np.int64)), out_mask=alone)
        assert_exact(alone, m_o, "mask alone")
    assert d.device_error() == 0
    d.close()


def random_dfa(rng, n_states, n_classes, live):
    """n_classes classes of bytes; `live` of them live in each state, with random targets."""
    cls = rng.permutation(np.arange(256) % n_classes)
    delta = np.zeros((n_states, 256), np.int32)
    for q in range(1, n_states):
        on = rng.permutation(n_classes)[:live]
        to = np.zeros(n_classes, np.int32)
        to[on] = 1 + (q + rng.permutation(n_states - 2)[np.arange(live) % (n_states - 2)]) % (n_states - 1)   # never q
        delta[q] = to[cls]
    live_q = np.ones(n_states, np.uint8)
    live_q[0] = 0
    return synth.Automaton(delta=delta, live=live_q, accepting=live_q.copy(), start=1, rules=None, max_depth=0, name="r")


def random_tokens(rng, n, alphabet, longest):
    toks = set()
    al = np.frombuffer(alphabet, np.uint8)
    while len(toks) < n - 1:
        toks.add(rng.choice(al, int(rng.integers(1, longest + 1))).tobytes())
    toks = sorted(toks)
    rng.shuffle(toks)
    toks = [bytes(t) for t in toks]
    toks.insert(n // 3, b"")
    return synth.Vocab.from_tokens(toks, eos_id=n // 3)


@pytest.mark.parametrize("classes,live", [(5, 5), (31, 9), (32, 32), (33, 12), (63, 63), (64, 20), (64, 64), (65, 10),
                                          (200, 200), (256, 40)])
@pytest.mark.parametrize("batch", [1, 9, 80])
def test_rows_class_counts_and_full_pools(classes, live, batch):
    rng = np.random.default_rng(classes * 1000 + live)
    a = random_dfa(rng, 40, classes, live)
    v = random_tokens(rng, 9001, bytes(range(256)) if classes > 5 else b"abcde", 4 if classes > 5 else 7)
    states = rng.integers(0, 40, batch).astype(np.int32)
    check(a, v, states, want_next=True)


@functools.lru_cache(maxsize=None)
def json_vocab():
    rng = np.random.default_rng(5)
    return synth.random_vocab(rng, 20011, bytes(range(256)), synth.geometric_lengths(4.0, 32), synth._mixed_bytes)


@pytest.mark.parametrize("batch", [106, 300])
def test_rows_loop_sets_with_a_stack(batch):
    rng = np.random.default_rng(6)
    a, _ = synth.json_pda(rng)
    pool = [synth.random_pda_walk(a, rng, int(rng.integers(0, 33))) for _ in range(40)]
    pool += [(q, []) for q in range(1, a.n_states)][:60]
    pick = rng.integers(0, len(pool), batch)
    states = np.array([pool[i][0] for i in pick], np.int32)
    stacks = np.array([synth.pack_stack(pool[i][1]) for i in pick], np.uint64)
    check(a, json_vocab(), states, stacks)


def test_rows_loop_sets_with_long_tokens_and_equivalent_states():
    """String states copied four times (the copies lead to one another), tokens
    of up to 400 bytes that stay in the string, leave it and come back."""
    rng = np.random.default_rng(8)
    n = 4
    delta = np.zeros((2 * n + 2, 256), np.int32)
    letters = b"abcdefgh"
    for k in range(n):
        s, q = 1 + k, 1 + n + k          # inside a string, after it
        for i, c in enumerate(letters):
            delta[s, c] = 1 + (k + i) % n
            delta[q, c] = 0
        delta[s, ord('"')] = 1 + n + k
        delta[q, ord('"')] = 1 + (k + 1) % n
        delta[q, ord(",")] = 2 * n + 1
    delta[2 * n + 1, ord('"')] = 1
    live = np.ones(2 * n + 2, np.uint8)
    live[0] = 0
    a = synth.Automaton(delta=delta, live=live, accepting=live.copy(), start=1, rules=None, max_depth=0, name="copies")
    toks = {b'"', b",", b'",', b'","', b"#"}
    al = np.frombuffer(letters, np.uint8)
    for L in (1, 2, 3, 250, 253, 254, 255, 256, 257, 300, 400):
        base = rng.choice(al, L).tobytes()
        toks |= {base, base + b'"', base + b'","' + base[:20], b'"' + base, b'""' + base + b'"x'}
    while len(toks) < 4200 - 1:
        parts = [rng.choice(al, int(rng.integers(0, 6))).tobytes() for _ in range(int(rng.integers(1, 5)))]
        t = rng.choice([b'"', b'","', b'""', b","]).join(parts)
        if t:
            toks.add(bytes(t))
    toks = sorted(toks)
    rng.shuffle(toks)
    v = synth.Vocab.from_tokens([bytes(t) for t in toks] + [b""], eos_id=len(toks))
    states = (np.arange(520) % (2 * n + 2)).astype(np.int32)
    check(a, v, states)


def test_rows_many_tokens_per_node():
    """Two live classes: every node holds hundreds of tokens, whole subtrees are long ranges."""
    rng = np.random.default_rng(9)
    delta = np.zeros((4, 256), np.int32)
    delta[1, 32:128] = 2
    delta[2, 32:80] = 1
    delta[2, 80:128] = 3
    delta[3, 32:128] = 3
    live = np.array([0, 1, 1, 1], np.uint8)
    a = synth.Automaton(delta=delta, live=live, accepting=live.copy(), start=1, rules=None, max_depth=0, name="two")
    v = random_tokens(rng, 40003, bytes(range(30, 128)), 6)
    check(a, v, np.tile(np.arange(4, dtype=np.int32), 14)[:53])


@pytest.mark.parametrize("kind", ["plain", "stack", "wide"])
@pytest.mark.parametrize("batch", [3, 90, 400])
def test_rows_full_pools_with_long_tokens(kind, batch):
    """Rows with more live nodes than the pool holds (tests/full_pools.py)."""
    a, v = full_pools.problem(kind)
    assert min(full_pools.widest_level(kind, q) for q in (1, 2)) > full_pools.POOL
    states, stacks = full_pools.configurations(kind, batch, 11)
    check(a, v, states, stacks, want_next=True)


def test_first_step_in_a_capture():
    """A step whose walk needs scratch is recorded without a call before it."""
    from paper_2403_06988_gb300 import _binding as B
    rng = np.random.default_rng(12)
    a = synth.random_sparse_dfa(rng, 300)
    v = synth.random_vocab(rng, 8000, bytes(range(256)), synth.geometric_lengths(4.0, 16), synth._mixed_bytes)
    states = torch.from_numpy(rng.integers(1, 300, 6).astype(np.int32)).cuda()
    lg = torch.randn((6, 8000), device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(torch.bfloat16)
    got = []
    for capture in (True, False):
        d = Domino.from_parts(a, v, device=0)
        mask = poison.empty((6, d.info()["n_words"]), torch.int32)
        arg, out = poison.empty(6, torch.int32), poison.empty(6, torch.int32)
        torch.cuda.synchronize()
        run = lambda: B.domino_step_decode(d.h, states, None, 6, lg.data_ptr(), B.DTYPE_BF16, 8000, mask, arg, None, None,
                                           out, None, torch.cuda.current_stream().cuda_stream)
        if capture:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                run()
            g.replay()
        else:
            run()
        torch.cuda.synchronize()
        got.append([t.cpu().numpy().copy() for t in (mask, arg, out)])
        assert d.device_error() == 0
        d.close()
    for x, y in zip(*got):
        assert_exact(x, y, "recorded")


@pytest.mark.parametrize("batch", [309, 701])
def test_rows_of_half_the_threads(batch):
    """More rows than run at once: CTAs of 256 threads, with and without loop sets, and with more than 64 classes."""
    rng = np.random.default_rng(13)
    v = synth.random_vocab(rng, 15987, bytes(range(256)), synth.geometric_lengths(4.0, 32), synth._mixed_bytes)
    a = synth.random_sparse_dfa(rng, 400)
    check(a, v, rng.integers(0, 400, batch).astype(np.int32), want_next=True)
    a, _ = synth.kv200_dfa(rng)
    check(a, v, rng.integers(0, 200, batch).astype(np.int32))
    a = random_dfa(rng, 400, 100, 12)
    check(a, v, rng.integers(0, 400, batch).astype(np.int32), want_next=True)


def test_recorded_step_outlives_larger_batches():
    """A graph recorded at a small batch is replayed after larger batches have grown the scratch."""
    from paper_2403_06988_gb300 import _binding as B
    rng = np.random.default_rng(14)
    a = synth.random_sparse_dfa(rng, 300)
    V = 8000
    v = synth.random_vocab(rng, V, bytes(range(256)), synth.geometric_lengths(4.0, 16), synth._mixed_bytes)
    d = Domino.from_parts(a, v, device=0)
    states = torch.from_numpy(rng.integers(1, 300, 300).astype(np.int32)).cuda()
    lg = torch.randn((300, V), device="cuda", generator=torch.Generator("cuda").manual_seed(2)).to(torch.bfloat16)
    mask = poison.empty((300, d.info()["n_words"]), torch.int32)
    arg, out = poison.empty(300, torch.int32), poison.empty(300, torch.int32)

    def run(n):
        B.domino_step_decode(d.h, states, None, n, lg.data_ptr(), B.DTYPE_BF16, V, mask, arg, None, None, out, None,
                             torch.cuda.current_stream().cuda_stream)
    run(4)
    want = arg[:4].cpu().numpy().copy()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        run(4)
    for n in (20, 90, 300):
        run(n)
    full = arg.cpu().numpy().copy()
    arg.fill_(-7)
    g.replay()
    torch.cuda.synchronize()
    assert_exact(arg[:4], want, "recorded")
    assert_exact(full[:4], want, "largest batch")
    assert d.device_error() == 0
    d.close()
