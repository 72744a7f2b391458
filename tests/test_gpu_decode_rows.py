"""The decode of one row by a CTA or a cluster of CTAs (decode.cuh) against
the oracle: bf16 and fp32 rows at every alignment, vocabularies around the
vector, word and segment sizes, 1 to 8 CTAs per row, sparse and dense masks,
masks with bits past V, rows with nothing allowed, ties, infinite logits, the
largest and lowest finite ones; masks that allow only the tokens around the
edges of rows, slices and segments; the Gumbel-max draw over the same rows; and
the mask step with the decode and the update folded in, over unaligned rows and
over rows that row_kernel walks token by token.  Tokens bit-exact.

Tolerance of lse and log-probabilities: a lane adds the sums of at most 36
vectors (140000 tokens over 512 lanes) of 8 terms (5 additions deep), and lanes,
warps and CTAs are merged in 12 steps: 53 roundings, 53 * 2^-24 = 3.2e-6
relative.  A term e^-d errs by 2^-22 (ex2) and d * 2^-23 (its exponent's two
roundings), 3e-7 of the sum at most.  So ln(sum) errs by less than 3.5e-6, and
the roundings of logf, m + ln(sum) and x - lse (below 32) by 2^-20 each: 6.4e-6,
1e-5 allowed.  Output buffers start as 0xAB bytes (tests/poison.py)."""
import functools
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2403_06988_gb300 import Domino, synth  # noqa: E402
from paper_2403_06988_gb300 import _binding as B  # noqa: E402
import full_pools  # noqa: E402
import poison  # noqa: E402
from poison import assert_exact, assert_no_poison  # noqa: E402

NT = os.cpu_count() or 1
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_06988_gb300 import build
    build.build()


@functools.lru_cache(maxsize=2)
def handle(V):
    toks = [b"%d" % i for i in range(V - 1)] + [b""]
    d = Domino(0)
    d.load_vocab(synth.Vocab.from_tokens(toks, eos_id=V - 1))
    return d


def rows(dt, batch, V, offset, pad, seed, sigma=3.0):
    """(the oracle's contiguous [batch][V] logits, device buffer, address of row 0, row stride): rows of V + pad
    elements, the first one `offset` elements past an allocation."""
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((batch, V + pad)) * sigma).astype(np.float32)
    x = x if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(x)
    buf = np.zeros(offset + batch * (V + pad), x.dtype)
    buf[offset:] = x.reshape(-1)
    t = torch.from_numpy(buf.view(np.int16) if dt == B.DTYPE_BF16 else buf).cuda()
    return np.ascontiguousarray(x[:, :V]), t, t.data_ptr() + offset * x.dtype.itemsize, V + pad


def masks(batch, V, share, seed):
    rng = np.random.default_rng([seed, 1])
    W = (V + 31) // 32
    bits = rng.random((batch, W * 32)) < share * (0.2 + 1.6 * rng.random((batch, 1)))
    if batch > 2:
        bits[1] = False
    return np.packbits(bits.reshape(batch, W, 32), axis=2, bitorder="little").view(np.uint32).reshape(batch, W)


def check(x, m, V, arg, lse, lp):
    import oracle
    clean = m.copy()
    if V % 32:
        clean[:, -1] &= (1 << (V % 32)) - 1
    a_o, l_o, p_o = oracle.mask_logits(x, clean, n_tokens=V, want_logprobs=lp is not None, n_threads=NT)
    assert_exact(arg, np.asarray(a_o, np.int32), "argmax")
    for name, got, want in (("lse", lse, l_o), ("log-probs", lp, p_o)):
        if got is None:
            continue
        assert_no_poison(got, name)
        g = got.cpu().numpy()
        fin = np.isfinite(want)
        assert (np.isfinite(g) == fin).all(), name
        assert np.abs(g[fin].astype(np.float64) - want[fin]).max(initial=0) < TOL, name


@pytest.mark.parametrize("dt", [B.DTYPE_BF16, B.DTYPE_F32])
@pytest.mark.parametrize("V,batch,offset,pad", [(1, 1, 0, 0), (7, 3, 1, 0), (33, 5, 3, 0), (1000, 1, 0, 0),
                                                (4099, 2, 5, 0), (8191, 24, 7, 0), (50001, 3, 2, 6), (32000, 64, 0, 0),
                                                (32001, 80, 0, 0), (131105, 9, 0, 7), (140000, 160, 1, 0),
                                                (300007, 2, 4, 1)])
@pytest.mark.parametrize("share", [0.003, 0.6])
def test_rows_of_any_alignment(dt, V, batch, offset, pad, share):
    import oracle
    x, t, ptr, stride = rows(dt, batch, V, offset, pad, V + batch)
    m = masks(batch, V, share, V)
    d = handle(V)
    mt = torch.from_numpy(m.view(np.int32)).cuda()
    for want_lp in (False, True):
        arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
        lp = poison.empty((batch, V), torch.float32) if want_lp else None
        B.domino_mask_logits(d.h, ptr, dt, batch, stride, mt, arg, lse, lp)
        check(x, m, V, arg, lse, lp)
    arg = poison.empty(batch, torch.int32)
    B.domino_mask_logits(d.h, ptr, dt, batch, stride, mt, arg)
    check(x, m, V, arg, None, None)
    tok = poison.empty(batch, torch.int32)
    B.domino_mask_sample(d.h, ptr, dt, batch, stride, mt, 0.7, 11, 5, tok)
    clean = m.copy()
    if V % 32:
        clean[:, -1] &= (1 << (V % 32)) - 1
    assert_exact(tok, np.asarray(oracle.mask_sample(x, clean, 0.7, 11, 5), np.int32), "drawn token")
    del t


def edge_tokens(V):
    """The tokens within 9 of the ends of the row, of the slices of 1 to 8 CTAs and of segments of 4096 mask words."""
    W = (V + 31) // 32
    edges = {0, V}
    for s in (1, 2, 4, 8):
        words = ((W + s - 1) // s + 3) // 4 * 4
        edges |= {32 * words * i for i in range(1, s)} | {131072 * i for i in range(1, V // 131072 + 1)}
    return np.array(sorted({t for e in edges for t in range(e - 9, e + 9) if 0 <= t < V}))


def edge_rows(dt, batch, V, seed):
    """(logits, allowed tokens per row): tokens that are not allowed are the largest; a row allows every edge token,
    with equal logits (lse = x + ln(n) then shows a token that is missing or taken twice), or one of them."""
    rng = np.random.default_rng(seed)
    edges = edge_tokens(V)
    x = np.full((batch, V), 50.0, np.float32)
    allowed = [edges if b % 3 == 0 else edges[[int(rng.integers(0, len(edges)))]] for b in range(batch)]
    for b in range(batch):
        x[b, allowed[b]] = 1.5
    return (x if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(x)), allowed


def check_edges(allowed, arg, lse, lp, V):
    a, l = arg.cpu().numpy(), lse.cpu().numpy()
    for b, t in enumerate(allowed):
        assert a[b] == t[0], (b, a[b], t[0])
        assert abs(float(l[b]) - (1.5 + np.log(len(t)))) < TOL, (b, len(t), l[b])
    if lp is not None:
        p = lp.cpu().numpy()
        for b, t in enumerate(allowed):
            assert (np.nonzero(np.isfinite(p[b]))[0] == t).all() and (p[b][~np.isfinite(p[b])] == -np.inf).all()
            assert np.abs(p[b][t] + np.log(len(t))).max() < TOL


def placed(x, dt, offset, pad):
    """(the device buffer, address of row 0, row stride) of rows of V + pad elements, `offset` elements in."""
    batch, V = x.shape
    buf = np.zeros(offset + batch * (V + pad), x.dtype)
    buf[offset:].reshape(batch, V + pad)[:, :V] = x
    t = torch.from_numpy(buf.view(np.int16) if dt == B.DTYPE_BF16 else buf).cuda()
    return t, t.data_ptr() + offset * x.dtype.itemsize, V + pad


def bits_of(allowed, V):
    m = np.zeros((len(allowed), (V + 31) // 32 * 32), np.uint8)
    for b, t in enumerate(allowed):
        m[b, t] = 1
    return np.packbits(m, axis=1, bitorder="little").view(np.uint32)


SHIFTS = [(B.DTYPE_BF16, k) for k in range(8)] + [(B.DTYPE_F32, k) for k in range(4)]


@pytest.mark.parametrize("dt,shift,V,batch",
                         [(dt, k, V, b) for dt, k in SHIFTS for V, b in ((1000, 9), (20001, 9), (20000, 40), (33000, 100),
                                                                         (140000, 3))] +
                         # more rows than SMs: one CTA a row, two segments (bf16 on 16-byte boundaries: the gather)
                         [(B.DTYPE_BF16, 0, 140000, 160), (B.DTYPE_BF16, 3, 140000, 160), (B.DTYPE_F32, 1, 140000, 160)])
def test_tokens_at_the_edges(dt, shift, V, batch):
    """Every shift of the vectors against the mask: rows of V elements (odd V: every row at another shift) or padded to
    whole 16 bytes (all rows at one)."""
    x, allowed = edge_rows(dt, batch, V, V + batch + shift)
    m = torch.from_numpy(bits_of(allowed, V).view(np.int32)).cuda()
    for pad in {0, -V % 8}:
        t, ptr, stride = placed(x, dt, shift, pad)
        arg, lse, lp = (poison.empty(n, d) for n, d in ((batch, torch.int32), (batch, torch.float32),
                                                        ((batch, V), torch.float32)))
        B.domino_mask_logits(handle(V).h, ptr, dt, batch, stride, m, arg, lse, lp)
        check_edges(allowed, arg, lse, lp, V)
        arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
        B.domino_mask_logits(handle(V).h, ptr, dt, batch, stride, m, arg, lse)
        check_edges(allowed, arg, lse, None, V)
        del t


@functools.lru_cache(maxsize=2)
def edge_grammar(V):
    """An automaton and a vocabulary whose allowed tokens are the edge tokens (state 1) or one of them (the others)."""
    edges = edge_tokens(V)
    n = len(edges)
    digits = lambda i: bytes([97 + i // 26 % 26, 97 + i % 26, 97 + i // 676])
    toks = [b"#%d" % t for t in range(V)]
    for i, t in enumerate(edges):
        toks[t] = digits(i)
    delta = np.zeros((4 + n, 256), np.int32)
    delta[1, 97:123], delta[2, 97:123], delta[3, 97:123] = 2, 3, 1    # any three letters
    live = np.ones(4 + n, np.uint8)
    live[0] = 0
    singles = []
    for i in range(0, n, 7):                                          # one token's letters only, then nothing
        q = len(singles) * 3 + 4
        if q + 3 > 4 + n:
            break
        a, b, c = digits(i)
        delta[q, a], delta[q + 1, b], delta[q + 2, c] = q + 1, q + 2, 1
        singles.append((q, i))
    a = synth.Automaton(delta=delta, live=live, accepting=np.zeros_like(live), start=1, rules=None, max_depth=0, name="edges")
    return a, synth.Vocab.from_tokens(toks, eos_id=-1), edges, singles


@pytest.mark.parametrize("dt,shift", SHIFTS)
@pytest.mark.parametrize("V,batch", [(20001, 9), (20001, 40), (20001, 100), (20001, 200), (140001, 5)])
def test_folded_tokens_at_the_edges(dt, shift, V, batch, monkeypatch):
    """The same with the decode folded into row_kernel."""
    monkeypatch.setenv("DOMINO_WALK", "tree")
    a, v, edges, singles = edge_grammar(V)
    rng = np.random.default_rng(batch + shift)
    pick = [None if b % 3 == 0 else singles[int(rng.integers(0, len(singles)))] for b in range(batch)]
    states = np.array([1 if p is None else p[0] for p in pick], np.int32)
    allowed = [edges if p is None else edges[[p[1]]] for p in pick]
    x = np.full((batch, V), 50.0, np.float32)
    for b in range(batch):
        x[b, allowed[b]] = 1.5
    t, ptr, stride = placed(x if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(x), dt, shift, 0)
    d = Domino.from_parts(a, v, device=0)
    mask = poison.empty((batch, (V + 31) // 32), torch.int32)
    arg, lse, lp = (poison.empty(n, k) for n, k in ((batch, torch.int32), (batch, torch.float32),
                                                    ((batch, V), torch.float32)))
    B.domino_step_decode(d.h, torch.from_numpy(states).cuda(), None, batch, ptr, dt, stride, mask, arg, lse, lp)
    assert_exact(mask, bits_of(allowed, V), "mask")
    check_edges(allowed, arg, lse, lp, V)
    assert d.device_error() == 0
    d.close()
    del t


@pytest.mark.parametrize("temperature", [1e-3, 0.05, 40.0])
def test_draws_at_extreme_temperatures(temperature):
    """Scores of up to about 1e4: the rounding of the bound on a variate must not drop the winner."""
    import oracle
    V, batch = 5003, 6
    x, t, ptr, stride = rows(B.DTYPE_F32, batch, V, 0, 0, 3, sigma=10.0)
    m = masks(batch, V, 0.7, 3)
    m[:, -1] &= (1 << (V % 32)) - 1
    tok = poison.empty(batch, torch.int32)
    B.domino_mask_sample(handle(V).h, ptr, B.DTYPE_F32, batch, stride, torch.from_numpy(m.view(np.int32)).cuda(),
                         temperature, 2, 9, tok)
    assert_exact(tok, np.asarray(oracle.mask_sample(x, m, temperature, 2, 9), np.int32), "drawn token")
    del t


@pytest.mark.parametrize("dt", [B.DTYPE_BF16, B.DTYPE_F32])
def test_infinite_logits(dt):
    """-inf logits never win and add nothing; a row of only -inf allowed logits decodes as nothing allowed; +inf wins."""
    V, batch = 2001, 4
    x, _, _, _ = rows(dt, batch, V, 0, 0, 21)
    f = x if dt == B.DTYPE_F32 else synth.bf16_bits_to_f32(x)
    f = f.copy()
    m = masks(batch, V, 0.5, 4)
    m[1] = m[0]
    m[:, -1] &= (1 << (V % 32)) - 1
    bits = np.unpackbits(m.view(np.uint8), bitorder="little").reshape(batch, -1)[:, :V].astype(bool)
    f[0, ::3] = -np.inf
    f[1] = -np.inf
    f[2, 900] = np.inf
    bits[2, 900] = True
    m[2, 900 // 32] |= np.uint32(1 << (900 % 32))
    raw = f if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(f)
    t = torch.from_numpy(raw.view(np.int16) if dt == B.DTYPE_BF16 else raw).cuda()
    arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
    B.domino_mask_logits(handle(V).h, t.data_ptr(), dt, batch, V, torch.from_numpy(m.view(np.int32)).cuda(), arg, lse)
    for b in range(batch):
        v = np.where(bits[b], f[b].astype(np.float64), -np.inf)
        if b == 1:
            assert arg[b] == -1 and lse[b] == -np.inf
        elif b == 2:
            assert arg[b] == 900 and lse[b] == np.inf
        else:
            assert arg[b] == int(np.argmax(v))
            assert abs(float(lse[b]) - np.logaddexp.reduce(v[np.isfinite(v)])) < TOL


def extreme_logits(dt, batch, V, seed):
    """float32 rows whose logits reach the type's ends: banned tokens at the lowest value and the like."""
    rng = np.random.default_rng(seed)
    top = float(torch.finfo(torch.bfloat16 if dt == B.DTYPE_BF16 else torch.float32).max)
    x = (rng.standard_normal((batch, V)) * 3).astype(np.float32)
    few = rng.random((batch, V)) < 0.02
    for b in range(batch):
        kind = b % 12
        if kind == 0:
            x[b] = -top                                                  # nothing but the lowest value
        elif kind == 1:
            x[b] = np.where(few[b], x[b], np.float32(-top))              # a few tokens left
        elif kind == 2:
            x[b] = np.where(few[b], np.float32(-top), x[b])              # a few tokens banned
        elif kind == 3:
            x[b] = top
        elif kind == 4:
            x[b] = np.where(few[b], np.float32(top), np.where(rng.random(V) < 0.5, np.float32(-top), x[b]))
        elif kind == 5:
            x[b] = rng.choice(np.array([-2.4e38, -2.3e38, -3e38], np.float32), V)
        elif kind == 6:
            x[b] = (rng.random(V) * 2 - 1).astype(np.float32) * np.float32(3.3e38)
        elif kind == 7:                                                  # every magnitude, either sign
            x[b] = np.where(rng.random(V) < 0.5, 1, -1) * np.exp(rng.random(V) * 88).astype(np.float32)
        elif kind == 8:
            x[b] = np.where(few[b], x[b], -np.exp(rng.random() * 88).astype(np.float32))
        elif kind == 9:                                                  # around the ends of the sum's reference
            x[b] = np.where(few[b], x[b], -np.exp2(28 + 5 * rng.random(V)).astype(np.float32))
        elif kind == 10:
            x[b] = (1 if b % 24 < 12 else -1) * np.exp2(28 + 5 * rng.random(V)).astype(np.float32)
        else:
            x[b] = np.where(few[b], -np.float32(2.36e38), np.float32(-top))
    return x


def check_extreme(x, m, V, arg, lse):
    """As check(); lse to TOL beside an fp32 rounding of the result."""
    import oracle
    a_o, l_o, _ = oracle.mask_logits(x, m, n_tokens=V, n_threads=NT)
    assert_exact(arg, np.asarray(a_o, np.int32), "argmax")
    g = lse.cpu().numpy().astype(np.float64)
    fin = np.isfinite(l_o)
    assert (np.isfinite(g) == fin).all() and not np.isnan(g).any()
    assert (np.abs(g[fin] - l_o[fin]) <= TOL + 2.0 ** -23 * np.abs(l_o[fin])).all()


@pytest.mark.parametrize("dt,batch", [(B.DTYPE_BF16, 24), (B.DTYPE_BF16, 200), (B.DTYPE_F32, 24), (B.DTYPE_F32, 200)])
@pytest.mark.parametrize("share", [0.01, 0.6])
def test_logits_at_the_ends_of_their_type(dt, batch, share):
    """Given masks: the cluster kernel, and the gather (bf16, more rows than SMs)."""
    V = 8000
    f = extreme_logits(dt, batch, V, batch)
    x = f if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(f)
    t = torch.from_numpy(x.view(np.int16) if dt == B.DTYPE_BF16 else x).cuda()
    m = masks(batch, V, share, 5)
    arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
    B.domino_mask_logits(handle(V).h, t.data_ptr(), dt, batch, V, torch.from_numpy(m.view(np.int32)).cuda(), arg, lse)
    check_extreme(x, m, V, arg, lse)


@pytest.mark.parametrize("dt", [B.DTYPE_BF16, B.DTYPE_F32])
@pytest.mark.parametrize("walk", ["tree", "token"])
@pytest.mark.parametrize("grammar", ["kv200", "sparse"])
def test_folded_logits_at_the_ends_of_their_type(dt, walk, grammar, monkeypatch):
    """The decode folded into either walk, over windows of few, some (the single bytes' window of the sparse grammar)
    and many allowed tokens."""
    import oracle
    monkeypatch.setenv("DOMINO_WALK", walk)
    rng = np.random.default_rng(31)
    V, batch = 12000, 96
    v = synth.random_vocab(rng, V, bytes(range(256)), synth.geometric_lengths(4.0, 32), synth._mixed_bytes)
    a = synth.kv200_dfa(rng)[0] if grammar == "kv200" else synth.random_sparse_dfa(rng, 300)
    states = rng.integers(1, a.n_states, batch)
    wide = 1 + np.nonzero((a.delta[1:] == np.arange(1, a.n_states)[:, None]).sum(1) > 64)[0]   # inside strings
    if grammar == "kv200":
        states = np.where(rng.random(batch) < 0.5, rng.choice(wide, batch), states)
    states = states.astype(np.int32)
    d = Domino.from_parts(a, v, device=0)
    m_o, _, _ = oracle.Problem.from_parts(a, v).step_mask(states, None, n_threads=NT)
    f = extreme_logits(dt, batch, V, 7)
    x = f if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(f)
    t = torch.from_numpy(x.view(np.int16) if dt == B.DTYPE_BF16 else x).cuda()
    mask = poison.empty((batch, d.info()["n_words"]), torch.int32)
    arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
    B.domino_step_decode(d.h, torch.from_numpy(states).cuda(), None, batch, t.data_ptr(), dt, V, mask, arg, lse)
    assert_exact(mask, m_o, "mask")
    check_extreme(x, m_o, V, arg, lse)
    d.close()


@pytest.mark.parametrize("dt,offset,pad", [(B.DTYPE_BF16, 0, 5), (B.DTYPE_BF16, 3, 0), (B.DTYPE_F32, 0, 0),
                                           (B.DTYPE_F32, 1, 2)])
@pytest.mark.parametrize("grammar,batch", [("json", 60), ("json", 170), ("sparse", 5), ("sparse", 200),
                                           ("sparse", 310), ("wide", 20), ("wide", 320)])
@pytest.mark.parametrize("walk", ["tree", None])
def test_whole_step_in_one_kernel(dt, offset, pad, grammar, batch, walk, monkeypatch):
    import oracle
    if walk:
        monkeypatch.setenv("DOMINO_WALK", walk)
    rng = np.random.default_rng(batch)
    V = 19997
    v = synth.random_vocab(rng, V, bytes(range(256)), synth.geometric_lengths(4.0, 32), synth._mixed_bytes)
    if grammar == "json":
        a, _ = synth.json_pda(rng)
        cfg = [synth.random_pda_walk(a, rng, int(rng.integers(0, 33))) for _ in range(30)]
        pick = rng.integers(0, len(cfg), batch)
        states = np.array([cfg[i][0] for i in pick], np.int32)
        stacks = np.array([synth.pack_stack(cfg[i][1]) for i in pick], np.uint64)
    else:
        a = synth.random_sparse_dfa(rng, 300, *((100, 12) if grammar == "wide" else ()))
        states, stacks = rng.integers(0, 300, batch).astype(np.int32), None
    d = Domino.from_parts(a, v, device=0)
    P = oracle.Problem.from_parts(a, v)
    x, t, ptr, stride = rows(dt, batch, V, offset, pad, 5)
    st = torch.from_numpy(states).cuda()
    sk = None if stacks is None else torch.from_numpy(stacks.view(np.int64)).cuda()
    mask = poison.empty((batch, d.info()["n_words"]), torch.int32)
    arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
    lp = poison.empty((batch, V), torch.float32)
    B.domino_step_decode(d.h, st, sk, batch, ptr, dt, stride, mask, arg, lse, lp, st, sk)
    m_o, _, bad = P.step_mask(states, stacks, n_threads=NT)
    assert bad == 0
    assert_exact(mask, m_o, "mask")
    check(x, m_o, V, arg, lse, lp)
    a_o, _, _ = oracle.mask_logits(x, m_o, n_tokens=V, n_threads=NT)
    s_o, k_o, _ = P.advance(states, stacks, a_o, a.start)
    assert_exact(st, s_o, "states")
    if sk is not None:
        assert_exact(sk, k_o, "stacks")
    assert d.device_error() == 0
    d.close()
    del t


@pytest.mark.parametrize("dt,offset,pad", [(B.DTYPE_BF16, 0, 0), (B.DTYPE_BF16, 3, 1), (B.DTYPE_F32, 0, 0),
                                           (B.DTYPE_F32, 1, 2)])
@pytest.mark.parametrize("kind", ["plain", "stack", "wide"])
@pytest.mark.parametrize("batch", [3, 60, 200, 400])
def test_whole_step_of_rows_that_fill_the_pool(dt, offset, pad, kind, batch, monkeypatch):
    """1 to 8 CTAs per row; the winner of most rows is a token of 14 to 60 classes, which the update walks."""
    import oracle
    monkeypatch.setenv("DOMINO_WALK", "tree")
    a, v = full_pools.problem(kind)
    V = v.n_tokens
    assert min(full_pools.widest_level(kind, q) for q in (1, 2)) > full_pools.POOL
    rng = np.random.default_rng(batch)
    states, stacks = full_pools.configurations(kind, batch, batch)
    P = oracle.Problem.from_parts(a, v)
    m_o, _, bad = P.step_mask(states, stacks, n_threads=NT)
    assert bad == 0
    f = (rng.standard_normal((batch, V)) * 2).astype(np.float32)
    lens = np.diff(v.offsets)
    bits = np.unpackbits(np.ascontiguousarray(m_o).view(np.uint8).reshape(batch, -1), axis=1, bitorder="little")[:, :V]
    for b in range(1, batch):
        far = np.nonzero(bits[b] & (lens >= 14))[0]
        if len(far) and b % 5:
            f[b, far[int(rng.integers(0, len(far)))]] = 20.0
    x = f if dt == B.DTYPE_F32 else synth.f32_to_bf16_bits(f)
    t, ptr, stride = placed(x, dt, offset, pad)
    d = Domino.from_parts(a, v, device=0)
    st = torch.from_numpy(states).cuda()
    sk = None if stacks is None else torch.from_numpy(stacks.view(np.int64)).cuda()
    mask = poison.empty((batch, d.info()["n_words"]), torch.int32)
    arg, lse = poison.empty(batch, torch.int32), poison.empty(batch, torch.float32)
    lp = poison.empty((batch, V), torch.float32)
    B.domino_step_decode(d.h, st, sk, batch, ptr, dt, stride, mask, arg, lse, lp, st, sk)
    assert_exact(mask, m_o, "mask")
    check(x, m_o, V, arg, lse, lp)
    a_o, _, _ = oracle.mask_logits(x, m_o, n_tokens=V, n_threads=NT)
    assert (lens[np.asarray(a_o)[1:]] >= 14).mean() > 0.4
    s_o, k_o, _ = P.advance(states, stacks, a_o, a.start)
    assert_exact(st, s_o, "states")
    if sk is not None:
        assert_exact(sk, k_o, "stacks")
    assert d.device_error() == 0
    d.close()
    del t
