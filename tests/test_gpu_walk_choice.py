"""The walk that is chosen for a mask step gives the same masks as either walk
and is not much slower than the better one, on random automata whose rows visit
1000 nodes of the prefix tree and more, with levels of 500 to 2800 live nodes and
of more than row_kernel's pool holds.  A row that does not fit the pool is walked
twice, which took 1.5 to 3.7 times the per-token walk's time here; the bound of
1.25 leaves room for the clock."""
import functools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2403_06988_gb300 import Domino, synth  # noqa: E402
from paper_2403_06988_gb300 import _binding as B  # noqa: E402

V, Q = 128256, 500


@functools.lru_cache(maxsize=1)
def vocab():
    return synth.random_vocab(np.random.default_rng(77), V, bytes(range(256)), synth.geometric_lengths(4.5, 32),
                              synth._mixed_bytes)


def mask_us(a, batch):
    """(time of a mask step, the masks) on a new handle: the shortest of 8 replays of 10 steps."""
    d = Domino.from_parts(a, vocab(), device=0)
    st = torch.from_numpy(np.random.default_rng(3).integers(1, Q, batch).astype(np.int32)).cuda()
    mask = torch.empty((batch, d.info()["n_words"]), dtype=torch.int32, device="cuda")
    run = lambda: B.domino_step_mask(d.h, st, None, batch, mask)
    for _ in range(3):
        run()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(10):
            run()
    us = []
    for _ in range(8):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        g.replay()
        e1.record()
        torch.cuda.synchronize()
        us.append(e0.elapsed_time(e1) * 100)
    out = mask.cpu().numpy().copy()
    d.close()
    return min(us), out


@pytest.mark.parametrize("classes,live,batch", [(66, 16, 32), (100, 20, 32), (256, 40, 32), (32, 14, 256), (48, 16, 256),
                                                (64, 20, 256), (66, 16, 256), (100, 20, 256), (256, 40, 256),
                                                # more visits, more rows before row_kernel pays
                                                (32, 12, 32), (32, 14, 32), (48, 16, 32), (32, 14, 96), (48, 16, 256),
                                                # rows too large for it
                                                (32, 18, 256), (32, 28, 256)])
def test_chosen_walk_is_not_much_slower_than_either(classes, live, batch, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a = synth.random_sparse_dfa(np.random.default_rng(5), Q, classes, live)
    monkeypatch.delenv("DOMINO_WALK", raising=False)
    chosen, m = mask_us(a, batch)
    monkeypatch.setenv("DOMINO_WALK", "token")
    token, want = mask_us(a, batch)
    monkeypatch.setenv("DOMINO_WALK", "tree")
    tree, same = mask_us(a, batch)
    assert (m == want).all() and (same == want).all()
    assert chosen < 1.25 * min(token, tree), (chosen, token, tree)
