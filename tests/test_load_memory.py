"""A load that runs out of host memory returns DOMINO_E_OOM: no exception
passes through the C ABI (which would end the process).  A child process limits
its own address space after the inputs are made."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import resource, sys
import numpy as np
sys.path.insert(0, %r)
from paper_2403_06988_gb300 import Domino, synth
from paper_2403_06988_gb300 import _binding as B

def limit(more):
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    resource.setrlimit(resource.RLIMIT_AS, (used + more, resource.getrlimit(resource.RLIMIT_AS)[1]))

V = 1 << 20
data = np.random.default_rng(1).integers(0, 256, 6 * V, dtype=np.uint8)
offsets = np.arange(V + 1, dtype=np.int64) * 6
a = synth.random_sparse_dfa(np.random.default_rng(2), 20, 200, 30)
a.delta = np.ascontiguousarray(a.delta, np.int32)
d = Domino(-1)
small = synth.Vocab.from_tokens([b"a", b"b", b""], eos_id=2)
part = %r
if part == "vocab":
    d.load_automaton(a)
    limit(4 << 20)
    call = lambda: B.domino_load_vocab(d.h, data, offsets, V, -1)
else:
    B.domino_load_vocab(d.h, data, offsets, V, -1)
    limit(24 << 20)
    call = lambda: d.load_automaton(a)
try:
    call()
    raise SystemExit("no error")
except B.DominoError as e:
    assert "out of memory" in str(e), e
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.getrlimit(resource.RLIMIT_AS)[1]))
d.load_vocab(small)       # the handle goes on
d.load_automaton(a)
assert d.info()["n_tokens"] == 3
d.close()
print("ok")
"""


@pytest.mark.parametrize("part", ["vocab", "automaton"])
def test_load_out_of_host_memory(part):
    r = subprocess.run([sys.executable, "-c", CHILD % (ROOT, part)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), (r.returncode, r.stdout, r.stderr[-2000:])
