"""The first overlaps of a process, from several threads with a context each: all take the same kernel (the
cluster's), so that they give the same bits.  Run in a process of its own, which has called nothing before."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import threading
import numpy as np
from paper_2507_05222_gb300 import inputs, qtt
T = 8
ctx = [qtt.Context(0) for _ in range(T)]
cores = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(20, 32, 3)]
g = [qtt.MPS.from_cores(c, cores) for c in ctx]
gate, v = threading.Barrier(T), [None] * T
def first(k):
    gate.wait()
    v[k] = qtt.mps_dot(ctx[k], g[k], g[k])
th = [threading.Thread(target=first, args=(k,)) for k in range(T)]
[t.start() for t in th]
[t.join() for t in th]
again = qtt.mps_dot(ctx[0], g[0], g[0])
assert all(x == again for x in v), (v, again)
"""


def test_first_calls_of_several_threads_agree():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
