"""One context per host thread: contexts that start with different sizes at the same time.  What the library keeps per
process (the shared memory a kernel may have, resident blocks) is first touched here, so each run is a fresh process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import sys, threading
sys.path.insert(0, sys.argv[1])
import numpy as np
import workloads as W
from paper_2012_11430_gb300 import Context, default_opts
from paper_2012_11430_gb300 import binding
binding.load()
SIZES = [(2, 9, 3), (2, 15, 12), (2, 23, 24), (2, 31, 45), (2, 50, 20), (3, 13, 10), (1, 60, 6), (2, 31, 64)]
probs = [W.make_problem(f"th{i}", d, n, m, 7600 + i) for i, (d, n, m) in enumerate(SIZES)]
start = threading.Barrier(4)
errors = []
def work(k):
    try:
        order = probs if k % 2 == 0 else probs[::-1]
        with Context(0) as ctx:
            start.wait()
            for prec in ("bf16x3", "fp32") if k < 2 else ("tf32x3", "fft32"):
                for p in order:
                    r = ctx.solve(p.grid, p.d, p.n, p.m, default_opts(precision=prec)) if prec != "fft32" or p.d < 3 else None
                    if r is not None:
                        te, ce = W.match_to_truth(r.t, r.c, p.t, p.c)
                        assert te <= 1e-6 and ce <= 1e-5, (k, prec, p.name, te, ce)
                    f = ctx.eval(p.t, p.c, np.zeros((4000, p.d), np.int32))
                    assert np.allclose(f, p.c.sum(), rtol=0, atol=1e-12 * p.m)
    except BaseException as e:
        errors.append(repr(e))
threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not errors, errors
"""


@pytest.mark.parametrize("run", range(3))
def test_contexts_of_threads_start_together(run):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
