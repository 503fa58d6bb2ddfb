"""Several threads create their first contexts at once, in a fresh process: every
one has the tensor-copy variant and computes the same field."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import threading
import numpy as np
from paper_2603_25282_gb300 import inputs, sgp

n, N = (512, 512), 12
psi = inputs.gaussian_random_phase(n, 16.0, seed=1)[None].astype(np.complex64)
sgp.lib()
start, out, bad = threading.Barrier(N), [None] * N, []

def work(k):
    try:
        start.wait()
        with sgp.Context(n, 16.0) as c:
            c.set_params(omega=0.5, gamma=1.0, c0=100.0, c1=-1.0, c2=2.0)
            c.set_state(psi, 0.0)
            if k % 2:
                c.set_plan((1, 4))          # refused where no encoder was found
                c.set_plan((0, 0))
            c.step(3, 1e-3)
            out[k] = c.get_state()
    except Exception as e:
        bad.append(repr(e))

t = [threading.Thread(target=work, args=(k,)) for k in range(N)]
[x.start() for x in t]
[x.join() for x in t]
assert not bad, bad
assert all(np.array_equal(o, out[0]) for o in out) and np.isfinite(out[0]).all()
print("same")
"""


def test_first_contexts_at_once():
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]
