"""The block-sum reduction of the observables at more blocks than its threads,
and the persistent ensemble kernel with one and with two tiles per work item.

Mass: FP64 sums of exact squares of FP32 values, at most 2^22 terms: the two
orders of summation differ by less than 22 u = 2.5e-15 relative; 1e-13 leaves
room for the blocks' inner order.
"""
import numpy as np
import pytest

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [((16, 16), 1), ((512, 1024), 2), ((1024, 768), 1), ((64, 64, 96), 2)])
def test_mass_of_many_blocks(n, batch):
    f = np.stack([inputs.random_field(n, 3 + m) for m in range(batch)]).astype(np.complex64)
    with sgp.Context(n, 4.0, batch=batch) as c:
        c.set_params(omega=0.1, gamma=0.2, c0=1.0)
        c.set_state(f, 0.0)
        cell = np.prod([8.0 / N for N in n])
        for m, o in enumerate(c.observables()):
            g = f[m].astype(np.complex128)
            want = [cell * float((g[k].real ** 2 + g[k].imag ** 2).sum()) for k in range(5)]
            assert np.allclose(o["comp_mass"], want, rtol=1e-13, atol=0.0)


@pytest.mark.parametrize("count", [2, 20])     # 64 tiles a pass, and 640: past 1.5 per CTA
def test_tiles_per_item(count):
    n, steps = (256, 256), 3
    out = []
    for persistent in (True, False):
        with sgp.Ensemble([(n, 8.0)] * count) as e:
            e.set_params([dict(omega=0.1 + 0.02 * m, gamma=1.0, c0=100.0 + m, c1=-1.0, c2=2.0) for m in range(count)])
            e.set_persistent(persistent)
            psi = inputs.gaussian_random_phase(n, 8.0, seed=2, amp=0.1).astype(np.complex64)
            for m in range(count):
                e.set_member_state(m, psi)
            e.step(steps, 1e-3)
            out.append([e.get_member_state(m) for m in range(count)])
            e.synchronize()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
