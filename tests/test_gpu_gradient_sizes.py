"""FP32 gradients against FP64 ones over the forms that their passes take: every
number of elements per thread, rows and columns per CTA of the component-parallel
passes, z-lines, several members, all schemes, and the plain passes on the other
side of the size rule; the tensor-copy line pass inside a 3D sweep.

Tolerances, n steps of f flow pairs: the state and its gradient go through about
2 f n passes each way, every element rounded about sqrt(2 log2 N) times at 0.6 u a
pass: at most 30 passes here, sqrt(30) * 2.7 u = 9e-7 in relative L2, the state's
error entering the gradient once more.  1e-5 leaves room for the flows' angles.
The parameters' derivatives are FP64 sums of terms with that rounding which cancel
in part: 1e-4 of the member's largest, the accuracy the gradients are specified to.
"""
import numpy as np
import pytest

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu


def _params(batch):
    return [dict(omega=0.6 + 0.05 * m, gamma=1.0 - 0.1 * m, c0=200.0 + 30.0 * m, c1=-2.0, c2=4.0 + m, gx=1.0, gy=1.3,
                 gz=1.5) for m in range(batch)]


def _gradient(n, batch, scheme, prec, nsteps=3, plan=None, graphs=True, interval=2):
    with sgp.Context(n, 6.0, batch=batch, prec=prec) as c:
        c.set_params_batch(_params(batch))
        c.set_graphs(graphs)
        if plan:
            c.set_plan(plan)
        psi = np.stack([inputs.gaussian_random_phase(n, 6.0, seed=20 + m % 3, amp=0.4) for m in range(batch)])
        g = np.stack([inputs.gaussian_random_phase(n, 6.0, seed=40 + m % 3, amp=1.0) for m in range(batch)])
        c.set_state(psi.astype(c.dtype), 0.2)
        c.record(nsteps, 1e-3, scheme, interval)
        return c.backward(g.astype(c.dtype))


SPLIT = [((16, 48), 2, "ts2_lnl"), ((48, 16), 1, "ts4"), ((96, 192), 1, "ts2"), ((192, 96), 2, "ts2"),
         ((768, 32), 1, "ts2"), ((32, 768), 1, "ts4_l"), ((1024, 16), 2, "ts2"), ((16, 1024), 2, "ts2"),
         ((512, 64), 1, "ts4"), ((64, 512), 2, "ts2_lnl"), ((384, 128), 1, "ts2"), ((32, 32), 128, "ts2"),
         ((16, 48, 32), 2, "ts2"), ((48, 32, 16), 1, "ts4_l"), ((32, 16, 96), 1, "ts2_lnl"), ((16, 16, 16), 24, "ts2")]
PLAIN = [((512, 512), 1, "ts2"), ((768, 384), 1, "ts2_lnl"), ((256, 256), 4, "ts2"), ((1024, 192), 1, "ts2"),
         ((32, 64), 96, "ts2"), ((64, 64, 64), 1, "ts2"), ((96, 48, 32), 2, "ts2"), ((32, 16, 16), 15, "ts4_l")]


@pytest.mark.parametrize("n,batch,scheme", SPLIT + PLAIN)
def test_fp32_against_fp64(n, batch, scheme):
    g32, p32 = _gradient(n, batch, scheme, "f32")
    g64, p64 = _gradient(n, batch, scheme, "f64")
    for m in range(batch):
        assert np.linalg.norm(g32[m] - g64[m]) <= 1e-5 * np.linalg.norm(g64[m]), m
        assert np.abs(p32[m] - p64[m]).max() <= 1e-4 * np.abs(p64[m]).max(), (m, p32[m], p64[m])


@pytest.mark.parametrize("graphs", [True, False])
def test_tensor_copies_in_a_3d_sweep(graphs):
    """The y-lines of a 3D sweep are the plan's, on the sweep's own buffers: the
    tensor map follows them."""
    n = (64, 64, 48)
    a = _gradient(n, 2, "ts2", "f32", nsteps=7, plan=(1, 1, 1), graphs=graphs)
    b = _gradient(n, 2, "ts2", "f32", nsteps=7, plan=(1, 4, 4), graphs=graphs)
    assert np.isfinite(a[0]).all() and np.isfinite(a[1]).all()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
