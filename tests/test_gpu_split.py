"""The component-parallel passes (variant 0 of small grids) and what variant 0
stands for by the size of the grid: every line length along x and along y
against the oracle's flows through an FP64 context and the plain kernels.

Tolerances: a pass rounds each element about sqrt(2 log2 N) times at 0.6 u, u
the unit roundoff; two TS2 steps are five passes, so N <= 1024 gives about 7 u
in relative L2.  Four times that, rounded up: FP32 2e-6, FP64 1e-14 (the flows'
own angles add another factor in FP64: 1e-13).
"""
import numpy as np
import pytest

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu

PRM = dict(omega=0.7, gamma=1.2, c0=300.0, c1=-4.0, c2=6.0, gx=1.0, gy=1.3, gz=1.5)
TOL = {"f32": 2e-6, "f64": 1e-13}
SIDES = (16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)


def rel(a, b):
    return np.linalg.norm(a.astype(np.complex128) - b) / np.linalg.norm(b)


def propagate(n, prec, plan=None, batch=1, nsteps=2, scheme="ts2", graphs=True):
    with sgp.Context(n, 6.0, batch=batch, prec=prec) as c:
        c.set_params_batch([dict(PRM, omega=0.7 + 0.05 * m, c0=300.0 - 20.0 * m) for m in range(batch)])
        c.set_graphs(graphs)
        if plan:
            c.set_plan(plan)
        psi = inputs.gaussian_random_phase(n, 6.0, seed=3, amp=0.2)
        c.set_state(np.stack([psi * (1.0 + 0.1 * m) for m in range(batch)]).astype(c.dtype), 0.25)
        for k in nsteps if isinstance(nsteps, tuple) else (nsteps,):
            c.step(k, 1e-3, scheme)
        return c.get_state()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("side", SIDES)
def test_every_line_length(prec, side):
    # the other side small, so that variant 0 is the component-parallel pass
    for n in ((side, 16), (16, side), (side, 48)):
        ref = propagate(n, "f64", plan=(1, 1))
        assert rel(propagate(n, prec), ref) < TOL[prec], n


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", [(48, 32, 16), (16, 96, 32), (64, 16, 48)])
def test_three_dimensions(prec, n):
    ref = propagate(n, "f64", plan=(1, 1, 1), scheme="ts4")
    assert rel(propagate(n, prec, scheme="ts4"), ref) < TOL[prec]


@pytest.mark.parametrize("n,batch", [((256, 256), 3), ((256, 256), 4), ((512, 512), 1), ((192, 128), 8),
                                     ((64, 32, 32), 1), ((64, 64, 32), 1)])
def test_both_sides_of_the_size_rule(n, batch):
    """FP32 at and past the sizes where variant 0 changes; FP64 alike."""
    plan = (1,) * len(n)
    ref = propagate(n, "f64", plan=plan, batch=batch)
    assert rel(propagate(n, "f64", batch=batch), ref) < TOL["f64"]
    assert rel(propagate(n, "f32", batch=batch), ref) < TOL["f32"]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("scheme", ["ts2", "ts4_l"])
def test_dependent_launches_in_graphs(prec, scheme):
    """130 steps: two replays of a captured chunk of 64 and a rest of 2, bit for
    bit the eager launches of the same runs (a run merges the substeps that
    meet at its step boundaries; the passes overlap their neighbours in both)."""
    a = propagate((96, 64), prec, nsteps=130, scheme=scheme)
    b = propagate((96, 64), prec, nsteps=(64, 64, 2), scheme=scheme, graphs=False)
    assert np.array_equal(a, b)


def test_host_windows_match():
    """Member windows run the kernels of the whole batch."""
    n, batch = (64, 48), 5
    psi = inputs.gaussian_random_phase(n, 6.0, seed=3, amp=0.2)
    host = np.stack([psi * (1.0 + 0.1 * m) for m in range(batch)]).astype(np.complex64)
    with sgp.Context(n, 6.0, batch=batch) as c:
        c.set_params(**PRM)
        c.set_state(host, 0.0)
        c.step(3, 1e-3, "ts2")
        want = c.get_state()
        for chunks in (1, 2, 5):
            assert np.array_equal(c.step_host(host, 0.0, 3, 1e-3, "ts2", chunks=chunks), want)


# ---------------------------------------------------------------------------
# the fixed-point transforms of the FP64 passes
# ---------------------------------------------------------------------------
def linear(f, n, plan=None, delta=0.03):
    with sgp.Context(n, 6.0, prec="f64") as c:
        c.set_params(**PRM)
        if plan:
            c.set_plan(plan)
        c.set_state(f[None].copy(), 0.0)
        c.substep("linear", delta)
        return c.get_state()[0]


@pytest.mark.parametrize("n", [(64, 48), (96, 32), (512, 16), (16, 384)])
def test_fixed_point_lines(n):
    """Lines of very different content: unstructured, one element, one
    component far below the others, zeros; and every power-of-two scale of a
    field (the common exponent of a line) gives the scaled result bit for bit."""
    f = inputs.random_field(n, 5)
    one = np.zeros_like(f)
    one[2, 3, 5] = 1.5 - 0.5j
    low = f.copy()
    low[3] *= 1e-18
    for g in (f, one, low):
        assert rel(linear(g, n), linear(g, n, plan=(1, 1))) < TOL["f64"]
    assert not linear(np.zeros_like(f), n).any()
    want = linear(f, n)
    for k in (-900, -40, 300, 900):
        assert np.array_equal(linear(f * 2.0 ** k, n), want * 2.0 ** k), k
    # components that do not mix keep their own relative accuracy
    with sgp.Context(n, 6.0, prec="f64") as c:
        c.set_params(omega=0.0, gamma=0.0)
        c.set_state(low[None].copy(), 0.0)
        c.substep("linear", 0.03)
        got = c.get_state()[0]
        c.set_plan((1, 1))
        c.set_state(low[None].copy(), 0.0)
        c.substep("linear", 0.03)
        assert rel(got[3], c.get_state()[0][3]) < TOL["f64"]


def test_fixed_point_not_finite():
    """A NaN or an infinity leaves nothing finite, as in the FP64 transforms,
    and the next state is clean again."""
    n = (48, 64)
    f = inputs.random_field(n, 5)
    for bad in (np.nan, np.inf, -np.inf):
        g = f.copy()
        g[1, 7, 9] = bad
        assert not np.isfinite(linear(g, n)).any()
        assert not np.isfinite(linear(g, n, plan=(1, 1))).any()
    assert np.isfinite(linear(f, n)).all()


def test_flow_tiers():
    """FP64 flow at one substep on every branch of its angles: Taylor degrees 3
    to 6 of the spin rotation and past them, both forms of the singlet and of
    the phase, against the plain kernels."""
    n = (32, 16)
    f = inputs.random_field(n, 8, scale=0.3)
    for c1 in (0.0, 1e-4, 1e-3, 5e-3, 1e-2, 2.0, 40.0):
        for c0, c2 in ((1.0, 0.01), (100.0, 2.0), (900.0, -300.0)):
            out = []
            for plan in ((0, 0), (1, 1)):
                with sgp.Context(n, 6.0, prec="f64") as c:
                    c.set_params(omega=0.3, gamma=0.5, c0=c0, c1=c1, c2=c2, gx=1.0, gy=1.5)
                    c.set_plan(plan)
                    c.set_state(f[None].copy(), 0.4)
                    c.substep("nonlinear", 0.01)
                    out.append(c.get_state())
            assert rel(out[0], out[1]) < TOL["f64"], (c0, c1, c2)
