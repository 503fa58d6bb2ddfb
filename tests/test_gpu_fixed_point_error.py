"""How far the fixed-point transforms of the FP64 passes are from exact ones, and
a captured run of them against the oracle.

A linear substep of length 1e-300 is a forward and an inverse transform along
every axis and nothing else: it gives its input back.  In fixed point the field is
rounded to doubles once per transform and once or twice in the mode's factor and
the scaling, at 0.6 u each: sqrt(6) * 0.6 * 1.1e-16 = 1.6e-16 in relative L2.  A
transform's own error, from an emulation of its integers, is 0.2e-16 to 1.3e-16 (the
most for smooth lines of 768 and 1024): four of them 2.6e-16, together 3.1e-16.  The
FP64 transforms of the plain kernels round every element sqrt(2 log2 N) times
more per axis: they are further off.
"""
import numpy as np
import pytest

from oracle import sgp_oracle as O
from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu


def _there_and_back(n, f, plan):
    with sgp.Context(n, 6.0, prec="f64") as c:
        c.set_params(omega=0.0, gamma=0.0)
        c.set_plan(plan)
        c.set_state(f[None].copy(), 0.0)
        c.substep("linear", 1e-300)
        out = c.get_state()[0]
    return np.linalg.norm(out - f) / np.linalg.norm(f)


@pytest.mark.parametrize("n", [(256, 256), (192, 128), (512, 64), (48, 1024), (96, 384), (768, 16), (32, 16)])
def test_closer_than_fp64_transforms(n):
    for f in (inputs.random_field(n, 5), inputs.gaussian_random_phase(n, 6.0, seed=2, amp=0.3)):
        fixed, plain = _there_and_back(n, f, (0, 0)), _there_and_back(n, f, (7, 7))
        assert fixed <= 3.1e-16, (fixed, plain)
        assert fixed < plain


@pytest.mark.parametrize("n,scheme", [((64, 48), "ts2"), ((32, 16, 16), "ts2")])
def test_captured_run_against_the_oracle(n, scheme):
    """130 steps: two replays of a captured chunk and a rest.  Errors of 260
    passes, 7 u each in quadrature: 1.3e-14; the phases' own rounding (angles up
    to delta c0 rho) about as much again per step: 1e-12."""
    prm = dict(omega=0.6, gamma=1.2, c0=200.0, c1=-2.0, c2=3.0, gx=1.0, gy=1.2, gz=1.5)
    psi = inputs.gaussian_random_phase(n, 6.0, seed=3, amp=0.5)
    ref = O.Propagator(O.Grid(n, 6.0), O.Params(**prm)).run(psi, 0.0, 1e-3, 130, scheme)[0]
    with sgp.Context(n, 6.0, prec="f64") as c:
        c.set_params(**prm)
        c.set_state(psi[None].copy(), 0.0)
        c.step(130, 1e-3, scheme)
        out = c.get_state()[0]
    assert O.rel_l2(out, ref) < 1e-12
