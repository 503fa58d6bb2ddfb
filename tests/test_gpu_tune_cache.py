"""The autotuner's process-wide plans of ensemble groups and of contexts are
apart: their variant 0 is another kernel, so neither may take the other's plan
without timing its own kernels."""
import numpy as np
import pytest

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu

PRM = dict(omega=0.5, gamma=1.0, c0=100.0, c1=-1.0, c2=2.0)


def _context(n, prec):
    c = sgp.Context(n, 8.0, prec=prec)
    c.set_params(**PRM)
    c.set_state(inputs.gaussian_random_phase(n, 8.0, seed=2)[None].astype(c.dtype), 0.0)
    return c


def _tuned(c):
    before = c.launch_count()
    c.autotune(reps=2)
    return c.launch_count() - before


def _ensemble(n, prec):
    with sgp.Ensemble([(n, 8.0)], prec=prec) as e:
        e.set_params([PRM])
        psi = inputs.gaussian_random_phase(n, 8.0, seed=2)
        e.set_member_state(0, psi.astype(np.complex64 if prec == "f32" else np.complex128), 0.0)
        e.autotune(reps=2)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_context_after_ensemble(prec):
    n = (64, 48)
    _ensemble(n, prec)
    with _context(n, prec) as c:
        assert _tuned(c) > 0                # its own kernels are timed
    with _context(n, prec) as c:
        assert _tuned(c) == 0               # and kept for the next context
