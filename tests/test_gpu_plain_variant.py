"""Variant 7, the plain kernels at any size: what variant 0 stands for in the
groups of an ensemble, a member's result the same alone and in any batch, the
gradient's passes plain too, and its place in the autotuner's table."""
import ctypes

import numpy as np
import pytest

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu

PRM = dict(omega=0.6, gamma=1.2, c0=200.0, c1=-2.0, c2=3.0, gx=1.0, gy=1.2, gz=1.5)


def _fields(n, batch, prec):
    return np.stack([inputs.gaussian_random_phase(n, 6.0, seed=3 + m, amp=0.4) for m in range(batch)]).astype(
        np.complex64 if prec == "f32" else np.complex128)


def _run(n, batch, prec, plan, grad=False):
    with sgp.Context(n, 6.0, batch=batch, prec=prec) as c:
        c.set_params(**PRM)
        c.set_plan(plan)
        f = _fields(n, batch, prec)
        c.set_state(f, 0.0)
        if not grad:
            c.step(4, 1e-3, "ts4")
            return c.get_state()
        c.record(4, 1e-3, "ts2")
        return c.backward(np.conj(f))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,batch", [((96, 64), 40), ((48, 32, 16), 12)])
def test_a_member_alone_and_in_a_batch(prec, n, batch):
    plan = (7,) * len(n)
    one, many = _run(n, 1, prec, plan), _run(n, batch, prec, plan)
    assert np.isfinite(many).all()
    assert np.array_equal(one[0], many[0])
    (g1, p1), (gb, pb) = _run(n, 1, prec, plan, True), _run(n, batch, prec, plan, True)
    assert np.array_equal(g1[0], gb[0]) and np.array_equal(p1[0], pb[0])


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_is_the_kernel_of_ensemble_groups(prec):
    n = (96, 64)
    f = _fields(n, 2, prec)
    with sgp.Ensemble([(n, 6.0)] * 2, prec=prec) as e:
        e.set_params([PRM] * 2)
        e.set_persistent(False)
        for m in range(2):
            e.set_member_state(m, f[m], 0.0)
        e.step(4, 1e-3, "ts4")
        got = [e.get_member_state(m) for m in range(2)]
    want = _run(n, 2, prec, (7, 7))
    for m in range(2):
        assert np.array_equal(got[m], want[m])


def test_autotuner_table():
    n = (512, 512)                 # variant 0 of the y-lines stands for variant 4
    with sgp.Context(n, 16.0) as c:
        c.set_params(**PRM)
        c.set_state(_fields(n, 1, "f32"), 0.0)
        plan, ms = c.autotune(reps=2, force=True, timings=True)
        assert ms[1][0] == ms[1][4] > 0
        assert all(ms[a][7] > 0 for a in range(2))
        # a caller with a table of 7 columns: nothing is written past it
        tab = (ctypes.c_double * 22)(*([123.0] * 22))
        assert sgp.lib().sgp_autotune(c.handle, 2, sgp.SGP_TUNE_FORCE, tab) == 0
        assert tab[21] == 123.0 and list(tab[14:21]) == [-1.0] * 7
        assert tab[0] > 0 and tab[7] > 0 and max(c.get_plan()) < 7
