"""A tile-load wait that gave up (the error word of the passes that bring their
tiles in by tensor copies) reaches every call that hands a result to the host,
also on the default kernels.  The word is set through the allocator's view of
the context's memory: no wait of a kernel is made to fail."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu

PRM = dict(omega=0.5, gamma=1.0, c0=100.0, c1=-1.0, c2=2.0)


# 19 sums per member, then the error word
OBS_BLOCK = {(19 * batch + 1) * 8 for batch in (1, 2)}


@pytest.fixture
def words():
    """The error words of contexts of one or two members."""
    held = {}

    def _alloc(size, device, stream, user):
        t = torch.empty(max(size, 16), dtype=torch.uint8, device="cuda:%d" % device)
        held[t.data_ptr()] = (size, t)
        return t.data_ptr()

    keep = (sgp.ALLOC_FN(_alloc), sgp.FREE_FN(lambda p, *a: held.pop(p, None)))
    assert sgp.lib().sgp_set_allocator(keep[0], keep[1], None) == 0
    yield lambda: [t[size - 8:size - 4].view(torch.int32) for size, t in held.values() if size in OBS_BLOCK]
    sgp.use_torch_allocator(False)


def _set(words):
    assert len(words()) == 1
    for w in words():
        w.fill_(1)
    torch.cuda.synchronize()


CALLS = {
    "get_state": lambda c, f: c.get_state(),
    "get_state_lab": lambda c, f: c.get_state_lab(),
    "observables": lambda c, f: c.observables(),
    "step_host": lambda c, f: c.step_host(f, 0.0, 1, 1e-3),
    "synchronize": lambda c, f: c.synchronize(),
    "health check": lambda c, f: c.step(1, 1e-3),
    "backward": lambda c, f: c.backward(f),
}


@pytest.mark.parametrize("call", CALLS)
def test_default_kernels_report_it(words, call):
    n = (512, 512)                          # above the component-parallel sizes: TMA y-lines
    f = inputs.gaussian_random_phase(n, 16.0, seed=1)[None].astype(np.complex64)
    with sgp.Context(n, 16.0) as c:
        c.set_params(**PRM)
        c.set_state(f, 0.0)
        if call == "health check":
            c.set_health_check(1, 1e-2)
        if call == "backward":
            c.record(2, 1e-3)
        else:
            c.step(2, 1e-3)
        c.synchronize()
        _set(words)
        with pytest.raises(sgp.SgpError, match="SGP_ETIMEOUT"):
            CALLS[call](c, f)
        with pytest.raises(sgp.SgpError):   # the state is undefined
            c.step(1, 1e-3)
        c.set_health_check(0, 0.0)
        c.set_state(f, 0.0)
        c.step(1, 1e-3)
        c.observables()
        c.synchronize()


def test_ensemble_reports_it(words):
    n = (128, 64)
    f = inputs.gaussian_random_phase(n, 8.0, seed=1).astype(np.complex64)
    for call in ("get", "host", "sync", "observables"):
        with sgp.Ensemble([(n, 8.0)] * 2) as e:
            e.set_params([PRM] * 2)
            e.set_persistent(False)
            e.set_member_state(0, f, 0.0)
            e.set_member_state(1, f, 0.0)
            e.autotune(reps=1, force=True)  # runs the tensor-copy variant
            e.synchronize()
            _set(words)
            with pytest.raises(sgp.SgpError, match="SGP_ETIMEOUT"):
                if call == "get":
                    e.get_member_state(0)
                elif call == "host":
                    e.step_host([f, f], 0.0, 1, 1e-3)
                elif call == "observables":
                    e.observables()
                else:
                    e.synchronize()
            with pytest.raises(sgp.SgpError):
                e.step(1, 1e-3)             # the states are undefined
            for m in (0, 1):
                e.set_member_state(m, f, 0.0)
            e.step(1, 1e-3)
            assert np.isfinite(e.get_member_state(0)).all()
