"""The rounded directions of the FP32 mode tables against the search with FP64
scores: read from the context's memory through a caller's allocator."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_25282_gb300 import inputs, sgp

pytestmark = pytest.mark.gpu


def _table(n, L):
    held = {}

    def _alloc(size, device, stream, user):
        t = torch.empty(max(size, 16), dtype=torch.uint8, device="cuda:%d" % device)
        held[t.data_ptr()] = t[:size]
        return t.data_ptr()

    keep = (sgp.ALLOC_FN(_alloc), sgp.FREE_FN(lambda p, *a: held.pop(p, None)))
    assert sgp.lib().sgp_set_allocator(keep[0], keep[1], None) == 0
    try:
        with sgp.Context(n, L) as c:
            c.set_params(omega=0.6, gamma=1.2)
            c.set_state(inputs.gaussian_random_phase(n, L, seed=1)[None].astype(np.complex64), 0.0)
            have = set(held)
            c.substep("linear", 1e-3)
            c.synchronize()
            shape = (n[0] // 2 + 1, n[1] // 2 + 1, 8)
            tab = [t for p, t in held.items() if p not in have and t.numel() == 4 * np.prod(shape)]
            assert len(tab) == 1
            return tab[0].view(torch.float32).cpu().numpy().reshape(shape)
    finally:
        sgp.use_torch_allocator(False)


@pytest.mark.parametrize("n,L", [((48, 32), (5.0, 6.0)), ((256, 512), (16.0, 16.0))])
def test_directions(n, L):
    tab = _table(n, L)
    z = tab[..., 6:8].astype(np.float64)
    # the axis modes are exact, zeros included
    assert (tab[0, 1:, 6] == 0).all() and (tab[0, 1:, 7] == 1).all()
    assert (tab[1:, 0, 6] == 1).all() and (tab[1:, 0, 7] == 0).all()
    # the others lie within 2.5 ulp of the direction (the rounded pair and two
    # more), and no worse in modulus than the rounded pair may be (2^-24)
    p, q = np.arange(n[0] // 2 + 1)[:, None] / L[0], np.arange(n[1] // 2 + 1)[None] / L[1]
    r = np.hypot(p, q)
    r[0, 0] = 1.0
    t = np.stack([p + 0 * q, q + 0 * p], -1) / r[..., None]
    t[0, 0] = (1.0, 0.0)
    ulp = np.spacing(np.abs(t).astype(np.float32)).astype(np.float64)
    assert (np.abs(z - t) <= 2.5 * ulp).all()
    assert (np.abs(np.hypot(z[..., 0], z[..., 1]) - 1.0) < 2.0 ** -24).all()
