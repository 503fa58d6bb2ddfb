"""Performance cases of the propagator: what a user's program has it do.

A case is a dict of plain values.  ``prepare`` makes the inputs on the GPU
from a seed, with the context (or ensemble) a program keeps; ``run`` is one
pass through the public entry points; ``exact`` is the same result in FP64 by
plain torch, written from the method (Sec. 3 of arXiv 2603.25282) and sharing
no code with the package.

Kinds of a case:
  run   set the state, advance nsteps, read the state back (device buffers);
        with obs the observables of the final state, with lab its lab-frame
        field, as a program that follows a simulation does at every output
  host  the same as one host-to-host call on page-locked buffers
  ens   independent runs on grids of different sizes, advanced together in one
        host-to-host call
  grad  a recorded run and its gradient (state and parameters)
"""
from __future__ import annotations

import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_2603_25282_gb300 import inputs, sgp

# parameter sets: the fast-rotating 2D system, the timing runs of the paper's
# Example 2, the dynamical laws of its Example 3, the 3D system with an
# anisotropic trap, the gradient workload
PARAMS = {
    "fast2d": dict(omega=0.9, gamma=1.5, c0=1000.0, c1=-5.0, c2=10.0, gx=1.0, gy=1.0, gz=1.0),
    "ex2": dict(omega=0.2, gamma=0.1, c0=10.0, c1=1.0, c2=1.0, gx=1.0, gy=1.0, gz=1.0),
    "ex3": dict(omega=0.2, gamma=0.9, c0=120.0, c1=1.0, c2=1.0, gx=1.0, gy=1.0, gz=1.0),
    "trap3d": dict(omega=0.7, gamma=1.0, c0=500.0, c1=-2.0, c2=5.0, gx=1.0, gy=1.0, gz=2.0),
    "grad": dict(omega=0.6, gamma=1.0, c0=400.0, c1=-1.0, c2=2.0, gx=1.0, gy=1.0, gz=1.0),
}
# initial data: component weights and width factor s of exp(-s |x|^2); the
# weights of the "gaussian" data are normalised to mass 1 on the grid
INITIAL = {
    "gaussian": ((1.0, 1.0, 1.0, 1.0, 1.0), 0.5),
    "ini1": ((1.0, 1.0, 2.0, 1.0, 1.0), 0.5),
    "ini3": ((1.0, 1.0, 6.0 * math.sqrt(7.0), 1.0, 1.0), 0.125),
}
SIDES = (16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)


def _case(name, kind, nx, ny, nz, L, batch, prec, scheme, nsteps, dt, prm, init, tune=False,
          obs=False, lab=False, chunks=0, count=0):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, L=L, batch=batch, prec=prec, scheme=scheme,
             nsteps=nsteps, dt=dt, prm=prm, init=init, tune=tune, obs=obs, lab=lab,
             chunks=chunks, count=count)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a program that looks at the state after every step of a small grid:
        # launches and latency are all there is
        _case("2d64_ts2_f32_one_step", "run", 64, 64, 1, 12.0, 1, "f32", "ts2", 1, 1e-3, "ex2", "ini1"),
        # the paper's timing run (Example 2) on a small grid, with the
        # lab-frame field for the output at its end
        _case("2d128_ts2_f32_example2", "run", 128, 128, 1, 12.0, 1, "f32", "ts2", 100, 1e-3, "ex2",
              "ini1", lab=True),
        # the same set-up in FP64, as its accuracy tables are computed; a
        # side with a factor 3
        _case("2d192_ts2_f64_example2", "run", 192, 192, 1, 12.0, 1, "f64", "ts2", 10, 1e-3, "ex2", "ini1"),
        # one production run on a large 2D grid, default kernels
        _case("2d512_ts4_f32", "run", 512, 512, 1, 16.0, 1, "f32", "ts4", 10, 5e-4, "fast2d", "gaussian"),
        # the benchmark's batch of such runs, tuned as the benchmark does:
        # the resident field is larger than L2
        _case("2d512_ts4_f32_batch32", "run", 512, 512, 1, 16.0, 32, "f32", "ts4", 4, 5e-4, "fast2d",
              "gaussian", tune=True),
        # the reference solution of such a run in FP64
        _case("2d512_ts4_f64", "run", 512, 512, 1, 16.0, 1, "f64", "ts4", 2, 5e-4, "fast2d", "gaussian"),
        # the benchmark's 3D runs
        _case("3d128_ts2_f32_batch4", "run", 128, 128, 128, 8.0, 4, "f32", "ts2", 5, 1e-3, "trap3d",
              "gaussian", tune=True),
        # a 3D grid with three different sides in FP64 (the temporal error
        # tables), default kernels
        _case("3d96x64x48_ts4_f64", "run", 96, 64, 48, 8.0, 1, "f64", "ts4", 2, 1e-3, "trap3d", "gaussian"),
        # a parameter study: runs on grids of sides 64 to 256 side by side
        _case("ens64_ts2_f32", "ens", 0, 0, 1, 8.0, 1, "f32", "ts2", 20, 1e-3, "ens", "gaussian", count=64),
        # one gradient of a terminal objective, forward run and backward sweep
        _case("grad256_ts2_f32", "grad", 256, 256, 1, 8.0, 1, "f32", "ts2", 100, 1e-3, "grad", "gaussian"),
        # the dynamical-laws series (Example 3): observables every ten steps
        _case("2d768_ts4_f32_observables", "run", 768, 768, 1, 24.0, 1, "f32", "ts4", 10, 1e-3, "ex3",
              "ini3", obs=True),
        # the benchmark's end-to-end call: states from page-locked host
        # memory, one step, back to host memory
        _case("2d512_ts4_f32_batch32_host", "host", 512, 512, 1, 16.0, 32, "f32", "ts4", 1, 5e-4, "fast2d",
              "gaussian", chunks=16),
    ]


def _log_choice(rng, values):
    """One of the (ascending) values, uniformly over the range's logarithm."""
    lo, hi = math.log(values[0]), math.log(values[-1])
    x = rng.uniform(lo, hi)
    return min(values, key=lambda v: abs(math.log(v) - x))


def draw(rng):
    what = rng.choice(["2d32", "2d32", "2d32", "2d64", "3d32", "3d64", "ens", "grad", "obs", "host"])
    scheme = rng.choice(["ts2", "ts2", "ts4", "ts4", "ts2_lnl", "ts4_l"])
    prm = rng.choice(["fast2d", "ex2", "ex3", "grad"])
    init = rng.choice(["gaussian", "ini1", "ini3"])
    L = 24.0 if init == "ini3" else rng.choice([8.0, 12.0, 16.0])
    dt = rng.choice([5e-4, 1e-3, 7e-4])
    tune = rng.random() < 0.3
    flows = 1 if scheme.startswith("ts2") else 3        # linear flows per step

    def steps(points, most):
        """A number of steps for that many points: short of the largest case."""
        return max(1, min(int(math.exp(rng.uniform(0.0, math.log(100.0)))), int(most / (points * flows))))

    if what in ("2d32", "obs", "host"):
        nx, ny = _log_choice(rng, SIDES[2:]), _log_choice(rng, SIDES[2:])
        if rng.random() < 0.5:
            ny = nx
        batch = _log_choice(rng, (1, 2, 3, 5, 8, 16, 32)) if what != "obs" else 1
        batch = max(1, min(batch, 8388608 // (nx * ny)))
        n = steps(nx * ny * batch, 5e7) if what != "host" else rng.choice([1, 2, 3])
        return _case(None, "host" if what == "host" else "run", nx, ny, 1, L, batch, "f32", scheme, n, dt, prm,
                     init, tune=tune, obs=what == "obs", lab=what == "2d32" and nx * ny * batch < 300000,
                     chunks=min(batch, 16) if what == "host" else 0)
    if what == "2d64":
        nx, ny = _log_choice(rng, SIDES[2:10]), _log_choice(rng, SIDES[2:10])
        if rng.random() < 0.5:
            ny = nx
        return _case(None, "run", nx, ny, 1, L, 1, "f64", scheme, min(steps(nx * ny, 1.5e6), 9 // flows), dt, prm, init,
                     obs=rng.random() < 0.3)
    if what == "3d32":
        n3 = [_log_choice(rng, SIDES[1:7]) for _ in range(3)]
        batch = rng.choice([1, 1, 2, 3])
        return _case(None, "run", n3[0], n3[1], n3[2], 8.0, batch, "f32", scheme,
                     steps(n3[0] * n3[1] * n3[2] * batch, 2.5e7), dt, "trap3d", "gaussian", tune=tune)
    if what == "3d64":
        n3 = [_log_choice(rng, SIDES[1:6]) for _ in range(3)]
        return _case(None, "run", n3[0], n3[1], n3[2], 8.0, 1, "f64", scheme,
                     min(steps(n3[0] * n3[1] * n3[2], 1.5e6), 9 // flows), dt, "trap3d", "gaussian")
    if what == "ens":
        return _case(None, "ens", 0, 0, 1, 8.0, 1, "f32", scheme, rng.choice([5, 10, 20]) // flows, dt, "ens",
                     "gaussian", count=rng.choice([12, 24, 40, 56]))
    nx = _log_choice(rng, (64, 96, 128, 192, 256, 384))
    ny = rng.choice([nx, _log_choice(rng, (64, 96, 128, 192, 256))])
    return _case(None, "grad", nx, ny, 1, 8.0, 1, "f32", rng.choice(["ts2", "ts4"]),
                 max(4, min(100, int(6e6 / (nx * ny * 3)))), 1e-3, "grad", "gaussian")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _n(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] > 1 else ())


def _grid(n, L, dev):
    """Coordinates (x, y[, z]), each shaped to broadcast over ([nz,] ny, nx)."""
    d = len(n)
    out = []
    for a, N in enumerate(n):
        x = torch.arange(N, device=dev, dtype=torch.float64) * (2.0 * L / N) - L
        out.append(x.reshape([N if k == d - 1 - a else 1 for k in range(d)]))
    return out


def _field(n, L, init, gen, amp=0.01, nmodes=8, kmax=3):
    """One member: the initial data's Gaussian with a smooth random phase in
    every component (eight cosines of low wave numbers), complex128."""
    w, s = INITIAL[init]
    X = _grid(n, L, "cuda")
    d = len(n)
    G = torch.exp(-s * sum(x * x for x in X))
    u = torch.rand(5, nmodes, generator=gen, dtype=torch.float64) * 2 - 1
    k = torch.randint(-kmax, kmax + 1, (5, nmodes, d), generator=gen)
    ph = torch.rand(5, nmodes, generator=gen, dtype=torch.float64) * 2 * math.pi
    psi = []
    for c in range(5):
        theta = torch.zeros_like(G)
        for j in range(nmodes):
            arg = sum(math.pi / L * int(k[c, j, a]) * X[a] for a in range(d)) + float(ph[c, j])
            theta = theta + float(u[c, j]) * torch.cos(arg)
        psi.append(w[c] * torch.polar(G, amp * theta))
    psi = torch.stack(psi)
    if init == "gaussian":
        cell = math.prod(2.0 * L / N for N in n)
        return psi / torch.sqrt(cell * (psi.abs() ** 2).sum())
    return psi / (math.sqrt(8.0) * math.pi ** (d / 4.0) if init == "ini1" else 32.0 * math.sqrt(math.pi))


def _dtype(case):
    return torch.complex64 if case["prec"] == "f32" else torch.complex128


def _states(case, seed):
    """The initial states of a case in its precision: (batch, 5, ...)."""
    gen = torch.Generator().manual_seed(int(seed))
    return torch.stack([_field(_n(case), case["L"], case["init"], gen) for _ in range(case["batch"])]).to(_dtype(case))


def _members(case):
    return inputs.ensemble_members(case["count"], 4)


def _cotangent(case, seed):
    """Gradient of the objective at the final state: another smooth field."""
    gen = torch.Generator().manual_seed(int(seed) + 1000003)
    g = _field(_n(case), case["L"], case["init"], gen, amp=1.0)
    return g[None].to(_dtype(case))


_stream = None


def _on_stream():
    """The stream of the program: every context issues its work on it."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    st = dict(case=case)
    stream = _on_stream().cuda_stream
    if case["kind"] == "ens":
        gen = torch.Generator().manual_seed(int(seed))
        mem = _members(case)
        ens = sgp.Ensemble([((m["n"], m["n"]), m["L"]) for m in mem], prec=case["prec"], stream=stream)
        ens.set_params([{k: m[k] for k in ("omega", "gamma", "c0", "c1", "c2", "gx", "gy", "gz")} for m in mem])
        src = [_field((m["n"], m["n"]), m["L"], case["init"], gen).to(_dtype(case)) for m in mem]
        flat = torch.empty(sum(f.numel() for f in src), dtype=_dtype(case), pin_memory=True)
        src = [f.cpu().pin_memory() for f in src]
        outs, at = [], 0
        for f in src:
            outs.append(flat[at:at + f.numel()].view(f.shape))
            at += f.numel()
        st.update(ens=ens, src=src, outs=outs, flat=flat)
    else:
        ctx = sgp.Context(_n(case), case["L"], batch=case["batch"], prec=case["prec"], stream=stream)
        ctx.set_params(**PARAMS[case["prm"]])
        psi = _states(case, seed)
        st.update(ctx=ctx, psi=psi, out=torch.empty_like(psi))
        if case["kind"] == "grad":
            st.update(g=_cotangent(case, seed), g0=torch.empty_like(psi))
        if case["lab"]:
            st.update(lab=torch.empty_like(psi))
        torch.cuda.synchronize()
        if case["tune"]:
            ctx.set_state(psi, 0.0)
            ctx.autotune(reps=10)
        if case["kind"] == "host":
            st.update(psi=psi.cpu().pin_memory(), out=torch.empty(psi.shape, dtype=psi.dtype, pin_memory=True))
    torch.cuda.synchronize()
    return st


_OBS = ("mass", "energy", "magnetization", "lz", "e_kin", "e_pot", "e_rot", "e_int", "e_soc")


def _obs_vector(o, dtype):
    return torch.tensor([o[k] for k in _OBS] + list(o["comp_mass"]) + list(o["width2"]), dtype=dtype)


def run(st):
    case = st["case"]
    if case["kind"] == "ens":
        # from page-locked host memory and back, the members' time starting at 0
        st["ens"].step_host(st["src"], 0.0, case["nsteps"], case["dt"], case["scheme"], outs=st["outs"])
        return st["flat"]
    ctx = st["ctx"]
    if case["kind"] == "host":
        return ctx.step_host(st["psi"], 0.0, case["nsteps"], case["dt"], case["scheme"],
                             chunks=case["chunks"], out=st["out"])
    ctx.set_state(st["psi"], 0.0)
    # observables and parameter gradients in the field's precision: their sums
    # are FP64, what they sum has the field's rounding
    real = torch.float32 if case["prec"] == "f32" else torch.float64
    if case["kind"] == "grad":
        ctx.record(case["nsteps"], case["dt"], case["scheme"])
        ctx.get_state(st["out"])
        _, dp = ctx.backward(st["g"], st["g0"])
        return {"psi": st["out"], "g0": st["g0"], "dprm": torch.from_numpy(dp).to(real)}
    ctx.step(case["nsteps"], case["dt"], case["scheme"])
    ctx.get_state(st["out"])
    res = {"psi": st["out"]}
    if case["obs"]:
        res["obs"] = torch.stack([_obs_vector(o, real) for o in ctx.observables()])
    if case["lab"]:
        res["lab"] = ctx.get_state_lab(st["lab"])
    return res


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    flows = 1 if case["scheme"].startswith("ts2") else 3
    size = 8 if case["prec"] == "f32" else 16
    grids = [(m["n"], m["n"]) for m in _members(case)] if case["kind"] == "ens" else [_n(case)] * case["batch"]
    nbytes = flops = 0.0
    for n in grids:
        pts = math.prod(n)
        # per point and flow pair: two transforms of five components along
        # every axis (5 log2 N each), the 5x5 mix and the nonlinear flow
        pair = sum(50.0 * math.log2(N) for N in n) + 450.0 + 500.0
        passes = 3.5 if case["kind"] == "grad" else 1.0       # forward, recomputation, adjoint
        flops += pts * pair * flows * case["nsteps"] * passes
        nbytes += pts * 5 * size * (4 if case["kind"] == "grad" else 3 if case["lab"] else 2)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in FP64, from the method
# ---------------------------------------------------------------------------
_R6H = math.sqrt(6.0) / 2.0


def _dot(wx, wy, wz, v):
    """(w.f) v for a real vector field w and the spin-2 matrices; v: five fields."""
    wp, wm = torch.complex(wx, wy), torch.complex(wx, -wy)
    return [2 * wz * v[0] + wm * v[1],
            wp * v[0] + wz * v[1] + _R6H * (wm * v[2]),
            _R6H * (wp * v[1] + wm * v[3]),
            _R6H * (wp * v[2]) - wz * v[3] + wm * v[4],
            wp * v[3] - 2 * wz * v[4]]


def _exp_spin(wx, wy, wz, v, sign):
    """exp(sign i w.f) v by its power series (entire in w)."""
    with torch.no_grad():
        r = 2.0 * float(torch.sqrt(wx * wx + wy * wy + wz * wz).max())
    terms, t = 1, r
    while t > 1e-19 and terms < 80:
        terms += 1
        t *= r / terms
    out, p = list(v), list(v)
    for k in range(1, terms + 1):
        p = [(sign * 1j / k) * x for x in _dot(wx, wy, wz, p)]
        out = [a + b for a, b in zip(out, p)]
    return out


def _even_series(x, shift):
    """sum (-x)^k / (2k + shift)!: cos(sqrt x) for shift 0, sin(sqrt x)/sqrt x for 1."""
    out, t = torch.ones_like(x), torch.ones_like(x)
    for k in range(1, 24):
        t = t * (-x) / ((2 * k - 1 + shift) * (2 * k + shift))
        out = out + t
    return out


class _Exact:
    """The rotating-frame propagation of one grid in complex128.  prm: FP64
    tensors that broadcast over (batch, ...)."""

    def __init__(self, n, L, prm, trap):
        self.n, self.L, self.prm, self.trap = n, L, prm, trap
        d = len(n)
        self.X = _grid(n, L, "cuda")
        self.nu = []
        for a, N in enumerate(n):
            p = torch.arange(N, device="cuda", dtype=torch.float64)
            p = torch.where(p < N // 2, p, p - N) * (math.pi / L)
            self.nu.append(p.reshape([N if k == d - 1 - a else 1 for k in range(d)]))
        self.axes = tuple(range(-d, 0))
        self.full = torch.zeros([1] + list(n[::-1]), device="cuda", dtype=torch.float64)

    def densities(self, v):
        a = [x.real ** 2 + x.imag ** 2 for x in v]
        rho = sum(a)
        Fz = 2 * (a[0] - a[4]) + a[1] - a[3]
        Fp = 2 * (v[0].conj() * v[1] + v[3].conj() * v[4]) + 2 * _R6H * (v[1].conj() * v[2] + v[2].conj() * v[3])
        A00 = (2 * v[0] * v[4] - 2 * v[1] * v[3] + v[2] * v[2]) / math.sqrt(5.0)
        return rho, Fz, Fp, A00

    def coords(self, t):
        ang = self.prm["omega"] * t
        co, si = torch.cos(ang), torch.sin(ang)
        return co * self.X[0] + si * self.X[1], co * self.X[1] - si * self.X[0]

    def potential(self, t):
        xr, yr = self.coords(t)
        V = 0.5 * (self.trap[0] ** 2 * xr * xr + self.trap[1] ** 2 * yr * yr)
        if len(self.n) == 3:
            V = V + 0.5 * self.trap[2] ** 2 * self.X[2] ** 2
        return V

    def nonlinear(self, v, d, t):
        p = self.prm
        rho, Fz, Fp, A00 = self.densities(v)
        k = p["c2"] * d
        x = k * k * (rho * rho / 25 - (A00.real ** 2 + A00.imag ** 2) / 5)
        cs, sn = _even_series(x, 0), k * _even_series(x, 1)
        ac = [v[4].conj(), -v[3].conj(), v[2].conj(), -v[1].conj(), v[0].conj()]
        b = [cs * v[c] + 1j * sn * (rho / 5 * v[c] - A00 * ac[c] / math.sqrt(5.0)) for c in range(5)]
        s = p["c1"] * d
        b = _exp_spin(s * Fp.real, s * Fp.imag, s * Fz, b, -1)
        ph = d * (self.potential(t) + (p["c0"] + p["c2"] / 5) * rho)
        e = torch.complex(torch.cos(ph), -torch.sin(ph))
        return [e * x for x in b]

    def linear(self, v, d):
        p = self.prm
        v = [torch.fft.fftn(x, dim=self.axes) for x in v]
        chi = 0.5 * d * sum(q * q for q in self.nu)
        e = torch.complex(torch.cos(chi), -torch.sin(chi))
        g = p["gamma"] * d
        v = _exp_spin(-g * self.nu[1] + self.full, g * self.nu[0] + self.full, -p["omega"] * d + self.full, v, 1)
        return [torch.fft.ifftn(e * x, dim=self.axes) for x in v]

    def step(self, psi, t, dt, scheme):
        c = 2.0 ** (1.0 / 3.0)
        a1, a2 = 1 / (2 * (2 - c)), (1 - c) / (2 * (2 - c))
        b1, b2 = 1 / (2 - c), -c / (2 - c)
        seq = {"ts2": "N0.5 L1 N0.5", "ts2_lnl": "L0.5 N1 L0.5"}.get(scheme)
        if seq:
            seq = [(s[0], float(s[1:])) for s in seq.split()]
        else:
            A, B = ("N", "L") if scheme == "ts4" else ("L", "N")
            seq = [(A, a1), (B, b1), (A, a2), (B, b2), (A, a2), (B, b1), (A, a1)]
        v = list(psi.unbind(1))
        for kind, f in seq:
            if kind == "N":
                v = self.nonlinear(v, f * dt, t)
            else:
                v = self.linear(v, f * dt)
                t = t + f * dt
        return torch.stack(v, 1)

    def steps(self, psi, nsteps, dt, scheme, grad=False):
        for s in range(nsteps):
            if grad:
                psi = checkpoint(self.step, psi, s * dt, dt, scheme, use_reentrant=False)
            else:
                psi = self.step(psi, s * dt, dt, scheme)
        return psi

    def observables(self, psi, t):
        """The vector of _OBS, component masses and widths, per member."""
        p, d = self.prm, len(self.n)
        v = list(psi.unbind(1))
        cell = math.prod(2.0 * self.L / N for N in self.n)
        total = lambda f: cell * (f + self.full).sum(dim=self.axes)   # noqa: E731
        rho, Fz, Fp, A00 = self.densities(v)
        grads = [[torch.fft.ifft(1j * self.nu[a] * torch.fft.fft(x, dim=-1 - a), dim=-1 - a) for x in v]
                 for a in range(d)]
        m = [total(x.real ** 2 + x.imag ** 2) for x in v]
        kin = total(0.5 * sum(g.real ** 2 + g.imag ** 2 for ga in grads for g in ga))
        im = lambda ga: sum((x.conj() * g).imag for x, g in zip(v, ga))   # noqa: E731
        lz = total(self.X[0] * im(grads[1]) - self.X[1] * im(grads[0]))
        # SOC energy: -gamma Re <Phi, S Phi> with S Phi = i (w.f) of the derivatives
        # (linear flow symbol Q = gamma (-nu_y f_x + nu_x f_y) in physical space)
        dx, dy = grads[0], grads[1]
        o, z = self.full + 1.0, self.full
        q = [a - b for a, b in zip(_dot(z, o, z, dx), _dot(o, z, z, dy))]
        soc = total(sum((x.conj() * (-1j) * y).real for x, y in zip(v, q)))
        e_soc = -p["gamma"].reshape(-1) * soc
        xr, yr = self.coords(t)
        z2 = self.X[2] ** 2 if d == 3 else self.full
        w = [total(xr * xr * rho), total(yr * yr * rho), total(z2 * rho)]
        pot = total(self.potential(t) * rho)
        F2 = Fz * Fz + Fp.real ** 2 + Fp.imag ** 2
        e_int = total(0.5 * (p["c0"] * rho * rho + p["c1"] * F2 + p["c2"] * (A00.real ** 2 + A00.imag ** 2)))
        rot = -p["omega"].reshape(-1) * lz
        mass = sum(m)
        mag = 2 * (m[0] - m[4]) + m[1] - m[3]
        vec = [mass, kin + pot + rot + e_int + e_soc, mag, lz, kin, pot, rot, e_int, e_soc] + m + w
        return torch.stack([x.reshape(-1).expand(psi.shape[0]) for x in vec], 1)

    def lab(self, psi, t):
        """psi_l(x) = exp(i l omega t) phi_l(R^T x): the rotation as three
        shears, each a Fourier translation of every line (|omega t| < pi/4)."""
        th = self.prm["omega"] * t
        rows, cols = -torch.tan(0.5 * th), torch.sin(th)

        def shear(f, axis, c, other):
            nu, dim = self.nu[axis], -1 - axis
            return torch.fft.ifft(torch.fft.fft(f, dim=dim) * torch.exp(1j * nu * (c * other)), dim=dim)

        out = []
        for k, f in enumerate(psi.unbind(1)):
            f = shear(f, 0, rows, self.X[1])
            f = shear(f, 1, cols, self.X[0])
            f = shear(f, 0, rows, self.X[1])
            out.append(torch.exp(1j * (2 - k) * th) * f)
        return torch.stack(out, 1)


def _prm(sets, d, grad=False):
    """Per-member parameter tensors shaped (batch, 1, ...), and the trap."""
    p = {k: torch.tensor([s[k] for s in sets], device="cuda", dtype=torch.float64)
         .reshape([-1] + [1] * d).requires_grad_(grad) for k in ("omega", "gamma", "c0", "c1", "c2")}
    return p, (sets[0]["gx"], sets[0]["gy"], sets[0]["gz"])


def exact(case, seed):
    T = case["nsteps"] * case["dt"]
    if case["kind"] == "ens":
        gen = torch.Generator().manual_seed(int(seed))
        mem = _members(case)
        src = [_field((m["n"], m["n"]), m["L"], case["init"], gen).to(_dtype(case)) for m in mem]
        outs = [None] * len(mem)
        for side in sorted({m["n"] for m in mem}):
            idx = [i for i, m in enumerate(mem) if m["n"] == side]
            p, trap = _prm([mem[i] for i in idx], 2)
            psi = torch.stack([src[i] for i in idx]).to(torch.complex128)
            res = _Exact((side, side), mem[idx[0]]["L"], p, trap).steps(psi, case["nsteps"], case["dt"], case["scheme"])
            for i, r in zip(idx, res):
                outs[i] = r.reshape(-1)
        return torch.cat(outs)
    grad = case["kind"] == "grad"
    p, trap = _prm([PARAMS[case["prm"]]], len(_n(case)), grad)
    ex = _Exact(_n(case), case["L"], p, trap)
    psi = _states(case, seed).to(torch.complex128).requires_grad_(grad)
    out = ex.steps(psi, case["nsteps"], case["dt"], case["scheme"], grad)
    if case["kind"] == "host":
        return out
    if grad:
        g = _cotangent(case, seed).to(torch.complex128)
        out.backward(g)
        dp = torch.stack([p[k].grad.reshape(-1) for k in ("omega", "gamma", "c0", "c1", "c2")], 1)
        return {"psi": out.detach(), "g0": psi.grad, "dprm": dp}
    res = {"psi": out}
    if case["obs"]:
        res["obs"] = ex.observables(out, T)
    if case["lab"]:
        res["lab"] = ex.lab(out, T)
    return res
