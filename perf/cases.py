"""The work a user of this package has it do, as measurable cases.

Five kinds, all through the public entry points (``solver.Solver``,
``ensemble.Ensemble``, ``wallmodel`` and the C ABI in ``binding``):

* ``step``: a block of time steps of one case, then the fields on the device, as
  a run between two snapshots;
* ``ensemble``: steps of several uneven cases, one graph launch per step;
* ``poisson``: the separable Poisson solve on device arrays;
* ``infer`` / ``gradient``: the wall model's network;
* ``coupled``: a coarse run stepped with the wall model.

Snapshots of a mixed-precision run are kept in FP32, its working precision, and
leave out the pressure: it is the divergence of FP32 velocities over the time
step, solved, so that two orders of the same sums differ by 1e-4 of it while the
velocities that it corrects agree to 1e-6.
"""
import math

import numpy as np
import torch

LX, LZ = 2 * math.pi, math.pi
FIELDS = ("u", "v", "w", "p", "cp", "cm", "Phi")
WIDTHS = (40, 128, 128, 128, 128, 5)          # the wall model's layers


def _step(name, nx, ny, nz, precision, steps, Re, lam, V, stretch, scheme="cn"):
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
            "Re": Re, "lam": lam, "V": V, "stretch": stretch, "scheme": scheme}


def listed():
    return [
        # the validation run (32x33x32, FP64): the smallest grid a user steps, bound by launches and latency
        _step("fp64_32x33x32", 32, 33, 32, "fp64", 20, 400.0, 0.05, 2.0, 2.0),
        # an all-FP64 run at the ensemble's larger grid: the reference side of a precision comparison
        _step("fp64_128x97x128", 128, 97, 128, "fp64", 2, 3000.0, 0.0158, 2.0, 2.5),
        # one case of the drag-against-voltage sweep: thousands of short steps on a small grid
        _step("mixed_64x65x64", 64, 65, 64, "mixed", 20, 3000.0, 0.0158, 2.0, 2.0),
        # the benchmark: turbulent Couette flow at 256x193x256
        _step("mixed_256x193x256", 256, 193, 256, "mixed", 5, 3000.0, 0.01, 2.0, 2.5),
        # the large single case
        _step("mixed_1024x385x512", 1024, 385, 512, "mixed", 1, 1.0e4, 0.005, 5.0, 3.0),
        # the approximately factorised scheme on a grid with an odd number of cells in y
        _step("af_256x150x128", 256, 150, 128, "mixed", 5, 3000.0, 0.01, 2.0, 2.5, scheme="af"),
        # a parameter sweep of uneven cases (four of each grid of the 48-case ensemble)
        {"name": "ensemble_8", "kind": "ensemble", "small": 4, "large": 4, "steps": 5},
        # a coarse run with the wall model in the loop, as the learned double layer is used
        {"name": "coupled_128x49x128", "kind": "coupled", "nx": 128, "ny": 49, "nz": 128, "steps": 5},
        # the network's outputs for all wall columns of that coarse grid
        {"name": "infer_32768", "kind": "infer", "rows": 32768},
        # one training batch
        {"name": "gradient_65536", "kind": "gradient", "rows": 65536},
        # a potential solve as a caller of the C ABI has it, at the benchmark's grid and at the smallest one
        {"name": "poisson_256x193x256", "kind": "poisson", "nx": 256, "ny": 193, "nz": 256, "bc": "dirichlet"},
        {"name": "poisson_32x33x32", "kind": "poisson", "nx": 32, "ny": 33, "nz": 32, "bc": "neumann"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("step", "ensemble", "poisson", "infer", "gradient", "coupled"), (50, 8, 12, 12, 12, 6))[0]
    if kind == "step":
        precision = rng.choices(("mixed", "fp64"), (70, 30))[0]
        most = 16.0e6 if precision == "mixed" else 2.0e6
        while True:
            nx, nz, ny = 2 ** rng.randint(4, 9), 2 ** rng.randint(4, 9), _log_int(rng, 17, 257)
            if nx * ny * nz <= most:
                break
        steps = max(1, min(20, int(4.0e7 / (nx * ny * nz) / (1 if precision == "mixed" else 12))))
        return {"kind": "step", "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
                "Re": rng.choice((400.0, 1000.0, 3000.0)), "lam": rng.choice((0.01, 0.0158, 0.05)),
                "V": rng.choice((0.5, 1.0, 2.0)), "stretch": rng.choice((1.5, 2.0, 2.5)),
                "scheme": rng.choices(("cn", "af"), (80, 20))[0]}
    if kind == "ensemble":
        return {"kind": "ensemble", "small": rng.randint(1, 6), "large": rng.randint(0, 3), "steps": rng.randint(2, 8)}
    if kind == "poisson":
        while True:
            nx, nz, ny = 2 ** rng.randint(4, 9), 2 ** rng.randint(4, 9), _log_int(rng, 9, 385)
            if nx * ny * nz <= 32.0e6:
                break
        return {"kind": "poisson", "nx": nx, "ny": ny, "nz": nz, "bc": rng.choice(("neumann", "dirichlet"))}
    if kind == "coupled":
        return {"kind": "coupled", "nx": 2 ** rng.randint(4, 7), "ny": rng.randint(17, 65), "nz": 2 ** rng.randint(4, 7),
                "steps": rng.randint(1, 10)}
    return {"kind": kind, "rows": _log_int(rng, 100, 131072)}


# ---- grids, parameters and time steps ------------------------------------------------------------------------------
def _bulk(lam, V):
    """Bulk concentration left by two Gouy-Chapman layers formed from c = 1."""
    b = 2.0 * lam * (math.cosh(0.5 * V) - 1.0)
    return (0.5 * (-b + math.sqrt(b * b + 4.0))) ** 2


def _dt(c):
    """A time step inside the explicit limits: advection (wall speed 1 along x, fluctuations of 0.3 across), x/z
    diffusion, ion drift across the wall cell and dielectric relaxation."""
    dx, dz, Re, lam, V, ny = LX / c["nx"], LZ / c["nz"], c["Re"], c["lam"], c["V"], c["ny"]
    cb, D, th = _bulk(lam, V), 1.0 / Re, math.tanh(c["stretch"])
    dy0 = 1.0 - math.tanh(c["stretch"] * (1.0 - 2.0 / (ny - 1))) / th
    dym = math.tanh(c["stretch"] * 2.0 / (ny - 1)) / th
    return min(0.25 * dx, 0.25 * min(dz, dym) / 0.3, 0.2 / (D * (1.0 / dx ** 2 + 1.0 / dz ** 2)),
               1.0 / (D * cb * (math.exp(V) + math.exp(-V)) / (2.0 * lam * lam)),
               0.25 * dy0 / (D * 2.0 * math.sqrt(cb) * math.sinh(0.5 * V) / lam))


def _members(case):
    """The cases of an ensemble: Re x Debye length x wall potential on its two grids."""
    got = []
    for n in range(case["small"] + case["large"]):
        large = n >= case["small"]
        got.append({"nx": 128 if large else 64, "ny": 97 if large else 65, "nz": 128 if large else 64,
                    "precision": "mixed", "steps": case["steps"], "Re": (1000.0, 3000.0)[n % 2],
                    "lam": (0.05, 0.0158)[n // 2 % 2], "V": (0.5, 2.0, 1.0)[n % 3], "stretch": 2.0, "scheme": "cn"})
    return got


def _coupled_member(case):
    return {"nx": case["nx"], "ny": case["ny"], "nz": case["nz"], "precision": "mixed", "steps": case["steps"],
            "Re": 3000.0, "lam": 0.0158, "V": 2.0, "stretch": 2.0, "scheme": "cn"}


def _solver(c, seed):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    s = Solver(c["nx"], c["ny"], c["nz"], LX, LZ, stretch=c["stretch"],
               precision=B.PNP_MIXED if c["precision"] == "mixed" else B.PNP_FP64)
    if c["scheme"] == "af":
        B.check(B.pnp_set_scheme(s.ctx, B.PNP_SCHEME_AF), "pnp_set_scheme")
    s.set_params(c["Re"], c["lam"], 1.0, c["V"], 0.5)
    s.init_state(B.PNP_IC_PB, seed, 0.1)
    return s


def _kept(single):
    return [f for f in FIELDS if not (single and f == "p")]


def _buffers(s, single):
    return {f: torch.empty(s.shape(f), dtype=torch.float64, device=s.device) for f in _kept(single)}


def _snapshot(s, buf, single):
    """The fields on the device, ordered before torch's own work."""
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import FIELD_NAMES

    out = {}
    with torch.cuda.stream(s.stream):
        for f, t in buf.items():
            B.check(B.pnp_get_state(s.ctx, FIELD_NAMES[f], t.data_ptr(), 1), "pnp_get_state")
            out[f] = t.float() if single else t
    torch.cuda.current_stream(s.device).wait_stream(s.stream)
    return out


# ---- the network ---------------------------------------------------------------------------------------------------
def _network_data(rows, seed):
    """Weights, normalisation, feature rows and labels of a network in use: near-wall features with their own means
    and spreads, labels that depend on them smoothly plus scatter (NumPy, from the seed)."""
    g = np.random.default_rng(seed)
    p = []
    for k, n in zip(WIDTHS[:-1], WIDTHS[1:]):
        a = math.sqrt(6.0 / k)
        p += [g.uniform(-a, a, n * k), 0.1 * g.standard_normal(n)]
    p = np.concatenate(p).astype(np.float32)
    y = (np.arange(8) + 0.5) * 0.01
    shift = np.concatenate([y, 0 * y, 1 + np.exp(-y / 0.02), 1 - 0.5 * np.exp(-y / 0.02), np.exp(-y / 0.02)])
    spread = np.concatenate([0.3 * y, 0.3 * y, 0.2 * np.exp(-y / 0.02), 0.1 * np.exp(-y / 0.02), 0.1 * np.exp(-y / 0.02)])
    shift, scale = shift.astype(np.float32), (1.0 / spread).astype(np.float32)
    out_shift = np.array([1.0, 0.0, 0.05, 0.0, 0.0], dtype=np.float32)
    out_scale = np.array([4.0, 4.0, 50.0, 500.0, 500.0], dtype=np.float32)
    gen = torch.Generator(device="cpu").manual_seed(seed)
    z = torch.randn((rows, WIDTHS[0]), generator=gen, dtype=torch.float32)
    X = z * torch.from_numpy(1.0 / scale) + torch.from_numpy(shift)
    n = torch.tanh(z[:, 0:40:8] + 0.5 * z[:, 1:40:8]) + 0.3 * torch.randn((rows, 5), generator=gen)
    T = n / torch.from_numpy(out_scale) + torch.from_numpy(out_shift)
    return p, (shift, scale, out_shift, out_scale), X, T


def _network(rows, p, norm):
    from paper_1701_02005_gb300 import wallmodel as wm

    m = wm.MLP(rows)
    m.set_params(p)
    m.set_normalization(*norm)
    return m


def _network_exact(p, norm, X, grad=False, T=None):
    """The network (or its loss and gradient) in FP64."""
    dev = X.device
    q = torch.from_numpy(p).to(dev).double().requires_grad_(grad)
    si, ci, so, co = (torch.from_numpy(a).to(dev).double() for a in norm)
    with torch.set_grad_enabled(grad):
        a, off = (X.double() - si) * ci, 0
        for l, (k, n) in enumerate(zip(WIDTHS[:-1], WIDTHS[1:])):
            a = a @ q[off:off + n * k].view(n, k).T + q[off + n * k:off + n * k + n]
            off += n * k + n
            if l < len(WIDTHS) - 2:
                a = torch.nn.functional.gelu(a)
        if not grad:
            return a.clamp(-6.0, 6.0) / co + so
        loss = (a - (T.double() - so) * co).square().mean()
        loss.backward()
    return q.grad, loss.detach()


# ---- the cases' states and passes ----------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        s = _solver(case, seed)
        return {"case": case, "s": s, "dt": _dt(case), "buf": _buffers(s, case["precision"] == "mixed")}
    if kind == "ensemble":
        from paper_1701_02005_gb300.ensemble import Ensemble

        members = _members(case)
        solvers = [_solver(c, seed + 7919 * n) for n, c in enumerate(members)]
        dts = [_dt(c) for c in members]
        return {"case": case, "e": Ensemble(solvers), "s": solvers, "dts": dts,
                "buf": [_buffers(s, True) for s in solvers]}
    if kind == "poisson":
        from paper_1701_02005_gb300 import binding as B
        from paper_1701_02005_gb300.solver import Solver

        s = Solver(case["nx"], case["ny"], case["nz"], LX, LZ, stretch=2.0, precision=B.PNP_FP64)
        rhs = _poisson_rhs(case, seed)
        s.stream.wait_stream(torch.cuda.current_stream())
        return {"case": case, "s": s, "rhs": rhs, "x": torch.empty_like(rhs),
                "bc": B.PNP_NEUMANN if case["bc"] == "neumann" else B.PNP_DIRICHLET}
    if kind == "coupled":
        from paper_1701_02005_gb300 import wallmodel as wm

        c = _coupled_member(case)
        s = _solver(c, seed)
        p, _, _, _ = _network_data(16, seed)
        # normalisation from the run's own features; outputs near the laminar wall values
        X = wm.features(s).double()
        sd = torch.maximum(X.std(0), 1e-2 * X.mean(0).abs().clamp(min=1e-2))
        out = (np.array([1.0, 0.0, 0.0, 0.0, 0.0]), np.array([10.0, 10.0, 100.0, 1e4, 1e4]))
        m = _network(X.shape[0], p, (X.mean(0).cpu().numpy(), (1.0 / sd).cpu().numpy(), *out))
        m.set_skip(*wm.PHI_SKIP)
        wm.set_coupling(s, 2, 0.3, 0.3, 0.3)
        return {"case": case, "s": s, "m": m, "dt": _dt(c), "buf": _buffers(s, True)}
    p, norm, X, T = _network_data(case["rows"], seed)
    return {"case": case, "m": _network(case["rows"], p, norm), "X": X.cuda(), "T": T.cuda()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        state["s"].step(case["steps"], state["dt"])
        return _snapshot(state["s"], state["buf"], case["precision"] == "mixed")
    if kind == "ensemble":
        state["e"].step(case["steps"], state["dts"])
        return [_snapshot(s, b, True) for s, b in zip(state["s"], state["buf"])]
    if kind == "poisson":
        from paper_1701_02005_gb300 import binding as B

        s = state["s"]
        B.check(B.pnp_poisson(s.ctx, state["bc"], state["rhs"].data_ptr(), state["x"].data_ptr()), "pnp_poisson")
        torch.cuda.current_stream(s.device).wait_stream(s.stream)
        return state["x"]
    if kind == "coupled":
        from paper_1701_02005_gb300 import wallmodel as wm

        wm.step_with_model(state["s"], state["m"], case["steps"], state["dt"])
        return _snapshot(state["s"], state["buf"], True)
    if kind == "infer":
        return state["m"].forward(state["X"])
    g, loss = state["m"].gradient(state["X"], state["T"])
    return {"gradient": g, "loss": np.float32(loss)}


# ---- bytes and operations ------------------------------------------------------------------------------------------
def _step_work(c):
    """Per cell and substage: the state and the stored explicit terms read and written once; the stencil, five y-solves,
    two Poisson solves (forward and inverse transforms of half-length spectra, one y-solve) and the projection."""
    cells = c["nx"] * (c["ny"] - 1) * c["nz"]
    per = 2 * (7 + 5) * 8 if c["precision"] == "fp64" else 2 * (4 * 4 + 2 * 8 + 4 + 5 * 4)
    flops = 250 + 5 * 6 + 2 * (2 * 2.5 * math.log2(c["nx"] * c["nz"]) + 12) + 12
    return {"bytes": 3.0 * c["steps"] * per * cells, "flops": 3.0 * c["steps"] * flops * cells}


def work(case):
    kind = case["kind"]
    if kind == "step":
        return _step_work(case)
    if kind == "ensemble":
        each = [_step_work(c) for c in _members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "poisson":
        cells = case["nx"] * (case["ny"] - 1) * case["nz"]
        return {"bytes": 16.0 * cells, "flops": cells * (2 * 2.5 * math.log2(case["nx"] * case["nz"]) + 12)}
    params = sum(k * n + n for k, n in zip(WIDTHS[:-1], WIDTHS[1:]))
    if kind == "coupled":
        w, rows = _step_work(_coupled_member(case)), 2 * case["nx"] * case["nz"]
        return {"bytes": w["bytes"] + case["steps"] * 4.0 * rows * 45, "flops": w["flops"] + case["steps"] * 2.0 * rows * params}
    if kind == "infer":
        return {"bytes": 4.0 * (case["rows"] * 45 + params), "flops": 2.0 * case["rows"] * params}
    return {"bytes": 4.0 * (case["rows"] * 45 + 2 * params), "flops": 6.0 * case["rows"] * params}


# ---- the same in 64 bits, in plain torch ---------------------------------------------------------------------------
def _poisson_rhs(case, seed):
    """A charge-like source: smooth waves along the walls, layers at them, and noise (device, FP64)."""
    nyc, nz, nx = case["ny"] - 1, case["nz"], case["nx"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    y = torch.linspace(-1.0, 1.0, nyc, dtype=torch.float64, device="cuda")[:, None, None]
    z = torch.arange(nz, dtype=torch.float64, device="cuda")[None, :, None] * (2 * math.pi / nz)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, None, :] * (2 * math.pi / nx)
    r = torch.exp(-(1.0 - y.abs()) / 0.1) * torch.sign(y) * (1.0 + 0.3 * torch.sin(x + (seed % 7)) * torch.cos(2 * z))
    return r + 0.1 * torch.randn((nyc, nz, nx), dtype=torch.float64, device="cuda", generator=gen)


class _Grid:
    def __init__(self, c, stretch, dev):
        self.nx, self.ny, self.nz, self.dev = c["nx"], c["ny"], c["nz"], dev
        s = np.arange(self.ny) * 2.0 / (self.ny - 1) - 1.0
        yf = s if stretch == 0.0 else np.tanh(stretch * s) / math.tanh(stretch)
        yf[0], yf[-1] = -1.0, 1.0
        self.yf, self.dy, self.yc = yf, yf[1:] - yf[:-1], 0.5 * (yf[1:] + yf[:-1])
        self.h = np.concatenate([[0.5 * self.dy[0]], self.yc[1:] - self.yc[:-1], [0.5 * self.dy[-1]]])
        self.dx, self.dz = LX / self.nx, LZ / self.nz
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)[:, None, None]  # noqa: E731
        self.Yf, self.Yc, self.Dy, self.H = t(yf), t(self.yc), t(self.dy), t(self.h)
        m, n = np.arange(self.nx // 2 + 1), np.arange(self.nz)
        kx2 = torch.as_tensor((2 - 2 * np.cos(2 * np.pi * m / self.nx)) / self.dx ** 2, device=dev)
        kz2 = torch.as_tensor((2 - 2 * np.cos(2 * np.pi * n / self.nz)) / self.dz ** 2, device=dev)
        self.kx2, self.kz2 = kx2[None, :], kz2[:, None]

    def cells(self, dirichlet):
        """(L q)_j on the cells as a dense matrix: wall value on the wall face, or no wall flux."""
        n = self.ny - 1
        lo, hi = 1.0 / (self.h[:-1] * self.dy), 1.0 / (self.h[1:] * self.dy)
        b = -lo - hi
        if not dirichlet:
            b[0] += lo[0]
            b[-1] += hi[-1]
        return np.diag(b) + np.diag(lo[1:], -1) + np.diag(hi[:-1], 1) if n > 1 else np.diag(b)

    def faces(self):
        """(L v)_j on the interior faces."""
        lo, hi = 1.0 / (self.dy[:-1] * self.h[1:-1]), 1.0 / (self.dy[1:] * self.h[1:-1])
        return np.diag(-lo - hi) + np.diag(lo[1:], -1) + np.diag(hi[:-1], 1)

    def solve(self, rhs, neumann):
        """(d_xx + d_zz + L_y) x = rhs; the constant mode of the Neumann problem is zero in its bottom cell."""
        L = self.cells(not neumann)
        a, b, c = np.diag(L, -1), np.diag(L), np.diag(L, 1)
        r, k2, n = torch.fft.rfft2(rhs), self.kx2 + self.kz2, self.ny - 1
        del rhs
        fac = torch.empty((n, self.nz, self.nx // 2 + 1), dtype=torch.float64, device=self.dev)
        for j in range(n):
            piv = b[j] - k2
            if j:
                piv = piv - a[j - 1] * fac[j - 1]
            if neumann and j == 0:
                piv[0, 0] = 1.0
                r[0, 0, 0] = 0.0
            r[j] = (r[j] - a[j - 1] * r[j - 1] if j else r[j]) / piv
            if j < n - 1:
                fac[j] = c[j] / piv
                if neumann and j == 0:
                    fac[0, 0, 0] = 0.0
        for j in range(n - 2, -1, -1):
            r[j] -= fac[j] * r[j + 1]
        return torch.fft.irfft2(r, s=(self.nz, self.nx))


def _xm(a):
    return a.roll(1, 2)


def _xp(a):
    return a.roll(-1, 2)


def _zm(a):
    return a.roll(1, 1)


def _zp(a):
    return a.roll(-1, 1)


def _walls(a):
    """Values on the interior faces with zero wall faces around them."""
    return torch.nn.functional.pad(a, (0, 0, 0, 0, 1, 1))


def _noise(seed, field, shape, dev):
    """Counter-based uniform numbers in [-1, 1): SplitMix64 of counter field 2^40 + index."""
    wrap = lambda v: (v & (2 ** 64 - 1)) - (2 ** 64 if v & 2 ** 63 else 0)  # noqa: E731
    shr = lambda t, k: (t >> k) & (2 ** (64 - k) - 1)  # noqa: E731
    n = math.prod(shape)
    t = torch.arange(1, n + 1, dtype=torch.int64, device=dev) + (field << 40)
    t = t * wrap(0x9E3779B97F4A7C15) + seed
    t = (t ^ shr(t, 30)) * wrap(0xBF58476D1CE4E5B9)
    t = (t ^ shr(t, 27)) * wrap(0x94D049BB133111EB)
    t = t ^ shr(t, 31)
    return (shr(t, 11).double() * 2.0 ** -52 - 1.0).view(shape)


def _divergence(g, u, v, w):
    return (_xp(u) - u) / g.dx + (v[1:] - v[:-1]) / g.Dy + (_zp(w) - w) / g.dz


def _project(g, u, v, w, scale):
    ph = g.solve(_divergence(g, u, v, w) / scale, True)
    v = v.clone()
    v[1:-1] -= scale * (ph[1:] - ph[:-1]) / g.H[1:-1]
    return u - scale * (ph - _xm(ph)) / g.dx, v, w - scale * (ph - _zm(ph)) / g.dz, ph


def _explicit(g, c, q, xz):
    """Advection, x/z diffusion (where explicit), Coulomb force and ion migration of the state q."""
    u, v, w, cp, cm, Phi = (q[f] for f in ("u", "v", "w", "cp", "cm", "Phi"))
    nu = D = 1.0 / c["Re"]
    K = 0.5 / (2.0 * c["Re"] ** 2 * c["lam"] ** 2)
    lap = lambda a: (_xp(a) - 2 * a + _xm(a)) / g.dx ** 2 + (_zp(a) - 2 * a + _zm(a)) / g.dz ** 2  # noqa: E731
    rho, hi = cp - cm, g.H[1:-1]
    gx, gz, gy = (Phi - _xm(Phi)) / g.dx, (Phi - _zm(Phi)) / g.dz, (Phi[1:] - Phi[:-1]) / hi
    vi, up = v[1:-1], lambda a: 0.5 * (a[1:] + a[:-1])  # noqa: E731
    H = {}
    f = 0.5 * (u + _xp(u))
    f = f * f
    H["u"] = -(f - _xm(f)) / g.dx
    f = _walls(0.5 * (_xm(vi) + vi) * up(u))
    H["u"] -= (f[1:] - f[:-1]) / g.Dy
    f = 0.5 * (_xm(w) + w) * 0.5 * (_zm(u) + u)
    H["u"] -= (_zp(f) - f) / g.dz + K * 0.5 * (_xm(rho) + rho) * gx
    f = 0.5 * (w + _zp(w))
    f = f * f
    H["w"] = -(f - _zm(f)) / g.dz
    f = _walls(0.5 * (_zm(vi) + vi) * up(w))
    H["w"] -= (f[1:] - f[:-1]) / g.Dy
    f = 0.5 * (_zm(u) + u) * 0.5 * (_xm(w) + w)
    H["w"] -= (_xp(f) - f) / g.dx + K * 0.5 * (_zm(rho) + rho) * gz
    mean = lambda a: (g.Dy[:-1] * a[:-1] + g.Dy[1:] * a[1:]) / (2.0 * hi)  # noqa: E731
    f = mean(u) * 0.5 * (_xm(vi) + vi)
    Hv = -(_xp(f) - f) / g.dx
    f = mean(w) * 0.5 * (_zm(vi) + vi)
    Hv -= (_zp(f) - f) / g.dz
    f = up(v)
    f = f * f
    Hv -= (f[1:] - f[:-1]) / hi + K * up(rho) * gy
    if xz:
        H["u"] += nu * lap(u)
        H["w"] += nu * lap(w)
        Hv += nu * lap(vi)
    H["v"] = Hv
    for name, a, s in (("cp", cp, 1.0), ("cm", cm, -1.0)):
        f = 0.5 * (_xm(a) + a) * (u - s * D * gx)
        if xz:
            f -= D * (a - _xm(a)) / g.dx
        h = -(_xp(f) - f) / g.dx
        f = 0.5 * (_zm(a) + a) * (w - s * D * gz)
        if xz:
            f -= D * (a - _zm(a)) / g.dz
        h -= (_zp(f) - f) / g.dz
        f = _walls(up(a) * (vi - s * D * gy))
        H[name] = h - (f[1:] - f[:-1]) / g.Dy
    return H


def _exact_steps(c, seed, dev):
    """The member case's fields after its steps: the scheme of the library, restated in FP64."""
    g = _Grid(c, c["stretch"], dev)
    shp, nu, V, af = (g.ny - 1, g.nz, g.nx), 1.0 / c["Re"], c["V"], c["scheme"] == "af"
    dt = _dt(c)
    u = g.Yc + 0.1 * (1 - g.Yc ** 2) * _noise(seed, 0, shp, dev)
    v = 0.1 * (1 - g.Yf ** 2) * _noise(seed, 1, (g.ny, g.nz, g.nx), dev)
    w = 0.1 * (1 - g.Yc ** 2) * _noise(seed, 2, shp, dev)
    u, v, w, ph = _project(g, u, v, w, 1.0)
    cb, t = _bulk(c["lam"], V), math.tanh(0.25 * V)
    kap = math.sqrt(cb) / c["lam"]
    lay = 4 * torch.atanh(t * torch.exp(-(1 - g.Yc) * kap)) - 4 * torch.atanh(t * torch.exp(-(1 + g.Yc) * kap))
    one = torch.ones_like(u)
    q = {"u": u, "v": v, "w": w, "p": torch.zeros_like(u), "cp": cb * torch.exp(-lay) * one, "cm": cb * torch.exp(lay) * one}
    del u, v, w, ph, one

    def potential():
        return V * g.Yc + g.solve(-(q["cp"] - q["cm"]) / (2.0 * c["lam"] ** 2), False)

    def apply(L, a):
        """L a for tridiagonal L along y."""
        L = [torch.as_tensor(np.diag(L, k).copy(), device=dev)[:, None, None] for k in (-1, 0, 1)]
        out = L[1] * a
        out[1:] += L[0] * a[:-1]
        out[:-1] += L[2] * a[1:]
        return out

    q["Phi"] = potential()
    Lw, Lf, Ln, old = g.cells(True), g.faces(), g.cells(False), None
    for n in range(3 * c["steps"]):
        gam, zet = ((8 / 15, 0.0), (5 / 12, -17 / 60), (3 / 4, -5 / 12))[n % 3]
        alp = gam + zet
        sub = 0.5 * alp * dt * nu                       # Sc = 1: ions and momentum diffuse alike
        H, p = _explicit(g, c, q, not af), q["p"]
        grad = {"u": (p - _xm(p)) / g.dx, "v": (p[1:] - p[:-1]) / g.H[1:-1], "w": (p - _zm(p)) / g.dz}
        new = {}
        for f, L in (("u", Lw), ("v", Lf), ("w", Lw), ("cp", Ln), ("cm", Ln)):
            a = q[f][1:-1] if f == "v" else q[f]
            r = gam * H[f] + alp * nu * apply(L, a)
            if zet:
                r += zet * old[f]
            if f in grad:
                r -= alp * grad[f]
            if f == "u":                                # the walls move at -1 and +1
                r[0] -= alp * nu / (g.h[0] * g.dy[0])
                r[-1] += alp * nu / (g.h[-1] * g.dy[-1])
            if af:
                r += alp * nu * ((_xp(a) - 2 * a + _xm(a)) / g.dx ** 2 + (_zp(a) - 2 * a + _zm(a)) / g.dz ** 2)
                r = torch.fft.irfft2(torch.fft.rfft2(r) / ((1 + sub * g.kx2) * (1 + sub * g.kz2)), s=(g.nz, g.nx))
            inv = torch.as_tensor(np.linalg.inv(np.eye(len(L)) - sub * L), device=dev)
            r = (inv @ (dt * r).reshape(len(L), -1)).view_as(a)
            new[f] = a + r
        q["cp"], q["cm"], old = new["cp"], new["cm"], H
        q["u"], q["v"], q["w"], ph = _project(g, new["u"], _walls(new["v"]), new["w"], alp * dt)
        q["p"] = p + ph
        q["Phi"] = potential()
    return {f: q[f] for f in _kept(c["precision"] == "mixed")}


def exact(case, seed):
    kind, dev = case["kind"], torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if kind == "step":
        return _exact_steps(case, seed, dev)
    if kind == "ensemble":
        return [_exact_steps(c, seed + 7919 * n, dev) for n, c in enumerate(_members(case))]
    if kind == "poisson":
        return _Grid(case, 2.0, dev).solve(_poisson_rhs(case, seed), case["bc"] == "neumann")
    if kind == "coupled":
        return None   # a BF16 network in the loop: no 64-bit value that the run stands for
    p, norm, X, T = _network_data(case["rows"], seed)
    if kind == "infer":
        return _network_exact(p, norm, X.to(dev))
    g, loss = _network_exact(p, norm, X.to(dev), True, T.to(dev))
    return {"gradient": g, "loss": loss}
