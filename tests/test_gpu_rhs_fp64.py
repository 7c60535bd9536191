"""The FP64 stencil that computes each face once, against the oracle and against
the per-cell kernel (launch code 16): tiles narrower than, as wide as and wider
than the row; rows of tiles; chunks of one and more planes; slip walls; x/z
diffusion explicit and implicit."""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import pnp_oracle as o
from tests import seeded

pytestmark = pytest.mark.gpu
H = ("Hu", "Hv", "Hw", "Hcp", "Hcm")


@pytest.mark.parametrize("af", [False, True])
@pytest.mark.parametrize("nx,ny,nz", [(32, 3, 4), (32, 10, 8), (64, 12, 4), (64, 34, 16), (128, 9, 4), (256, 6, 8),
                                      (128, 40, 64)])
def test_faces_computed_once_match_the_oracle(nx, ny, nz, af):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(nx, ny, nz, 2 * math.pi, math.pi, stretch=1.5)
    prm = o.Params(Re=50.0, lam=0.3, Sc=1.0, V=1.0, beta=0.5, af=af)
    st = o.initial_state(g, prm, o.IC_PB, seed=3, amp=0.2)
    shp = (g.nyc, nz, nx)
    st.cp = st.cp * seeded.positive_field(4, shp, 0.8, 1.2)
    st.cm = st.cm * seeded.positive_field(5, shp, 0.8, 1.2)
    st.Phi = o.potential_from_ions(g, prm, st.cp, st.cm)
    st.p = seeded.field(6, shp, 0.1)
    s = Solver(nx, ny, nz, g.Lx, g.Lz, y_faces=g.yf)
    if af:
        B.check(B.pnp_set_scheme(s.ctx, B.PNP_SCHEME_AF), "pnp_set_scheme")
    s.set_params(prm.Re, prm.lam, prm.Sc, prm.V, prm.beta, prm.Uw)
    out = {}
    for code in (32, 16):
        B.check(B.pnp_set_launch_config(s.ctx, (C.c_int * 4)(code, 128, 64, 32)), "pnp_set_launch_config")
        s.set_state(st)
        s.step(2, 1e-3)
        out[code] = {n: s.get(n) for n in ("u", "v", "w", "p", "cp", "cm", "Phi") + H}
    ref = o.step(g, prm, st, 1e-3, 2)
    for n, a in out[32].items():
        scale = np.max(np.abs(getattr(ref, n))) + 1e-300
        assert np.max(np.abs(a - getattr(ref, n))) <= 1e-10 * scale, n
        assert np.max(np.abs(a - out[16][n])) <= 1e-11 * scale, n
    s.close()


def test_slip_walls_agree_with_the_per_cell_kernel():
    import torch

    from paper_1701_02005_gb300 import binding as B, wallmodel as wm
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(64, 17, 8, 2 * math.pi, math.pi, stretch=1.5)
    prm = o.Params(Re=50.0, lam=0.3, Sc=1.0, V=1.0, beta=0.5)
    st = o.initial_state(g, prm, o.IC_PB, seed=3, amp=0.2)
    s = Solver(g.nx, g.ny, g.nz, g.Lx, g.Lz, y_faces=g.yf)
    s.set_params(prm.Re, prm.lam, prm.Sc, prm.V, prm.beta, prm.Uw)
    out = {}
    for code in (32, 16):
        B.check(B.pnp_set_launch_config(s.ctx, (C.c_int * 4)(code, 128, 64, 32)), "pnp_set_launch_config")
        s.set_state(st)
        X = wm.features(s, 8)
        Y = torch.from_numpy(1.0 + seeded.field(7, (X.shape[0], 5), 0.2)).float().cuda()
        wm.set_slip(s, X, Y)
        s.step(1, 1e-3)
        out[code] = {n: s.get(n) for n in ("u", "w") + H}
    for n, a in out[32].items():
        assert np.max(np.abs(a - out[16][n])) <= 1e-11 * (np.max(np.abs(a)) + 1e-300), n
    s.close()
