"""The twisted spectral y-solves against the oracle's one-sided elimination: the
fewest rows, odd and even numbers of them around the batch of four, and columns
streamed or held in shared memory."""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import pnp_oracle as o
from tests import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [3, 4, 5, 6, 9, 10, 18, 35])
def test_fp64_solve_matches_the_oracle(ny):
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(16, ny, 4, 2 * math.pi, math.pi, stretch=1.5)
    rhs = seeded.field(ny, (g.nyc, g.nz, g.nx), 1.0)
    s = Solver(g.nx, g.ny, g.nz, g.Lx, g.Lz, y_faces=g.yf)
    for bc, name in ((0, o.NEUMANN), (1, o.DIRICHLET)):
        x, ref = s.poisson(rhs, bc), o.poisson_solve(g, rhs, name)
        assert np.max(np.abs(x - ref)) <= 1e-11 * np.max(np.abs(ref)), bc
    s.close()


@pytest.mark.parametrize("ny,code", [(3, 16), (3, 32), (4, 16), (4, 32), (10, 16), (10, 32), (35, 16), (35, 32),
                                     (500, 16), (500, 32), (700, 64)])
def test_mixed_step_matches_the_oracle(ny, code):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(16, ny, 8, 2 * math.pi, math.pi, stretch=1.5)
    prm = o.Params(Re=300.0, lam=0.3 if ny < 8 else 0.05, Sc=1.0, V=1.0, beta=0.5)
    st = o.initial_state(g, prm, o.IC_PB, seed=25, amp=0.1)
    s = Solver(g.nx, g.ny, g.nz, g.Lx, g.Lz, precision=B.PNP_MIXED, y_faces=g.yf)
    s.set_params(prm.Re, prm.lam, prm.Sc, prm.V, prm.beta, prm.Uw)
    B.check(B.pnp_set_launch_config(s.ctx, (C.c_int * 4)(16, 128, code, 32)), "pnp_set_launch_config")
    s.set_state(st)
    s.step(2, 1e-3)
    ref = o.step(g, prm, st, 1e-3, 2)
    for name in ("u", "v", "w", "cp", "cm", "Phi"):
        b = getattr(ref, name)
        scale = max(np.max(np.abs(b)), 1.0 if name in ("u", "v", "w") else 1e-300)
        assert np.max(np.abs(s.get(name) - b)) <= 1e-5 * scale, name
    assert s.status() == 0
    s.close()
