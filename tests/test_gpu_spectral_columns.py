"""The spectral y-solves with the columns in shared memory and streamed: the same
bits, at every remainder of the sweeps' batches of four and eight rows, from the
fewest rows of a sweep, and around the most shared memory without and with opt-in."""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import pnp_oracle as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [3, 4, 5, 6, 7, 8, 9, *range(16, 36), 65, 130, 185, 186, 187, 188, 878, 879, 880])
def test_columns_in_shared_memory_equal_streamed_ones(ny):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(16, ny, 16, 2 * math.pi, math.pi, stretch=1.5)
    out = []
    for code in (16, 32):
        s = Solver(g.nx, g.ny, g.nz, g.Lx, g.Lz, precision=B.PNP_MIXED, y_faces=g.yf)
        s.set_params(300.0, 0.3, 1.0, 1.0, 0.5)
        B.check(B.pnp_set_launch_config(s.ctx, (C.c_int * 4)(16, 128, code, 32)), "pnp_set_launch_config")
        s.init_state(B.PNP_IC_PB, 25, 0.1)
        s.step(2, 1e-3)
        out.append({n: s.get(n) for n in ("u", "v", "w", "p", "cp", "cm", "Phi")})
        assert s.status() == 0
        s.close()
    for n, a in out[0].items():
        assert np.isfinite(a).all() and np.array_equal(a, out[1][n]), n
