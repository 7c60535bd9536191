"""FP64 transforms whose columns are packed over the planes: every register length of
the z-transform, with numbers of columns that end a plane, a block and the last block
at every remainder, against the oracle."""
import math

import numpy as np
import pytest

from oracle import pnp_oracle as o
from tests import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [16, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("nx,ny", [(4, 3), (16, 5), (32, 33), (64, 16), (128, 7)])
def test_poisson_matches_the_oracle(nx, ny, nz):
    from paper_1701_02005_gb300.solver import Solver

    g = o.Grid(nx, ny, nz, 2 * math.pi, math.pi, stretch=1.5)
    rhs = seeded.field(nx + nz, (g.nyc, g.nz, g.nx), 1.0)
    s = Solver(g.nx, g.ny, g.nz, g.Lx, g.Lz, y_faces=g.yf)
    for bc, name in ((0, o.NEUMANN), (1, o.DIRICHLET)):
        x, ref = s.poisson(rhs, bc), o.poisson_solve(g, rhs, name)
        assert np.max(np.abs(x - ref)) <= 1e-11 * np.max(np.abs(ref)), bc
    s.close()
