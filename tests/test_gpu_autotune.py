"""What the autotuner chooses from: codes that stand for different launches."""
import ctypes as C
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,stencil,spectral", [(0, 64, (16, 32), (64,)), (0, 16, (16, 32), (64,)),
                                                           (1, 64, (16, 32, 64, 128), (16, 32))])
def test_chosen_codes(precision, nx, stencil, spectral):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    s = Solver(nx, 33, 32, 2 * math.pi, math.pi, stretch=2.0, precision=precision)
    s.set_params(1000.0, 0.05, 1.0, 1.0, 0.5)
    cfg, ms = (C.c_int * 4)(), (C.c_double * 4)()
    B.check(B.pnp_autotune(s.ctx, 1e-3, cfg, ms), "pnp_autotune")
    assert cfg[0] in stencil and cfg[2] in spectral and cfg[3] == 32
    assert all(0.0 < m < 1e3 for m in ms)
    got = (C.c_int * 4)()
    B.check(B.pnp_get_launch_config(s.ctx, got), "pnp_get_launch_config")
    assert list(got) == list(cfg)
    s.close()
