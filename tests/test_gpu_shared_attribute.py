"""Contexts on different grids side by side: the opt-in shared memory of a kernel is
one attribute for the whole process, so a small grid's launches must not take from a
large grid's what it needs."""
import math
import threading

import numpy as np
import pytest

from oracle import pnp_oracle as o

pytestmark = pytest.mark.gpu


def _mixed(ny):
    from paper_1701_02005_gb300 import binding as B
    from paper_1701_02005_gb300.solver import Solver

    s = Solver(16, ny, 16, 2 * math.pi, math.pi, precision=B.PNP_MIXED,
               y_faces=o.Grid(16, ny, 16, 2 * math.pi, math.pi, stretch=1.5).yf)
    s.set_params(300.0, 0.3, 1.0, 1.0, 0.5)
    s.init_state(B.PNP_IC_PB, 25, 0.1)
    return s


def test_uneven_columns_in_several_threads():
    # columns of 186 and of 213 rows: 48 and 55 KB; a new step size captures the step again
    errors = []

    def work(ny):
        try:
            s = _mixed(ny)
            for n in range(400):
                s.step(1, 1e-3 * (1 + n % 2))
            assert s.status() == 0
            s.close()
        except Exception as e:   # noqa: BLE001: reported by the test's own thread
            errors.append((ny, e))

    ts = [threading.Thread(target=work, args=(ny,)) for ny in (187, 214) * 3]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def test_ensemble_of_uneven_columns_equals_the_cases_alone():
    from paper_1701_02005_gb300.ensemble import Ensemble

    sizes = (400, 214, 187, 33)
    cases = [_mixed(ny) for ny in sizes]
    e = Ensemble(cases)
    e.step(3, [1e-3] * len(cases))
    e.synchronize()
    for ny, s in zip(sizes, cases):
        alone = _mixed(ny)
        alone.step(3, 1e-3)
        for f in ("u", "v", "w", "p", "cp", "cm", "Phi"):
            assert np.array_equal(s.get(f), alone.get(f)), (ny, f)
        alone.close()
    e.close()
    for s in cases:
        s.close()
