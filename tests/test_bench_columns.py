"""The benchmark's byte model of the mixed y-solves in the form that runs: columns in
shared memory move 32 B per spectral point, streamed ones 64."""
import pytest

import bench


# four blocks on an SM up to 214 rows; beyond, two waves of 152 SMs
@pytest.mark.parametrize("nx,ny,nz,code,columns", [
    (256, 193, 256, 0, True), (256, 193, 256, 64, True), (256, 193, 256, 16, True), (256, 193, 256, 32, False),
    (512, 215, 512, 0, True), (512, 216, 512, 0, False), (128, 385, 128, 0, True), (256, 385, 256, 0, False),
    (1024, 385, 512, 0, False), (1024, 385, 512, 16, True), (16, 879, 16, 0, True), (16, 880, 16, 16, False)])
def test_form_of_the_solves(nx, ny, nz, code, columns):
    assert bench.columns_in_smem(nx, ny, nz, code) is columns


def test_bytes_follow_the_form():
    half = (bench.WL["nx"] // 2 + 1) / bench.WL["nx"]
    for site in ("p_thomas", "e_thomas"):
        assert bench.site_cost(site, "mixed", None, True, True)["bytes"] == 32 * half
        assert bench.site_cost(site, "mixed", None, True, False)["bytes"] == 64 * half


def test_step_traffic_is_quoted_for_the_captured_launches_only():
    ok = bench.step_ncu_launches
    assert ok(None, True, True) and ok([64, 128, 16, 32], True, True) and ok([64, 64, 64, 8], True, True)
    assert not any((ok(None, False, True), ok(None, True, False), ok([32, 64, 16, 32], True, True),
                    ok([64, 32, 16, 32], True, True), ok([64, 64, 16, 64], True, True)))
