"""The potential solve where its V-cycle changes shape: grids whose coarse levels all run in one
kernel from the fine level down, from the first or second coarse level, grids whose one axis runs
out of cells before the other, odd sizes, periodic axes and insulating walls; and far fields and
residuals far outside FP32's range, which the scaled FP32 correction must not notice.
FP64: the stated 1e-13 residual, and the oracle's potential within 1e-11 (the bound of the
solver's parity test).  Mixed: the residual below its tolerance."""
import numpy as np
import pytest

import oracle
from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu

SIZES = [(4, 4, {}), (5, 7, {}), (16, 16, {}), (17, 15, {}), (64, 32, {}), (65, 32, {}), (66, 33, {}), (128, 63, {}),
         (4, 300, {}), (300, 5, {}), (96, 48, dict(mag_bc=1)), (64, 40, dict(periodic_x=1)), (20, 40, dict(periodic_x=1)),
         (90, 31, dict(mag_bc=1)), (31, 10, {})]


@pytest.mark.parametrize("nx,ny,kw", SIZES)
def test_levels_fp64_against_oracle(nx, ny, kw):
    c = I.case(nx, ny, radius=0.35 * min(nx, ny), H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0, **kw)
    ref = oracle.Oracle(c)
    ref.step(1)
    s = lbfs.Solver(precision=lbfs.FP64, max_cases=1)
    s.set_case(0, c)
    st = s.step(1)[0]
    phi = s.field(0, I.PHI)
    s.close()
    assert st["pot_resid"] <= 1e-13 and st["pot_cycles"] >= 1
    assert np.max(np.abs(phi - ref.get(I.PHI))) <= 1e-11 * np.max(np.abs(ref.get(I.PHI)))


@pytest.mark.parametrize("nx,ny,kw", SIZES[4:8] + SIZES[10:12])
def test_levels_mixed_converge(nx, ny, kw):
    c = I.case(nx, ny, radius=0.35 * min(nx, ny), H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0, **kw)
    s = lbfs.Solver(precision=lbfs.MIXED, max_cases=1, use_graph=True)
    s.set_case(0, c)
    st = s.step(5)[0]
    s.close()
    assert st["pot_resid_max"] <= 1e-6


@pytest.mark.parametrize("H0", [1e-60, 1e-25, 1e-5, 1e20])
def test_field_strength_does_not_change_the_fp64_solve(H0):
    """the problem is linear in H0: the same potential per unit field, in about as many cycles"""
    out = []
    for h in (1.0, H0):
        s = lbfs.Solver(precision=lbfs.FP64, max_cases=1)
        # sigma = 0 and no Kelvin force to speak of: only the potential is looked at
        s.set_case(0, I.case(80, 40, radius=14.0, H0=h, bo_m=0.0, field_angle_deg=40.0))
        s.set_fields(0, {I.PHI: np.zeros((40, 80))})
        status, st = s.step(1, raise_on_error=False)
        out.append((s.field(0, I.PHI) / h, st[0]["pot_resid"], st[0]["pot_cycles"]))
        s.close()
    assert out[1][1] <= 1e-13
    assert abs(out[1][2] - out[0][2]) <= 1
    assert np.max(np.abs(out[1][0] - out[0][0])) <= 1e-11 * np.max(np.abs(out[0][0]))
