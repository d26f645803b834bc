"""The FP64 warm start extrapolated from one, two and three earlier potentials, through the step on
which three begin to be used and after a state is set again: every step meets 1e-13, and the
potential is that of a solver that starts each step from an imported state, which has no history, to
1e-11 (the bound of the solver's parity test; both solve to 1e-13)."""
import numpy as np
import pytest

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu
STATE = [I.PHI, I.HE, I.P, I.C, I.MX, I.MY, I.FSPREV]


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("nx,ny", [(31, 17), (128, 64)])
def test_history_does_not_change_the_potential(nx, ny, graph):
    c = I.case(nx, ny, radius=0.37 * ny, H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0)
    warm = lbfs.Solver(precision=lbfs.FP64, max_cases=1, use_graph=graph)
    cold = lbfs.Solver(precision=lbfs.FP64, max_cases=1)
    for s in (warm, cold):
        s.set_case(0, c)
    for n in range(12):
        if n == 9:
            warm.set_fields(0, warm.fields(0, STATE))
        cold.set_fields(0, warm.fields(0, STATE))
        st = warm.step(1)[0]
        cold.step(1)
        a, b = warm.field(0, I.PHI), cold.field(0, I.PHI)
        assert st["pot_resid"] <= 1e-13
        assert np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b))
    warm.close()
    cold.close()
