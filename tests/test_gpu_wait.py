"""The wait between the blocks of the cycles' kernel is bounded: with a limit of one poll it runs
out while one block solves the coarse levels (tens of microseconds), lbfs_step says so, the device
stays usable, and the default limit is not met."""
import numpy as np
import pytest

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbfs.FP64, lbfs.MIXED])
def test_a_wait_that_runs_out_is_an_error_status(precision):
    c = I.case(256, 128, radius=50.0, H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0)
    s = lbfs.Solver(precision=precision, max_cases=1, mg_wait_polls=1)
    s.set_case(0, c)
    status, _ = s.step(1, raise_on_error=False)
    assert status == lbfs.ETIMEOUT
    for n in (1, 3):   # the context launches its cycles from now on, and its checks sum whole residuals
        st = s.step(n)[0]
        assert 0.0 < st["pot_resid_max"] <= s.mg_tol_used()
    s.close()
    out = []
    for plain in (False, True):
        s = lbfs.Solver(precision=precision, max_cases=1, mg_plain_cycles=plain)
        s.set_case(0, c)
        s.step(3)
        out.append(s.field(0, I.PHI))
        s.close()
    assert np.array_equal(*out)
