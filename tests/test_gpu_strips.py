"""The stage kernel's strips at the sizes where they can go wrong: grids that end at, one short
of and one past a strip's edge in either direction, narrower than a strip's halo, with walls
on every side or periodic, half-cell and other streaming steps; one case (whose coefficients
are kernel arguments) and a batch (whose coefficients are in shared memory) alike.
FP64 against the oracle within 1e-9 of each field's scale (the parity bound of the FP64
path); a batch against each of its cases alone bitwise, in both precisions."""
import numpy as np
import pytest

import oracle
from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

from parity import assert_parity, set_both

pytestmark = pytest.mark.gpu
IDS = [I.HE, I.P, I.C, I.MX, I.MY, I.PHI, I.FSPREV]

GRIDS = [
    (4, 5, {}), (25, 9, {}), (26, 4, {}), (27, 12, {}), (29, 7, {}), (52, 8, {}), (54, 17, {}), (79, 33, {}),
    (30, 13, dict(dts=0.4)), (53, 25, dict(dts=0.4, contact_angle_deg=64.0)),
    (28, 10, dict(periodic_x=1)), (52, 16, dict(periodic_x=1, dts=0.4)), (27, 12, dict(periodic_y=1, mag_bc=1, chi_l=0.0, chi_s=0.0)),
    (31, 11, dict(mag_bc=1)), (33, 9, dict(thermal_dirichlet=(1, 1, 1, 1), wall_T=(-0.5, 0.2, -1.0, 0.3), gravity=-1e-4)),
]


def _case(nx, ny, kw):
    return I.case(nx, ny, radius=0.4 * min(nx, 2 * ny), H0=0.03, field_angle_deg=35.0, stefan=0.0, latent=5.0, **kw)


@pytest.mark.parametrize("nx,ny,kw", GRIDS)
def test_strip_edges_fp64_against_oracle(nx, ny, kw):
    c = _case(nx, ny, kw)
    st = I.random_state(nx, ny, seed=nx + ny, latent=5.0, noise=0.02)
    ref = oracle.Oracle(c)
    s = lbfs.Solver(precision=lbfs.FP64, max_cases=1)
    s.set_case(0, c)
    set_both(s, 0, ref, st)
    ref.step(3)
    s.step(3)
    assert_parity(s, 0, ref, 1e-9)
    s.close()


@pytest.mark.parametrize("precision", [lbfs.MIXED, lbfs.FP64])
@pytest.mark.parametrize("half", [True, False])
def test_batch_of_strips_equals_each_case_alone(precision, half):
    cases = [(nx, ny, kw) for nx, ny, kw in GRIDS if ("dts" not in kw) == half]

    def run(group):
        s = lbfs.Solver(precision=precision, max_cases=len(group))
        for k, (nx, ny, kw) in enumerate(group):
            s.set_case(k, _case(nx, ny, kw))
            s.set_fields(k, I.random_state(nx, ny, seed=nx + ny, latent=5.0, noise=0.02))
        s.step(3)
        out = [s.fields(k, IDS) for k in range(len(group))]
        s.close()
        return out

    batch = run(cases)
    for k, c in enumerate(cases):
        alone = run([c])[0]
        for f in IDS:
            assert np.array_equal(batch[k][f], alone[f]), (c, I.FIELD_NAMES[f])
