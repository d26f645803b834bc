"""The refinement cycles in one cooperative kernel: the same bits as a kernel per phase, on grids
whose coarse levels begin at the fine level, that take one and several tiles per group of threads,
with a coarsest level solved by itself, and in a batch of unlike depths; and every cycle reduces the
residual by at least a half (the method's contraction is below 0.25), on grids of many more tiles
than run at once, where a tile must not read what a neighbour has already overwritten."""
import numpy as np
import pytest

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu


def _case(nx, ny, **kw):
    return I.case(nx, ny, radius=0.35 * min(nx, ny), H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0, **kw)


GRIDS = {"tail": [_case(24, 16)], "one leg": [_case(128, 64)], "ragged": [_case(505, 253)],
         "many tiles": [_case(1100, 520)], "coarsest alone": [_case(126, 64, periodic_x=1)],
         "batch": [_case(24, 16), _case(126, 64, periodic_x=1), _case(300, 150), _case(77, 40, chi_g=0.0), _case(512, 256)]}


@pytest.mark.parametrize("prec", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("grid", list(GRIDS))
def test_same_bits_as_a_kernel_per_phase(prec, grid):
    out = []
    for plain in (False, True):
        s = lbfs.Solver(precision=prec, max_cases=len(GRIDS[grid]), mg_plain_cycles=plain, use_graph=not plain)
        for k, c in enumerate(GRIDS[grid]):
            s.set_case(k, c)
        st = s.step(4)
        out.append([(s.field(k, I.PHI), st[k]["pot_resid_max"], st[k]["pot_cycles"]) for k in range(len(GRIDS[grid]))])
        s.close()
    for (pa, ra, ca), (pb, rb, cb) in zip(*out):
        assert np.array_equal(pa, pb) and ra == rb and ca == cb


@pytest.mark.parametrize("prec", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("nx,ny", [(1024, 512), (1500, 700), (4096, 512)])
def test_every_cycle_contracts(prec, nx, ny):
    phi0 = np.random.default_rng(3).uniform(-1, 1, (ny // 8, nx // 8)).repeat(8, 0).repeat(8, 1)
    phi0 = np.pad(phi0, ((0, ny - phi0.shape[0]), (0, nx - phi0.shape[1])))
    last = None
    for n in (1, 2, 3, 4):
        s = lbfs.Solver(precision=prec, max_cases=1, mg_max_cycles=n, mg_tol=1e-30)
        s.set_case(0, _case(nx, ny))
        s.set_fields(0, {I.PHI: phi0})
        status, st = s.step(1, raise_on_error=False)
        s.close()
        assert st[0]["pot_cycles"] == n
        assert last is None or st[0]["pot_resid"] <= 0.5 * last
        last = st[0]["pot_resid"]
