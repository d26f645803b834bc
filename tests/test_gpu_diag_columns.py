"""The diagnostics kernel where its split shows: widths around its 32-column blocks, fewer rows
than its 32 warps and rows that split unevenly, and speeds for which its upper bound must not hide
the largest: tiny and huge momenta, one fast cell anywhere, a gas as dense as the liquid and a C far
outside [0, 1] whose mixture density cancels.  The state is exported exactly and evaluated by the
oracle in FP64; 1e-12, some thousand roundings, is the bound of the diagnostics' parity test."""
import numpy as np
import pytest

import oracle
from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu
STATE = [I.PHI, I.HE, I.P, I.C, I.MX, I.MY, I.FSPREV]


def _compare(prec, case, st):
    s = lbfs.Solver(precision=prec, max_cases=1)
    s.set_case(0, case)
    s.set_fields(0, st)
    dg, qg = s.diagnostics(0)
    kept = s.fields(0, STATE)
    s.close()
    ref = oracle.Oracle(case)
    ref.set_state(kept)
    dr, qr = ref.diagnostics()
    for k in ("H_m", "U_max", "Pe", "Q_wall"):
        assert abs(dg[k] - dr[k]) <= 1e-12 * max(abs(dr[k]), 1e-300), (k, dg[k], dr[k])
    assert np.max(np.abs(qg - qr)) <= 1e-12 * max(np.max(np.abs(qr)), 1e-300)


@pytest.mark.parametrize("prec", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 5), (32, 32), (33, 31), (64, 33), (65, 127), (97, 130)])
def test_sizes(prec, nx, ny):
    c = I.case(nx, ny, radius=0.4 * min(nx, ny), stefan=0.0, latent=10.0, rho_s=0.9)
    _compare(prec, c, I.random_state(nx, ny, seed=nx, latent=10.0, noise=0.2))


@pytest.mark.parametrize("prec", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("what", ["tiny", "huge", "still", "one", "dense gas", "wide C"])
def test_speeds(prec, what):
    nx, ny = 70, 45
    c = I.case(nx, ny, radius=15.0, stefan=0.0, latent=10.0, rho_s=0.9, rho_g=1.7 if what == "dense gas" else 0.1)
    st = I.random_state(nx, ny, seed=5, latent=10.0, noise=0.2)
    scale = {"tiny": 1e-36, "huge": 1e15, "still": 0.0}.get(what, 1.0)
    st[I.MX], st[I.MY] = st[I.MX] * scale, st[I.MY] * scale
    if what == "one":
        j, i = np.argwhere(st[I.C] > 0.6)[-7]
        st[I.MY][j, i] = 0.5
    if what in ("wide C", "dense gas"):
        st[I.C] = 0.5 + 2.6 * (st[I.C] - 0.5)
    _compare(prec, c, st)
