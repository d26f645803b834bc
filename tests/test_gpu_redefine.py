"""A case slot of a living batch defined again on the same grid: the statistics and diagnostics of
every case are those of a context that never held the earlier case, bitwise (the same kernels on
the same data), in both precisions, with and without a recorded graph, after steps and after the
autotuner."""
import numpy as np
import pytest

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu


def _case(**kw):
    return I.case(100, 52, radius=20.0, H0=0.04, field_angle_deg=30.0, **kw)


@pytest.mark.parametrize("precision", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("before", ["step", "autotune"])
def test_statistics_after_a_slot_is_defined_again(precision, graph, before):
    def run(s, reused):
        shape = 0
        if reused:
            for k in range(2):
                s.set_case(k, _case(stefan=0.5))
            if before == "step":
                s.step(3)
            else:
                shape, _ = s.autotune(1)
        for k in range(2):
            s.set_case(k, _case(stefan=(0.2, 0.9)[k]))
        st = s.step(5)
        out = (st, [s.diagnostics(k)[0] for k in range(2)], [s.field(k, I.HE) for k in range(2)])
        s.close()
        return out, shape

    got, shape = run(lbfs.Solver(precision=precision, max_cases=2, use_graph=graph), True)
    want, _ = run(lbfs.Solver(precision=precision, max_cases=2, use_graph=graph, tile=shape), False)
    for k in range(2):
        assert got[0][k]["t"] > 0.0
        assert got[0][k] == want[0][k]
        assert got[1][k] == want[1][k]
        assert np.array_equal(got[2][k], want[2][k])
