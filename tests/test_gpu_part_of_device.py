"""A context whose stream owns a part of the device's multiprocessors (a green context's stream):
the cycles' kernel, whose blocks wait on one another, must not count on the others.  Every step
succeeds and the fields are those of a stream with the whole device, bitwise."""
import ctypes as ct

import numpy as np
import pytest

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

pytestmark = pytest.mark.gpu
IDS = [I.HE, I.PHI, I.C, I.MX]


class Resource(ct.Structure):   # CUdevResource
    _fields_ = [("type", ct.c_int), ("pad", ct.c_ubyte * 92), ("sm_count", ct.c_uint), ("rest", ct.c_ubyte * 44)]


@pytest.fixture
def small_stream():
    """a stream of 16 multiprocessors"""
    cu = ct.CDLL("libcuda.so.1")
    keep = lbfs.Solver(max_cases=1)   # the device's primary context is active

    def call(name, *args):
        if not hasattr(cu, name) or getattr(cu, name)(*args) != 0:
            pytest.skip(f"{name}: no green contexts here")

    every, some, n = Resource(), Resource(), ct.c_uint(1)
    desc, ctx, stream = ct.c_void_p(), ct.c_void_p(), ct.c_void_p()
    call("cuDeviceGetDevResource", 0, ct.byref(every), 1)
    call("cuDevSmResourceSplitByCount", ct.byref(some), ct.byref(n), ct.byref(every), None, 0, 16)
    call("cuDevResourceGenerateDesc", ct.byref(desc), ct.byref(some), 1)
    call("cuGreenCtxCreate", ct.byref(ctx), desc, 0, 1)
    call("cuGreenCtxStreamCreate", ct.byref(stream), ctx, 1, 0)
    assert n.value == 1 and 16 <= some.sm_count < every.sm_count
    yield stream.value
    call("cuStreamDestroy_v2", stream)
    call("cuGreenCtxDestroy", ctx)
    keep.close()


@pytest.mark.parametrize("precision", [lbfs.FP64, lbfs.MIXED])
@pytest.mark.parametrize("graph", [False, True])
def test_fields_on_a_part_of_the_device(small_stream, precision, graph):
    c = I.case(512, 256, radius=90.0, H0=0.04, field_angle_deg=40.0, chi_l=2.0, chi_s=2.0)
    out, launches = [], []
    for stream in (None, small_stream):
        s = lbfs.Solver(precision=precision, max_cases=1, use_graph=graph, stream=stream)
        s.set_case(0, c)
        for _ in range(3):
            status, _st = s.step(2, raise_on_error=False)
            assert status == lbfs.OK
        launches.append(s.last_launch_count())
        out.append(s.fields(0, IDS))
        s.close()
    print(f"launches of two steps: {launches}")
    for f in IDS:
        assert np.array_equal(out[0][f], out[1][f]), I.FIELD_NAMES[f]
