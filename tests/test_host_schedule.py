"""The host code of the library followed call by call on a fake CUDA runtime (tests/hostlib.py):
what orders its memory, what its kernels are launched with, and what it does when a call fails."""
import ctypes as ct

import pytest

import hostlib
from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

BOTH = [lbfs.FP64, lbfs.MIXED]


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    return hostlib.build(tmp_path_factory.mktemp("host"))


@pytest.fixture
def fake(host_lib, monkeypatch):
    monkeypatch.setattr(lbfs, "_lib", None)
    f = hostlib.Fake(lbfs.load(host_lib))
    f.clear()
    return f


def _case(nx=64, ny=32, **kw):
    return I.case(nx, ny, radius=9.0, H0=0.03, field_angle_deg=40.0, **kw)


def _torch_memory(monkeypatch, offset=0):
    """torch's caching allocator over the host's memory, `offset` bytes past a multiple of 64; the
    list of its calls"""
    torch = pytest.importorskip("torch")
    libc = ct.CDLL(None)
    libc.aligned_alloc.restype, libc.aligned_alloc.argtypes = ct.c_void_p, [ct.c_size_t, ct.c_size_t]
    libc.free.argtypes = [ct.c_void_p]
    calls = []

    class Stream:
        def synchronize(self):
            calls.append("waited")

    def alloc(n, device):
        calls.append("allocated")
        return libc.aligned_alloc(64, (n + 127) // 64 * 64) + offset

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", lambda p: libc.free(p - offset))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: Stream())
    return calls


def test_torch_memory_is_free_of_pending_work_before_it_is_used(fake, monkeypatch):
    """A block of torch's caching allocator may still be in use by kernels queued on torch's
    current stream; the library's stream is not ordered behind them."""
    calls = _torch_memory(monkeypatch)
    s = lbfs.Solver(precision=lbfs.MIXED, max_cases=1, torch_alloc=True)
    s.set_case(0, _case())
    s.step(1)
    s.fields(0, [I.C])
    s.close()
    assert len(calls) > 6 and calls == ["allocated", "waited"] * (len(calls) // 2)


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("graph", [False, True])
def test_lists_arrive_before_the_kernels_that_read_them(fake, precision, graph):
    """Every upload is in the order of the kernels' own stream (one on the default stream is not
    ordered before a non-blocking stream's kernels) and has ended before its host copy goes."""
    s = lbfs.Solver(precision=precision, max_cases=2, use_graph=graph)
    for k in range(2):
        s.set_case(k, _case(300, 150))
    fake.clear()
    s.step(2)
    s.autotune(1)
    s.close()
    log = fake.log()
    assert not [w for w in log if w[0] == "copy-unordered"]
    stream = {w[1] for w in log if w[0] == "launch"} - {w[1] for w in log if w[0] == "record"}
    assert len(stream) == 1 and {w[1] for w in log if w[0] == "copy"} == stream
    kinds = [w[0] for w in log]
    uploads = [k for k in range(kinds.index("set")) if kinds[k] == "copy"]
    assert uploads and "sync" in kinds[uploads[-1]:kinds.index("set")]


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("tune", [False, True])
def test_a_redefined_case_keeps_its_strip_count(fake, precision, tune):
    """A batch launch reads a case's strip count from its table, which defining the case clears."""
    s = lbfs.Solver(precision=precision, max_cases=2)
    for k in range(2):
        s.set_case(k, _case())
    if tune:
        s.autotune(1)
    else:
        s.step(1)
    s.set_case(0, _case(stefan=0.7))   # the same grid, so as many strips as before
    fake.clear()
    s.step(1)
    s.close()
    stages = [w for w in fake.log() if w[0] == "stage"]
    assert len(stages) == 3 and all(w[2:] == ["batch"] for w in stages), stages


def test_a_failed_upload_is_made_up_for(fake):
    """After a copy that failed, the next step uploads the counts again."""
    s = lbfs.Solver(precision=lbfs.FP64, max_cases=2)
    for k in range(2):
        s.set_case(k, _case())
    for n in range(1, 4):
        fake.set("failing_copies", n)
        status, _ = s.step(1, raise_on_error=False)
        assert status in (lbfs.ECUDA, lbfs.ENOMEM)
    fake.set("failing_copies", 0)
    fake.clear()
    s.step(1)
    s.close()
    stages = [w for w in fake.log() if w[0] == "stage"]
    assert len(stages) == 3 and all(w[2:] == ["batch"] for w in stages), stages


@pytest.mark.parametrize("precision", BOTH)
def test_a_step_changes_no_limit_of_a_kernel(fake, precision):
    """A kernel's shared-memory limit is the whole process's: a context of small cases, stepped by
    another thread between a larger one's set-up of the limit and its launch, must not lower it."""
    large = [_case(91, 45), _case(126, 64, periodic_x=1), _case(6, 2700, periodic_x=1)]   # coarsest 4050 cells
    small = [_case(8, 8)]
    solvers = []
    for cases in (large, small):
        s = lbfs.Solver(precision=precision, max_cases=len(cases), mg_plain_cycles=len(solvers) == 1)
        for k, c in enumerate(cases):
            s.set_case(k, c)
        solvers.append(s)
    fake.clear()
    for _ in range(2):
        for s in solvers:
            s.step(2)
    for s in solvers:
        s.close()
    log = fake.log()
    assert not [w for w in log if w[0] == "limit"]
    sizes = [(int(w[6]), int(w[8])) for w in log if w[0] in ("launch", "cooperative")]
    assert max(n for n, _ in sizes) > 48 * 1024 and all(n <= limit for n, limit in sizes)


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("graph", [False, True])
def test_a_wait_that_ran_out_is_reported_as_such(fake, precision, graph):
    """LBFS_ETIMEOUT, not a potential that has not converged; the counts that the blocks left
    behind are cleared, and the next step solves the potential afresh."""
    s = lbfs.Solver(precision=precision, max_cases=2, use_graph=graph)
    for k in range(2):
        s.set_case(k, _case(300, 150))
    s.step(2)
    fake.set("wait_runs_out", 1)
    s.set_case(1, _case(300, 150))
    status, _ = s.step(1, raise_on_error=False)
    fake.set("wait_runs_out", 0)
    fake.clear()
    again, _ = s.step(1, raise_on_error=False)
    third, _ = s.step(1, raise_on_error=False)
    s.close()
    log = fake.log()
    assert status == lbfs.ETIMEOUT and again == third == lbfs.OK
    assert not [w for w in log if w[0] == "cooperative"]   # launched from now on
    assert [w[0] for w in log].count("replay") == (1 if graph else 0)
    assert {w[2] for w in log if w[0] == "ticket"} == {"0"}


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("first", [1, 40])   # cycles of the first solve: fewer and more than are launched anyway
def test_a_refused_cooperative_launch_falls_back(fake, precision, graph, first):
    """On a stream with fewer multiprocessors than the device has, the cycles are launched phase by
    phase, as many as the kernel would have run; the refused launch is not tried again and never
    part of a recording."""
    s = lbfs.Solver(precision=precision, max_cases=2, use_graph=graph, mg_max_cycles=first)
    for k in range(2):
        s.set_case(k, _case(300, 150))
    fake.set("cooperative_limit", 2)
    fake.clear()
    s.step(3)
    log = fake.log()
    kinds = [w[0] for w in log]
    assert kinds.count("refused") == 1 and "cooperative" not in kinds
    if graph:
        assert kinds.index("refused") < kinds.index("record")
    fake.clear()
    s.set_case(1, _case(300, 150))   # a new recording
    s.step(3)
    s.close()
    fake.set("cooperative_limit", 1 << 20)
    log = fake.log()
    assert not [w for w in log if w[0] in ("refused", "cooperative")]
    tails = [k for k, w in enumerate(log) if w[0] == "launch" and w[2].startswith("k_tail")]
    if graph:   # one recorded warm step: its checks are of the step's start and after each cycle
        a, b = [[w[0] for w in log].index(x) for x in ("record", "recorded")]
        checks = [k for k, w in enumerate(log) if w[0] == "launch" and w[2].startswith("k_residual") and a < k < b]
        warm = 12 if precision == lbfs.FP64 else 3
        assert len(checks) == warm + 1 and sum(a < k < b for k in tails) == warm


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("offset", [0, 8, 24, 40])
def test_a_callers_allocator_need_not_align_to_a_quad(fake, monkeypatch, precision, offset):
    """The kernels read a cell's quantities 16 and 32 bytes at a time."""
    _torch_memory(monkeypatch, offset)
    for cases in (1, 2):
        s = lbfs.Solver(precision=precision, max_cases=cases, torch_alloc=True)
        for k in range(cases):
            s.set_case(k, _case())
        fake.clear()
        s.step(1)
        s.close()
        stages = [w for w in fake.log() if w[0] == "stage"]
        assert len(stages) == 3 and not [w for w in stages if "misplaced" in w]


@pytest.mark.parametrize("tune", [False, True])
def test_lists_are_allocated_on_the_contexts_device(fake, tune):
    """Whichever device the calling thread used last."""
    fake.set("devices", 2)
    second = lbfs.Solver(precision=lbfs.MIXED, max_cases=1, device=1)
    second.set_case(0, _case())
    first = lbfs.Solver(precision=lbfs.MIXED, max_cases=1, device=0)
    fake.clear()
    if tune:
        second.autotune(1)
    else:
        second.step(1)
    log = fake.log()
    for s in (first, second):
        s.close()
    fake.set("devices", 1)
    assert {w[3] for w in log if w[0] == "malloc"} == {"1"}
