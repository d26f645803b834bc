"""The library's host code linked with the CUDA runtime of tests/host/fake_cuda.cpp: what it
allocates, copies, waits for and launches can be followed on a machine without a GPU, and a
failing call can be faked.  Kernels do nothing there."""
import ctypes as ct
import os
import shutil
import subprocess

from paper_2511_10257_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCES = [os.path.join(B.CSRC, f) for f in ("lbfs_api.cu", "lbfs_potential.cu", "lbfs_fields.cu", "lbfs_stage.cu")]


def build(folder) -> str:
    """compile (device code only as far as PTX, unoptimised) and link; the path of the library"""
    toolkit = os.path.dirname(os.path.dirname(shutil.which(B.nvcc()) or B.nvcc()))
    inc = ["-I", os.path.join(B.ROOT, "include"), "-I", B.CSRC, "-I", os.path.join(toolkit, "include")]
    nvcc = [B.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-O1", "-Xcicc", "-O0", "-Xcompiler", "-fPIC"]
    procs, objs = [], []
    for src in SOURCES + [os.path.join(HERE, "host", f) for f in ("fake_stage.cu", "fake_cuda.cpp")]:
        objs.append(os.path.join(str(folder), os.path.splitext(os.path.basename(src))[0] + ".o"))
        cmd = (nvcc if src.endswith(".cu") else ["g++", "-O1", "-fPIC"]) + ["-std=c++17"] + inc + ["-c", src, "-o", objs[-1]]
        procs.append(subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT))
    for p in procs:
        out, _ = p.communicate()
        assert p.returncode == 0, out.decode(errors="replace")
    lib = os.path.join(str(folder), "liblbfs_host.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib] + objs, check=True)
    return lib


class Fake:
    """the fake runtime behind a loaded library"""

    def __init__(self, L):
        self._L = L
        L.fake_log.restype = ct.c_char_p
        L.fake_set.argtypes = [ct.c_char_p, ct.c_longlong]

    def set(self, what: str, value: int):
        self._L.fake_set(what.encode(), value)

    def clear(self):
        self._L.fake_clear()

    def log(self):
        """the calls since the last clear, each as its list of words"""
        return [line.split() for line in self._L.fake_log().decode().splitlines()]
