"""What the library's host code hands to kernels, on a fake CUDA runtime
(tests/host_uploads.cpp): constants have arrived before a kernel on the
caller's stream may read them, and an allocation that failed and is made up
for leaves no error for the next launch to report.  And which streams a product
that is written over its input runs on."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2503_22227_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_22227_gb300", "csrc")


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(_cuda_include(), "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("uploads") / "host_uploads.so")
    srcs = [os.path.join(ROOT, "tests", "host_uploads.cpp")]
    srcs += [os.path.join(CSRC, f) for f in ("ops.cpp", "context.cpp", "mmaplan.cpp", "hostmath.cpp")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), "-I", _cuda_include(), *srcs, "-o", out,
                    "-Wl,-z,lazy", "-Wl,-Bsymbolic"], check=True)
    return out


# The other launchers are not called, so their symbols stay open: a library
# bound lazily, in a process of its own.
LOADER = """
import ctypes, sys
dl = ctypes.CDLL(None)
dl.dlopen.restype = dl.dlsym.restype = ctypes.c_void_p
dl.dlopen.argtypes, dl.dlsym.argtypes = [ctypes.c_char_p, ctypes.c_int], [ctypes.c_void_p, ctypes.c_char_p]
dl.dlerror.restype = ctypes.c_char_p
h = dl.dlopen(sys.argv[1].encode(), 1)
assert h, dl.dlerror()
f = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_char_p, ctypes.c_int)(dl.dlsym(h, b"host_uploads"))
print(f(sys.argv[2].encode(), int(sys.argv[3])))
"""


def _run(program, what, scheme):
    r = subprocess.run([sys.executable, "-c", LOADER, program, what, str(scheme)],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    return int(r.stdout)


@pytest.mark.parametrize("scheme", [W.CKKS, W.BFV, W.BGV])
def test_constants_arrive_before_the_kernels_that_read_them(program, scheme):
    assert _run(program, "encrypt", scheme) == 0


def test_no_memory_for_an_image_leaves_the_integer_form_usable(program):
    assert _run(program, "nomem", W.CKKS) == 0


def test_fused_products_over_their_inputs_run_on_one_stream(program):
    """The result's ciphertexts are a limb shorter than the input's, so that the
    second half's results lie in the first half's inputs."""
    assert _run(program, "over", W.CKKS) == 1
