"""The host side of the tensor-core base conversion, without a device: which
form a launch takes, at the sizes where both were measured."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_22227_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("mma") / "host_mma.so")
    srcs = [os.path.join(ROOT, "tests", "host_mma.cpp")]
    srcs += [os.path.join(CSRC, f) for f in ("mmaplan.cpp", "hostmath.cpp")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-I", cuda, *srcs, "-o", out], check=True)
    return ctypes.CDLL(out)


def _rule(lib, shapes, items, log_n, beside, split=1, sms=152):
    n = len(shapes)
    K, T = ((ctypes.c_int * n)(*(s[i] for s in shapes)) for i in (0, 1))
    return bool(lib.mma_rule(n, K, T, split, ctypes.c_uint64(items << log_n), sms,
                             int(beside)))


@pytest.mark.parametrize("shapes,items,log_n,beside,tensor", [
    # digits of 8 primes to the 4 special ones, halves of 8, 4, 3 and 2
    ([(8, 4)], 8, 15, True, False), ([(8, 4)], 4, 16, True, False), ([(8, 4)], 3, 16, True, False),
    ([(8, 4)], 8, 14, True, False), ([(7, 4)], 4, 16, True, False),
    # alone
    ([(8, 4)], 3, 16, False, True), ([(8, 4)], 2, 16, False, True), ([(8, 4)], 16, 13, False, True),
    # ModDown by 8 primes to 4, halves of 2 and 8
    ([(8, 4)], 4, 16, True, False), ([(8, 4)], 16, 16, True, True),
    # more targets: as alone
    ([(8, 5), (1, 12)], 2, 15, True, True), ([(8, 20)] * 3, 4, 16, True, True),
    ([(5, 23)], 8, 16, True, True), ([(8, 12)] * 2, 2, 14, True, True),
    # a launch too small for the matrix's start
    ([(3, 5)], 1, 12, False, False), ([(8, 20)] * 3, 1, 12, False, True)])
def test_form_of_a_conversion(lib, shapes, items, log_n, beside, tensor):
    assert _rule(lib, shapes, items, log_n, beside) == tensor


def test_other_layouts_take_the_tensor_cores(lib):
    for beside in (False, True):
        assert _rule(lib, [(9, 2)], 1, 12, beside, split=0)


def test_form_follows_the_devices_size(lib):
    """The same launch spreads its start over fewer coefficients per SM on a
    larger device."""
    assert _rule(lib, [(8, 4)], 2, 16, False)
    assert not _rule(lib, [(8, 4)], 2, 16, False, sms=304)
    assert _rule(lib, [(8, 4)], 4, 16, False, sms=304)
    assert _rule(lib, [(8, 4)], 1, 16, False, sms=76)
    assert not _rule(lib, [(8, 4)], 1, 16, False)
