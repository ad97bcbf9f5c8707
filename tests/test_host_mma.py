"""The host side of the tensor-core base conversion, without a device: which
form a launch takes, at the sizes where both were measured, and the images of
its plans, read as the kernel reads them and compared with big integers."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
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


MAGIC = 12582912.0  # 3 * 2^22


class Image:
    """A plan's image, taken apart as conv_mma.cu does."""

    def __init__(self, lib, src, pre, dst, post):
        cap = 1 << 16
        img = np.zeros(cap, dtype=np.uint64)
        arrs = [np.array(v, dtype=np.uint64) for v in (src, pre, dst, post)]
        p = [a.ctypes.data_as(ctypes.c_void_p) for a in arrs]
        words = lib.mma_plan(len(src), p[0], p[1], len(dst), p[2], p[3],
                             img.ctypes.data_as(ctypes.c_void_p), cap)
        assert words > 0
        img = img[:words]
        head, self.counts = int(img[0]), int(img[1])
        self.K, self.blocks, self.cores, self.six = head & 0xff, head >> 8 & 0xff, head >> 16 & 0xff, head >> 32
        self.src = img[2:2 + 6 * self.K].reshape(self.K, 6)
        t0 = 2 + 6 * self.K
        self.tgt = img[t0:t0 + 18 * self.blocks].reshape(self.blocks, 3, 6)
        b0 = (t0 + 18 * self.blocks + 15) & ~15
        self.matrix = img[b0:].view(np.float16).reshape(self.cores, 16 * self.blocks, 8)

    def convert(self, r, plus, above):
        """Targets' words from the sources' residues r; plus: the other
        representative of y below 2 m."""
        row = np.zeros((self.cores, 8), dtype=np.int64)
        fr = 1 << 26
        for i in range(self.K):
            m, w, _, c = (int(x) for x in self.src[i, :4])
            y = r[i] * w % m + (m if plus else 0)
            row[i] = [(y >> 8 * e & 255) - 128 for e in range(8)]
            fr += ((y >> (c >> 32)) * (c & 0xffffffff)) >> 32
        assert fr < 1 << 32
        v = fr >> 27
        if fr & ((1 << 27) - 1) >= (1 << 27) - 3 * self.K:
            v = (fr - (1 << 26) >> 27) + above
        row[self.K, 0] = v
        weights = self.matrix.astype(np.int64)
        assert np.array_equal(weights, self.matrix)  # whole numbers
        sums = np.einsum("ke,kce->c", row, weights)
        # any order of the products stays a whole number below 2^24
        assert np.einsum("ke,kce->c", np.abs(row), np.abs(weights)).max() < 1 << 22
        offset = 3072 * weights[self.K, :, 1]
        out = {}
        for b in range(self.blocks):
            D = 6 if self.six >> b & 1 else 5
            for j in range(self.counts >> 4 * b & 15):
                cols = slice(16 * b + j * D, 16 * b + (j + 1) * D)
                assert (offset[cols] == 3 << 22).all()
                f = (sums[cols] + offset[cols]).astype(np.float32)
                bits = [int(x) for x in f.view(np.uint32)]
                o = self.tgt[b, j]
                k = np.array([o[2], o[3]], dtype=np.uint64).view(np.float32).astype(np.float64)
                q = np.float32(float(f[D - 3]) * k[2] + k[3])
                q = np.float32(float(f[D - 2]) * k[1] + float(q))
                q = np.float32((float(f[D - 1]) - MAGIC) * k[0] + float(q))
                e = int(np.float32(q + np.float32(MAGIC)).view(np.uint32))
                acc = int(o[0]) + sum(x << 10 * d for d, x in enumerate(bits)) + e * int(o[1])
                out[int(o[4])] = acc % (1 << 64)
        return [out[t] for t in sorted(out)]


@pytest.mark.parametrize("K,src_bits,dst_bits", [
    (1, 50, (50, 60)), (2, 33, (41, 42)), (3, 60, (50, 60)), (5, 60, (50,) * 7), (7, 41, (45, 41)),
    (8, 50, (50, 51, 60)), (8, 60, (60,) * 5), (14, 50, (50, 49)), (12, 60, (60, 41)), (15, 33, (50,))])
def test_images_convert_as_big_integers(lib, K, src_bits, dst_bits):
    sympy = pytest.importorskip("sympy")
    rng = np.random.default_rng(K * 100 + src_bits)
    p, primes = 1 << src_bits, []
    for _ in range(K):
        p = sympy.prevprime(p)
        primes.append(p)
    dst = []
    for bits in dst_bits:
        p = sympy.prevprime(1 << bits)
        while p in primes or p in dst:
            p = sympy.prevprime(p)
        dst.append(p)
    draw = lambda m: int(rng.integers(1, m))
    for pre, post in (([1] * K, [1] * len(dst)), ([draw(m) for m in primes], [draw(m) for m in dst])):
        image = Image(lib, primes, pre, dst, post)
        M = 1
        for m in primes:
            M *= m
        vals = [(M - 1) // 2, (M + 1) // 2, (M - 3) // 2, (M + 3) // 2, 0, 1, M - 1, M - 2,
                (M - 1) // 2 - (M >> 40), (M + 1) // 2 + (M >> 40), M // 3]
        vals += [int.from_bytes(rng.bytes(K * 8), "little") % M for _ in range(20)]
        for x in vals:
            # the sources are residues whose product with pre is x
            r = [x * pow(f, -1, m) % m for f, m in zip(pre, primes)]
            above = x > (M - 1) // 2
            for plus in (False, True):
                got = image.convert(r, plus, above)
                for g, q, f in zip(got, dst, post):
                    assert g % q == (x - M * above) * f % q
                    assert 2 * q < 5 * g < 8 * q
