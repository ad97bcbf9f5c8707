"""The lift of a decrypted polynomial to 64-bit integers at the centring
boundary and at the ends of its range, for 1 to 32 primes, against Python
integers: with c1 = 0 the decryption is c0 itself."""
import numpy as np
import pytest

from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


@pytest.mark.parametrize("bits", [(50,) * 24, (20, 21, 61), (60,) * 15, (40,) * 32, (61,) * 9],
                         ids=lambda b: f"{len(b)}x{b[0]}")
def test_decrypt_at_the_edges(bits):
    p = W.Preset("edges", W.CKKS, 12, bits, (60,), 1, log_n_max=12)
    ctx = api.Context(p)
    keys = ctx.keygen(W.seed_for("edges"))
    rng = np.random.default_rng(5)
    for level in sorted({1, 2, len(bits) // 2 + 1, len(bits)}):
        qs = [int(q) for q in ctx.q[:level]]
        M = 1
        for q in qs:
            M *= q
        vals = [0, 1, M - 1, (M - 1) // 2, (M + 1) // 2, (M - 3) // 2, (M + 3) // 2]
        vals += [int.from_bytes(rng.bytes(300), "little") % M for _ in range(57)]
        ct = np.zeros((1, 2, level, ctx.n), dtype=np.uint64)
        for i, q in enumerate(qs):
            ct[0, 0, i] = np.resize(np.array([v % q for v in vals], dtype=np.uint64), ctx.n)
        got = ctx.decrypt(keys, ctx.import_ct(ct))
        want = [(v - M if v > (M - 1) // 2 else v) & ((1 << 64) - 1) for v in vals]
        want = np.resize(np.array(want, dtype=np.uint64), ctx.n).view(np.int64)
        assert np.array_equal(got, want), level
