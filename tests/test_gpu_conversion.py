"""The tensor-core base conversion against the oracle and against the integer
kernels: source counts from 3 to 15, one and two passes of targets, part-filled
column blocks, five- and six-digit targets, constants on both sides (BGV), full
reduction (BFV), and values next to the centring boundary.

A batch of 32 ciphertexts takes the tensor-core kernel where a single one may
take the integer kernel, so batches are also compared with single calls."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402

COUNT = 32
PRESETS = [
    W.Preset("k8_t20", W.CKKS, 12, (50,) * 24, (60,) * 4, 3, log_n_max=12),
    W.Preset("k8_t24_two_passes", W.CKKS, 12, (50,) * 24, (60,) * 8, 3, log_n_max=12),
    W.Preset("k15", W.CKKS, 12, (50,) * 30, (50,) * 14, 2, log_n_max=12),
    W.Preset("k7_k6_small_primes", W.CKKS, 12, (41,) * 13, (45,) * 3, 2, log_n_max=12),
    W.Preset("six_digit_targets", W.CKKS, 12, (45, 51, 60) * 3, (59,) * 5, 2, log_n_max=12),
    W.Preset("bgv", W.BGV, 12, (55,) * 9, (60,) * 4, 2, t=65537, log_n_max=12),
    W.Preset("bfv", W.BFV, 12, (50,) * 6, (60,) * 3, 2, t=65537, log_n_max=12),
    W.Preset("bfv_12_primes", W.BFV, 12, (50,) * 12, (60,) * 4, 3, t=65537, log_n_max=12),
    # 61-bit primes: the integer scale-and-round
    W.Preset("bfv_61", W.BFV, 12, (61,) * 3, (61,), 3, t=65537, log_n_max=12, b_bits=61),
]


def _octx(p):
    return oracle.Context(p.scheme, p.log_n, p.q_bits, p.p_bits, p.dnum, t=p.t,
                          log_n_max=p.log_n_max, b_bits=p.b_bits)


@pytest.mark.parametrize("p", PRESETS, ids=lambda p: p.name)
def test_batches_match_oracle_and_single_calls(p):
    ctx, octx = api.Context(p), _octx(p)
    keys, okeys = ctx.keygen(W.seed_for("conv-keys")), octx.keygen(W.seed_for("conv-keys"))
    seed = W.seed_for("conv-in")
    for level in sorted({p.L, p.L - 1, p.L // 2 + 1} if p.scheme != W.BFV else {p.L}):
        a = [octx.ct_uniform(seed, i, level) for i in range(3)]
        da = ctx.import_ct(np.stack(a))
        big = da.repeat(COUNT // 3 + 1, 1, 1, 1)[:COUNT].contiguous()
        other = torch.roll(big, 1, 0).contiguous()
        got = ctx.mul_relin(keys, big, other)
        want = octx.mul_relin(okeys, a[1], a[0])
        assert np.array_equal(ctx.export_ct(got[1:2])[0], want), level
        for i in range(3):
            one = ctx.mul_relin(keys, da[i:i + 1], da[(i - 1) % 3:(i - 1) % 3 + 1])
            for j in range(i + 3, COUNT, 3):
                assert torch.equal(got[j:j + 1], one), (level, j)
        if p.scheme == W.CKKS:
            fused = ctx.mul_relin_rescale(keys, big, other)
            assert np.array_equal(ctx.export_ct(fused[1:2])[0], octx.rescale(want)), level
            assert torch.equal(fused, ctx.rescale(got)), level


def test_values_at_the_centring_boundary():
    """Digits equal to (M-1)/2, (M+1)/2 and their neighbours (where the
    fixed-point quotient cannot decide) and to 0, 1, M-1."""
    p = PRESETS[0]
    ctx, octx = api.Context(p), _octx(p)
    keys, okeys = ctx.keygen(W.seed_for("edge-keys")), octx.keygen(W.seed_for("edge-keys"))
    g = ctx.galois_elt(1)
    keys.gen_galois(g)
    okeys.gen_galois(g)
    a = octx.ct_uniform(W.seed_for("edge-in"), 0, p.L)
    alpha = ctx.alpha
    for d in range(0, p.L, alpha):
        qs = [int(q) for q in ctx.q[d:d + alpha]]
        M = 1
        for q in qs:
            M *= q
        vals = [(M - 1) // 2, (M + 1) // 2, (M - 3) // 2, (M + 3) // 2, 0, 1, M - 1,
                (M - 1) // 2 - (1 << 60), (M + 1) // 2 + (1 << 60)]
        for i, q in enumerate(qs):
            a[1, d + i] = np.resize(np.array([v % q for v in vals], dtype=np.uint64), ctx.n)
    da = ctx.import_ct(a).repeat(COUNT, 1, 1, 1).contiguous()
    got = ctx.rotate(keys, da, g)
    assert np.array_equal(ctx.export_ct(got[:1])[0], octx.rotate(okeys, a, g))
    assert torch.equal(got, got[:1].expand_as(got))
