"""Lifts from a single prime inside the transform that reads them (digits of
one prime, rescale, ModDown by one prime) against the oracle: every schedule of
every ring degree, sources below, at and far above their targets' size, factors
on both sides (BGV), the coefficient-form combine (BFV), and residues next to
the centring boundary."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


def _pair(p):
    ctx = api.Context(p)
    octx = oracle.Context(p.scheme, p.log_n, p.q_bits, p.p_bits, p.dnum, t=p.t,
                          log_n_max=p.log_n_max, b_bits=p.b_bits)
    seed = W.seed_for("lift-keys")
    return ctx, octx, ctx.keygen(seed), octx.keygen(seed)


def _edge_ct(octx, ctx, level):
    """Uniform, with the last limb's coefficients at the boundary and the ends."""
    ct = octx.ct_uniform(W.seed_for("lift-in"), 0, level)
    m = int(ctx.q[level - 1])
    vals = [(m - 1) // 2, (m + 1) // 2, 0, 1, m - 1, (m - 3) // 2]
    ct[0, level - 1] = np.resize(np.array(vals, dtype=np.uint64), ctx.n)
    return ct


@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
def test_every_schedule_matches_oracle(log_n):
    p = W.Preset("lift", W.CKKS, log_n, (50, 58, 50), (60,), 3, log_n_max=16)
    ctx, octx, keys, okeys = _pair(p)
    a = _edge_ct(octx, ctx, p.L)
    b = octx.ct_uniform(W.seed_for("lift-in"), 1, p.L)
    prod = octx.mul_relin(okeys, a, b)
    scaled = octx.rescale(a)
    da, db = ctx.import_ct(a), ctx.import_ct(b)
    _, count, _ = ctx.ntt_schedule()
    for k in range(count):
        ctx.set_ntt_schedule(k)
        assert np.array_equal(ctx.export_ct(ctx.mul_relin(keys, da, db))[0], prod), k
        assert np.array_equal(ctx.export_ct(ctx.rescale(da))[0], scaled), k


@pytest.mark.parametrize("scheme,q_bits,p_bits", [
    (W.CKKS, (30, 31, 30, 61), (60,)),      # far larger sources, targets below 2^33
    (W.CKKS, (61, 61, 40), (61,)),          # a source below its targets
    (W.CKKS, (50, 51, 52), (52,)),          # sources up to four times the target
    (W.BGV, (55, 55, 30), (60,)),
    (W.BFV, (55, 40, 55), (60,)),
    (W.BFV, (55, 55, 55), (55,)),
], ids=str)
def test_prime_sizes_match_oracle(scheme, q_bits, p_bits):
    t = 0 if scheme == W.CKKS else 257
    p = W.Preset("lift-sizes", scheme, 12, q_bits, p_bits, len(q_bits), t=t, log_n_max=12)
    ctx, octx, keys, okeys = _pair(p)
    g = ctx.galois_elt(3)
    keys.gen_galois(g)
    okeys.gen_galois(g)
    a = _edge_ct(octx, ctx, p.L)
    b = octx.ct_uniform(W.seed_for("lift-in"), 1, p.L)
    da, db = ctx.import_ct(a), ctx.import_ct(b)
    assert np.array_equal(ctx.export_ct(ctx.mul_relin(keys, da, db))[0],
                          octx.mul_relin(okeys, a, b))
    assert np.array_equal(ctx.export_ct(ctx.rotate(keys, da, g))[0], octx.rotate(okeys, a, g))
    if scheme != W.BFV:
        assert np.array_equal(ctx.export_ct(ctx.rescale(da))[0], octx.rescale(a))
