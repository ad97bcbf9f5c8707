"""Multiplications without a tensor kernel (few words: the inverse transform
and the inner product form the products) against those with it (batches of more
than 2^19 words per launch) and against the oracle: 1 to 9 digits, partly used
last digits, 41- to 61-bit primes, every transform schedule, gathered entries of
a batch, and results written over an input."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


@pytest.mark.parametrize("scheme,dnum,bits", [
    (W.CKKS, 1, (50, 58, 61)), (W.CKKS, 2, (41, 50, 59, 60)), (W.CKKS, 3, (50,) * 5),
    (W.CKKS, 4, (50,) * 8), (W.BGV, 5, (55,) * 5), (W.CKKS, 6, (45,) * 11), (W.CKKS, 7, (61,) * 7),
    (W.BGV, 8, (55,) * 8), (W.CKKS, 8, (60,) * 8), (W.CKKS, 9, (50,) * 9)])
def test_products_equal_the_tensor_kernel(scheme, dnum, bits):
    t = 0 if scheme == W.CKKS else 65537
    special = 61 if dnum < 8 else 60  # (digits + 1) q < 2^64
    p = W.Preset("product", scheme, 12, bits, (special,) * -(-len(bits) // dnum), dnum, t=t,
                 log_n_max=12)
    ctx = api.Context(p)
    octx = oracle.Context(p.scheme, 12, p.q_bits, p.p_bits, p.dnum, t=t, log_n_max=12)
    seed = W.seed_for(f"product-{dnum}-{bits[0]}")
    keys, okeys = ctx.keygen(seed), octx.keygen(seed)
    for level in sorted({p.L, max(2, p.L - 1)}):
        count = 128 // level + 3  # one launch of more than 2^19 words
        a = torch.cat([ctx.ct_uniform(seed, 2 * j, level) for j in range(count)])
        b = torch.cat([ctx.ct_uniform(seed, 2 * j + 1, level) for j in range(count)])
        want = ctx.mul_relin(keys, a, b)
        ha, hb = ctx.export_ct(a[:1])[0], ctx.export_ct(b[:1])[0]
        assert np.array_equal(ctx.export_ct(want[:1])[0], octx.mul_relin(okeys, ha, hb))
        for j in (0, 1, count - 1):
            assert torch.equal(ctx.mul_relin(keys, a[j:j + 1], b[j:j + 1]), want[j:j + 1]), j
        few = min(4, 128 // level)
        assert torch.equal(ctx.mul_relin(keys, a[:few], b[:few]), want[:few])
        over = a[:few].clone()
        ctx.mul_relin(keys, over, b[:few], out=over)
        assert torch.equal(over, want[:few])
        same = ctx.mul_relin(keys, a[:1], a[:1])
        assert np.array_equal(ctx.export_ct(same)[0], octx.mul_relin(okeys, ha, ha))
        if scheme == W.CKKS:
            wr = ctx.mul_relin_rescale(keys, a, b)
            assert torch.equal(ctx.mul_relin_rescale(keys, a[:1], b[:1]), wr[:1])
        # gathered: single entries of one batch, merged on one lane
        outs = [torch.full_like(want[:1], -1) for _ in range(few)]
        ins = [(a[j:j + 1].clone(), b[j:j + 1].clone()) for j in range(few)]
        api.run_batch([api.make_op(api.OP_MUL_RELIN, ctx, x, o, keys=keys, b=y)
                       for (x, y), o in zip(ins, outs)], lanes=1)
        torch.cuda.synchronize()
        for j in range(few):
            assert torch.equal(outs[j], want[j:j + 1]), (level, j)


@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
def test_products_under_every_schedule(log_n):
    p = W.Preset("product-sched", W.CKKS, log_n, (50, 58, 61), (61,), 3, log_n_max=16)
    ctx = api.Context(p)
    seed = W.seed_for(f"product-sched-{log_n}")
    keys = ctx.keygen(seed)
    big = (1 << 19) // (3 << log_n) + 1
    a = torch.cat([ctx.ct_uniform(seed, 2 * j, 3) for j in range(big)])
    b = torch.cat([ctx.ct_uniform(seed, 2 * j + 1, 3) for j in range(big)])
    _, count, _ = ctx.ntt_schedule()
    for k in range(count):
        ctx.set_ntt_schedule(k)
        want = [ctx.mul_relin_rescale(keys, a, b), ctx.mul_relin(keys, a, b)]
        assert torch.equal(ctx.mul_relin_rescale(keys, a[:1], b[:1]), want[0][:1]), k
        assert torch.equal(ctx.mul_relin(keys, a[:1], b[:1]), want[1][:1]), k
