"""Which multiplications have no tensor kernel (the inverse transform and the
inner product form the products), seen from the kernels a call launches, and
their results: against the oracle under every schedule of every ring degree, and
against single calls on both sides of the rule."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


def _launches(f):
    f()  # constants, opt-ins
    before = api.kernel_launches()
    out = f()
    return out, api.kernel_launches() - before


def _uniform(ctx, seed, count, level, first=0):
    return torch.cat([ctx.ct_uniform(seed, first + j, level) for j in range(count)])


# (N, limbs, ciphertexts, tensor kernel): 24 primes in digits of 8, 4 special
# primes; the line is 2^20 words of (digits + 2) (limbs + 4) N per ciphertext,
# or up to 2^19 words of at most 3 ciphertexts of at least 4 limbs
@pytest.mark.parametrize("log_n,level,count,tensor", [
    (12, 2, 8, False), (12, 2, 16, True), (12, 8, 7, False), (12, 8, 16, True), (12, 24, 3, False),
    (12, 24, 5, True), (13, 3, 4, False), (13, 5, 8, True), (13, 9, 5, True), (14, 3, 3, False),
    (14, 3, 4, False), (14, 2, 16, True), (14, 9, 5, True), (14, 16, 2, False), (14, 16, 4, True),
    (15, 2, 1, False), (15, 2, 2, True), (15, 2, 4, True), (15, 16, 1, False), (15, 17, 1, True),
    (16, 3, 1, True), (16, 4, 1, False), (16, 8, 1, False), (16, 9, 1, True), (16, 2, 8, True)])
def test_route_and_results(log_n, level, count, tensor):
    p = W.Preset("route", W.CKKS, log_n, (50,) * 24, (60,) * 4, 3, log_n_max=16)
    ctx = api.Context(p)
    seed = W.seed_for(f"route-{log_n}-{level}-{count}")
    keys = ctx.keygen(seed)
    a, b = _uniform(ctx, seed, count, level), _uniform(ctx, seed, count, level, 100)
    # one ciphertext at N = 2^12 is below the line at every level
    q = W.Preset("route-small", W.CKKS, 12, (50,) * 24, (60,) * 4, 3, log_n_max=16)
    cs = api.Context(q)
    ks = cs.keygen(seed)
    x = cs.ct_uniform(seed, 0, level)
    _, base = _launches(lambda: cs.mul_relin(ks, x, x))
    got, n = _launches(lambda: ctx.mul_relin(keys, a, b))
    parts = 2 if count >= 4 and log_n >= 14 else 1
    assert n == parts * (base + (1 if tensor else 0))
    for j in {0, count // 2, count - 1}:
        assert torch.equal(ctx.mul_relin(keys, a[j:j + 1], b[j:j + 1]), got[j:j + 1]), j


@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
def test_both_routes_match_the_oracle_under_every_schedule(log_n):
    p = W.Preset("route-sched", W.CKKS, log_n, (50, 58, 61, 45), (61,), 4, log_n_max=16)
    ctx = api.Context(p)
    octx = oracle.Context(p.scheme, log_n, p.q_bits, p.p_bits, p.dnum, log_n_max=16)
    seed = W.seed_for(f"route-sched-{log_n}")
    keys, okeys = ctx.keygen(seed), octx.keygen(seed)
    parts = 2 if log_n >= 14 else 1
    many = parts * max(4, (1 << 20) // (6 * 5 << log_n) + 1)  # past the line in each part
    a, b = _uniform(ctx, seed, many, 4), _uniform(ctx, seed, many, 4, 1000)
    want = octx.mul_relin(okeys, ctx.export_ct(a[:1])[0], ctx.export_ct(b[:1])[0])
    scaled = octx.rescale(want)
    _, count, _ = ctx.ntt_schedule()
    for k in range(count):
        ctx.set_ntt_schedule(k)
        one, n1 = _launches(lambda: ctx.mul_relin(keys, a[:1], b[:1]))
        all_, n = _launches(lambda: ctx.mul_relin(keys, a, b))
        assert n == parts * (n1 + 1), k
        assert np.array_equal(ctx.export_ct(one)[0], want), k
        assert np.array_equal(ctx.export_ct(all_[:1])[0], want), k
        one, n1 = _launches(lambda: ctx.mul_relin_rescale(keys, a[:1], b[:1]))
        all_, n = _launches(lambda: ctx.mul_relin_rescale(keys, a, b))
        assert n == parts * (n1 + 1), k
        assert np.array_equal(ctx.export_ct(one)[0], scaled), k
        assert np.array_equal(ctx.export_ct(all_[:1])[0], scaled), k


@pytest.mark.parametrize("scheme,dnum", [(W.CKKS, 1), (W.CKKS, 3), (W.BGV, 8)])
def test_gathered_products_of_two_and_three(scheme, dnum):
    """Entries of one batch merged on one lane, with one digit to eight."""
    t = 0 if scheme == W.CKKS else 65537
    p = W.Preset("route-gathered", scheme, 12, (55,) * 8, (60,) * -(-8 // dnum), dnum, t=t,
                 log_n_max=12)
    ctx = api.Context(p)
    seed = W.seed_for(f"route-gathered-{dnum}")
    keys = ctx.keygen(seed)
    for count in (2, 3):
        ins = [(ctx.ct_uniform(seed, 2 * j, 8), ctx.ct_uniform(seed, 2 * j + 1, 8))
               for j in range(count)]
        want = [ctx.mul_relin(keys, x, y) for x, y in ins]
        outs = [torch.full_like(w, -1) for w in want]
        api.run_batch([api.make_op(api.OP_MUL_RELIN, ctx, x, o, keys=keys, b=y)
                       for (x, y), o in zip(ins, outs)], lanes=1)
        torch.cuda.synchronize()
        for j in range(count):
            assert torch.equal(outs[j], want[j]), (count, j)


@pytest.mark.parametrize("count,level", [(4, 3), (5, 9), (3, 4)])
def test_fused_products_over_their_inputs(count, level):
    """The result, a limb shorter, in the buffer of either input."""
    p = W.Preset("route-over", W.CKKS, 14, (50,) * 24, (60,) * 4, 3, log_n_max=16)
    ctx = api.Context(p)
    seed = W.seed_for(f"route-over-{count}")
    keys = ctx.keygen(seed)
    a, b = _uniform(ctx, seed, count, level), _uniform(ctx, seed, count, level, 100)
    want = ctx.mul_relin_rescale(keys, a, b)
    for which in (0, 1):
        ins = [a.clone(), b.clone()]
        out = ins[which].view(-1)[:want.numel()].view(want.shape)
        ctx.mul_relin_rescale(keys, ins[0], ins[1], out=out)
        assert torch.equal(out, want), which
