"""Which form a call's base conversions take, read from the library's count of
tensor-core conversions, that the results do not depend on it, and BFV's rounding
next to the boundary of its first conversion."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402
from test_gpu_conversion import COUNT, PRESETS  # noqa: E402


def _counted(f):
    before = api.tensor_conversions()
    out = f()
    return out, api.tensor_conversions() - before


# 24 primes in digits of 8: with 4 special primes ModUp at 8 limbs has 4
# targets and at 24 limbs 20, with 8 special primes ModDown at 4 limbs has 4
@pytest.mark.parametrize("log_n,specials,level,count,tensor", [
    (14, 4, 8, 16, 0), (14, 4, 8, 5, 0), (15, 4, 8, 11, 0), (13, 4, 8, 16, 1), (14, 4, 24, 4, 4),
    (15, 8, 4, 8, 0)])
def test_halves_take_the_integer_form_to_few_targets(log_n, specials, level, count, tensor):
    p = W.Preset("form", W.CKKS, log_n, (50,) * 24, (60,) * specials, 3, log_n_max=16)
    ctx = api.Context(p)
    seed = W.seed_for(f"form-{log_n}-{level}-{count}")
    keys = ctx.keygen(seed)
    g = ctx.galois_elt(1)
    keys.gen_galois(g)
    a = torch.cat([ctx.ct_uniform(seed, j, level) for j in range(count)])
    for call in (lambda x: ctx.mul_relin(keys, x, x), lambda x: ctx.rotate(keys, x, g)):
        got, n = _counted(lambda: call(a))
        assert n == tensor
        for j in (0, count - 1):
            assert torch.equal(call(a[j:j + 1]), got[j:j + 1]), j


# the conversions of one product of test_gpu_conversion's batches (its COUNT)
# that take the tensor cores: ModUp and ModDown, BFV's two lifts and its rounding
@pytest.mark.parametrize("name,least", [
    ("k8_t20", 2), ("k8_t24_two_passes", 2), ("k15", 2), ("k7_k6_small_primes", 1),
    ("six_digit_targets", 2), ("bgv", 1), ("bfv", 3), ("bfv_12_primes", 3), ("bfv_61", 0)])
def test_batches_reach_the_tensor_cores(name, least):
    p = next(p for p in PRESETS if p.name == name)
    ctx = api.Context(p)
    seed = W.seed_for("form-presets")
    keys = ctx.keygen(seed)
    a = torch.cat([ctx.ct_uniform(seed, j, p.L) for j in range(COUNT)])
    _, n = _counted(lambda: ctx.mul_relin(keys, a, a))
    assert n >= least and (n == 0) == (least == 0)


@pytest.mark.parametrize("name", ["bfv", "bfv_12_primes", "bfv_61"])
def test_bfv_rounding_next_to_its_boundary(name):
    """Products by the constant 1: t x mod Q next to Q/2, where the fixed-point
    quotient of the rounding's first conversion cannot decide, and up to four
    times as far from it as it can be off."""
    p = next(p for p in PRESETS if p.name == name)
    ctx = api.Context(p)
    octx = oracle.Context(p.scheme, p.log_n, p.q_bits, p.p_bits, p.dnum, t=p.t,
                          log_n_max=p.log_n_max, b_bits=p.b_bits)
    seed = W.seed_for(f"round-edges-{name}")
    keys, okeys = ctx.keygen(seed), octx.keygen(seed)
    qs = [int(q) for q in ctx.q[:p.L]]
    Q = 1
    for q in qs:
        Q *= q
    near = [0, 1, 2, Q >> 60, Q >> 40, Q >> 30] + [j * p.L * (Q >> 27) for j in (1, 3, 12)]
    vals = [(Q - 1) // 2 - d for d in near] + [(Q + 1) // 2 + d for d in near] + [0, 1, Q - 1]
    xs = [v * pow(p.t, -1, Q) % Q for v in vals]
    a = np.zeros((2, p.L, ctx.n), dtype=np.uint64)
    one = np.zeros((2, p.L, ctx.n), dtype=np.uint64)
    for i, q in enumerate(qs):
        a[0, i] = np.resize(np.array([x % q for x in xs], dtype=np.uint64), ctx.n)
        a[1, i] = np.resize(np.array([x % q for x in xs[::-1]], dtype=np.uint64), ctx.n)
    one[0, :, 0] = 1
    da, db = ctx.import_ct(a), ctx.import_ct(one)
    got, n = _counted(lambda: ctx.mul_relin(keys, da, db))
    assert (n > 0) == (name != "bfv_61")
    assert np.array_equal(ctx.export_ct(got)[0], octx.mul_relin(okeys, a, one))
    many = ctx.mul_relin(keys, da.repeat(COUNT, 1, 1, 1), db.repeat(COUNT, 1, 1, 1))
    assert torch.equal(many, got.expand_as(many))
