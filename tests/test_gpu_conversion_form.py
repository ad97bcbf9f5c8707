"""Which form a call's base conversions take, read from the library's count of
tensor-core conversions, and that the results do not depend on it."""
import pytest

from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


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
