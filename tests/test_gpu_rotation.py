"""Rotations with the permutation in the result's last kernel: every NTT
schedule of every ring degree (each has its own chunk sizes, which the
permuted store works on) against the oracle, steps in both directions and the
conjugation, and results written over their inputs."""
import numpy as np
import pytest

import oracle
from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402


@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
def test_rotation_matches_oracle_under_every_schedule(log_n):
    p = W.Preset("rot", W.CKKS, log_n, (50, 58), (60,), 1, log_n_max=16)
    ctx = api.Context(p)
    octx = oracle.Context(p.scheme, log_n, p.q_bits, p.p_bits, p.dnum, log_n_max=16)
    seed = W.seed_for(f"rot-keys-{log_n}")
    keys, okeys = ctx.keygen(seed), octx.keygen(seed)
    a = octx.ct_uniform(W.seed_for("rot-in"), log_n, p.L)
    da = ctx.import_ct(a)
    gs = [ctx.galois_elt(1), ctx.galois_elt(-3), 2 * ctx.n - 1]
    want = []
    for g in gs:
        keys.gen_galois(g)
        okeys.gen_galois(g)
        want.append(octx.rotate(okeys, a, g))
    _, count, _ = ctx.ntt_schedule()
    for k in range(count):
        ctx.set_ntt_schedule(k)
        hoisted = ctx.rotate_hoisted(keys, da, gs)
        for j, g in enumerate(gs):
            assert np.array_equal(ctx.export_ct(ctx.rotate(keys, da, g))[0], want[j]), (k, g)
            assert np.array_equal(ctx.export_ct(hoisted[j])[0], want[j]), (k, g)


@pytest.mark.parametrize("scheme,count", [(W.CKKS, 2), (W.CKKS, 5), (W.BGV, 1), (W.BFV, 1),
                                          (W.BFV, 5)])
def test_rotation_over_its_input(scheme, count):
    t = 0 if scheme == W.CKKS else 65537
    p = W.Preset("rot-in-place", scheme, 14, (50,) * 3, (60,), 3, t=t, log_n_max=14)
    ctx = api.Context(p)
    keys = ctx.keygen(W.seed_for("rot-in-place"))
    seed = W.seed_for("rot-in-place-in")
    a = torch.cat([ctx.ct_uniform(seed, i, p.L) for i in range(count)])
    for g in (ctx.galois_elt(5), 2 * ctx.n - 1):
        keys.gen_galois(g)
        want = ctx.rotate(keys, a, g)
        same = a.clone()
        ctx.rotate(keys, same, g, out=same)
        assert torch.equal(same, want), g


@pytest.mark.parametrize("log_n,dnum,L", [(12, 1, 3), (12, 2, 4), (12, 3, 5), (13, 8, 8),
                                          (12, 9, 9), (14, 1, 2), (14, 4, 7), (15, 5, 5)])
def test_paired_rotations_equal_single_ones(log_n, dnum, L):
    """1 to 9 digits (pairs from 2 to 8), every remainder of the pairs over one
    and two streams, one ciphertext (one buffer), two and five, a level with a
    partly used last digit, and an element given twice."""
    p = W.Preset("rot-pairs", W.CKKS, log_n, (50,) * L, (60,) * 4, dnum, log_n_max=16)
    ctx = api.Context(p)
    keys = ctx.keygen(W.seed_for(f"rot-pairs-{log_n}-{dnum}"))
    gs = [ctx.galois_elt(r) for r in (1, -3, 5, 2, 7)] + [2 * ctx.n - 1, ctx.galois_elt(1)]
    for g in gs:
        keys.gen_galois(g)
    seed = W.seed_for("rot-pairs-in")
    for level in {L, max(1, L - 1)}:
        for count in (1, 2, 5):
            a = torch.cat([ctx.ct_uniform(seed, i, level) for i in range(count)])
            want = [ctx.rotate(keys, a, g) for g in gs]
            for n_rot in range(1, len(gs) + 1):
                out = ctx.rotate_hoisted(keys, a, gs[:n_rot])
                for j in range(n_rot):
                    assert torch.equal(out[j], want[j]), (level, count, n_rot, j)
