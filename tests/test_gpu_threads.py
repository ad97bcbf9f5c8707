"""Two host threads on one context: their first calls, which build the kept
constants, plans, lift tables and encoder tables, at the same time, each on its
own stream with its own workspace and levels, against a context that one thread
uses."""
import threading

import numpy as np
import pytest

from paper_2503_22227_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_22227_gb300 import api  # noqa: E402

P = W.Preset("threads", W.CKKS, 12, (50,) * 8, (60,) * 2, 3, log_n_max=12, log_scale=40)
SEED = W.seed_for("threads")


def _calls(ctx, keys, g, level):
    """One call of each kind that keeps something in the context."""
    a, b = (ctx.ct_uniform(SEED, i, level) for i in (0, 1))
    slots = W.complex_slots(W.rng_for(f"threads-{level}"), ctx.n)
    return [ctx.encode_ckks(slots, 2.0 ** 40, level), ctx.mul_relin(keys, a, b),
            ctx.mul_relin_rescale(keys, a, b), ctx.rotate(keys, a, g), ctx.rescale(a),
            ctx.rotate_hoisted(keys, a, [g, g]),
            torch.from_numpy(ctx.decrypt(keys, a)),
            torch.from_numpy(np.ascontiguousarray(ctx.decode_ckks(keys, a, 2.0 ** 40)))]


def _context():
    ctx = api.Context(P)
    keys = ctx.keygen(SEED)
    g = ctx.galois_elt(1)
    keys.gen_galois(g)
    return ctx, keys, g


def test_first_calls_of_two_threads():
    levels = ((8, 5, 3), (7, 6, 4))
    ctx, keys, g = _context()
    want = {l: [t.cpu() for t in _calls(ctx, keys, g, l)] for ls in levels for l in ls}
    for trial in range(8):
        ctx, keys, g = _context()
        torch.cuda.synchronize()
        start, got, errors = threading.Barrier(2), {}, []

        def work(own):
            try:
                with torch.cuda.stream(torch.cuda.Stream()):
                    start.wait()
                    for l in own:
                        got[l] = [t.cpu() for t in _calls(ctx, keys, g, l)]
            except Exception as e:  # shown by the main thread
                errors.append(e)

        threads = [threading.Thread(target=work, args=(ls,)) for ls in levels]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors
        for l, outs in want.items():
            for i, (x, y) in enumerate(zip(got[l], outs)):
                assert torch.equal(x, y), (trial, l, i)
