"""What a session costs and codes, by its number of steps (needs a GPU)."""
import time

import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [edpc.EDPC_FP32, edpc.EDPC_BF16])
@pytest.mark.parametrize("steps", [16, 24, 32])
def test_a_short_session_costs_no_more_a_step_than_a_shorter_one(prec, steps):
    """A fixed cost and one per step: n times the steps cost at most n times the time."""
    b, K = 4, 16
    cfg = edpc.make_cfg(streams=b, precision=prec)
    x = synth.markov_bytes(b * (K + steps), 1, 0.1, steps)
    best = {8: 1e9, steps: 1e9}
    for _ in range(15):
        for n in best:
            part = x[:b * (K + n)]
            t = time.perf_counter()
            edpc.compress(part, cfg)
            best[n] = min(best[n], time.perf_counter() - t)
    assert best[steps] <= steps / 8 * best[8]


@pytest.mark.parametrize("prec", [edpc.EDPC_FP32, edpc.EDPC_BF16])
@pytest.mark.parametrize("steps", [1023, 1024, 1037])
def test_long_sessions_code_the_same_bytes(prec, steps):
    """On both sides of the length from which several steps share a graph."""
    b = 3
    dims = dict(context=8, embed_dim=8, latent=64, hidden=64, blocks=1, branches=2, seed=5)
    x = synth.markov_bytes(b * (8 + steps) - 1, 1, 0.1, steps)
    ref = edpc.compress(x, edpc.make_cfg(streams=b, precision=prec, flags=edpc.EDPC_FLAG_NO_GRAPH, **dims))
    cfg = edpc.make_cfg(streams=b, precision=prec, **dims)
    assert edpc.compress(x, cfg) == ref
    assert np.array_equal(edpc.decompress(ref), x)
    with edpc.Encoder(cfg, x) as e:  # odd advances, profiling turned on and off between them
        for k, n in enumerate((1, 8, 3, 70, 64, 40)):
            e.profile(k % 2 == 1)
            e.run(n)
        e.profile(False)
        assert e.finish() == ref
