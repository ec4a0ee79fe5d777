"""Profiling a short session does not pay for graphs that a long one would need (needs a GPU)."""
import time

import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [edpc.EDPC_FP32, edpc.EDPC_BF16])
def test_one_step_more_costs_less_than_half_again(prec):
    """63 and 64 steps, each timed as a whole: opening, profiling, running and closing."""
    b, K = 4, 16
    cfg = edpc.make_cfg(streams=b, precision=prec)
    x = synth.markov_bytes(b * (K + 64), 1, 0.1, 5)
    best = {63: 1e9, 64: 1e9}
    for _ in range(12):
        for n in best:
            t = time.perf_counter()
            with edpc.Encoder(cfg, x[:b * (K + n)]) as e:
                e.profile(True)
                e.run(n)
                e.profile(False)
                e.finish()
                samples = e.stats().fdm_samples
            best[n] = min(best[n], time.perf_counter() - t)
            assert samples == n
    assert best[64] <= 1.5 * best[63]
