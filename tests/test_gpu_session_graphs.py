"""Sessions advance through multi-step graphs, one-step graphs and, while
profiling, graphs with event records: every mix codes the same bytes (needs a GPU).
"""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu

DIMS = dict(context=8, embed_dim=8, latent=64, hidden=64, blocks=2, branches=2, seed=5)


@pytest.mark.parametrize("prec,flags", [(edpc.EDPC_FP32, 0), (edpc.EDPC_BF16, 0),
                                        (edpc.EDPC_BF16, edpc.EDPC_FLAG_DELAYED_UPDATE),
                                        (edpc.EDPC_BF16, edpc.EDPC_FLAG_OVERLAP_FDM)])
@pytest.mark.parametrize("steps", [1, 15, 16, 17, 64, 209])
def test_any_advance_codes_the_same_bytes(prec, flags, steps):
    b = 6
    x = synth.markov_bytes(b * (8 + steps), 1, 0.1, steps)
    eager = edpc.make_cfg(streams=b, precision=prec, flags=flags | edpc.EDPC_FLAG_NO_GRAPH, **DIMS)
    cfg = edpc.make_cfg(streams=b, precision=prec, flags=flags, **DIMS)
    ref = edpc.compress(x, eager)
    assert edpc.compress(x, cfg) == ref
    with edpc.Encoder(cfg, x) as e:  # odd advances, profiling turned on and off between them
        for k, n in enumerate((1, 16, 3, 70, 64, 40)):
            e.profile(k % 2 == 1)
            e.run(n)
        e.profile(False)
        assert e.finish() == ref
        st = e.stats()
    assert st.fdm_samples == min(max(steps - 154, 0), 40)  # counted since profiling was last turned on
    if not flags & edpc.EDPC_FLAG_OVERLAP_FDM:
        assert np.array_equal(edpc.decompress(ref), x)
