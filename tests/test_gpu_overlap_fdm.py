"""The FDM update on its own stream gives the fused adjoint's results: the same container,
which any decoder reads (needs a GPU)."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [edpc.EDPC_BF16, edpc.EDPC_FP8E4M3])
@pytest.mark.parametrize("latent", [0, 8, 72, 128, 200, 256, 384, 512, 1024])  # 0: the FDM is F x F, F = 128
def test_overlapped_update_codes_the_same_container(prec, latent):
    b, steps = (40, 100) if latent <= 256 else (12, 70)
    kw = dict(streams=b, precision=prec, context=8, embed_dim=16, latent=latent, hidden=64, blocks=2, branches=2, seed=3)
    x = synth.markov_bytes(b * (8 + steps) - 5, 1, 0.1, latent)
    bits = edpc.compress(x, edpc.make_cfg(flags=edpc.EDPC_FLAG_OVERLAP_FDM, **kw))
    assert np.array_equal(edpc.decompress(bits), x)
    assert bits == edpc.compress(x, edpc.make_cfg(**kw))
