"""FP32 GEMM tiles: logits and gradients of models whose layers take each tile and
leave remainders in every direction, against the FP64 oracle (needs a GPU).

The benchmark spec's bounds hold: |dz| <= 1e-3 max|z|, |dg| <= 1e-3 max|g| a tensor.
"""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
from oracle.model import Config, Model as OModel, softmax  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("context,embed_dim,latent,hidden,branches,b", [
    (5, 8, 8, 24, 1, 1),        # 8 x 8 tiles, one row
    (11, 8, 72, 40, 3, 37),     # 8 x 8 tiles, remainders
    (25, 16, 40, 136, 2, 150),  # 8 x 16 and 16 x 32 tiles
    (36, 8, 16, 392, 2, 331),   # 16 x 32 and 32 x 64 tiles
    (65, 16, 8, 1032, 1, 1030),  # 64 x 64 tiles in every layout
])
def test_logits_and_gradients(context, embed_dim, latent, hidden, branches, b):
    dims = dict(context=context, embed_dim=embed_dim, latent=latent, hidden=hidden, blocks=2, branches=branches, seed=3)
    m = edpc.Model(edpc.make_cfg(precision=edpc.EDPC_FP32, **dims), b)
    om = OModel(Config(**dims), b)
    rng = np.random.default_rng(b)
    ctx = rng.integers(0, 256, size=(b, context)).astype(np.uint8)
    tg = rng.integers(0, 256, size=b).astype(np.uint8)
    z, _ = m.forward(ctx)
    g, _ = m.backward(ctx, tg, np.ones(b, np.uint8))
    zo, cache = om.forward(ctx.astype(np.int64))
    assert np.abs(z - zo).max() <= 1e-3 * np.abs(zo).max()
    dz = softmax(zo)
    dz[np.arange(b), tg] -= 1
    go, _ = om.backward(cache, dz / b)
    o = 0
    for name, shape, _ in om.layout:
        n = int(np.prod(shape))
        ref = np.asarray(go[name], np.float64).reshape(-1)
        assert np.abs(g[o:o + n] - ref).max() <= 1e-3 * np.abs(ref).max(), name
        o += n
