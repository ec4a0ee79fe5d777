"""Embedding adjoint with few distinct bytes vs the FP64 oracle (needs a GPU).

Frequent bytes fill the adjoint's position lists and copy stages; the cases put
their edges (embedding widths whose rows do not divide a stage, position counts
that are no multiple of a block, several position chunks) against the oracle's
gradient. FP32, so the benchmark spec's bound holds: |dg| <= 1e-3 max|g| an element.
"""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
from oracle.model import Config, Model as OModel, softmax  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("context,embed_dim,b,symbols", [(3, 8, 1, 1), (11, 24, 37, 2), (32, 16, 130, 1),
                                                         (7, 40, 85, 3), (5, 64, 53, 2), (64, 16, 300, 2),
                                                         (128, 8, 160, 1)])
def test_frequent_bytes(context, embed_dim, b, symbols):
    dims = dict(context=context, embed_dim=embed_dim, latent=16, hidden=16, blocks=1, branches=1, lr=1e-3, seed=3)
    m = edpc.Model(edpc.make_cfg(precision=edpc.EDPC_FP32, **dims), b)
    om = OModel(Config(**dims), b)
    rng = np.random.default_rng(b)
    ctx = rng.integers(0, symbols, size=(b, context)).astype(np.uint8) * 127
    ctx[rng.random(ctx.shape) < 0.02] = 255
    tg = rng.integers(0, 256, size=b).astype(np.uint8)
    g, _ = m.backward(ctx, tg, np.ones(b, np.uint8))
    zo, cache = om.forward(ctx.astype(np.int64))
    dz = softmax(zo)
    dz[np.arange(b), tg] -= 1
    go, _ = om.backward(cache, dz / b)
    n = 256 * embed_dim
    ref = OModel.flat_grads(om.layout, go)[:n].reshape(256, -1)
    got = g[:n].reshape(256, -1)
    assert np.abs(got - ref).max() <= 1e-3 * np.abs(ref).max()
    used = np.unique(ctx)
    assert not got[np.setdiff1d(np.arange(256), used)].any()
