"""Forward passes of an FP8 model may be repeated without end (needs a GPU)."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402

pytestmark = pytest.mark.gpu


def test_fp8_forward_repeats_and_leaves_the_gradient_alone():
    b = 20
    cfg = edpc.make_cfg(precision=edpc.EDPC_FP8E4M3, context=8, embed_dim=8, latent=64, hidden=64, blocks=3, branches=2)
    rng = np.random.default_rng(1)
    ctx = rng.integers(0, 256, (b, 8)).astype(np.uint8)
    tg = rng.integers(0, 256, b).astype(np.uint8)
    on = np.ones(b, np.uint8)
    fresh, m = edpc.Model(cfg, b), edpc.Model(cfg, b)
    g, gu = fresh.backward(ctx, tg, on)
    z, _ = m.forward(ctx)
    for _ in range(130):  # more than a step has side-stream forks to give
        zk, _ = m.forward(ctx)
    assert np.array_equal(zk, z)
    gk, guk = m.backward(ctx, tg, on)
    assert np.array_equal(gk, g) and np.array_equal(guk, gu)
    for _ in range(130):
        m.forward(ctx)
    m.train_step(ctx, tg, on)
    fresh.close()
    m.close()
