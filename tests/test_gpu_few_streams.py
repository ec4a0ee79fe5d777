"""The GEMMs with the streams on the MMA's N side give the 128-row kernels' bits:
logits and gradients with the default plan against tile code 17 (persistent
kernel, N tiles of 32) at every site (needs a GPU).
"""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("context,embed_dim,latent,hidden,branches,b", [
    (5, 8, 8, 8, 1, 1),         # one K block, one stream
    (5, 8, 40, 40, 3, 31),      # 32-unit sections with a remainder
    (11, 8, 72, 200, 2, 33),    # 64-unit sections with a remainder; two stream tiles
    (32, 16, 256, 256, 2, 512),  # the 64 MiB mix's layers
    (16, 16, 136, 136, 1, 129),  # 128-unit tiles with a remainder
    (64, 16, 64, 512, 3, 700),  # more than eight K blocks; 64-stream tiles in the widest layers
    (40, 16, 16, 72, 2, 1500),  # 64-stream tiles
])
def test_same_bits_as_the_row_kernels(context, embed_dim, latent, hidden, branches, b):
    cfg = edpc.make_cfg(precision=edpc.EDPC_BF16, context=context, embed_dim=embed_dim, latent=latent, hidden=hidden,
                        blocks=2, branches=branches, seed=b)
    rng = np.random.default_rng(b)
    ctx = rng.integers(0, 256, size=(b, context)).astype(np.uint8)
    tg = rng.integers(0, 256, size=b).astype(np.uint8)
    on = (rng.random(b) < 0.9).astype(np.uint8)
    on[0] = 1
    out = []
    for code in (0, 17):
        m = edpc.Model(cfg, b)
        if code:
            m.set_tiles(np.full(200, code, np.uint8))
        z, p = m.forward(ctx)
        g, gu = m.backward(ctx, tg, on)
        out.append((z, p, g, gu))
        m.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
