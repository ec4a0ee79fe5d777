"""Kraskov counts at the edges of the distance tiles and panels vs the oracle (needs a GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
from oracle.mi import ksg_counts, ksg_mi  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dz,dy,k", [(2, 1, 3, 1), (64, 32, 36, 2), (65, 33, 4, 33), (129, 31, 65, 32), (192, 4, 64, 64),
                                       (3001, 3, 2, 5)])  # the last needs several row panels
@pytest.mark.parametrize("offset", [0, 1])  # base addresses on and off a 16-byte boundary
def test_counts(n, dz, dy, k, offset):
    rng = np.random.default_rng(n + dz)
    Z = rng.normal(size=(n, dz)).astype(np.float32)
    Y = (0.5 * Z[:, :1] + rng.normal(size=(n, dy))).astype(np.float32)
    dev = []
    for a in (Z, Y):
        buf = torch.zeros(a.size + 4, device="cuda")
        buf[offset:offset + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
        dev.append(buf)
    cz = torch.zeros(n, dtype=torch.int32, device="cuda")
    cy = torch.zeros_like(cz)
    mi = edpc.ksg_mi(dev[0].data_ptr() + 4 * offset, dev[1].data_ptr() + 4 * offset, n, dz, dy, k, cz.data_ptr(),
                     cy.data_ptr())
    _, oz, oy = ksg_counts(Z, Y, k)
    assert np.array_equal(cz.cpu().numpy(), oz) and np.array_equal(cy.cpu().numpy(), oy)
    assert abs(mi - ksg_mi(Z, Y, k)) < 1e-9
