"""Whole-stream range encoding: windows at every alignment and carries that run
far back, against the oracle's coder, byte for byte (needs a GPU).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
from oracle.coder import RangeEncoder, quantize_cdf  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(pairs, cap):
    """pairs[s]: (cum, f) of stream s; streams shorter than the longest skip the rest."""
    streams, nsym = len(pairs), max(len(p) for p in pairs)
    sym = np.full((max(nsym, 1), streams), 0xFFFFFFFF, dtype=np.uint32)
    for s, p in enumerate(pairs):
        for t, (c, f) in enumerate(p):
            sym[t, s] = c | ((f - 1) << 16)
    sd = torch.from_numpy(sym.view(np.int32)).cuda()
    out = torch.full((streams * cap,), 0xAB, dtype=torch.uint8, device="cuda")
    ln = torch.zeros(streams, dtype=torch.int32, device="cuda")
    edpc.range_encode(sd.data_ptr(), nsym, streams, out.data_ptr(), cap, ln.data_ptr())
    out, ln = out.cpu().numpy(), ln.cpu().numpy()
    for s, p in enumerate(pairs):
        e = RangeEncoder()
        for c, f in p:
            e.encode(c, f)
        ref = e.finish()
        assert bytes(out[s * cap:s * cap + ln[s]]) == ref, (s, cap)


def _straddle(rng, steps):
    """Symbols whose intervals all hold the point 0x80 00 00 ... less one unit of a far byte, then the top symbol:
    low runs as 7F FF FF ... until the last symbol carries through all of it."""
    low, R, n = 0, 0xFFFFFFFF, 4
    pairs = []
    for k in range(steps + 1):
        f, cum = quantize_cdf(rng.dirichlet(np.full(256, 0.3)).astype(np.float32))
        r = R >> 16
        x = 255
        if k < steps:
            point = (0x80 << (8 * (n - 1))) - 1
            x = int(np.searchsorted(cum, min(max(point - low, 0) // r, 65535), side="right")) - 1
        c, w = int(cum[x]), int(f[x])
        pairs.append((c, w))
        low += r * c
        R = R - r * c if c + w == 65536 else r * w
        while R < 1 << 24:
            R <<= 8
            low <<= 8
            n += 1
    return pairs


@pytest.mark.parametrize("streams,nsym,cap", [(1, 0, 8), (1, 1, 9), (33, 7, 79), (5, 8, 81), (3, 9, 82), (70, 41, 147)])
def test_windows_of_any_alignment(streams, nsym, cap):
    rng = np.random.default_rng(streams * 100 + nsym)
    pairs = []
    for s in range(streams):
        n = nsym if s % 3 else max(0, nsym - s % 5)
        f, cum = quantize_cdf(rng.dirichlet(np.full(256, 0.2), size=max(n, 1)).astype(np.float32))
        x = rng.integers(0, 256, size=max(n, 1))
        pairs.append([(int(cum[t, x[t]]), int(f[t, x[t]])) for t in range(n)])
    _run(pairs, cap)


def test_carries_run_back():
    rng = np.random.default_rng(9)
    _run([_straddle(rng, steps) for steps in range(1, 60)], 2 * 61 + 65)
