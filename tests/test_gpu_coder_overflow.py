"""A stream that does not fit its window: the window holds the stream's first bytes,
whatever carries come after it is full (needs a GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
from oracle.coder import RangeEncoder  # noqa: E402

pytestmark = pytest.mark.gpu


def _run_of_ff(steps, tail, over):
    """(cum, f) whose intervals hold the point 0x80 00 00 ..., so that low runs as 7F FF FF ..., for `steps`
    symbols; then one below the point (no carry) or above it (a carry through all of them); then `tail` more."""
    low, R, n = 0, 0xFFFFFFFF, 4
    pairs = []
    for k in range(steps + 1):
        point, r = 0x80 << (8 * (n - 1)), R >> 16
        at = min(max((point - low) // r, 1), 65530)  # the unit that holds the point
        c, f = (at - 1, 3) if k < steps else ((at + 2, 1) if over else (at - 1, 1))
        pairs.append((c, f))
        low, R = low + r * c, r * f
        while R < 1 << 24:
            R, low, n = R << 8, low << 8, n + 1
    return pairs + [(7 * k, 1) for k in range(tail)]


@pytest.mark.parametrize("encode", [edpc.range_encode, edpc.range_encode_noalloc])
@pytest.mark.parametrize("cap", [1, 2, 3, 4, 5, 6, 7, 8, 13, 16, 21])
def test_truncated_windows_hold_the_streams_first_bytes(encode, cap):
    pairs = [_run_of_ff(steps, tail, over) for steps in range(1, 14) for tail in (0, 5) for over in (False, True)]
    full = []
    for p in pairs:
        e = RangeEncoder()
        for c, f in p:
            e.encode(c, f)
        e.finish()
        full.append(bytes(e.out))  # with its trailing zeros
    assert any(b"\x7f\xff\xff\xff\xff\xff" in b for b in full) and any(b"\x80\x00\x00\x00\x00\x00" in b for b in full)
    sym = np.full((max(map(len, pairs)), len(pairs)), 0xFFFFFFFF, dtype=np.uint32)
    for s, p in enumerate(pairs):
        sym[:len(p), s] = [c | ((f - 1) << 16) for c, f in p]
    sd = torch.from_numpy(sym.view(np.int32)).cuda()
    out = torch.full((len(pairs) * cap,), 0xAB, dtype=torch.uint8, device="cuda")
    ln = torch.zeros(len(pairs), dtype=torch.int32, device="cuda")
    assert max(map(len, full)) > cap
    with pytest.raises(RuntimeError):
        encode(sd.data_ptr(), sym.shape[0], len(pairs), out.data_ptr(), cap, ln.data_ptr())
    out, ln = out.cpu().numpy().reshape(-1, cap), ln.cpu().numpy()
    for s, b in enumerate(full):
        if len(b) > cap:
            assert ln[s] == cap and bytes(out[s]) == b[:cap], s
        else:
            assert bytes(out[s, :ln[s]]) == b.rstrip(b"\x00"), s
