"""A launch with several incoming dependencies waits for all of them in full (needs a GPU).

The library's kernels are launched with programmatic dependent launch only where
the preceding kernel on the stream is all they follow; where the stream has also
waited on an event they are launched without it. Eager steps are captured into a
graph here, and its edges are read back.
"""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

import paper_2507_18969_gb300 as edpc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu

EAGER = edpc.EDPC_FLAG_NO_GRAPH | edpc.EDPC_FLAG_NO_PIPELINE
THREAD_LOCAL, PROGRAMMATIC = 1, 1


class EdgeData(C.Structure):
    _fields_ = [("from_port", C.c_ubyte), ("to_port", C.c_ubyte), ("type", C.c_ubyte), ("reserved", C.c_ubyte * 5)]


def _captured_edges(enc, stream, steps):
    rt = C.CDLL("libcudart.so.13")
    st, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t()
    assert rt.cudaStreamBeginCapture(st, THREAD_LOCAL) == 0
    try:
        enc.run(steps, sync=False)
    finally:
        assert rt.cudaStreamEndCapture(st, C.byref(graph)) == 0
    assert rt.cudaGraphGetEdges(graph, None, None, None, C.byref(n)) == 0
    a, b, e = (C.c_void_p * n.value)(), (C.c_void_p * n.value)(), (EdgeData * n.value)()
    assert rt.cudaGraphGetEdges(graph, a, b, e, C.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return [(a[k], b[k], e[k].type) for k in range(n.value)]


@pytest.mark.parametrize("prec,flags", [(edpc.EDPC_FP32, 0), (edpc.EDPC_BF16, 0), (edpc.EDPC_FP8E4M3, 0),
                                        (edpc.EDPC_BF16, edpc.EDPC_FLAG_OVERLAP_FDM),
                                        (edpc.EDPC_FP32, edpc.EDPC_FLAG_DELAYED_UPDATE),
                                        (edpc.EDPC_BF16, edpc.EDPC_FLAG_DELAYED_UPDATE)])
def test_programmatic_edges_lead_to_kernels_with_one_dependency(prec, flags):
    b = 6
    cfg = edpc.make_cfg(streams=b, precision=prec, flags=flags | EAGER, context=8, embed_dim=8, latent=64, hidden=64,
                        blocks=2, branches=2, seed=5)
    stream = torch.cuda.Stream()
    with edpc.Encoder(cfg, synth.markov_bytes(b * 40, 1, 0.1, 3), stream=stream.cuda_stream) as enc:
        enc.run(2)  # beyond the first step of every schedule
        edges = _captured_edges(enc, stream, 4)
    assert any(t == PROGRAMMATIC for _, _, t in edges)
    several = {v for _, v, _ in edges if sum(v == w for _, w, _ in edges) > 1}
    assert not [v for _, v, t in edges if t == PROGRAMMATIC and v in several]
