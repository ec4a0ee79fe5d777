"""What the performance of this framework is measured on.

Each case is work that a user has the library do, through the Python binding of
its C ABI (``paper_2507_18969_gb300``): whole compressions and decompressions of
host buffers, one model step with its gradient, and the single device kernels
that the ABI exports. The model dimensions are those of the repository's
configurations: the library's default configuration, the 64 MiB mix (512
streams, F = 512, F' = 256), the 1 GiB mix (4096 streams, F = 1024, F' = 512),
file sets, archives of independent models, and odd sizes as the tests use them.
A whole 64 MiB input takes 130,000 model steps per stream and would only repeat
the same step, so the inputs here are prefixes: every stream holds its context
and then some hundred bytes.

The FP8 precision, the delayed-update schedule and the FDM update on its own
stream are kept for comparison (slower, or much worse in size, at the measured
dimensions) and the model without the LTE is an ablation: none is a case.
File sets time their GEMM tiles when they are written, so two containers of the
same files may differ; the file-set case therefore decodes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_18969_gb300 as edpc

PRECISION = {"fp32": edpc.EDPC_FP32, "bf16": edpc.EDPC_BF16}
DIMS = ("context", "embed_dim", "latent", "hidden", "blocks", "branches")
SMALL = dict(context=16, embed_dim=16, latent=128, hidden=128, blocks=2, branches=2)   # the default configuration
MIX64M = dict(context=32, embed_dim=16, latent=256, hidden=256, blocks=4, branches=2)  # the 64 MiB mix
MIX1G = dict(context=64, embed_dim=16, latent=512, hidden=512, blocks=6, branches=2)   # the 1 GiB mix
ODD = dict(context=11, embed_dim=8, latent=72, hidden=40, blocks=3, branches=3)        # no dimension a multiple of a tile


def listed():
    return [
        # a short buffer under the default configuration (FP32, four streams): latency and launches only
        dict(name="small_compress_fp32", kind="compress", precision="fp32", streams=4, steps=512, **SMALL),
        # the 64 MiB mix, the benchmark's workload, in both directions
        dict(name="mix64m_compress_bf16", kind="compress", precision="bf16", streams=512, steps=768, **MIX64M),
        dict(name="mix64m_decompress_bf16", kind="decompress", precision="bf16", streams=512, steps=768, **MIX64M),
        # the 1 GiB mix: the largest model and batch
        dict(name="mix1g_compress_bf16", kind="compress", precision="bf16", streams=4096, steps=96, **MIX1G),
        # the plain FP32 arithmetic at the 64 MiB mix's dimensions
        dict(name="mix64m_compress_fp32", kind="compress", precision="fp32", streams=512, steps=192, **MIX64M),
        # a small batch of odd sizes: ragged streams, three branches, tails of every tile
        dict(name="odd_compress_bf16", kind="compress", precision="bf16", streams=37, steps=500, **ODD),
        # reading back a file set of uneven sizes (one model, masked streams)
        dict(name="files_decompress_bf16", kind="files", precision="bf16", streams=900, files=60, longest=20000, **MIX64M),
        # an archive whose files each have a model of their own
        dict(name="independent_compress_bf16", kind="independent", precision="bf16", files=12, longest=40000,
             stream_len=512, **MIX64M),
        # the model API: logits and the gradient of one step
        dict(name="gradient_bf16", kind="gradient", precision="bf16", streams=64, **MIX64M),
        # the quantizer on the rows of the 1000-file set's batch
        dict(name="cdf_quantize", kind="quantize", rows=32291),
        # the range coder on the 1 GiB mix's streams
        dict(name="range_encode", kind="encode", streams=4096, nsym=1024),
        # the mutual-information estimate between a block's input and output
        dict(name="ksg_mi", kind="ksg", samples=2048, dims=512, k=3),
    ]


# ---- drawn cases --------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng):
    """Model dimensions over the library's range as the configurations and the tests use it."""
    return dict(context=rng.choice([5, 8, 11, 16, 32, 32, 64]), embed_dim=rng.choice([8, 16, 16]),
                latent=rng.choice([40, 64, 128, 200, 256, 256, 512]), hidden=rng.choice([40, 64, 128, 256, 256, 512]),
                blocks=rng.randint(1, 6), branches=rng.choice([1, 2, 2, 2, 3]))


def _step_seconds(c):
    """A generous estimate of one model step, to bound what a drawn case costs."""
    p = _gemm_weights(c)
    b = c["streams"]
    rate = 6e12 if c["precision"] == "fp32" else 1e14
    return (60e-6 + 70e-6 * c["blocks"]) + 28.0 * b * c["latent"] ** 2 / 4e12 + 6.0 * b * p / rate


def draw(rng):
    kind = rng.choice(["compress", "compress", "compress", "decompress", "decompress", "files", "independent",
                       "gradient", "quantize", "encode", "ksg"])
    if kind == "quantize":
        return dict(kind=kind, rows=_log(rng, 64, 65535))
    if kind == "encode":
        streams = _log(rng, 4, 16384)
        return dict(kind=kind, streams=streams, nsym=max(16, min(_log(rng, 16, 4096), (4 << 20) // streams)))
    if kind == "ksg":
        samples = _log(rng, 64, 2048)
        return dict(kind=kind, samples=samples, dims=_log(rng, 2, 512), k=rng.randint(1, 8))
    c = dict(kind=kind, precision=rng.choice(["bf16", "bf16", "fp32"]), **_dims(rng))
    if kind == "gradient":
        return dict(c, streams=min(_log(rng, 1, 512), max(1, (1 << 23) // c["latent"] ** 2)))
    if kind == "files":
        return dict(c, precision="bf16", streams=_log(rng, 30, 300), files=rng.randint(2, 30), longest=_log(rng, 800, 8000))
    if kind == "independent":
        # one model per file: few streams each, bounded so that the longest stream stays short
        return dict(c, precision="bf16", files=rng.randint(2, 10), longest=_log(rng, 2000, 30000),
                    stream_len=_log(rng, 128, 400))
    c["streams"] = _log(rng, 1, 4096)
    c["steps"] = max(8, min(_log(rng, 60, 700), int(0.35 / _step_seconds(c))))
    return c


# ---- inputs -------------------------------------------------------------------------------
def _media(n, rng):
    """n bytes shaped like the multimedia mix: thirds of image rows, 16-bit PCM and text."""
    parts = [n - 2 * (n // 3), n // 3, n // 3]
    i = np.arange(parts[0])
    x, y = i % 512, i // 512
    img = 128 + 0.2 * x - 0.1 * (y % 512) + 30 * np.cos(0.02 * x + 0.01 * y + rng.uniform(0, 6)) + rng.normal(0, 4, i.size)
    t = np.arange(parts[1] // 2 + 1) / 44100.0
    pcm = sum(a * np.sin(2 * np.pi * f * t) for a, f in zip(rng.uniform(1000, 8000, 3), rng.uniform(50, 4000, 3)))
    pcm = np.clip(pcm + rng.normal(0, 200, t.size), -32768, 32767).astype("<i2")
    words = rng.integers(97, 123, size=(2000, 6)).astype(np.uint8)
    words[np.arange(2000), rng.integers(2, 6, 2000)] = 32
    text = words[np.minimum(rng.zipf(1.3, parts[2] // 6 + 1) - 1, 1999)].reshape(-1)
    return np.concatenate([np.clip(np.rint(img), 0, 255).astype(np.uint8), pcm.view(np.uint8)[:parts[1]],
                           text[:parts[2]]])


def _cfg(c, **kw):
    return edpc.make_cfg(precision=PRECISION[c["precision"]], **{d: c[d] for d in DIMS}, **kw)


def _file_sizes(c):
    """Log-uniform sizes up to the longest (one file has it), as the uneven file set's: the case's own, for any seed."""
    rng = np.random.default_rng([c["files"], c["longest"]])
    s = np.exp(rng.uniform(np.log(c["longest"] / 40), np.log(c["longest"]), c["files"])).astype(int)
    s[0] = c["longest"]
    return [int(v) for v in s]


def _tensors(c):
    """Shapes of the shared parameters in the ABI's canonical order, with the scale of their initial values."""
    F, H, L, k = c["context"] * c["embed_dim"], c["hidden"], c["latent"], c["branches"]
    out = [((256, c["embed_dim"]), 3 ** 0.5)]
    for _ in range(c["blocks"]):
        out += [((F,), None), ((F,), 0.0), ((k * H, F), F ** -0.5), ((k * H,), F ** -0.5), ((F, H), H ** -0.5),
                ((F,), H ** -0.5)]
    return out + [((L, F), F ** -0.5), ((L,), F ** -0.5), ((F, L), L ** -0.5), ((F,), L ** -0.5), ((256, F), F ** -0.5),
                  ((256,), F ** -0.5)]


def _gradient_inputs(c, seed):
    """Parameters like the library's initial ones, contexts, targets, and some streams that have ended."""
    rng = np.random.default_rng([seed, 7])
    shared = [(np.ones(s) if a is None else rng.uniform(-1, 1, s) * a).astype(np.float32) for s, a in _tensors(c)]
    b, L = c["streams"], c["latent"]
    fdm = ((rng.random((b, L, L), dtype=np.float32) * 2 - 1) * np.float32((3 / L) ** 0.5))
    ctx = rng.integers(0, 256, (b, c["context"])).astype(np.uint8)
    targets = rng.integers(0, 256, b).astype(np.uint8)
    active = (rng.random(b) < 0.9).astype(np.uint8)
    active[0] = 1
    return shared, fdm, ctx, targets, active


def _whole(container, n, rows):
    """A container's bytes and length in an array whose size does not depend on them (n bytes coded in `rows` rows)."""
    out = np.zeros(2 * n + 512 * rows + 4096, np.uint8)
    out[:len(container)] = np.frombuffer(container, np.uint8)
    return out, len(container)


def prepare(case, seed):
    c, kind = case, case["kind"]
    rng = np.random.default_rng([seed, 11])
    if kind in ("compress", "decompress"):
        # every stream holds its context and `steps` more bytes; the last few streams are one byte shorter
        n = c["streams"] * (c["context"] + c["steps"]) - min(3, c["streams"] - 1)
        data, cfg = _media(n, rng), _cfg(c, streams=c["streams"])
        return (kind, edpc.compress(data, cfg)) if kind == "decompress" else (kind, data, cfg)
    if kind == "files":
        files = [_media(n, rng) for n in _file_sizes(c)]
        return kind, edpc.compress_many(files, _cfg(c, streams=c["streams"]))
    if kind == "independent":
        return kind, [_media(n, rng) for n in _file_sizes(c)], _cfg(c), c["stream_len"]
    if kind == "gradient":
        shared, fdm, ctx, targets, active = _gradient_inputs(c, seed)
        m = edpc.Model(_cfg(c, streams=c["streams"]), c["streams"])
        m.set_state(P=np.concatenate([t.reshape(-1) for t in shared]), U=fdm.reshape(-1))
        return kind, m, ctx, targets, active
    g = torch.Generator("cuda").manual_seed(seed)
    if kind == "quantize":
        # softmax rows from flat to peaked, as a model's predictions are
        z = torch.randn(c["rows"], 256, device="cuda", generator=g)
        z *= torch.rand(c["rows"], 1, device="cuda", generator=g) * 4
        return (kind, torch.softmax(z, 1), torch.empty(c["rows"], 256, device="cuda", dtype=torch.int32),
                torch.empty(c["rows"], 257, device="cuda", dtype=torch.int32))
    if kind == "encode":
        # symbols drawn from 64 integer CDFs of 2 to 8 bits of entropy
        p = rng.dirichlet(np.full(256, 0.05), 32).tolist() + rng.dirichlet(np.full(256, 1.0), 32).tolist()
        f = 1 + np.floor(np.array(p) * 65280).astype(np.int64)
        f[np.arange(64), f.argmax(1)] += 65536 - f.sum(1)
        cum = np.cumsum(f, 1) - f
        row = rng.integers(0, 64, (c["nsym"], c["streams"]))
        u = rng.integers(0, 65536, row.shape)
        x = np.empty_like(row)
        for r in range(64):
            at = row == r
            x[at] = np.searchsorted(cum[r], u[at], side="right") - 1
        sym = torch.from_numpy((cum[row, x] | (f[row, x] - 1) << 16).astype(np.uint32).view(np.int32)).cuda()
        cap = 2 * c["nsym"] + 64
        return (kind, sym, torch.zeros(c["streams"], cap, device="cuda", dtype=torch.uint8),
                torch.zeros(c["streams"], device="cuda", dtype=torch.int32))
    z = torch.randn(c["samples"], c["dims"], device="cuda", generator=g)
    y = 0.7 * z + 0.7 * torch.randn(z.shape, device="cuda", generator=g)
    cnt = [torch.zeros(c["samples"], device="cuda", dtype=torch.int32) for _ in range(2)]
    return kind, z, y, c["k"], cnt


def run(state):
    kind = state[0]
    if kind == "compress":
        return _whole(edpc.compress(state[1], state[2]), state[1].size, state[2].streams)
    if kind == "decompress":
        return edpc.decompress(state[1])
    if kind == "files":
        return np.concatenate(edpc.decompress_many(state[1]))
    if kind == "independent":
        _, files, cfg, stream_len = state
        return _whole(edpc.compress_independent(files, cfg, stream_len=stream_len), sum(f.size for f in files), len(files))
    if kind == "gradient":
        _, m, ctx, targets, active = state
        z, p = m.forward(ctx)
        g, gu = m.backward(ctx, targets, active)
        return {"logits": z, "probs": p, "shared": g, "fdm": gu}
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "quantize":
        _, p, freq, cum = state
        edpc.cdf_quantize(p.data_ptr(), p.shape[0], freq.data_ptr(), cum.data_ptr(), stream)
        return freq, cum
    if kind == "encode":
        _, sym, out, length = state
        edpc.range_encode(sym.data_ptr(), sym.shape[0], sym.shape[1], out.data_ptr(), out.shape[1], length.data_ptr(),
                          stream)
        return out, length
    _, z, y, k, cnt = state
    mi = edpc.ksg_mi(z.data_ptr(), y.data_ptr(), z.shape[0], z.shape[1], y.shape[1], k, cnt[0].data_ptr(),
                     cnt[1].data_ptr(), stream)
    return {"mi": mi, "counts": cnt}


# ---- what a pass cannot do without --------------------------------------------------------
def _gemm_weights(c):
    F = c["context"] * c["embed_dim"]
    return c["blocks"] * (c["branches"] + 1) * F * c["hidden"] + 2 * F * c["latent"] + 256 * F


def work(case):
    c, kind = case, case["kind"]
    if kind == "quantize":
        return {"bytes": c["rows"] * 4.0 * (256 + 256 + 257), "flops": 256.0 * c["rows"]}
    if kind == "encode":
        # about five bits a symbol come out
        return {"bytes": c["nsym"] * c["streams"] * (4 + 5 / 8), "flops": 0}
    if kind == "ksg":
        # a subtraction and a maximum for each coordinate of each pair
        return {"bytes": 8.0 * c["samples"] * c["dims"], "flops": 4.0 * c["samples"] ** 2 * c["dims"]}
    # A step reads and writes each active stream's FDM and its two moments (24 bytes an element) and reads it once more
    # to predict; its Linear layers multiply every weight three times (forward, input and weight gradient).
    fdm, p = c["latent"] ** 2, _gemm_weights(c)
    if kind == "gradient":
        b = c["streams"]  # two forward passes and an adjoint; the FDM in, its gradient out
        return {"bytes": b * fdm * 12.0 + 8.0 * p, "flops": 8.0 * b * p}
    if kind in ("compress", "decompress"):
        rows = float(c["streams"] * c["steps"])
    else:
        # file sizes are log-uniform over a factor of 40, one of them the longest
        rows = c["longest"] * (1 + (c["files"] - 1) * (1 - 1 / 40) / math.log(40))
    return {"bytes": rows * fdm * 28.0, "flops": rows * 6.0 * p}


# ---- the same in 64 bits ------------------------------------------------------------------
def _exact_gradient(c, seed):
    shared, fdm, ctx, targets, active = _gradient_inputs(c, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    P = [torch.from_numpy(t).to(dev, torch.float64).requires_grad_() for t in shared]
    U = torch.from_numpy(fdm).to(dev, torch.float64).requires_grad_()
    at = iter(P)
    x = next(at)[torch.from_numpy(ctx).to(dev).long()].reshape(c["streams"], -1)
    nloc, H, k = c["blocks"] // 2, c["hidden"], c["branches"]
    lte = P[1 + 6 * c["blocks"]:]
    for j in range(c["blocks"] + 1):
        if j == nloc:
            h = x @ lte[0].T + lte[1]
            x = torch.einsum("si,sij->sj", h, U) @ lte[2].T + lte[3]
        if j == c["blocks"]:
            break
        g, b, W, cb, Wo, co = (next(at) for _ in range(6))
        a = torch.nn.functional.layer_norm(x, x.shape[1:], g, b, 1e-5) @ W.T + cb
        f = torch.ones_like(a[:, :H])
        for i in range(k):
            f = f * a[:, i * H:(i + 1) * H]
        x = torch.nn.functional.gelu(f) @ Wo.T + co + x
    z = x @ lte[4].T + lte[5]
    logp = torch.log_softmax(z, 1)
    on = torch.from_numpy(active).to(dev).double()
    hit = logp.gather(1, torch.from_numpy(targets).to(dev).long()[:, None])[:, 0]
    (-(hit * on).sum() / on.sum()).backward()
    grads = torch.cat([(t.grad if t.grad is not None else torch.zeros_like(t)).reshape(-1) for t in P])
    return {"logits": z.detach(), "probs": logp.detach().exp(), "shared": grads, "fdm": U.grad.reshape(-1)}


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    if case["kind"] == "ksg":
        _, z, y, k, _ = prepare(case, seed)
        z, y = z.double(), y.double()
        n = z.shape[0]
        dz, dy = torch.cdist(z, z, p=float("inf")), torch.cdist(y, y, p=float("inf"))
        off = torch.full((n,), float("inf"), device=z.device, dtype=torch.float64).diag()
        eps = (torch.maximum(dz, dy) + off).kthvalue(k, 1).values[:, None]
        cz, cy = ((d + off < eps).sum(1) for d in (dz, dy))
        psi = lambda v: torch.digamma(torch.as_tensor(v).double().cpu())  # noqa: E731
        mi = psi(k) + psi(n) - (psi(cz + 1) + psi(cy + 1)).mean()
        return {"mi": mi.reshape(()), "counts": None}
    return None  # bytes and whole numbers only
