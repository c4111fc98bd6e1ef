"""Timing cases for the feature-map codec: what a program that uses the library has it do.

A program calibrates a layer once (fit the transform, count the symbols, build the code table) and
then encodes and decodes that layer's feature maps for as long as it runs: one map at a time next
to a single inference, a batch at a time in serving or training, or the whole list of a network's
layers in one call.  The cases cover those calls over the layer shapes, batch sizes, bit widths and
code-table granularities of the library's configurations, tests and benchmark, from a single
14 x 14 map to a batch of 4096.

Inputs are synthetic post-ReLU maps with correlated channels: a geometric spectrum (`decay`) mixed
by a random orthogonal matrix, blurred over 3 x 3 pixels, shifted by a per-channel bias (or by the
bias that makes a share `zeros` of the values ReLU zeros) and clamped at zero.
"""
import math
from statistics import NormalDist

import numpy as np
import torch

import paper_1905_10830_b200 as tc

CALIBRATION_PIXELS = 50_000      # pixels of the calibration maps that a layer's model is computed from

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # one fp32 map of a residual network's first stage next to a single inference: latency
        dict(name="encode one 64x56x56 f32", op="encode", layers="64x56x56", n=1, dtype="f32", bits=8, tables="layer",
             decay=0.85, zeros=0.0, keep=1.0),
        # the same at a later stage, read back, with a code table per coefficient channel
        dict(name="decode one 256x14x14 f32", op="decode", layers="256x14x14", n=1, dtype="f32", bits=6, tables="channel",
             decay=0.85, zeros=0.0, keep=1.0),
        # a shape off every grid: odd map sides (rows start at any 2-byte address), a last tile that is
        # nearly empty, leading coefficients only, a code table per channel
        dict(name="round trip 80x27x19 ragged", op="roundtrip", layers="80x27x19", n=37, dtype="bf16", bits=6,
             tables="channel", decay=0.9, zeros=0.0, keep=0.6),
        # every block output of a 34-layer residual network at batch 64, one call for the list
        dict(name="encode 16 layers", op="encode_many", layers="64x56x56*3 128x28x28*4 256x14x14*6 512x7x7*3", n=64,
             dtype="bf16", bits=4, tables="layer", decay=0.9, zeros=0.0, keep=1.0),
        dict(name="decode 16 layers", op="decode_many", layers="64x56x56*3 128x28x28*4 256x14x14*6 512x7x7*3", n=64,
             dtype="bf16", bits=4, tables="layer", decay=0.9, zeros=0.0, keep=1.0),
        # the widest map of an inverted-residual network: few channels, many pixels, dense symbols
        dict(name="encode 96x112x112", op="encode", layers="96x112x112", n=128, dtype="bf16", bits=5, tables="layer",
             decay=0.95, zeros=0.6, keep=1.0),
        # wide expansion maps: more channels than a basis in shared memory allows, each direction
        dict(name="decode 576x14x14", op="decode", layers="576x14x14", n=128, dtype="bf16", bits=5, tables="layer",
             decay=0.95, zeros=0.6, keep=1.0),
        dict(name="encode 960x7x7", op="encode", layers="960x7x7", n=128, dtype="bf16", bits=5, tables="layer",
             decay=0.95, zeros=0.6, keep=1.0),
        # the benchmark's layer at its full batch and default rate, each direction
        dict(name="encode 256x14x14 b4096", op="encode", layers="256x14x14", n=4096, dtype="bf16", bits=4, tables="layer",
             decay=0.9, zeros=0.0, keep=1.0),
        dict(name="decode 256x14x14 b4096", op="decode", layers="256x14x14", n=4096, dtype="bf16", bits=4, tables="layer",
             decay=0.9, zeros=0.0, keep=1.0),
        # the same layer near-lossless: long codes, hardly any runs
        dict(name="round trip 256x14x14 8 bits", op="roundtrip", layers="256x14x14", n=1024, dtype="bf16", bits=8,
             tables="layer", decay=0.9, zeros=0.0, keep=1.0),
        # calibration of that layer: fit, symbol statistics, code table
        dict(name="calibrate 256x14x14", op="calibrate", layers="256x14x14", n=256, dtype="bf16", bits=4, tables="layer",
             decay=0.9, zeros=0.0, keep=1.0),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) - 0.2))))


def draw(rng):
    """One more case of the same ranges: 16 to 960 channels, maps of 7 to 112 pixels a side, batches up to
    the values and operations of the largest listed case."""
    op = rng.choice(["encode", "encode", "encode", "decode", "decode", "decode", "roundtrip", "roundtrip", "encode_many", "decode_many",
                     "calibrate"])
    bits = rng.choice([2, 3, 4, 4, 5, 5, 6, 7, 8])
    decay, zeros = rng.choice([(0.85, 0.0), (0.9, 0.0), (0.95, 0.6)])
    base = dict(op=op, dtype="bf16", bits=bits, tables="layer", decay=decay, zeros=zeros, keep=1.0)
    if op.endswith("many"):
        n, parts = _log_int(rng, 1, 96), []
        for _ in range(rng.randint(2, 6)):
            side = rng.choice([7, 14, 14, 28, 56])
            c = 16 * _log_int(rng, 1, 2 * (7 * 64 // side) // 4)
            parts.append(f"{c}x{side}x{side}*{rng.randint(1, 3)}")
        return dict(base, layers=" ".join(parts), n=n)
    if op == "calibrate":
        c, side = 16 * _log_int(rng, 4, 24), rng.choice([7, 14, 28])
        return dict(base, layers=f"{c}x{side}x{side}", n=max(2, _log_int(rng, 3000, 50_000) // (side * side)))
    if rng.random() < 0.2:                                    # single fp32 maps, on the exact kernels
        c = 16 * _log_int(rng, 2, 32)
        h = max(7, min(56, round(math.sqrt(rng.uniform(0.3, 1.0) * 200_000 / c))))
        return dict(base, layers=f"{c}x{h}x{max(7, h - rng.randint(0, 3))}", n=1, dtype="f32", tables=rng.choice(["layer", "channel"]))
    c = 16 * _log_int(rng, 1, 60)
    h = _log_int(rng, 7, 112)
    w = h if rng.random() < 0.6 else max(7, h - rng.randint(1, 9))
    tables = "channel" if c <= 256 and rng.random() < 0.2 else "layer"
    keep = rng.choice([0.25, 0.5, 0.75]) if rng.random() < 0.2 else 1.0
    most = min(200e6 / c, 50e9 / (c * c)) * (0.3 if op == "roundtrip" else 1.0)      # pixels
    return dict(base, layers=f"{c}x{h}x{w}", n=max(1, int(_log_int(rng, 200, int(most)) / (h * w))), tables=tables, keep=keep)


def _layers(case):
    """[(c, h, w)] of the case, repeats written out."""
    out = []
    for part in case["layers"].split():
        shape, _, times = part.partition("*")
        out += [tuple(int(v) for v in shape.split("x"))] * int(times or 1)
    return out


def _kept(case, c):
    return max(16, int(c * case["keep"]) // 16 * 16) if case["keep"] < 1.0 else c


class _MapSource:
    """Feature maps of one layer, from its own random numbers."""

    def __init__(self, c, h, w, case, gen):
        dev = gen.device
        q, r = torch.linalg.qr(torch.randn(c, c, generator=gen, device=dev, dtype=torch.float64))
        q = q * torch.sign(torch.diagonal(r))
        lam = case["decay"] ** torch.arange(c, device=dev, dtype=torch.float64)
        mix = q * (lam * (c / lam.sum())).sqrt()
        if case["zeros"]:
            beta = -(mix.square().sum(1) / 9.0).sqrt() * NormalDist().inv_cdf(case["zeros"])
        else:
            beta = 0.2 + 0.1 * torch.randn(c, generator=gen, device=dev, dtype=torch.float64)
        self.mix, self.beta, self.gen = mix.float(), beta.float().view(1, c, 1, 1), gen
        self.shape, self.dtype = (c, h, w), DTYPES[case["dtype"]]

    def maps(self, n):
        c, h, w = self.shape
        out = torch.empty(n, c, h, w, dtype=self.dtype, device=self.gen.device)
        step = max(1, (32 << 20) // (c * h * w))
        for i in range(0, n, step):
            m = min(step, n - i)
            z = torch.randn(m, c, h * w, generator=self.gen, device=self.gen.device)
            s = torch.matmul(self.mix, z).view(m, c, h, w)
            s = torch.nn.functional.avg_pool2d(s, 3, stride=1, padding=1)
            out[i:i + m] = torch.clamp_min(s + self.beta, 0.0)
        return out


def _stream_buffers(model, cb, x):
    """The buffers a program keeps for a layer's stream, as tc_encode would allocate them."""
    lay = tc.tc_encode_bound(model, cb, x)
    return tc.EncodedStream(torch.zeros(max(lay.stream_bytes, 16), dtype=torch.uint8, device=x.device),
                            torch.zeros(max(lay.n_chunks + (lay.n_chunks & 1), 2), dtype=torch.int16, device=x.device),
                            torch.zeros(lay.n_tiles + 1, dtype=torch.int64, device=x.device), lay)


def _deployed_layer(ctx, case, cal, k):
    """Model and code table as a deployed program has them: computed once (here from the maps `cal`, in
    double precision) and imported."""
    n, c, h, w = cal.shape
    v = cal.transpose(0, 1).reshape(c, -1).double()
    mean = v.mean(1)
    v -= mean[:, None]
    eig, vec = torch.linalg.eigh(v @ v.T / (v.shape[1] - 1))
    basis = vec.T.flip(0).to(cal.dtype).double()
    y = basis[:k] @ v
    top = (1 << case["bits"]) - 1
    step = float(y[0].max() - y[0].min()) / top
    lo = -step * round(-float(y[0].min()) / step)             # zero is a level of the grid
    q = ((y - lo) / step).round_().clamp_(0, top).long()
    if case["tables"] == "channel":
        hist = torch.stack([torch.bincount(row, minlength=top + 1) for row in q])
    else:
        hist = torch.bincount(q.view(-1), minlength=top + 1)[None]
    lengths = np.stack([tc.tc_host_huffman_lengths(row) for row in hist.cpu().numpy()])
    model = tc.tc_model_import(ctx, basis=basis.cpu().numpy(), mean=mean.cpu().numpy(), lo=lo, step=step, bits=case["bits"],
                               basis_dtype=tc.binding.TC_F32 if cal.dtype == torch.float32 else tc.binding.TC_BF16, k=k,
                               eig=eig.flip(0).cpu().numpy())
    return model, tc.tc_codebook_import(ctx, lengths, case["bits"])


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    ctx = tc.tc_create(0)
    if case["op"] == "calibrate":
        (c, h, w), = _layers(case)
        return dict(case=case, ctx=ctx, maps=_MapSource(c, h, w, case, gen).maps(case["n"]))
    items, known = [], {}
    for c, h, w in _layers(case):
        if (c, h, w) not in known:          # blocks of one shape share the layer's statistics, not its maps
            src = _MapSource(c, h, w, case, gen)
            cal = src.maps(max(2, CALIBRATION_PIXELS // (h * w)))
            known[c, h, w] = src, *_deployed_layer(ctx, case, cal, _kept(case, c))
        src, model, cb = known[c, h, w]
        x = src.maps(case["n"])
        enc = _stream_buffers(model, cb, x)
        item = dict(model=model, cb=cb, enc=enc, shape=x.shape, dtype=x.dtype)
        if case["op"] in ("encode", "encode_many", "roundtrip"):
            item["x"] = x
        if case["op"] in ("decode", "decode_many"):
            tc.tc_encode(ctx, model, cb, x, out=enc)
        if case["op"] not in ("encode", "encode_many"):
            item["x_hat"] = torch.empty_like(x)
        items.append(item)
    if tc.tc_get_status(ctx) != 0:
        raise RuntimeError("the streams to decode could not be made")
    return dict(case=case, ctx=ctx, items=items)


def _stream(enc):
    return {"words": enc.words, "chunk_len": enc.chunk_len, "tile_off": enc.tile_off}


def run(state):
    ctx, op = state["ctx"], state["case"]["op"]
    if op == "calibrate":
        maps = state["maps"]
        model = tc.tc_fit_pca(ctx, maps, bits=state["case"]["bits"])
        stats = tc.tc_stats(ctx, model, None, maps, groups=1)
        cb = tc.tc_build_codebook(ctx, model, stats.hist, groups=1)
        m = tc.tc_model_export(model)
        return {"basis": m["basis"], "mean": m["mean"], "eig": m["eig"], "lo": m["lo"], "step": m["step"],
                "hist": stats.hist.double(), "entropy": stats.entropy, "mse": stats.mse,
                "lengths": tc.tc_codebook_export(cb).astype("float64")}
    items = state["items"]
    if op == "encode_many":
        encs = tc.tc_encode_many(ctx, [(i["model"], i["cb"], i["x"]) for i in items], outs=[i["enc"] for i in items])
        return [_stream(e) for e in encs]
    if op == "decode_many":
        return tc.tc_decode_many(ctx, [(i["model"], i["cb"], i["enc"], i["shape"], i["dtype"]) for i in items],
                                 outs=[i["x_hat"] for i in items])
    i, = items
    if op != "decode":
        enc = tc.tc_encode(ctx, i["model"], i["cb"], i["x"], out=i["enc"])
        if op == "encode":
            return _stream(enc)
    x_hat = tc.tc_decode(ctx, i["model"], i["cb"], i["enc"], i["shape"], i["dtype"], out=i["x_hat"])
    return x_hat if op == "decode" else {"x_hat": x_hat, "chunk_len": i["enc"].chunk_len}


def work(case):
    """The tensor once per direction and the stream with its side information once per direction; the
    projection's multiply-adds once per direction.  The stream's rate is the one such maps have."""
    rate = 1.13 + 0.75 * max(0, case["bits"] - 4) + (0.5 if case["zeros"] else 0.0)          # bits per coefficient
    size = 4 if case["dtype"] == "f32" else 2
    total = {"bytes": 0.0, "flops": 0.0}
    for c, h, w in _layers(case):
        p, k = case["n"] * h * w, _kept(case, c)
        if case["op"] == "calibrate":       # maps read once; covariance (one triangle), coefficients and reconstruction
            total["bytes"] += p * c * size + c * c * 8
            total["flops"] += p * c * c + 4.0 * p * c * k
            continue
        ways = 2 if case["op"] == "roundtrip" else 1
        total["bytes"] += ways * (p * c * size + p * k * rate / 8)
        total["flops"] += ways * 2.0 * p * c * k
    return total


def tolerance(case):
    # A stream is bytes: the same symbols give the same stream, whatever codes them.
    if case["op"] in ("encode", "encode_many"):
        return "exact"
    # fp32 maps are evaluated in fp64 in the order of the definition: one result, rounded once.
    if case["dtype"] == "f32":
        return "exact"
    # Fit in fp64, basis rounded to bf16: sums in another order move the eigenvectors by far less than
    # a bf16 rounding step, so that now and then an entry lands on the neighbouring bf16 number.
    if case["op"] == "calibrate":
        return {"rel": 1e-4, "max": 0.01}
    # fp32 accumulation of exact products, output rounded to bf16: against the fp64 kernels up to 2 values
    # in 10^4 land on the neighbouring bf16 number (one step is 2^-7 of the value at most), 2e-5 overall.
    # A round trip also meets rounding ties of the quantiser: such a symbol moves one pixel by a step and
    # its chunk by a few bits (3e-4 overall and 8e-4 of the chunks at 8 bits).
    if case["op"] == "roundtrip":
        return {"rel": 1.2e-3, "max": 0.3, "differ": 4e-3}
    return {"rel": 1e-4, "max": 0.01}
