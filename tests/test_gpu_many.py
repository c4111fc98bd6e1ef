"""tc_encode_many / tc_decode_many (Section 3.1: every layer has its own encoder and decoder):
the sixteen-layer set of the ResNet-34 configuration plus an fp32 map, a layer on the streaming
kernels and an empty tensor in one call each -- every item equal to the per-tensor entry points
byte for byte, and checked against the oracle's coder and reconstruction."""
import numpy as np
import pytest
import torch

import oracle
import paper_1905_10830_b200 as tc
from synth import featuremaps as fm
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


def _layer_set(ctx):
    """(model, codebook, x, oracle side, dtype) per item: cfg 3's shapes with their multiplicities (two
    images per item), one fp32 map (exact kernels, symbols parked in the arena) and an empty tensor."""
    w = fm.workload(3)
    items = []
    for spec, mult in zip(w.layers, w.repeats):
        o = H.oracle_side(spec, 4, 6, 2 * mult, torch.bfloat16, False)
        model = H.import_model(tc, ctx, o["model"], torch.bfloat16)
        cb = tc.tc_codebook_import(ctx, o["lengths"], 4)
        x = o["x"].cuda()
        for j in range(mult):
            items.append((model, cb, x[2 * j: 2 * j + 2].contiguous(), o, torch.bfloat16, slice(2 * j, 2 * j + 2)))
    o = H.oracle_side(fm.LayerSpec(48, 12, 12, 0.9, None, 8800), 6, 6, 3, torch.float32, True)
    model = H.import_model(tc, ctx, o["model"], torch.float32)
    cb = tc.tc_codebook_import(ctx, o["lengths"], 6)
    items.append((model, cb, o["x"].cuda(), o, torch.float32, slice(0, 3)))
    items.append((model, cb, o["x"].cuda()[:0].contiguous(), o, torch.float32, slice(0, 0)))
    return items


def test_many_equals_the_per_tensor_calls_and_the_oracle(ctx):
    w = fm.workload(3)
    assert sum(w.repeats) == 16
    items = _layer_set(ctx)
    encs = tc.tc_encode_many(ctx, [(m, cb, x) for m, cb, x, *_ in items])
    assert tc.tc_get_status(ctx) == 0
    outs = tc.tc_decode_many(ctx, [(m, cb, e, x.shape, x.dtype) for (m, cb, x, *_), e in zip(items, encs)])
    assert tc.tc_get_status(ctx) == 0
    routes = set()
    for (model, cb, x, o, dtype, sl), enc, xhat in zip(items, encs, outs):
        if x.shape[0] == 0:
            assert enc.total_bits() == 0
            continue
        alone = tc.tc_encode(ctx, model, cb, x, debug=True, k=o["model"].k)
        routes.add(tc.tc_last_path(ctx))
        assert enc.total_bits() == alone.total_bits()
        assert np.array_equal(H.stream_words(enc), H.stream_words(alone))
        assert np.array_equal(H.chunk_len(enc), H.chunk_len(alone)) and np.array_equal(H.tile_off(enc), H.tile_off(alone))
        xhat_alone = tc.tc_decode(ctx, model, cb, alone, x.shape, dtype)
        assert torch.equal(xhat, xhat_alone)
        # against the oracle: symbols within the tie allowance, its coder bit for bit on those symbols,
        # its reconstruction within the output tolerance
        pix = x.shape[2] * x.shape[3]
        rows = slice(sl.start * pix, sl.stop * pix)
        q_gpu = alone.symbols.cpu().numpy()
        bad = q_gpu != o["q"][rows]
        assert bad.mean() <= 1e-4
        ref = oracle.encode(q_gpu, o["lengths"], o["model"].bits, chunk_pixels=enc.layout.chunk_pixels,
                            pixel_splits=enc.layout.pixel_splits, tile_pixels=128)
        assert enc.total_bits() == ref.total_bits and np.array_equal(H.stream_words(enc), ref.words)
        assert np.array_equal(H.chunk_len(enc), ref.chunk_len) and np.array_equal(H.tile_off(enc), ref.tile_off)
        want = oracle.reconstruct(o["model"], q_gpu, x.shape, out_bf16=(dtype == torch.bfloat16))
        got = xhat.float().cpu().numpy()
        if dtype == torch.float32:
            assert np.array_equal(got, want)
        else:
            ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-30))) - 7)
            assert np.all(np.abs(got - want) <= np.maximum(1e-3 * np.maximum(np.abs(want), o["model"].step), ulp))
            assert H.count_output_flips(got, want) <= H.flip_allowance(H.expected_output_flips(o["model"], q_gpu))
    assert routes == {0, 1, 3}          # exact kernels, resident-basis and streaming tensor-core kernels all took part


def test_many_reuses_buffers_and_rejects_a_bad_item_before_launching(ctx):
    items = _layer_set(ctx)[:5]
    layers = [(m, cb, x) for m, cb, x, *_ in items]
    first = tc.tc_encode_many(ctx, layers)
    want = [H.stream_words(e).copy() for e in first]
    for e in first:
        e.words.fill_(0x5A)
    again = tc.tc_encode_many(ctx, layers, outs=first)
    assert tc.tc_get_status(ctx) == 0
    for e, w_ in zip(again, want):
        assert np.array_equal(H.stream_words(e), w_)
    # a misaligned stream buffer in the last item: refused, and the buffers of the others stay as they were
    for e in first:
        e.words.fill_(0x33)
    last = first[-1]
    skewed = tc.EncodedStream(last.words[8:], last.chunk_len, last.tile_off, last.layout)
    with pytest.raises(tc.TcError):
        tc.tc_encode_many(ctx, layers, outs=first[:-1] + [skewed])
    torch.cuda.synchronize()
    assert all(bool((e.words == 0x33).all()) for e in first)


def test_tensors_that_share_a_stream_and_its_workspace(ctx):
    # 24 items on eight streams, every one with workspace of another size: wide layers, unaligned maps, per-channel code tables,
    # fp32 maps and one wide layer that takes several passes; three follow each other on a stream.  Byte for byte the
    # single calls, twice (the second call meets the first one's leftovers) and in another order.
    shapes = [(320, 7, 7, 40, torch.bfloat16, False), (576, 14, 14, 9, torch.bfloat16, False), (272, 28, 28, 200, torch.bfloat16, False),
              (960, 7, 7, 30, torch.bfloat16, False), (80, 27, 19, 37, torch.bfloat16, True), (48, 5, 3, 300, torch.bfloat16, False),
              (256, 14, 14, 60, torch.bfloat16, True), (64, 9, 9, 3, torch.bfloat16, True), (48, 12, 12, 3, torch.float32, True),
              (128, 10, 10, 2, torch.float32, False), (1024, 4, 4, 5, torch.bfloat16, False), (16, 28, 28, 20, torch.bfloat16, True)]
    items = []
    for i, (c, h, w, n, dtype, per_channel) in enumerate(shapes):
        params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 8900 + i))
        cal = fm.make_maps(params, max(8, 2 * c // (h * w) + 1), calib=True, dtype=dtype, device="cuda")
        m = tc.tc_fit_pca(ctx, cal, 4 + i % 3)
        groups = c if per_channel else 1
        cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=groups).hist, groups=groups)
        x = fm.make_maps(params, n, dtype=dtype, device="cuda")
        items += [(m, cb, x), (m, cb, x[: (n + 1) // 2].contiguous())]
    want = []
    for m, cb, x in items:
        e = tc.tc_encode(ctx, m, cb, x)
        want.append((e, tc.tc_decode(ctx, m, cb, e, x.shape, x.dtype)))
    assert tc.tc_get_status(ctx) == 0
    outs = decs = None
    for order in (range(24), range(24), [5 * i % 24 for i in range(24)]):
        outs = [outs[i] for i in order] if outs else None
        decs = [torch.full_like(d, 7.0) for d in decs] if decs else None
        decs = [decs[i] for i in order] if decs else None
        if outs:
            for e in outs:
                e.words.fill_(0x5A)
        outs = tc.tc_encode_many(ctx, [items[i] for i in order], outs=outs)
        decs = tc.tc_decode_many(ctx, [(items[i][0], items[i][1], e, items[i][2].shape, items[i][2].dtype) for i, e in zip(order, outs)], outs=decs)
        assert tc.tc_get_status(ctx) == 0
        for i, e, d in zip(order, outs, decs):
            n = want[i][0].total_bits() // 8
            assert torch.equal(e.tile_off, want[i][0].tile_off) and torch.equal(e.words[:n], want[i][0].words[:n])
            assert torch.equal(e.chunk_len[:e.layout.n_chunks], want[i][0].chunk_len[:e.layout.n_chunks])
            assert torch.equal(d, want[i][1])
    for m, cb, _ in items[::2]:
        m.close(); cb.close()


# Tensors that share launches: more than a launch holds, more kernels than one (symbol pairs up to 6 bits, private runs where they
# fit, a table per channel, a non-linearity behind the decoder), tensors of one tile beside tensors of many, and beside them others that
# have kernels of their own.
def test_long_mixed_lists_equal_the_per_tensor_calls(ctx):
    shapes = [(64, 14, 14, 5, 4, False), (16, 4, 2, 1, 3, False), (256, 14, 14, 3, 8, False), (48, 10, 6, 2, 7, False), (80, 12, 12, 2, 5, True),
              (320, 7, 7, 3, 4, False), (96, 13, 13, 2, 4, False), (128, 28, 28, 2, 2, False)]
    sides, items, relus = [], [], []
    for i, (c, h, w, n, bits, per_channel) in enumerate(shapes):
        o = H.oracle_side(fm.LayerSpec(c, h, w, 0.9, None, 8700 + i), bits, max(3, 2 * c // (h * w) + 1), n, torch.bfloat16, per_channel)
        model = H.import_model(tc, ctx, o["model"], torch.bfloat16)
        sides.append((model, tc.tc_codebook_import(ctx, o["lengths"], bits), o["x"].cuda()))
    for j in range(70):
        model, cb, x = sides[(j * 5) % len(sides)]
        items.append((model, cb, x[:1 + j % x.shape[0]].contiguous()))
        relus.append(j % 3 == 0)
    encs = tc.tc_encode_many(ctx, items)
    assert tc.tc_get_status(ctx) == 0
    with pytest.raises(ValueError):
        tc.tc_decode_many(ctx, [(*i[:2], e, i[2].shape, torch.bfloat16) for i, e in zip(items, encs)], relu=relus[1:])
    for relu in (False, True, relus):
        outs = tc.tc_decode_many(ctx, [(*i[:2], e, i[2].shape, torch.bfloat16) for i, e in zip(items, encs)], relu=relu)
        assert tc.tc_get_status(ctx) == 0
        for i, out in enumerate(outs):
            model, cb, x = items[i]
            alone = tc.tc_encode(ctx, model, cb, x)
            assert alone.total_bits() == encs[i].total_bits()
            assert np.array_equal(H.stream_words(encs[i]), H.stream_words(alone)) and np.array_equal(H.chunk_len(encs[i]), H.chunk_len(alone))
            assert torch.equal(out, tc.tc_decode(ctx, model, cb, alone, x.shape, torch.bfloat16, relu=relus[i] if relu is relus else relu))
    assert tc.tc_get_status(ctx) == 0


# The route that a list reports: that of the item launched last, those that share launches first, and none by an empty tensor.
def test_the_route_that_a_list_reports(ctx):
    sides = {}
    for c, dtype in ((64, torch.bfloat16), (320, torch.bfloat16), (48, torch.float32)):
        o = H.oracle_side(fm.LayerSpec(c, 8, 8, 0.9, None, 8600 + c), 4, 2 * c // 64 + 3, 2, dtype, False)
        sides[c] = H.import_model(tc, ctx, o["model"], dtype), tc.tc_codebook_import(ctx, o["lengths"], 4), o["x"].cuda()
    encs = {c: tc.tc_encode(ctx, *sides[c]) for c in sides}
    for lst, route in (([64], 1), ([64, -64], 1), ([-320, 64], 1), ([64, 320], 3), ([320, -64], 3), ([64, 48], 0), ([-48], None)):
        own = tc.tc_create(0)
        before = tc.tc_last_path(own), tc.tc_last_path(own, True)
        items = [(sides[abs(c)][0], sides[abs(c)][1], sides[abs(c)][2][:2 if c > 0 else 0].contiguous()) for c in lst]
        out = tc.tc_encode_many(own, items)
        got = tc.tc_last_path(own)
        tc.tc_decode_many(own, [(*i[:2], encs[c] if c > 0 else e, i[2].shape, i[2].dtype) for c, i, e in zip(lst, items, out)])
        assert (got, tc.tc_last_path(own, True)) == (before if route is None else (route, route)), lst
        assert tc.tc_get_status(own) == 0
        own.close()
