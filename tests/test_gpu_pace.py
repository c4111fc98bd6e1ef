"""Calls that a choice of launch once made several times slower than the work they hold: times beside those of calls with more work, or the same
work laid out otherwise."""
import pytest
import torch

import paper_1905_10830_b200 as tc
from synth import featuremaps as fm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


def _queued_us(*calls, times=20, rounds=9):
    """us of each call among others of its kind, the least of several rounds taken in turn."""
    best = [float("inf")] * len(calls)
    for _ in range(rounds):
        for i, call in enumerate(calls):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            call()
            torch.cuda.synchronize()
            torch.cuda._sleep(400_000)                         # the calls are queued by the time that the first runs
            a.record()
            for _ in range(times):
                call()
            b.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], a.elapsed_time(b) * 1e3 / times)
    return best


def _layer(ctx, c, h, w, n, bits, tables, dtype):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.93, None, 41000 + c))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=dtype, device="cuda")
    x = fm.make_maps(params, n, dtype=dtype, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=tables).hist, groups=tables)
    return m, cb, x


# The exact inverse behind the entropy decoder: its blocks, early, all on some of the SMs took as long for 10 tiles as for 20 (47.0 and 49.4 us;
# 31.6 and 49.4 kept apart).
def test_exact_decodes_of_half_the_tiles(ctx):
    m, cb, x = _layer(ctx, 256, 8, 16, 20, 5, 1, torch.float32)
    half, whole = (tc.tc_encode(ctx, m, cb, v) for v in (x[:10], x))
    out = torch.empty_like(x)
    few, many = _queued_us(lambda: tc.tc_decode(ctx, m, cb, half, x[:10].shape, x.dtype, out=out[:10]),
                           lambda: tc.tc_decode(ctx, m, cb, whole, x.shape, x.dtype, out=out))
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 0
    assert few < 0.8 * many, (few, many)
    m.close(); cb.close()


# Decodes of one stream as maps of a pixel, two and three take about what larger maps of as many pixels take (208 channels as 1x3 82 us, as 14x12 26 when
# channels of small maps left as rows; twice the time is the line).
@pytest.mark.parametrize("w", [1, 2, 3])
def test_decodes_of_small_maps(ctx, w):
    m, cb, x = _layer(ctx, 208, 14, 12, 600, 4, 1, torch.bfloat16)
    enc = tc.tc_encode(ctx, m, cb, x)
    small = (x.shape[0] * 168 // w, 208, 1, w)
    out, as_small = torch.empty_like(x), torch.empty(small, dtype=x.dtype, device="cuda")
    large, us = _queued_us(lambda: tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, out=out), lambda: tc.tc_decode(ctx, m, cb, enc, small, x.dtype, out=as_small))
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    assert us < 2.0 * large, (us, large)
    m.close(); cb.close()


# The entropy coder with a table per channel keeps its blocks apart as the one with a table for the layer does (480x14x14 x 195, 299 blocks: three an SM
# on two thirds of the SMs took 160 us where one table takes 73; 1.6 times is the line).
def test_encodes_with_a_table_per_channel(ctx):
    us = []
    for tables in (1, 480):
        m, cb, x = _layer(ctx, 480, 14, 14, 195, 7, tables, torch.bfloat16)
        enc = tc.tc_encode(ctx, m, cb, x)
        us += _queued_us(lambda: tc.tc_encode(ctx, m, cb, x, out=enc))
        assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 3
        m.close(); cb.close()
    assert us[1] < 1.6 * us[0], us


# The pixel rows in front of a wide encode, early and all on some of the SMs, took half as long again as for more of the same (128 channels of maps of a
# pixel: 146 tiles 32.2 us, 292 tiles 33).
def test_wide_encodes_of_half_the_tiles(ctx):
    m, cb, x = _layer(ctx, 128, 1, 1, 37376, 4, 1, torch.bfloat16)
    halves = [x[:18688], x]
    encs = [tc.tc_encode(ctx, m, cb, v, pixel_splits=4) for v in halves]
    few, many = _queued_us(*[lambda v=v, e=e: tc.tc_encode(ctx, m, cb, v, out=e, pixel_splits=4) for v, e in zip(halves, encs)])
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 3
    assert few < 0.85 * many, (few, many)
    m.close(); cb.close()
