"""The reductions of a calibration (Section 3: mean, covariance, range of coefficient 0, squared error) against numpy in fp64, at the
edges of their tiles, of their vector loads and of a tensor's alignment."""
import numpy as np
import pytest
import torch

import paper_1905_10830_b200 as tc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


def _maps(n, c, h, w, dtype, offset, seed):
    """Maps that start `offset` elements into an aligned buffer."""
    x = torch.randn(n, c, h, w, generator=torch.Generator().manual_seed(seed)) * 3 + 1
    buf = torch.empty(n * c * h * w + offset, dtype=dtype, device="cuda")
    out = buf[offset:].view(n, c, h, w)
    out.copy_(x)
    return out


# Channels about the 64 of a covariance tile and the 8 of a block of sums, pixels about the 32 of a slab and the four images of a
# step, rows of every vector width, addresses that rule the wider ones out.
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,c,h,w,offset", [(1, 1, 1, 3, 0), (2, 7, 3, 3, 0), (5, 63, 2, 2, 0), (4, 64, 4, 2, 2), (9, 65, 5, 7, 0), (3, 129, 8, 8, 1),
                                            (6, 200, 4, 4, 4), (1, 300, 31, 1, 0), (33, 16, 1, 1, 0)])
def test_sums_and_outer_products(ctx, n, c, h, w, offset, dtype):
    x = _maps(n, c, h, w, dtype, offset, 31 + n + c)
    st = tc.tc_fit_state_create(ctx, c)
    tc.tc_fit_state_update(ctx, st, x)
    count, s1, s2 = tc.tc_fit_state_export(ctx, st)
    v = x.permute(1, 0, 2, 3).reshape(c, -1).double().cpu().numpy()
    assert count == v.shape[1]
    # fp64 sums of m terms in any order: at most m roundings of the sum of the terms' sizes
    m = v.shape[1] * 2.0 ** -52
    assert np.all(np.abs(s1 - v.sum(1)) <= m * np.abs(v).sum(1))
    assert np.all(np.abs(s2 - v @ v.T) <= 2 * m * (np.abs(v) @ np.abs(v).T))
    assert np.array_equal(s2, s2.T)


# One-shot fit of the same maps: mean, and the range of coefficient 0 (which sets step and lo) in the order of the definition.
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,c,h,w,offset", [(40, 16, 3, 3, 1), (7, 33, 9, 9, 0), (3, 64, 16, 8, 0), (2, 96, 14, 14, 2)])
def test_mean_and_range(ctx, n, c, h, w, offset, dtype):
    x = _maps(n, c, h, w, dtype, offset, 77 + c)
    m = tc.tc_model_export(tc.tc_fit_pca(ctx, x, 5, zero_level=False))
    v = x.permute(1, 0, 2, 3).reshape(c, -1).double().cpu().numpy()
    assert np.abs(m["mean"] - v.mean(1)).max() <= v.shape[1] * 2.0 ** -52 * np.abs(v).max()
    y = np.zeros(v.shape[1])
    for a in range(c):
        y = y + m["basis"][0, a] * (v[a] - m["mean"][a])
    assert m["lo"] == y.min() and m["step"] == (y.max() - y.min()) / 31


# Squared error and zeros behind tc_stats: whole and ragged pieces of 16 bytes, the exact route and the tensor-core one.
@pytest.mark.parametrize("dtype,n,c,h,w,offset", [(torch.float32, 1, 17, 3, 3, 0), (torch.float32, 2, 16, 5, 5, 1), (torch.float32, 2, 32, 8, 8, 0),
                                                  (torch.bfloat16, 3, 32, 4, 4, 0), (torch.bfloat16, 5, 48, 6, 6, 4), (torch.bfloat16, 4, 40, 3, 3, 0)])
def test_stats_error_and_zeros(ctx, dtype, n, c, h, w, offset):
    x = torch.relu(_maps(n, c, h, w, dtype, offset, 5 + c))
    buf = torch.empty(x.numel() + offset, dtype=dtype, device="cuda")
    y = buf[offset:].view(x.shape)
    y.copy_(x)
    model = tc.tc_fit_pca(ctx, y, 4)
    stats = tc.tc_stats(ctx, model, None, y)
    cb = tc.tc_build_codebook(ctx, model, stats.hist)
    enc = tc.tc_encode(ctx, model, cb, y)
    x_hat = tc.tc_decode(ctx, model, cb, enc, y.shape, y.dtype)
    want = float(((y.double() - x_hat.double()) ** 2).mean())
    assert abs(stats.mse - want) <= 1e-12 * want
    assert abs(stats.zero_fraction * y.numel() - int((y == 0).sum())) < 1e-6
