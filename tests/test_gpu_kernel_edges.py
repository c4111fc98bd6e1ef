"""Kernel branches that the parity cases do not separate, each at the sizes where it can go wrong."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1905_10830_b200 as tc
from synth import featuremaps as fm
from tests import helpers as H
from tests.test_gpu_parity import check_stream_against_oracle, check_symbols

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


def _same_stream(a, b):
    n = a.total_bits() // 8
    return a.total_bits() == b.total_bits() and torch.equal(a.words[:n], b.words[:n]) and torch.equal(a.tile_off, b.tile_off) \
        and torch.equal(a.chunk_len[:a.layout.n_chunks], b.chunk_len[:b.layout.n_chunks])


# Resident-basis encoder.  Rows of 8 k elements in a 16-byte aligned tensor are copied 16 bytes at a
# time, others 8; the last tile is partly or nearly empty; panels of 64 channels end in remainders.
@pytest.mark.parametrize("offset", [0, 4, 8])
@pytest.mark.parametrize("c,h,w,n,bits", [(16, 4, 2, 1, 4), (80, 8, 8, 3, 5), (208, 12, 12, 2, 4), (256, 14, 14, 1, 6), (48, 2, 10, 13, 8)])
def test_resident_encoder_copies(ctx, c, h, w, n, bits, offset):
    spec = fm.LayerSpec(c, h, w, 0.9, None, 11000 + c + h)
    o = H.oracle_side(spec, bits, max(3, 2 * c // (h * w) + 1), n, torch.bfloat16, False)
    m = H.import_model(tc, ctx, o["model"], torch.bfloat16)
    cb = tc.tc_codebook_import(ctx, o["lengths"], bits)
    buf = torch.empty(o["x"].numel() + 16, dtype=torch.bfloat16, device="cuda")
    x = buf[offset:offset + o["x"].numel()].view(o["x"].shape)
    x.copy_(o["x"])
    enc = tc.tc_encode(ctx, m, cb, x, debug=True)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    q = enc.symbols.cpu().numpy()
    check_symbols(q, o, exact=False)
    check_stream_against_oracle(enc, q, o["lengths"], bits)
    # the kernel without the debug outputs writes the same stream
    assert _same_stream(tc.tc_encode(ctx, m, cb, x), enc)
    assert tc.tc_get_status(ctx) == 0
    m.close(); cb.close()


# Resident-basis encoder with four groups a block (up to 128 coefficients): fewer tiles a block than groups and more than all groups'
# slots hold, one chunk a pixel, parts of one and several pixels a chunk, every code table, private runs and two passes, maps of
# more spread than the calibration's (tiles coded again, and straight into global memory).  The debug outputs take the kernel with two groups,
# whose streams the parity cases check: the same bytes.
@pytest.mark.parametrize("c,k,hw,n,bits,tables,cp,splits,spread", [
    (16, 16, 12, 1, 4, 1, 0, 0, 1.0), (128, 128, 64, 1500, 4, 1, 0, 0, 1.0), (128, 128, 16, 1184, 8, 1, 0, 0, 1.0), (64, 64, 196, 2300, 4, 1, 0, 0, 2.5),
    (96, 96, 196, 1300, 5, 1, 1, 2, 1.0), (128, 64, 100, 1600, 6, 1, 1, 4, 1.0), (80, 48, 64, 700, 3, 48, 0, 0, 1.0), (32, 32, 3136, 90, 7, 1, 16, 1, 3.0),
    (112, 112, 4, 20000, 2, 1, 0, 0, 1.0), (128, 128, 196, 600, 8, 128, 0, 0, 2.0), (144, 128, 36, 900, 4, 1, 0, 0, 1.0)])
def test_four_groups_a_block(ctx, c, k, hw, n, bits, tables, cp, splits, spread):
    params = fm.layer_params(fm.LayerSpec(c, hw // 4, 4, 0.9, None, 22000 + c + k + bits))
    cal = fm.make_maps(params, max(4, 30000 // hw), calib=True, dtype=torch.bfloat16, device="cuda")
    x = fm.make_maps(params, n, dtype=torch.bfloat16, device="cuda") * spread
    m = tc.tc_fit_pca(ctx, cal, bits, k=k)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=tables).hist, groups=tables)
    want = tc.tc_encode(ctx, m, cb, x, chunk_pixels=cp, pixel_splits=splits, debug=True)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    for _ in range(3):
        assert _same_stream(tc.tc_encode(ctx, m, cb, x, chunk_pixels=cp, pixel_splits=splits), want)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    m.close(); cb.close()


# Device eigensolver: every row / block shape of its kernel (blocks of 16 columns up to 512 rows, of 8
# beyond; 33 and 65 columns leave column blocks that are empty), and spectra that reach below zero.
@pytest.mark.parametrize("n,shift", [(16, 0.0), (31, 0.5), (33, 0.0), (65, 0.3), (130, 0.0), (300, 0.5), (384, 0.0), (513, 0.4), (640, 0.0)])
def test_device_eigh_block_shapes_and_indefinite(ctx, n, shift):
    rng = np.random.default_rng(300 + n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.sort(rng.uniform(0.0, 1.0, n) - shift)[::-1]
    a = (q * lam) @ q.T
    a = (a + a.T) / 2
    evals, evecs, sweeps = tc.tc_device_eigh(ctx, torch.from_numpy(a).cuda())
    evals, evecs = evals.cpu().numpy(), evecs.cpu().numpy()
    assert 1 <= sweeps <= 40
    # off-diagonal inner products stop at 8 sqrt(n) eps of the norms; (1.25 |A|_F + |A|) of it in V A V^T
    tol = 8 * np.sqrt(max(n, 16)) * 2.0 ** -52
    frob = np.linalg.norm(a)
    assert np.abs(evecs @ evecs.T - np.eye(n)).max() <= 2 * tol
    assert np.abs(evecs @ a @ evecs.T - np.diag(evals)).max() <= 6 * tol * frob
    assert np.abs(evals - np.linalg.eigvalsh(a)[::-1]).max() <= tol * frob


# Per-channel codes decoded from their bounds: one-symbol-dominated, flat and maximum-length (12 bit)
# tables side by side, every kernel that reads them (fp64 kernels with 1, 2 and 4 chunks a pixel and
# runs that are no multiple of 16, the tiled product's decoder, and -- without workspace (mode 4), or with the run-skipping
# decoder left out (mode 3) -- the resident and streaming tensor-core decoders).
@pytest.mark.parametrize("c,k,s,n,bits,dtype,cp,splits,mode", [
    (16, 16, 3, 1, 8, torch.float32, 0, 0, 0), (40, 24, 9, 2, 6, torch.float32, 0, 0, 0), (256, 256, 7, 2, 5, torch.float32, 0, 0, 0),
    (512, 512, 4, 1, 8, torch.float32, 0, 0, 0), (64, 64, 9, 2, 1, torch.float32, 4, 1, 0), (48, 48, 9, 2, 7, torch.bfloat16, 0, 0, 0),
    (256, 256, 14, 1, 6, torch.bfloat16, 0, 0, 0), (128, 128, 7, 3, 8, torch.bfloat16, 0, 0, 2), (320, 320, 5, 2, 4, torch.bfloat16, 0, 0, 0),
    (256, 256, 14, 1, 6, torch.bfloat16, 0, 0, 3), (48, 48, 9, 2, 7, torch.bfloat16, 0, 0, 4), (128, 128, 7, 3, 8, torch.bfloat16, 0, 0, 4),
    (320, 320, 5, 2, 4, torch.bfloat16, 0, 0, 4), (256, 256, 7, 2, 5, torch.float32, 0, 0, 4)])
def test_per_channel_codes_from_bounds(ctx, c, k, s, n, bits, dtype, cp, splits, mode):
    spec = fm.LayerSpec(c, s, s, 0.9, None, 12000 + c + bits)
    o = H.oracle_side(spec, bits, max(3, 2 * c // (s * s) + 1), n, dtype, True, k=k)
    lengths, nsym = o["lengths"].copy(), 1 << bits
    flat = np.full(nsym, bits, dtype=np.uint8)
    # the longest code a table can hold: 1, 2, 3, ... bits down to `deep` symbols of one length
    steep = np.sort(np.r_[np.arange(1, nsym), nsym - 1]).astype(np.uint8) if nsym <= 8 else None
    if steep is None:
        counts = np.array([4 ** max(0, 14 - i) for i in range(nsym)], dtype=np.uint64)
        steep = tc.tc_host_huffman_lengths(counts, 12)
        assert steep.max() == 12
    for j in range(0, k, 3):
        lengths[j] = flat if j % 2 else steep[::-1]
    m = H.import_model(tc, ctx, o["model"], dtype)
    cb = tc.tc_codebook_import(ctx, lengths, bits)
    x = o["x"].cuda()
    tc.tc_force_exact_path(ctx, mode)
    try:
        enc = tc.tc_encode(ctx, m, cb, x, chunk_pixels=cp, pixel_splits=splits, debug=True, k=k)
        xhat = tc.tc_decode(ctx, m, cb, enc, x.shape, dtype)
        assert tc.tc_get_status(ctx) == 0
        q = enc.symbols.cpu().numpy()
        ref = check_stream_against_oracle(enc, q, lengths, bits)
        assert np.array_equal(oracle.decode_symbols(ref, lengths, bits), q)
        want = oracle.reconstruct(o["model"], q, tuple(x.shape), out_bf16=dtype == torch.bfloat16)
        got = xhat.float().cpu().numpy()
        if dtype == torch.float32:
            assert np.array_equal(got, want)
        else:                                       # fp32 accumulation: the parity cases' bound
            flips, expected = H.count_output_flips(got, want), H.expected_output_flips(o["model"], q)
            assert flips <= H.flip_allowance(expected)
    finally:
        tc.tc_force_exact_path(ctx, 0)
    m.close(); cb.close()


# Run-skipping decoder: one to eight warps per group, two to eight groups per block, every group with
# several tiles (more than eight tiles a block), rows that allow 16-byte stores and rows that do not;
# against the fp64 kernels on the same stream.
@pytest.mark.parametrize("c,k,h,w,bits", [(16, 16, 56, 56, 4), (32, 32, 14, 14, 5), (64, 64, 56, 56, 4), (96, 48, 28, 28, 6), (144, 144, 14, 14, 5),
                                          (192, 192, 8, 8, 3), (256, 256, 14, 14, 4), (256, 96, 27, 28, 8), (80, 80, 9, 7, 4)])
def test_run_skipping_decoder_groups(ctx, c, k, h, w, bits):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 13000 + c + k))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=torch.bfloat16, device="cuda")
    x = fm.make_maps(params, 148 * 9 * 128 // (h * w) + 3, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits, k=k)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x)
    got = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    tc.tc_force_exact_path(ctx, 1)
    want = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0
    tc.tc_force_exact_path(ctx, 0)
    # one rounding to bf16 on each side of the same value: neighbours at most, and for 0.1 % of the values
    # (the cap of the parity cases)
    a, b = got.float(), want.float()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-6 * float(b.abs().max())).all())
    assert float((a != b).double().mean()) <= 1e-3
    m.close(); cb.close()


# Wide layers as tiled products: blocks of coefficients and channels with remainders, pixel rows of 1, 2 and
# 4-element alignment, fewer units than SMs and more, several passes over the workspace, every chunk
# shape, both table granularities, few and many decoder warps an SM.  Against the fused kernel (debug outputs take it), whose symbols the
# parity cases check, and the fp64 kernels.
@pytest.mark.parametrize("c,k,h,w,n,bits,tables,offset", [
    (272, 272, 3, 3, 1, 4, 1, 0), (320, 320, 5, 5, 40, 5, 1, 0), (576, 576, 14, 14, 9, 5, 1, 0), (960, 960, 7, 7, 30, 5, 1, 0),
    (1024, 1024, 12, 12, 160, 2, 1, 0), (512, 512, 7, 7, 64, 8, 1, 0), (400, 208, 6, 6, 50, 6, 208, 0), (960, 16, 7, 7, 5, 8, 1, 0),
    (80, 48, 27, 19, 37, 6, 48, 0), (64, 64, 9, 9, 1, 4, 1, 0), (256, 256, 7, 9, 90, 3, 1, 0), (128, 128, 14, 14, 6, 4, 1, 1), (48, 32, 5, 3, 700, 7, 1, 0),
    (272, 112, 28, 28, 97, 5, 1, 0), (272, 48, 28, 28, 194, 5, 1, 0)])
def test_wide_layers_as_tiled_products(ctx, c, k, h, w, n, bits, tables, offset):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.95, None, 14000 + c + k + h))
    cal = fm.make_maps(params, max(4, 4 * c // (h * w) + 1), calib=True, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits, k=k)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=tables).hist, groups=tables)
    maps = fm.make_maps(params, n, dtype=torch.bfloat16, device="cuda")
    buf = torch.empty(maps.numel() + 8, dtype=torch.bfloat16, device="cuda")
    x = buf[offset:offset + maps.numel()].view(maps.shape)
    x.copy_(maps)
    fused = tc.tc_encode(ctx, m, cb, x, debug=True, k=k)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 3
    enc = tc.tc_encode(ctx, m, cb, x)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 3
    assert _same_stream(enc, fused)
    got = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, relu=True)
    assert tc.tc_get_status(ctx) == 0
    if c > 256:
        assert tc.tc_last_path(ctx, True) == 3
    tc.tc_force_exact_path(ctx, 1)
    want = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, relu=True)
    assert tc.tc_get_status(ctx) == 0
    tc.tc_force_exact_path(ctx, 0)
    # (neighbouring bf16 numbers for at most 0.1 % of the values: the parity cases' cap)
    a, b = got.float(), want.float()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-6 * float(b.abs().max())).all())
    assert float((a != b).double().mean()) <= 1e-3
    m.close(); cb.close()


# Covariance of the fit in 64 x 64 blocks of channel pairs over slabs of 32 pixels: one block, blocks with
# remainders, a single partial slab, slabs that cross images.  The basis rows are rounded to fp32
# (2^-24 of an entry), so the covariance put together from the model is off by at most
# 2 * 2^-24 * sum_j eig_j |b_ja| |b_jb| <= 2^-23 * max(eig); as much again for the sums' order and the
# eigenvectors' residual.
@pytest.mark.parametrize("c,h,w,n,dtype", [(2, 3, 3, 1, torch.float32), (33, 5, 7, 3, torch.float32), (64, 14, 14, 2, torch.float32),
                                           (65, 4, 8, 9, torch.float32), (200, 7, 7, 30, torch.float32)])
def test_covariance_blocks(ctx, c, h, w, n, dtype):
    g = torch.Generator(device="cuda").manual_seed(c)
    x = torch.randn(n, c, h, w, generator=g, device="cuda", dtype=torch.float64) * torch.linspace(2.0, 0.5, c, device="cuda", dtype=torch.float64).view(1, c, 1, 1)
    x = (x + 3.0 + 0.5 * x.mean(1, keepdim=True)).to(dtype)
    m = tc.tc_fit_pca(ctx, x, 6)
    e = tc.tc_model_export(m)
    v = x.double().transpose(0, 1).reshape(c, -1).cpu().numpy()
    v = v - v.mean(1, keepdims=True)
    want = v @ v.T / (v.shape[1] - 1)
    basis, eig = np.asarray(e["basis"], dtype=np.float64).reshape(c, c), np.asarray(e["eig"], dtype=np.float64)
    got = basis.T @ (eig[:, None] * basis)
    assert np.abs(got - want).max() <= 2.0 ** -22 * eig.max()
    m.close()


# One map of 2^26 pixels: the channels that a loader copies together lie further apart than 32 bits count.  The
# same pixels as sixteen maps are the same stream.
def test_channels_more_than_4_gb_apart(ctx):
    c, side, parts = 48, 8192, 16
    g = torch.Generator(device="cuda").manual_seed(17)
    x = torch.empty(1, c, side, side, dtype=torch.bfloat16, device="cuda")
    for i in range(c):
        x[0, i] = torch.randn(side, side, generator=g, device="cuda")
    cal = x[:, :, :64, :64].contiguous()
    m = tc.tc_fit_pca(ctx, cal, 4)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    y = x.view(c, parts, side // parts, side).permute(1, 0, 2, 3).contiguous()
    assert _same_stream(enc, tc.tc_encode(ctx, m, cb, y))
    a = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    b = tc.tc_decode(ctx, m, cb, enc, y.shape, y.dtype)
    assert tc.tc_get_status(ctx) == 0
    assert torch.equal(a.view(c, parts, side // parts, side).permute(1, 0, 2, 3), b)
    m.close(); cb.close()


# Blocks of modal symbols are passed over after a test that adds the bias up differently from the quantiser.  With a mean of
# 2048 quantiser ranges (identity basis, channel 5 `d` of a level above the modal one) fp32 places the two up to
# 0.03 of a level apart: a position next to the rounding boundary must not pass as the modal symbol.  The debug
# outputs switch the passing over off.
@pytest.mark.parametrize("d", [0.486, 0.499, 0.501, 0.515])
def test_passing_over_modal_blocks_far_from_zero_mean(ctx, d):
    c, bits, modal, offset = 64, 8, 127, 2048.0
    mean = np.full(c, offset)
    mean[5] -= d / 255
    m = tc.tc_model_import(ctx, basis=np.eye(c), mean=mean, lo=-modal / 255, step=1 / 255, bits=bits, basis_dtype=1, eig=np.full(c, 1e-12))
    counts = np.ones(256, dtype=np.uint64)
    counts[modal] = 1 << 30
    cb = tc.tc_codebook_import(ctx, tc.tc_host_huffman_lengths(counts, 12), bits)
    x = torch.full((2, c, 16, 16), offset, dtype=torch.bfloat16, device="cuda")
    enc = tc.tc_encode(ctx, m, cb, x)
    dbg = tc.tc_encode(ctx, m, cb, x, debug=True)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    q = dbg.symbols.cpu().numpy()
    assert np.all(np.delete(q, 5, axis=1) == modal) and np.all((q[:, 5] == modal) | (q[:, 5] == modal + 1))
    assert _same_stream(enc, dbg)
    m.close(); cb.close()


# Resident-basis encoder with several tiles per group and staging buffers that hold one, one and a half or many of
# them: the place of a new tile has to wait for the copy of the one before.  The same maps in pieces of one tile per
# block write the same words.
@pytest.mark.parametrize("c,bits,ratio", [(256, 8, 0.9), (256, 8, 0.99), (256, 6, 0.97), (208, 7, 0.98), (64, 8, 0.98)])
def test_staging_ring_of_the_resident_encoder(ctx, c, bits, ratio):
    params = fm.layer_params(fm.LayerSpec(c, 14, 14, ratio, None, 15000 + c + bits))
    cal = fm.make_maps(params, 256, calib=True, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    x = fm.make_maps(params, 32 * 40, dtype=torch.bfloat16, device="cuda")             # 1960 tiles, pieces of 49
    enc = tc.tc_encode(ctx, m, cb, x)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    base, chunks = 0, 0
    for i in range(0, x.shape[0], 32):
        part = tc.tc_encode(ctx, m, cb, x[i:i + 32])
        assert tc.tc_get_status(ctx) == 0
        n, bits_n, t0 = part.total_bits() // 8, part.total_bits(), i // 32 * 49
        assert torch.equal(enc.words[base // 8: base // 8 + n], part.words[:n])
        assert torch.equal(enc.tile_off[t0:t0 + 50] - base, part.tile_off)
        assert torch.equal(enc.chunk_len[chunks:chunks + part.layout.n_chunks], part.chunk_len[:part.layout.n_chunks])
        base, chunks = base + bits_n, chunks + part.layout.n_chunks
    assert base == enc.total_bits()
    m.close(); cb.close()


# Run-skipping decoder, how channel rows leave: 16 and 8 bytes a thread and a pixel a thread (H*W a multiple of 8, of 4, of neither;
# tensors that start anywhere), one item for the whole block and several, one block of 128 channels and two with remainders, last
# tiles of a pixel, 64 and 127, images shorter than a tile.  The stream does not depend on how the pixels are laid out: one image of one row is the
# same tensor through other stores.  Against the fp64 kernels too (neighbouring bf16 numbers).
@pytest.mark.parametrize("c,h,w,n", [(16, 1, 1, 1), (16, 8, 8, 3), (32, 4, 3, 11), (48, 7, 7, 5), (64, 3, 43, 1), (80, 16, 16, 1), (128, 9, 7, 65), (128, 2, 2, 600),
                                     (144, 2, 64, 3), (176, 14, 14, 7), (208, 5, 5, 51), (256, 1, 129, 1), (256, 8, 12, 199), (112, 1, 1, 19000)])
def test_rows_of_the_run_skipping_decoder(ctx, c, h, w, n):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 21000 + c + h))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=torch.bfloat16, device="cuda")
    x = fm.make_maps(params, n, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, 4)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x)
    got = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    row = got.transpose(0, 1).reshape(c, -1)
    for shape in ((1, c, 1, n * h * w), (n * h * w, c, 1, 1)):
        assert torch.equal(row, tc.tc_decode(ctx, m, cb, enc, shape, x.dtype).transpose(0, 1).reshape(c, -1))
    for offset in (1, 2, 4):
        buf = torch.full((x.numel() + 16,), 7.0, dtype=x.dtype, device="cuda")
        part = buf[offset:offset + x.numel()].view(x.shape)
        tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, out=part)
        assert torch.equal(part, got)
        assert bool((buf[:offset] == 7.0).all()) and bool((buf[offset + x.numel():] == 7.0).all())
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    tc.tc_force_exact_path(ctx, 1)
    want = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0
    tc.tc_force_exact_path(ctx, 0)
    a, b = got.float(), want.float()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-6 * float(b.abs().max())).all())
    m.close(); cb.close()


# The run-skipping decoder is what runs on this build: kernels that come out with too few registers for its roles, or buffers that do not fit, leave
# the tensor to decoders that report the same path and are several times slower.
@pytest.mark.parametrize("c,h,w,n,bits,k,cp,splits", [(16, 1, 1, 1, 2, 0, 0, 0), (64, 56, 56, 4, 4, 0, 0, 0), (128, 14, 14, 9, 8, 0, 0, 0), (176, 7, 7, 40, 5, 0, 0, 0), (256, 14, 14, 9, 4, 0, 0, 0),
                                                      (256, 14, 14, 9, 8, 0, 0, 0), (256, 9, 7, 30, 8, 0, 0, 0), (256, 3, 1, 500, 6, 0, 0, 0), (240, 14, 14, 5, 6, 48, 0, 0), (256, 14, 14, 4, 4, 0, 1, 4),
                                                      (128, 14, 14, 4, 5, 0, 16, 1)])
def test_the_run_skipping_decoder_runs(ctx, c, h, w, n, bits, k, cp, splits):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 24000 + c))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=torch.bfloat16, device="cuda")
    x = fm.make_maps(params, n, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits, k=k)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x, chunk_pixels=cp, pixel_splits=splits)
    runs = tc.load_library().tc_last_decode_skipped_runs
    runs.argtypes = [ctypes.c_void_p]
    for switch, want in ((0, 1), (3, 0), (0, 1)):
        tc.tc_force_exact_path(ctx, switch)
        for relu in (False, True):
            tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, relu=relu)
            assert tc.tc_get_status(ctx) == 0 and runs(ctx.ptr) == want and (not want or tc.tc_last_path(ctx, True) == 1)
    tc.tc_decode_many(ctx, [(m, cb, enc, x.shape, x.dtype)] * 2)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1 and runs(ctx.ptr) == 1
    m.close(); cb.close()


# Maps of up to four pixels, whose channels leave side by side: 2, 4 and 8 bytes a thread (tensors that start anywhere), one item and several, a
# last tile of a pixel or a map, channels that end inside a warp's 32, maps that begin in the tile before (three pixels), the non-linearity.
@pytest.mark.parametrize("c,h,w,n", [(16, 1, 2, 5), (48, 3, 1, 43), (128, 1, 3, 700), (144, 1, 3, 1), (176, 1, 1, 129), (208, 4, 1, 33), (256, 1, 2, 20000), (240, 2, 2, 6000),
                                     (80, 1, 1, 38000), (112, 1, 3, 25000)])
def test_small_maps_of_the_run_skipping_decoder(ctx, c, h, w, n):
    test_rows_of_the_run_skipping_decoder(ctx, c, h, w, n)
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 23000 + c))
    cal, x = (fm.make_maps(params, m, calib=m > n, dtype=torch.bfloat16, device="cuda") for m in (max(n + 1, 12000), n))
    m = tc.tc_fit_pca(ctx, cal, 5)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x)
    got = [tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, relu=r) for r in (False, True)]
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1 and torch.equal(got[0].clamp(min=0), got[1])
    m.close(); cb.close()


# Run-skipping decoder, stream buffers sized by the rate: three groups and one work item per tile (128 and 112
# channels), buffers above 16 KB, segments that fit no buffer, and hints that are too small or too large -- the hint
# changes how tiles are staged, never the tensor.  Against the fp64 kernels on the same stream.
@pytest.mark.parametrize("c,h,w,bits,ratio,cp", [(128, 28, 28, 8, 0.9, 0), (112, 28, 28, 8, 0.98, 2), (160, 28, 28, 8, 0.9, 0), (208, 14, 14, 8, 0.98, 0),
                                                 (224, 14, 14, 8, 0.98, 0), (80, 28, 28, 8, 0.9, 0), (64, 56, 56, 7, 0.95, 0), (144, 28, 28, 6, 0.9, 0)])
def test_run_skipping_decoder_stream_buffers(ctx, c, h, w, bits, ratio, cp):
    params = fm.layer_params(fm.LayerSpec(c, h, w, ratio, None, 16000 + c))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=torch.bfloat16, device="cuda")
    x = fm.make_maps(params, 148 * 9 * 128 // (h * w) + 3, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x, chunk_pixels=cp)
    got = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    for hint in (1, 5000, 12000, 60000, 2 ** 31 - 1):
        assert torch.equal(got, tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype, mean_tile_bytes=hint))
    again = tc.tc_codebook_import(ctx, tc.tc_codebook_export(cb), bits)          # without counts
    assert torch.equal(got, tc.tc_decode(ctx, m, again, enc, x.shape, x.dtype))
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    tc.tc_force_exact_path(ctx, 1)
    want = tc.tc_decode(ctx, m, cb, enc, x.shape, x.dtype)
    assert tc.tc_get_status(ctx) == 0
    tc.tc_force_exact_path(ctx, 0)
    # (neighbouring bf16 numbers for at most 0.1 % of the values: the parity cases' cap)
    a, b = got.float(), want.float()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-6 * float(b.abs().max())).all())
    assert float((a != b).double().mean()) <= 1e-3
    for h_ in (m, cb, again):
        h_.close()


# Resident-basis encoder, private runs shorter than the codes: a model whose eigenvalues say too little (or nothing) and
# maps of more spread than the calibration's.  Tiles are then coded once more into the staging buffer, over the runs
# behind it, or into global memory; the words are those of a plan that allows for everything (eigenvalues 100 times
# too large), and those of the streaming kernels' coder on the same symbols.
@pytest.mark.parametrize("c,bits,tables,spread", [(256, 4, 1, 1), (256, 4, 1, 2), (256, 4, 1, 6), (64, 4, 1, 5), (128, 6, 1, 3), (128, 8, 1, 1),
                                                  (208, 5, 1, 3), (16, 2, 1, 4), (96, 4, 96, 3), (256, 3, 256, 5), (240, 8, 1, 8)])
def test_runs_shorter_than_the_codes(ctx, c, bits, tables, spread):
    params = fm.layer_params(fm.LayerSpec(c, 14, 14, 0.9, None, 17000 + c + bits))
    cal = fm.make_maps(params, 256, calib=True, dtype=torch.bfloat16, device="cuda")
    m = tc.tc_fit_pca(ctx, cal, bits)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=tables).hist, groups=tables)
    d = tc.tc_model_export(m)
    mean = torch.from_numpy(d["mean"]).float().cuda().view(1, c, 1, 1)
    x = ((fm.make_maps(params, 1500, dtype=torch.float32, device="cuda") - mean) * spread + mean).to(torch.bfloat16)      # several tiles a group
    x[7] = cal[0]                                                     # tiles that do fit between those that do not
    args = dict(basis=d["basis"], mean=d["mean"], lo=d["lo"], step=d["step"], bits=bits, basis_dtype=1, k=d["k"])
    ample = tc.tc_model_import(ctx, eig=d["eig"] * 100, **args)
    ref = tc.tc_encode(ctx, ample, cb, x, debug=True)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == 1
    check_stream_against_oracle(tc.tc_encode(ctx, ample, cb, x[:9], debug=True), ref.symbols[:9 * 196].cpu().numpy(), tc.tc_codebook_export(cb), bits)
    for eig in (d["eig"], d["eig"] / 100, np.full(c, 1e-9), None):
        own = tc.tc_model_import(ctx, eig=eig, **args)
        assert _same_stream(tc.tc_encode(ctx, own, cb, x), ref)
        assert tc.tc_get_status(ctx) == 0
        own.close()
    for h in (m, cb, ample):
        h.close()


# The decoder's side of it: eight channel rows of 2^29 pixels are further apart than 32 bits count.
def test_decoded_rows_more_than_2_32_elements_apart(ctx):
    c, h, w, parts = 16, 16384, 32768, 64
    g = torch.Generator(device="cuda").manual_seed(18)
    x = torch.empty(1, c, h, w, dtype=torch.bfloat16, device="cuda")
    for i in range(c):
        x[0, i] = torch.randn(h, w, generator=g, device="cuda")
    cal = x[:, :, :256, :256].contiguous()
    m = tc.tc_fit_pca(ctx, cal, 3)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal).hist)
    enc = tc.tc_encode(ctx, m, cb, x, capacity=6 << 30)
    assert tc.tc_get_status(ctx) == 0
    del x
    a = tc.tc_decode(ctx, m, cb, enc, (1, c, h, w), torch.bfloat16)
    b = tc.tc_decode(ctx, m, cb, enc, (parts, c, h // parts, w), torch.bfloat16)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == 1
    for i in range(c):
        assert torch.equal(a[0, i].view(parts, h // parts, w), b[:, i])
    m.close(); cb.close()


# Entropy coder and decoder with a tile dealt to several blocks: tiles few enough for two and four blocks (and one more), last tiles
# whose later blocks have a pixel or none, chunks of several pixels, one, two and four a pixel, tables per layer and per channel, codes
# of one bit and of twelve.  (Most of them leave the coder, which deals from 384 coefficients on, one block a tile: more of its cases below.)
# Against the one-thread-per-pixel kernels, which run without workspace.
@pytest.mark.parametrize("c,pixels,bits,dtype,per_channel,cp,splits", [
    (64, 1, 4, torch.float32, False, 0, 0), (64, 33, 4, torch.float32, False, 0, 0), (64, 128 * 37, 3, torch.float32, False, 4, 1),
    (64, 128 * 37 + 1, 5, torch.float32, True, 0, 0), (96, 65, 8, torch.float32, True, 0, 0), (128, 128 * 74 - 31, 4, torch.float32, False, 0, 0),
    (128, 128 * 74 + 97, 4, torch.float32, False, 0, 0), (64, 200, 2, torch.float32, False, 64, 1), (64, 200, 2, torch.float32, False, 32, 1),
    (256, 96, 6, torch.float32, True, 0, 0), (256, 300, 1, torch.float32, False, 0, 0), (512, 129, 8, torch.float32, False, 0, 0),
    (512, 128 * 5 + 34, 4, torch.float32, True, 0, 0), (320, 49 * 3, 4, torch.bfloat16, False, 0, 0), (320, 49 * 100, 8, torch.bfloat16, False, 0, 0),
    (576, 49 * 7, 5, torch.bfloat16, False, 0, 0), (256, 49 * 3, 6, torch.bfloat16, True, 0, 0), (512, 49 * 500, 4, torch.bfloat16, False, 0, 0)])
def test_a_tile_dealt_to_several_blocks(ctx, c, pixels, bits, dtype, per_channel, cp, splits):
    _deal_and_compare(ctx, c, pixels, bits, dtype, per_channel, cp, splits)


# The coder deals a tile to a cluster from 384 coefficients on.  Two blocks a tile (38 and 74 tiles; 75 leave one) and four; last tiles that
# leave the later blocks no pixel or one; chunks of several pixels, up to what a block has; codes of one bit, and codes of eight
# throughout, which exceed the staging (four bits a symbol), so that the cluster clears the stream and writes to it.
@pytest.mark.parametrize("c,pixels,bits,dtype,per_channel,cp,splits,flat", [
    (512, 128 * 3 + 1, 1, torch.float32, False, 0, 0, False), (384, 128 * 2 + 33, 2, torch.float32, False, 4, 1, False),
    (384, 128 + 97, 2, torch.float32, False, 32, 1, False), (384, 128 * 5, 1, torch.float32, False, 64, 1, False),
    (512, 128 * 5 + 65, 3, torch.float32, False, 16, 1, False), (384, 128 * 37 + 1, 4, torch.float32, False, 0, 0, False),
    (384, 128 * 37 + 64, 4, torch.float32, True, 0, 0, False), (384, 128 * 73 + 65, 3, torch.float32, False, 0, 0, False),
    (384, 128 * 74 + 1, 3, torch.float32, False, 0, 0, False), (960, 49 * 100, 5, torch.bfloat16, False, 0, 0, False),
    (512, 129, 8, torch.float32, False, 0, 0, True), (384, 128 * 2 + 34, 8, torch.float32, True, 0, 0, True), (384, 128 * 38 + 33, 8, torch.float32, False, 0, 0, True)])
def test_a_tile_coded_by_a_cluster(ctx, c, pixels, bits, dtype, per_channel, cp, splits, flat):
    enc = _deal_and_compare(ctx, c, pixels, bits, dtype, per_channel, cp, splits, flat)
    if flat:
        assert int(enc.tile_off[1] - enc.tile_off[0]) > 4 * 128 * c


def _deal_and_compare(ctx, c, pixels, bits, dtype, per_channel, cp, splits, flat=False):
    rng = np.random.default_rng(c + pixels)
    h, n = (7, pixels // 49) if dtype == torch.bfloat16 else (1, 1)
    w = pixels // (n * h)
    basis, _ = np.linalg.qr(rng.standard_normal((c, c)))
    if dtype == torch.bfloat16:
        basis = torch.from_numpy(basis).to(torch.bfloat16).double().numpy()
    else:
        basis = basis.astype(np.float32).astype(np.float64)
    scale = 4.0 * 0.97 ** np.arange(c) + 1e-3
    top = (1 << bits) - 1
    step = 12.0 / top if bits > 1 else 6.0
    lo = -step * round(6.0 / step)
    x = torch.from_numpy(((rng.standard_normal((n * h * w, c)) * scale) @ basis).reshape(n, h * w, c).transpose(0, 2, 1).reshape(n, c, h, w).copy()).to(dtype).cuda()
    counts = rng.integers(0, 50, (c if per_channel else 1, top + 1))
    counts[..., top // 2] = 2000 if bits > 1 else 1
    counts[..., 0] = 0
    if flat:
        counts[:] = 1
    lengths = np.stack([tc.tc_host_huffman_lengths(row) for row in counts])
    m = tc.tc_model_import(ctx, basis=basis, mean=np.zeros(c), lo=lo, step=step, bits=bits, basis_dtype=tc.binding.TC_BF16 if dtype == torch.bfloat16 else tc.binding.TC_F32,
                           eig=scale ** 2)
    cb = tc.tc_codebook_import(ctx, lengths, bits)
    kw = dict(chunk_pixels=cp, pixel_splits=splits) if cp else {}
    enc = tc.tc_encode(ctx, m, cb, x, **kw)
    x_hat = tc.tc_decode(ctx, m, cb, enc, x.shape, dtype)
    assert tc.tc_get_status(ctx) == 0
    tc.tc_force_exact_path(ctx, 4)
    want = tc.tc_encode(ctx, m, cb, x, **kw)
    want_hat = tc.tc_decode(ctx, m, cb, enc, x.shape, dtype)
    tc.tc_force_exact_path(ctx, 0)
    assert tc.tc_get_status(ctx) == 0
    if dtype == torch.float32:
        assert _same_stream(enc, want) and torch.equal(x_hat, want_hat)
    else:           # fp32 accumulation in another order: a symbol at a rounding tie, bf16 neighbours now and then
        assert abs(enc.total_bits() - want.total_bits()) <= 1e-3 * want.total_bits() + 256
        assert (x_hat != want_hat).double().mean() <= 1e-3 and (x_hat.double() - want_hat.double()).abs().max() <= 2.0 ** -7 * want_hat.double().abs().max()
    m.close(); cb.close()
    return enc


# The resident-basis encoder's look-back arrays, two of a context in turn, each cleared by the call that follows its use: calls large and small
# on one context, with those in between that leave the arrays alone (over 8192 tiles, captured, a list) or end early (a buffer that is
# too small).  Every stream that of a context of its own.
def test_look_back_arrays_in_turn(ctx):
    c, bits = 16, 4
    basis = torch.linalg.qr(torch.randn(c, c, dtype=torch.float64, generator=torch.Generator().manual_seed(4)))[0].to(torch.bfloat16).double().numpy()
    counts = np.full(16, 5)
    counts[7] = 2000
    m = tc.tc_model_import(ctx, basis=basis, mean=np.zeros(c), lo=-3.0, step=0.4, bits=bits, basis_dtype=tc.binding.TC_BF16, eig=4.0 * 0.7 ** np.arange(c))
    cb = tc.tc_codebook_import(ctx, np.stack([tc.tc_host_huffman_lengths(counts)]), bits)
    gen = torch.Generator(device="cuda").manual_seed(9)
    maps = {tiles: torch.randn(1, c, tiles * 32, 4, device="cuda", generator=gen).to(torch.bfloat16) for tiles in (1, 3, 148, 700, 5000, 8192, 8193)}
    want = {}
    for tiles, x in maps.items():
        own = tc.tc_create(0)
        want[tiles] = tc.tc_encode(own, m, cb, x)
        assert tc.tc_get_status(own) == 0 and tc.tc_last_path(own) == 1
        own.close()

    def check(enc, tiles):
        n = want[tiles].total_bits() // 8
        assert torch.equal(enc.tile_off, want[tiles].tile_off) and torch.equal(enc.words[:n], want[tiles].words[:n])
        assert torch.equal(enc.chunk_len[:enc.layout.n_chunks], want[tiles].chunk_len[:enc.layout.n_chunks])

    own = tc.tc_create(0)
    for tiles in (5000, 3, 5000, 1, 1, 700, 8192, "short", 700, "short", 8192, 8193, 148, "graph", 5000, "list", 5000, "list", 3, "graph", 8192, 1, 8192):
        if tiles == "short":
            tc.tc_encode(own, m, cb, maps[700], capacity=want[700].total_bits() // 16)
            assert tc.tc_get_status(own) == 3
        elif tiles == "graph":
            out = tc.tc_encode(own, m, cb, maps[700])
            torch.cuda.synchronize()
            graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            with torch.cuda.stream(side):
                graph.capture_begin()
                tc.tc_encode(own, m, cb, maps[700], out=out)
                graph.capture_end()
            torch.cuda.synchronize()
            for _ in range(3):
                out.words.zero_()
                graph.replay()
                torch.cuda.synchronize()
                check(out, 700)
        elif tiles == "list":
            for t, enc in zip((148, 5000, 3), tc.tc_encode_many(own, [(m, cb, maps[t]) for t in (148, 5000, 3)])):
                check(enc, t)
        else:
            check(tc.tc_encode(own, m, cb, maps[tiles]), tiles)
    assert tc.tc_get_status(own) == 0
    own.close()
