"""Kernels that start before the end of the one ahead of them in the stream: what that one writes, they read only once it is done.

The kernel ahead is one of the test's own.  It lets the kernel behind it start at once, waits, and only then rewrites the call's inputs in
place, so that a read ahead of the wait meets the data of the turn before."""
import numpy as np
import pytest
import torch

import paper_1905_10830_b200 as tc
from synth import featuremaps as fm

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32
TURNS = 10

SOURCE = """
extern "C" __global__ void late_copy(uint4 *dst, const uint4 *src, unsigned long long pieces, unsigned long long delay_ns)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int i = 0; i < 8000000; ++i) {            // (ends by itself whatever the clock says)
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 > delay_ns) break;
        __nanosleep(1000);
    }
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < pieces; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


@pytest.fixture(scope="module")
def ctx():
    c = tc.tc_create(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def late_copy():
    """late_copy(dst, src, delay_us): copies `src` over `dst` on the current stream, `delay_us` after the kernel behind it may start."""
    from cuda.bindings import driver, nvrtc

    def ok(result):
        err, *rest = result
        assert int(err) == 0, err
        return rest[0] if len(rest) == 1 else rest
    torch.zeros(1, device="cuda")                  # the primary context is current
    prog = ok(nvrtc.nvrtcCreateProgram(SOURCE.encode(), b"late_copy.cu", 0, [], []))
    ok(nvrtc.nvrtcCompileProgram(prog, 1, [b"--gpu-architecture=sm_100a"]))
    cubin = b" " * ok(nvrtc.nvrtcGetCUBINSize(prog))
    ok(nvrtc.nvrtcGetCUBIN(prog, cubin))
    kernel = ok(driver.cuModuleGetFunction(ok(driver.cuModuleLoadData(cubin)), b"late_copy"))

    def run(dst, src, delay_us):
        nbytes = dst.numel() * dst.element_size()
        assert nbytes == src.numel() * src.element_size() and nbytes % 16 == 0 and dst.data_ptr() % 16 == 0 and src.data_ptr() % 16 == 0
        args = [np.array([v], dtype=np.uint64) for v in (dst.data_ptr(), src.data_ptr(), nbytes // 16, int(delay_us * 1000))]
        params = np.array([a.ctypes.data for a in args], dtype=np.uint64)
        ok(driver.cuLaunchKernel(kernel, 4, 1, 1, 256, 1, 1, 0, torch.cuda.current_stream().cuda_stream, params.ctypes.data, 0))
    return run


def _layer(ctx, c, h, w, n, bits, tables, dtype, turns, k=0, seed=0):
    params = fm.layer_params(fm.LayerSpec(c, h, w, 0.9, None, 31000 + c + bits + seed))
    cal = fm.make_maps(params, max(4, 30000 // (h * w)), calib=True, dtype=dtype, device="cuda")
    maps = fm.make_maps(params, n * turns, dtype=dtype, device="cuda").view(turns, n, c, h, w)
    m = tc.tc_fit_pca(ctx, cal, bits, k=k)
    cb = tc.tc_build_codebook(ctx, m, tc.tc_stats(ctx, m, None, cal, groups=tables).hist, groups=tables)
    return m, cb, maps


def _packed(lay):
    """A stream's three arrays in one buffer: (buffer, EncodedStream of its parts)."""
    up = lambda v: (v + 255) // 256 * 256
    sizes = (max(lay.stream_bytes, 16), 2 * (lay.n_chunks + (lay.n_chunks & 1)), 8 * (lay.n_tiles + 1))
    at = np.concatenate([[0], np.cumsum([up(s) for s in sizes])])
    buf = torch.zeros(int(at[-1]), dtype=torch.uint8, device="cuda")
    part = [buf[int(a):int(a) + s] for a, s in zip(at, sizes)]
    return buf, tc.EncodedStream(part[0], part[1].view(torch.int16), part[2].view(torch.int64), lay)


# The run-skipping decoder (one block of channels and two, rows of every kind, one item and several), and the entropy decoders that leave
# symbols for the tiled product (wide layers, a table per channel) and for the exact inverse.
DECODES = [(64, 14, 14, 40, 4, 1, BF16, 1), (256, 14, 14, 30, 4, 1, BF16, 1), (256, 7, 7, 9, 8, 1, BF16, 1), (16, 2, 2, 1, 2, 1, BF16, 1),
           (576, 14, 14, 20, 5, 1, BF16, 3), (64, 14, 14, 20, 6, 64, BF16, 1), (256, 14, 14, 1, 6, 256, F32, 0), (48, 10, 10, 3, 5, 1, F32, 0)]


@pytest.mark.parametrize("c,h,w,n,bits,tables,dtype,path", DECODES)
def test_decodes_wait_for_the_stream(ctx, late_copy, c, h, w, n, bits, tables, dtype, path):
    m, cb, maps = _layer(ctx, c, h, w, n, bits, tables, dtype, TURNS)
    shape = maps.shape[1:]
    streams = [_packed(tc.tc_encode_bound(m, cb, x)) for x in maps]
    for x, (_, enc) in zip(maps, streams):
        tc.tc_encode(ctx, m, cb, x, out=enc)
    want = [tc.tc_decode(ctx, m, cb, enc, shape, dtype) for _, enc in streams]
    buf, live = _packed(streams[0][1].layout)
    got = [torch.empty_like(x) for x in maps]
    torch.cuda.synchronize()
    for (src, _), out in zip(streams, got):
        late_copy(buf, src, 40)
        tc.tc_decode(ctx, m, cb, live, shape, dtype, out=out)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == path
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    m.close(); cb.close()


# The exact projection, the pixel rows in front of the tiled product (7x7 and aligned maps), and the resident-basis encoder, which starts in
# its turn.
ENCODES = [(64, 28, 28, 1, 8, 1, F32, 0), (256, 14, 14, 1, 6, 256, F32, 0), (960, 7, 7, 30, 5, 1, BF16, 3), (320, 8, 8, 12, 4, 1, BF16, 3),
           (128, 14, 14, 30, 4, 1, BF16, 1)]


@pytest.mark.parametrize("c,h,w,n,bits,tables,dtype,path", ENCODES)
def test_encodes_wait_for_the_maps(ctx, late_copy, c, h, w, n, bits, tables, dtype, path):
    m, cb, maps = _layer(ctx, c, h, w, n, bits, tables, dtype, TURNS)
    want = [tc.tc_encode(ctx, m, cb, x) for x in maps]
    got = [_packed(e.layout)[1] for e in want]
    live = torch.zeros_like(maps[0])
    torch.cuda.synchronize()
    for x, out in zip(maps, got):
        late_copy(live, x, 40)
        tc.tc_encode(ctx, m, cb, live, out=out)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx) == path
    for a, b in zip(got, want):
        bits_a, chunks = a.total_bits(), a.layout.n_chunks
        assert bits_a == b.total_bits() and torch.equal(a.words[:bits_a // 8], b.words[:bits_a // 8])
        assert torch.equal(a.tile_off, b.tile_off) and torch.equal(a.chunk_len[:chunks], b.chunk_len[:chunks])
    m.close(); cb.close()


# A tensor that the kernel ahead still reads is written only once that is done, also across streams.
@pytest.mark.parametrize("c,h,w,n,bits,tables,dtype,path", DECODES)
def test_decodes_wait_for_readers_of_the_tensor(ctx, late_copy, c, h, w, n, bits, tables, dtype, path):
    m, cb, maps = _layer(ctx, c, h, w, n, bits, tables, dtype, TURNS)
    shape = maps.shape[1:]
    streams = [tc.tc_encode(ctx, m, cb, x) for x in maps]
    want = [tc.tc_decode(ctx, m, cb, enc, shape, dtype) for enc in streams]
    size = max(16, (maps[0].numel() * maps[0].element_size() + 15) // 16 * 16) // maps[0].element_size()
    room = torch.zeros(size, dtype=dtype, device="cuda")
    out = room[:maps[0].numel()].view(shape)
    kept = torch.zeros(TURNS, size, dtype=dtype, device="cuda")
    side, ready = torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    for i, enc in enumerate(streams):
        on = torch.cuda.current_stream() if i % 3 else side       # the reader's stream
        if not i % 3:
            ready.record(); side.wait_event(ready)
        with torch.cuda.stream(on):
            if i:
                late_copy(kept[i - 1], room, 40)
        if not i % 3:
            ready.record(side); torch.cuda.current_stream().wait_event(ready)
        tc.tc_decode(ctx, m, cb, enc, shape, dtype, out=out)
    kept[-1].copy_(room)
    assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == path
    for got, b in zip(kept, want):
        assert torch.equal(got[:b.numel()].view(shape), b)
    m.close(); cb.close()


# A kernel ahead that takes longer than a decoder's own waits are allowed to (two seconds): they begin when it is done.
def test_a_long_kernel_ahead_is_no_timeout(ctx, late_copy):
    m, cb, maps = _layer(ctx, 64, 14, 14, 40, 4, 1, BF16, 2)
    streams = [_packed(tc.tc_encode_bound(m, cb, x)) for x in maps]
    for x, (_, enc) in zip(maps, streams):
        tc.tc_encode(ctx, m, cb, x, out=enc)
    want = tc.tc_decode(ctx, m, cb, streams[1][1], maps.shape[1:], BF16)
    buf, live = _packed(streams[0][1].layout)
    buf.copy_(streams[0][0])
    torch.cuda.synchronize()
    late_copy(buf, streams[1][0], 2.6e6)
    got = tc.tc_decode(ctx, m, cb, live, maps.shape[1:], BF16)
    assert tc.tc_get_status(ctx) == 0 and torch.equal(got, want)
    m.close(); cb.close()


# Tables are read ahead of the wait: a codebook is complete when the call that makes it returns, also for streams that do not wait for the
# legacy one.
@pytest.mark.parametrize("c,tables,dtype,path", [(64, 1, BF16, 1), (256, 256, BF16, 1), (256, 256, F32, 0), (576, 1, BF16, 3)])
def test_a_new_codebook_on_a_stream_of_its_own(ctx, c, tables, dtype, path):
    m, cb, maps = _layer(ctx, c, 14, 14, 2, 8, tables, dtype, 1)
    x, rng = maps[0], np.random.default_rng(c)
    lengths = [np.stack([tc.tc_host_huffman_lengths(rng.integers(0, 10 ** rng.integers(1, 6), 256)) for _ in range(tables)]) for _ in range(TURNS)]
    books = [tc.tc_codebook_import(ctx, l, 8) for l in lengths]
    streams = [tc.tc_encode(ctx, m, b, x) for b in books]
    want = tc.tc_decode(ctx, m, books[0], streams[0], x.shape, dtype)
    assert tc.tc_get_status(ctx) == 0
    got = [torch.empty_like(x) for _ in lengths]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        made = [tc.tc_codebook_import(ctx, lengths[0], 8)]
        for l, enc, out in zip(lengths, streams, got):
            made.append(tc.tc_codebook_import(ctx, l, 8))
            tc.tc_decode(ctx, m, made[-1], enc, x.shape, dtype, out=out)
        assert tc.tc_get_status(ctx) == 0 and tc.tc_last_path(ctx, True) == path
    assert all(torch.equal(g, want) for g in got)
    for h in [m, cb] + books + made:
        h.close()
