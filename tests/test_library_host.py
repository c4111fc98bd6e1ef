"""CPU-side checks of the CUDA library: it loads, exports every symbol the header declares,
refuses to run without a device, and its host algorithms (Huffman lengths, eigensolver) agree
with the oracle / numpy."""
import os
import re

import numpy as np
import pytest

import oracle
import paper_1905_10830_b200 as tc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1905_10830_b200 import build
    build.build_library()
    return tc.load_library()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "tc.h")).read()
    declared = set(re.findall(r"\b(tc_[a-z0-9_]+)\s*\(", header))
    assert declared, "no declarations found"
    assert declared == set(tc.binding.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_no_device_means_error_not_fallback(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    with pytest.raises(tc.TcError):
        tc.tc_create(0)


def test_host_huffman_matches_oracle_lengths(lib):
    rng = np.random.default_rng(3)
    for _ in range(200):
        n = 1 << int(rng.integers(1, 9))
        counts = (rng.integers(0, 12, n) ** int(rng.integers(1, 8))).astype(np.uint64)
        for lmax in (12, max(8, int(np.log2(n)))):
            assert np.array_equal(tc.tc_host_huffman_lengths(counts, lmax), oracle.huffman_lengths(counts, lmax)[0])


def test_host_huffman_rejects_bad_arguments(lib):
    with pytest.raises(tc.TcError):
        tc.tc_host_huffman_lengths(np.zeros(256, dtype=np.uint64), 7)     # 2^7 < 256 symbols


@pytest.mark.parametrize("n", [1, 2, 17, 96, 256])
def test_host_eigh_against_numpy(lib, n):
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = 0.9 ** np.arange(n)
    a = (q * lam) @ q.T
    a = (a + a.T) / 2
    ev, vt = tc.tc_host_eigh(a)
    assert np.allclose(ev, np.sort(np.linalg.eigvalsh(a))[::-1], rtol=0, atol=1e-13)
    assert np.all(np.diff(ev) <= 0)
    assert np.allclose(vt @ vt.T, np.eye(n), atol=1e-12)
    assert np.allclose(vt @ a @ vt.T, np.diag(ev), atol=1e-13)
    for row in vt:
        assert row[np.argmax(np.abs(row))] > 0


def test_host_eigh_repeated_eigenvalues(lib):
    ev, vt = tc.tc_host_eigh(np.diag([2.0, 2.0, 1.0, 2.0]))
    assert np.allclose(ev, [2, 2, 2, 1])
    assert np.allclose(vt @ vt.T, np.eye(4), atol=1e-14)


# Shared memory that keeps the blocks of kernels that start early apart: as many as an SM would get fit it, and not one more.
@pytest.mark.parametrize("own", [2176, 5696, 10368, 15488])
def test_blocks_kept_apart_fit_their_sm(lib, own):
    import ctypes as C
    spread = lib.tc_spread_bytes
    spread.restype, spread.argtypes = C.c_size_t, [C.c_longlong, C.c_int, C.c_size_t]
    sms, sm, block = 148, 228 * 1024, 1024                     # bytes of an SM, and what the system keeps of a block's
    for blocks in (1, 2, 147, 148):
        assert 2 * (spread(blocks, sms, own) + own + block) > sm and spread(blocks, sms, own) + own <= 227 * 1024
    for per_sm in range(2, 9):
        for blocks in ((per_sm - 1) * sms + 1, per_sm * sms):
            each = spread(blocks, sms, own) + own + block
            assert per_sm * each <= sm < (per_sm + 1) * each
    assert spread(8 * sms + 1, sms, own) == 0


# The resident-basis encoder's issuing warp when one of its waits runs out: no products of what has not landed, no stage handed back, no
# accumulator handed on, and it leaves when what it has issued is done.
@pytest.mark.parametrize("groups,tiles,panels,stages", [(4, 1, 1, 8), (4, 9, 4, 6), (2, 3, 8, 8), (2, 5, 7, 6)])
def test_nothing_is_issued_after_a_wait_that_ran_out(lib, groups, tiles, panels, stages):
    import ctypes as C
    call = lib.tc_issue_events
    call.restype, call.argtypes = C.c_int, [C.c_int, C.c_longlong, C.c_int, C.c_int, C.c_int, C.POINTER(C.c_int32), C.c_int]
    room = (C.c_int32 * 4096)()

    def events(fails):
        n = call(groups, tiles, panels, stages, fails, room, len(room))
        assert 0 < n <= len(room)
        return list(room[:n])
    want, at = [], 0
    for tl in range(tiles):
        want += [100 + (at + i) % stages for i in range(panels)] + [200 + tl % groups]
        at += panels
    assert events(-1) == want + [300]
    assert events(0) == [-1]                                   # the basis: nothing has been issued
    for fails in range(1, 1 + tiles * (1 + panels)):
        tl, i = divmod(fails - 1, 1 + panels)                  # wait i of a tile: its accumulator, then its panels
        issued = want[:tl * (panels + 1) + max(0, i - 1)]
        assert events(fails) == issued + [-1, 300]


@pytest.fixture(scope="module")
def encode_classes(lib):
    """Kernel classes of tensors (c, k, bits, tables, tiles, bits per coefficient) of a list, or of a call with one: bit 0 a table per channel, bit 1 symbol
    pairs, bit 2 private runs, bit 3 four epilogue groups a block."""
    import ctypes as C

    def run(*tensors):
        n, out = len(tensors), (C.c_int * len(tensors))()
        ints = [(C.c_int * n)(*[t[j] for t in tensors]) for j in range(4)]
        lib.tc_encode_classes(n, *ints, (C.c_longlong * n)(*[t[4] for t in tensors]), (C.c_float * n)(*[t[5] for t in tensors]), 148, 227 * 1024, out)
        return list(out)
    return run


# Four epilogue groups where a block has several tiles, two where it has few and above 128 coefficients.
@pytest.mark.parametrize("k,tiles,four", [(16, 1, 1), (32, 1, 0), (48, 148, 0), (48, 149, 1), (64, 2 * 148, 0), (64, 2 * 148 + 1, 1), (128, 2 * 148, 0), (128, 2 * 148 + 1, 1), (16, 10 ** 7, 1), (144, 10 ** 7, 0)])
def test_epilogue_groups_by_tiles(encode_classes, k, tiles, four):
    assert encode_classes((max(k, 160), k, 4, 1, tiles, 1.3)) == [6 + 8 * four]


# Lists: short ones in one launch; longer ones, where wide tensors take a launch anyway, in theirs -- the class with two groups being that of the plan with two
# groups, which has room for private runs where four leave none -- and long ones with four groups for narrow tensors.
def test_epilogue_groups_of_lists(encode_classes):
    assert encode_classes((32, 32, 4, 1, 17, 1.3), (256, 256, 4, 1, 55, 1.3), (64, 64, 4, 1, 50, 1.3)) == [6, 6, 6]
    narrow, wide = (240, 128, 6, 1, 500, 4.5), (256, 256, 4, 1, 700, 1.3)
    assert encode_classes((*narrow[:4], 5000, 4.5)) == [10]
    assert encode_classes(narrow, wide) == [6, 6]
    assert encode_classes((128, 128, 4, 1, 1500, 1.3), (64, 64, 4, 1, 500, 1.3)) == [14, 14]
    assert encode_classes((128, 128, 4, 1, 5000, 1.3), (256, 256, 4, 1, 3000, 1.3)) == [14, 6]
