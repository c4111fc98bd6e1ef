"""How the SMs of the device are dealt to the tensors of a list: tensors that share launches, a class per kernel, and tensors with
kernels of their own."""
import ctypes as C
import random

import pytest

import paper_1905_10830_b200 as tc

SMS, ITEMS = 148, 32                       # of the device; tensors that a launch holds


@pytest.fixture(scope="module")
def deal():
    from paper_1905_10830_b200 import build
    build.build_library()
    f = tc.load_library().tc_deal_list
    f.restype = C.c_int

    def run(classes, others_us=0.0, others=0):
        flat = [t for c in classes for t in c]
        out = (C.c_int * len(classes))()
        rest = f(len(classes), (C.c_int * len(classes))(*map(len, classes)), (C.c_longlong * len(flat))(*[t for t, _ in flat]),
                 (C.c_double * len(flat))(*[us for _, us in flat]), C.c_double(others_us), others, SMS, out)
        return list(out), rest
    return run


def test_no_sms_are_held_back_for_tiles_that_are_not_there(deal):
    assert deal([[(1, 2.0)]], 10_000.0, 1) == ([1], SMS - 1)
    assert deal([[(1, 2.0)] * 5, [], [(2, 4.0)]], 10_000.0, 2) == ([5, 0, 2], SMS - 7)
    # a small tensor beside large ones takes eight, and those that would not save the large ones' blocks a tile
    sms, rest = deal([[(1000, 2.0)]], 100.0, 1)
    assert rest >= 8 and sms == [SMS - rest] and -(-1000 // sms[0]) == -(-1000 // (SMS - 8))
    # as much work of either kind: about half each
    sms, rest = deal([[(1000, 2.0)]], 2000.0, 1)
    assert abs(rest - 0.5 * SMS) < 0.15 * SMS


def test_a_kernel_of_many_small_tensors_beside_a_large_tensor(deal):
    # 30 tensors of a tile each: a place for each, not one after the other; the large tensor keeps the rest
    for others in (0, 1):
        sms, rest = deal([[(784, 10.7)], [(1, 2.0)] * 30], 50.0 * others, others)
        assert sms[1] == 30 and -(-784 // sms[0]) == -(-784 // (SMS - 30 - 8 * others))


def test_one_kernel_alone_has_the_device(deal):
    assert deal([[], [(3, 2.0), (1, 2.0)]]) == ([0, SMS], 0)


@pytest.mark.parametrize("seed", range(40))
def test_shares_of_any_list(deal, seed):
    rng = random.Random(seed)
    n_classes, others = rng.randint(1, 8), rng.choice([0, 0, 1, 3, 20])
    classes = [sorted(((rng.randint(1, 10 ** rng.randint(0, 4)), rng.uniform(1.2, 50.0)) for _ in range(rng.choice([0, 1, 2, 5, 31, 33, 70, 200]))),
                      key=lambda t: -t[0] * t[1]) for _ in range(n_classes)]
    others_us = others * 10 ** rng.uniform(1, 5)
    sms, rest = deal(classes, others_us, others)
    n = sum(1 for c in classes if c)
    if n == 0:
        assert rest == SMS
        return
    assert sum(sms) + rest == SMS
    assert rest >= 8 if others else rest == 0
    for share, c in zip(sms, classes):
        assert (share > 0) == bool(c)
        if c:
            launches = -(-len(c) // min(ITEMS, share))
            assert launches <= -(-len(c) // min(ITEMS, (SMS - 8 if others else SMS) // n))      # as many as a fair share allows, or fewer
            assert not others or share <= sum(t for t, _ in c)
    if others:      # the quarter, or what balance wants
        quarter = min(SMS // 4 // n, min(max(sum(t for t, _ in c[r::-(-len(c) // ITEMS)]) for r in range(-(-len(c) // ITEMS))) for c in classes if c))
        assert sum(sms) >= min(quarter, 8)


# Measured on a B200, us of one SM a tile over 100 000 pixels and more: (kind, c, bits of code a coefficient, encode, decode).  Widths, rates,
# tables and kernels other than those that the rule was first made with (512 channels at 4 bits).
@pytest.mark.parametrize("kind,c,rate,encode,decode", [
    ("layer", 320, 1.1, 24.0, 17.5), ("layer", 384, 1.1, 29.3, 22.5), ("layer", 512, 1.1, 40.0, 28.0), ("layer", 576, 1.1, 50.5, 36.8),
    ("layer", 576, 3.2, 52.8, 39.4), ("layer", 768, 1.1, 66.1, 49.0), ("layer", 960, 1.1, 97.0, 70.3), ("layer", 1024, 2.6, 105.8, 80.2),
    ("channel", 272, 1.2, 25.6, 21.9), ("channel", 960, 1.0, 120.3, 88.2), ("channel", 64, 1.7, None, 3.9), ("channel", 128, 4.9, None, 8.0),
    ("layer", 128, 1.3, 8.0, None), ("layer", 192, 1.3, 10.8, None), ("fp32", 40, 2.2, 11.4, 14.5), ("fp32", 136, 1.3, 54.2, 49.5),
    ("fp32", 200, 1.2, 104.0, 96.7), ("exact", 64, 1.5, 38.4, 36.1), ("exact", 128, 1.2, 120.2, 106.1), ("exact", 256, 1.1, 415.1, 358.2),
    ("exact", 512, 1.0, 1397.3, 1245.4)])
def test_work_of_tensors_with_kernels_of_their_own(kind, c, rate, encode, decode):
    from paper_1905_10830_b200 import build
    build.build_library()
    f = tc.load_library().tc_list_own_us
    f.restype = C.c_double
    for want, enc in ((encode, True), (decode, False)):
        got = f(C.c_longlong(10), c, c, C.c_double(rate * c), C.c_bool(kind == "channel"), C.c_bool(kind in ("layer", "channel")), C.c_bool(kind == "exact"), C.c_bool(enc))
        assert want is None or abs(got / 10 / want - 1.0) <= 0.33, (got / 10, want)
