"""The 16-bit arithmetic of the streaming passes (ssd_internal.cuh's out2, not_never2 and expiry minimum, and
ssd_stream.cu's merge of several routers by two running maxima), restated here and compared with
the distances for every stored value, at clocks on both sides of every wrap and windows from 1 to 65534."""
import numpy as np
import pytest

NEVER = 65535
ALL = np.arange(65536, dtype=np.int64)
CLOCKS = [0, 1, 5, 16, 58, 59, 60, 61, 1000, 32766, 32767, 32768, 65473, 65533, 65534]
WINDOWS = [1, 2, 17, 60, 300, 32768, 65533, 65534]


def u16(x):
    return x & 0xFFFF


def add_max(a, b, c):   # the fused add-maximum: the sum wraps at 16 bits
    return np.maximum(u16(a + b), c)


def add_min(a, b, c):
    return np.minimum(u16(a + b), c)


def distance(x, tm):
    return np.where(x == NEVER, 65535, np.where(x <= tm, tm - x, tm - x + 65535))


def clock(tm, k):
    """(wrap, -lo, klim - 1, 1 - klim, -xe) of make_clock and fused_operands."""
    wrap = tm + 1 < k
    lo = tm + 65536 - k if wrap else tm + 1 - k
    klim = k + 1 if wrap else k
    xe = 0 if tm + 1 >= 65535 else tm + 1
    return wrap, u16(-lo), klim - 1, u16(1 - klim), u16(-xe)


def out2(x, neg_lo, top, neg_top):
    return add_min(add_max(x, neg_lo, top), neg_top, 1)


@pytest.mark.parametrize("tm", CLOCKS)
@pytest.mark.parametrize("k", WINDOWS)
def test_window_and_expiry_of_one_router(tm, k):
    wrap, neg_lo, top, neg_top, neg_xe = clock(tm, k)
    inside = distance(ALL, tm) < k
    out = out2(ALL, neg_lo, top, neg_top)
    not_never = add_min(ALL, 1, 1)
    assert np.array_equal(not_never, (ALL != NEVER).astype(np.int64))
    # a lane counts both halves together: outside the 16-bit range, and with a window that wraps not kNever
    assert np.array_equal(not_never - out if wrap else 1 - out, inside.astype(np.int64))
    # the minimum of x - xe is 0 exactly for the recorder whose distance reaches 65535
    assert np.array_equal(add_min(ALL, neg_xe, NEVER) == 0, (ALL != NEVER) & (distance(ALL, tm) == 65534))


@pytest.mark.parametrize("tm", CLOCKS)
def test_merge_by_running_maxima(tm):
    other = np.unique(np.clip(np.concatenate([np.arange(-3, 4) + v for v in (0, tm, 300, 30000, 65534)]
                                             + [np.arange(0, 65536, 1733)]), 0, NEVER))
    to_p, st_p, never, from_p = u16(-(tm + 1)), u16(-(tm + 2)), 65534 - tm, tm + 1
    x = ALL[:, None]
    y = other[None, :]
    hi = add_max(y, to_p, add_max(x, to_p, 0))
    newest = add_max(y, 1, add_max(x, 1, 0))
    merged = np.where(hi == never, u16(newest + st_p), hi)
    want = np.minimum(distance(x, tm), distance(y, tm))
    stored = u16(merged + from_p)
    assert np.array_equal(distance(stored, tm), want)
    for k in WINDOWS:
        wrap, neg_lo, top, neg_top, _ = clock(tm, k)
        # the window test on p; without a wrap the first maximum alone decides
        p = merged if wrap else hi
        out = out2(p, u16(tm + 1 + neg_lo), top, neg_top)
        if wrap:
            out = out | (p == never)
        assert np.array_equal(out == 0, want < k), k


def test_bits_of_a_vector():
    """One bit per recorder from the four words' 0/1 halves, each in a place of its own."""
    seen = {}
    for i in range(8):
        o = [0x00010001] * 4
        o[i // 2] &= ~(1 << (16 * (i % 2)))
        inside = (o[0] + 2 * o[1] + 4 * o[2] + 8 * o[3]) ^ 0x000F000F
        seen[i] = (inside | (inside >> 12)) & 0xFF
    assert sorted(seen.values()) == [1 << b for b in range(8)]


@pytest.mark.parametrize("k", WINDOWS)
def test_window_of_distances(k):
    """Recorders holding distances (the allocation-free regain's input): the range [0, k)."""
    assert np.array_equal(out2(ALL, 0, k - 1, u16(1 - k)) == 0, ALL < k)
