"""The floating-point arithmetic of the point test (csrc/thin_simd.cuh), restated in numpy on the CPU.

u8 pixels are halves 1024 + v, u16 pixels floats 2^23 + v.  Saturated differences are comparisons, sums of
their multiples index the decision table, and the low bits of a sum are its integer.  Checked for every
pair of u8 values and every lambda, and for u16 values and lambdas at their ends: the comparisons are exact,
no sum rounds or leaves its lane, the index is the ternary number of the ring's states (twice its all-deep
half at lambda = 0), the marks' bits are right, and alpha^- comes out of the modular add-max."""
import numpy as np
import pytest

V8 = np.arange(256)


def half(x):
    return np.asarray(x, np.float64).astype(np.float16)


def bits(x):
    return np.asarray(x).view(np.uint16 if x.dtype == np.float16 else np.uint32).astype(np.int64)


def sat(a, b):
    return np.clip(a - b, 0, 1).astype(a.dtype)  # (numpy rounds the difference to the type, as the kernel's add does)


def test_half_bias_is_exact_for_every_pixel():
    assert (bits(half(1024 + V8)) == 0x6400 + V8).all()


@pytest.mark.parametrize("lams", [range(0, 128), range(128, 256)])
def test_u8_comparisons(lams):
    c, n = half(1024 + V8)[:, None], half(1024 + V8)[None, :]
    assert (sat(c, n) == (V8[None, :] < V8[:, None])).all()
    for lam in lams:
        lamh = (half(1024 + lam) - half(1024)).astype(np.float16)
        low = (c - lamh).astype(np.float16)
        assert (low.astype(np.float64) == 1024 + V8[:, None] - lam).all()
        assert (sat(low, n) == (V8[None, :] < V8[:, None] - lam)).all()
        top = (c + lamh).astype(np.float16)
        assert (top.astype(np.float64) == 1024 + V8[:, None] + lam).all()
        assert (sat(n, top) == (V8[None, :] > V8[:, None] + lam)).all()


def test_u8_sums_and_index_stay_in_their_lane():
    t = np.arange(3 ** 8)
    d = [(t // 3 ** k) % 3 for k in range(8)]  # state of each neighbour: 0 not lower, 1 shallow, 2 deep
    for deep_only in (False, True):
        lo, hi = half(np.full(t.size, 1024)), half(np.full(t.size, 1024))
        for step in (1,) if deep_only else (1, 2):  # lambda = 0 makes one pass
            for k in range(4):
                w = half(3 ** k)
                lo = half(((d[k] >= step) * w).astype(np.float64) + lo.astype(np.float64))
                hi = half(((d[k + 4] >= step) * w).astype(np.float64) + hi.astype(np.float64))
        i = (bits(hi) & 0xff) * 81 + bits(lo)
        base = 0x6400
        want = t
        if deep_only:
            i, base = i << 1, 2 * 0x6400
            want = 2 * sum((d[k] >= 1) * 3 ** k for k in range(8))
        assert i.max() < 1 << 16  # two lanes to a word: nothing is carried over
        assert (i - base == want).all()


def test_u8_mark_bits():
    m = np.arange(256)
    s = half(np.full(256, 1024))
    for k in range(8):
        s = half(((m >> k) & 1) * float(1 << k) + s.astype(np.float64))
    assert (bits(s) & 0xff == m).all()
    for k in range(8):  # taking marks away again never goes below the bias
        s = half(s.astype(np.float64) - ((m >> k) & 1) * float(1 << k))
    assert (bits(s) == 0x6400).all()


def test_u8_alpha_by_add_max():
    rng = np.random.default_rng(0)
    c = rng.integers(0, 256, (20000, 2))
    nb = rng.integers(0, 256, (20000, 2, 8))
    nb[:10000] = np.clip(c[:10000, :, None] + rng.integers(-3, 4, (10000, 2, 8)), 0, 255)  # close values, equal ones
    word = (0x6400 + c[:, 0]) | ((0x6400 + c[:, 1]) << 16)
    neg = ((~word & 0xffffffff) + 0x00010001) & 0xffffffff
    for lane in range(2):
        m = (neg >> (16 * lane)) & 0xffff
        assert (m == (-(0x6400 + c[:, lane])) & 0xffff).all()
        best = np.zeros(len(c), np.int64)
        for k in range(8):
            best = np.maximum((0x6400 + nb[:, lane, k] + m) & 0xffff, best)
        low = np.where(nb[:, lane] < c[:, lane, None], nb[:, lane], -1).max(1)
        got = ((0x6400 + c[:, lane] + best) & 0xffff) - 0x6400
        assert (got == low)[low >= 0].all()


ENDS = np.unique(np.concatenate([[0, 1, 2, 255, 256, 4095, 32767, 32768, 65533, 65534, 65535],
                                 np.random.default_rng(1).integers(0, 65536, 300)]))


@pytest.mark.parametrize("lam", [0, 1, 30, 4095, 65534, 65535])
def test_u16_comparisons(lam):
    f = np.float32
    c, n = f(2 ** 23) + ENDS.astype(f)[:, None], f(2 ** 23) + ENDS.astype(f)[None, :]
    assert (bits(c) == 0x4b000000 + ENDS[:, None]).all()
    assert (sat(c, n) == (ENDS[None, :] < ENDS[:, None])).all()
    low, top = c - f(lam), c + f(lam)
    assert (low.astype(np.float64) == 2.0 ** 23 + ENDS[:, None] - lam).all()
    assert (top.astype(np.float64) == 2.0 ** 23 + ENDS[:, None] + lam).all()
    assert (sat(low, n) == (ENDS[None, :] < ENDS[:, None] - lam)).all()
    assert (sat(n, top) == (ENDS[None, :] > ENDS[:, None] + lam)).all()


def test_u16_sums_and_alpha():
    f = np.float32
    assert bits(f(2 ** 23) + np.arange(3 ** 8).astype(f)).tolist() == list(range(0x4b000000, 0x4b000000 + 3 ** 8))
    c = ENDS[:, None]
    n = ENDS[None, :]
    diff = (n - c) & 0xffffffff  # the bias cancels
    assert ((diff > 0xffff) == (n < c)).all()  # so the largest one belongs to the largest neighbour below
    assert (((c + diff) & 0xffffffff) == n)[n < c].all()
