"""The integer form of the conversion of an FP64 number to fp32 and to the 3xTF32 split (hi with 13 bits cut off, lo the
rounded rest), restated in numpy, against IEEE conversions and subtractions: the same bits at every exponent the
form takes, with carries, ties and empty rests."""
import numpy as np
import pytest


def split_integer(x):
    u = x.view(np.uint64)
    e = ((u >> np.uint64(52)) & np.uint64(0x7FF)).astype(np.int64)
    assert e.min() >= 949 and e.max() <= 1149
    sg = (u >> np.uint64(63)).astype(np.uint32)
    m = (u & np.uint64(2 ** 52 - 1)) | np.uint64(2 ** 52)
    q = ((m + np.uint64(0xFFFFFFF) + ((m >> np.uint64(29)) & np.uint64(1))) >> np.uint64(29)).astype(np.uint32)
    fb = (sg << np.uint32(31)) | (((e - 897).astype(np.uint32) << np.uint32(23)) + q)
    d = m.astype(np.int64) - ((q & np.uint32(0xFFFFE000)).astype(np.int64) << 29)
    d = np.where(sg == 1, -d, d)
    dh, dl = (d >> 18), d & 0x3FFFF
    assert np.abs(dh).max() <= 2 ** 24
    # one rounding, as the fma (the sum is exact in FP64)
    s = (dh.astype(np.float64) * 2.0 ** 18 + dl).astype(np.float32)
    lo = s * ((e - 948).astype(np.uint32) << np.uint32(23)).view(np.float32)
    return fb, fb & np.uint32(0xFFFFE000), lo.view(np.uint32)


@pytest.mark.parametrize("kind", ["random", "low bits zero", "low bits one", "tie", "carry", "short"])
def test_split_has_the_bits_of_fp64_arithmetic(kind):
    rng = np.random.default_rng(len(kind))
    N = 100000
    m = rng.integers(0, 1 << 52, N, dtype=np.uint64)
    if kind == "low bits zero":
        m &= ~np.uint64(2 ** 42 - 1)
    elif kind == "low bits one":
        m |= np.uint64(2 ** 42 - 1)
    elif kind == "tie":
        m = (m & ~np.uint64(2 ** 29 - 1)) | np.uint64(2 ** 28)
    elif kind == "carry":
        m |= np.uint64(2 ** 52 - 2 ** 28)
    elif kind == "short":
        m &= np.uint64(2 ** 20 - 1) << np.uint64(32)
    e = rng.integers(949, 1150, N).astype(np.uint64)
    x = (m | (e << np.uint64(52)) | (rng.integers(0, 2, N).astype(np.uint64) << np.uint64(63))).view(np.float64)
    f = x.astype(np.float32)
    h = (f.view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32)
    lo = (x - h.astype(np.float64)).astype(np.float32)
    got = split_integer(x)
    assert np.array_equal(got[0], f.view(np.uint32))
    assert np.array_equal(got[1], h.view(np.uint32))
    assert np.array_equal(got[2], lo.view(np.uint32))
