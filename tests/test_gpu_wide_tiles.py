"""Emulated products of many tiles and long sums (128 x 64 tiles, one CTA per SM) against the same products one at a
time (128 x 32 tiles, two CTAs per SM): the same bits, in every form of the epilogue, with ragged rows, columns
and K, two K chunks, odd leading dimensions, and scales at the ends of the range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
PLAIN, SKEW, GJ = 0, 1, 2


@pytest.fixture(scope="module")
def pkg():
    import paper_2105_01088_gb300 as p
    return p


@pytest.mark.parametrize("batch,m,n,k,kw", [
    (76, 129, 65, 241, dict()),
    (76, 129, 65, 256, dict()),
    (76, 200, 131, 257, dict(beta=1.0)),
    (120, 128, 66, 300, dict(alpha=0.7, beta=-0.3, diag=2.0)),
    (120, 65, 128, 511, dict(trans_a=True, trans_b=True)),
    (80, 140, 180, 700, dict(alpha=-2.0, beta=1.0)),
    (40, 257, 257, 257, dict(mode=SKEW, beta=1.0)),
    (40, 300, 300, 300, dict(mode=SKEW, alpha=0.3, antisym_b=True)),
    (40, 300, 300, 300, dict(antisym_b=True, alpha=-1.0)),
    (40, 320, 320, 260, dict(mode=GJ, gj=(30, 260), beta=1.0)),
    (76, 129, 70, 512, dict(scale=1e158)),
    (76, 129, 70, 512, dict(scale=1e-158)),
])
def test_wide_equals_narrow(pkg, batch, m, n, k, kw):
    kw = dict(kw)
    scale, asym = kw.pop("scale", 1.0), kw.pop("antisym_b", False)
    rng = np.random.default_rng(m + n + k)
    A = scale * rng.standard_normal((batch, m, k)) * 10.0 ** rng.uniform(-3, 3, (batch, m, 1))
    B = scale * rng.standard_normal((batch, k, n)) * 10.0 ** rng.uniform(-3, 3, (batch, 1, n))
    A[1] = B[1] = 1.0                                       # sums of one sign
    A[2, :, 0] *= 1e12                                      # rows of uneven magnitudes
    A[3, m // 2] = 0.0
    if asym:
        B = B - np.swapaxes(B, 1, 2)
        kw["b_antisym"] = True
    if kw.pop("trans_a", False):
        A, kw["trans_a"] = np.swapaxes(A, 1, 2).copy(), True
    if kw.pop("trans_b", False):
        B, kw["trans_b"] = np.swapaxes(B, 1, 2).copy(), True
    Cin = rng.standard_normal((batch, m, n)) if "beta" in kw else None
    got = pkg.batched_gemm(A, B, Cin=Cin, **kw)
    for b in [0, 1, 2, 3, batch // 2, batch - 1]:
        one = pkg.batched_gemm(A[b:b + 1], B[b:b + 1], Cin=None if Cin is None else Cin[b:b + 1], **kw)
        assert np.array_equal(got[b], one[0], equal_nan=True)
