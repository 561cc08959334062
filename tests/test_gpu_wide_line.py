"""Emulated products on both sides of the wide tiles' line (K = 224): a batch of many tiles against its entries one at a
time, which have too few for wide tiles: the same bits, also with a last slab of 15 and 16 steps and ragged K."""
import numpy as np
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [223, 224, 225, 239, 240])
@pytest.mark.parametrize("form", ["general", "skew", "gj"])
def test_same_bits_across_the_line(k, form):
    rng = np.random.default_rng(k)
    b, m = 60, 250
    A = rng.standard_normal((b, m, k)) * 10.0 ** rng.uniform(-3, 3, (b, m, 1))
    B = rng.standard_normal((b, k, m))
    Cin = rng.standard_normal((b, m, m))
    kw = {"general": dict(alpha=0.5, beta=1.5), "skew": dict(mode=1, beta=1.0),
          "gj": dict(mode=2, gj=(4, k), beta=1.0)}[form]
    got = sgs.batched_gemm(A, B, Cin=Cin, **kw)
    for i in (0, 1, b // 2, b - 1):
        assert np.array_equal(got[i], sgs.batched_gemm(A[i:i + 1], B[i:i + 1], Cin=Cin[i:i + 1], **kw)[0])
