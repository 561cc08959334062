"""log|det| of matrices whose pivots sit at the ends of the FP64 range: subnormal ones (whose reciprocals are still
finite) and ones near overflow, several in a panel and over two panels, in the one-CTA and the cluster panel."""
import numpy as np
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 300])
@pytest.mark.parametrize("n", [4, 33, 70])
@pytest.mark.parametrize("d", [2.0 ** -1023, 3.0 * 2.0 ** -1024, 2.0 ** 1021, 2.0 ** -1000, 1.5])
def test_log_determinant(n, batch, d):
    v = np.ones(n)
    v[1::2] = d
    v[2::4] = -1.25
    S = np.broadcast_to(np.diag(v), (batch, n, n)).copy()
    inv, ld = sgs.batched_inverse(S)
    want = np.log(np.abs(v)).sum()
    # one rounding each of the product's mantissa, its logarithm, the exponent's multiple and the sum
    assert np.abs(ld - want).max() <= 4 * n * 2.0 ** -53 * max(abs(want), 1.0)
    assert np.array_equal(inv[-1], np.diag(1.0 / v))
