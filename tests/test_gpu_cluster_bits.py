"""The Gauss-Jordan panel by clusters of 8, 4 or 2 CTAs gives the one-CTA form's bits (inverse and log|det|), so the form
that a batch takes does not show in its results: one matrix in batches on every side of the lines (40, 80, 320
matrices), rows that the cluster does not divide, exact ties between pivot candidates, zeros in the columns."""
import numpy as np
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "skew":
        X = rng.standard_normal((n, n))
        return X - X.T + (n % 2) * np.eye(n)             # (an odd skew matrix is singular)
    if kind == "ties":                      # entries +-1: every pivot search of a column starts with ties
        return np.where(rng.random((n, n)) < 0.5, -1.0, 1.0)
    X = np.where(rng.random((n, n)) < 0.9, 0.0, rng.standard_normal((n, n)))
    return X + np.roll(np.eye(n), 3, axis=0)


@pytest.mark.parametrize("kind", ["skew", "ties", "sparse"])
@pytest.mark.parametrize("n", [16, 31, 33, 66, 130, 164])
@pytest.mark.parametrize("path", [sgs.FP64_EMULATED, sgs.FP64_FMA])
def test_same_bits(kind, n, path):
    A = matrix(kind, n)
    inv, ld = sgs.batched_inverse(A[None], path)
    assert np.abs(A @ inv[0] - np.eye(n)).max() < 1e-9            # condition numbers up to 1e4
    for batch in (40, 41, 80, 81, 320, 321):
        X, l = sgs.batched_inverse(np.broadcast_to(A, (batch, n, n)), path)
        for b in {0, batch // 2, batch - 1}:
            assert np.array_equal(X[b], inv[0]) and l[b] == ld[0]
