"""Gauss-Jordan inverse and complex Pfaffian on batches that take the panels' cluster forms (few matrices: 8, 4 or 2
CTAs each) and the one-CTA form (many), at sizes around the edges of a CTA's rows, of the panels and of the
smallest matrix a cluster takes, against numpy and the oracle's Pfaffian."""
import numpy as np
import pytest

from oracle import sgs_oracle as orc

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def skew(rng, b, n, cplx=False):
    X = rng.standard_normal((b, n, n))
    if cplx:
        X = X + 1j * rng.standard_normal((b, n, n))
    return X - np.swapaxes(X, 1, 2)


@pytest.mark.parametrize("path", [sgs.FP64_EMULATED, sgs.FP64_FMA])
@pytest.mark.parametrize("n,batch", [(2, 1), (14, 3), (16, 3), (18, 41), (64, 40), (66, 2), (130, 79), (164, 81), (258, 161), (66, 256), (66, 257),
                                     (330, 3), (1030, 1)])
def test_inverse(n, batch, path):
    S = skew(np.random.default_rng(n * 1000 + batch), batch, n)
    inv, ld = sgs.batched_inverse(S, path)
    for b in {0, batch // 2, batch - 1}:
        # backward stable elimination: |S X - 1| <= c n u |S| |X| in norms, c = 8 for pivot growth and the
        # emulated products' row-wise bound
        nrm = np.linalg.norm(S[b], 2) * np.linalg.norm(inv[b], 2)
        assert np.abs(S[b] @ inv[b] - np.eye(n)).max() <= 8 * n * U * nrm
        _, ref = np.linalg.slogdet(S[b])
        assert abs(ld[b] - ref) <= 8 * n * U * np.linalg.norm(S[b], 2) * (1.0 / np.linalg.svd(S[b])[1]).sum() + 4 * U * abs(ref)


@pytest.mark.parametrize("path", [sgs.FP64_EMULATED, sgs.FP64_FMA])
@pytest.mark.parametrize("n,batch", [(2, 1), (8, 2), (16, 3), (32, 1), (34, 63), (66, 125), (66, 2), (164, 10), (164, 126),
                                     (260, 5), (420, 2)])
def test_pfaffian(n, batch, path):
    Y = skew(np.random.default_rng(n * 1000 + batch), batch, n, True)
    ph, la = sgs.batched_pfaffian(Y, path)
    for b in {0, batch // 2, batch - 1}:
        rp, rl = orc.pfaffian_log(Y[b])
        # d log Pf = tr(Y^-1 dY) / 2 for the backward error |dY| <= 8 n u |Y|
        s = np.linalg.svd(Y[b])[1]
        bar = 8 * n * U * s[0] * (1.0 / s).sum() + 4 * U * abs(rl)
        assert abs(la[b] - rl) <= bar
        assert abs(ph[b] - rp) <= bar


def test_singular_and_zero():
    S = skew(np.random.default_rng(5), 2, 40)
    S[1, :, 7] = S[1, 7, :] = 0.0
    with pytest.raises(sgs.SGSError):
        sgs.batched_inverse(S)
    Y = skew(np.random.default_rng(6), 2, 40, True)
    Y[1, :, 7] = Y[1, 7, :] = 0.0
    ph, la = sgs.batched_pfaffian(Y)
    rp, rl = orc.pfaffian_log(Y[0])
    assert abs(la[0] - rl) <= 1e-10 and abs(ph[0] - rp) <= 1e-10
    assert la[1] == -np.inf
