"""The Gram matrix's conditioning in the health report: after the direct amplitude solve and after the Jacobi one, at ranks
around a warp, several reports of one solve; and the report does not repeat the eigenproblem that the direct solve
saves (128 x 128 Jacobi on one CTA takes some 100 ms, the report's own work well under 1 ms)."""
import time

import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def solver(M, spread):
    m = sgs.build_anderson(5, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(m.n_modes, M, np.random.default_rng(M), 1, spread=spread)
    return sgs.Solver(m, g, None)


@pytest.mark.parametrize("M,spread", [(1, 1.0), (2, 1.0), (5, 1.0), (31, 2.0), (33, 2.0), (64, 2.0), (5, 1e-5)])
def test_gram_ratio(M, spread):
    s = solver(M, spread)
    s.energy()
    w = np.linalg.eigvalsh(s.pair_matrices()[0])
    got = [s.health()["gram_eig_ratio"] for _ in range(2)]
    s.close()
    assert got[0] == got[1]
    # normwise backward stable: 16 M u on each eigenvalue, relative to the largest
    assert abs(got[0] - w[0] / w[-1]) <= 32 * M * 2.0 ** -53


def test_report_is_quick():
    s = solver(64, 2.0)
    t = []
    for _ in range(3):
        s.energy()
        t0 = time.perf_counter()
        s.health()
        t.append(time.perf_counter() - t0)
    s.close()
    assert min(t) < 0.03
