"""The amplitude solve on the GPU against scipy's generalised eigensolver on the same (G, h): the direct route
(independent states) at ranks around a warp, a block of rows and the largest, and the Jacobi route (nearly
dependent states, where canonical orthogonalisation drops eigenvalues of G)."""
import numpy as np
import pytest
import scipy.linalg

import sgs_inputs as inp
from oracle import sgs_oracle as orc

pkg = pytest.importorskip("paper_2105_01088_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,spread", [(1, 1.0), (2, 1.0), (3, 1.0), (8, 1.5), (9, 1.5), (31, 2.0), (32, 2.0), (33, 2.0),
                                      (64, 2.0), (5, 1e-8)])
def test_amplitudes(M, spread):
    n_bath = 5
    model = pkg.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(M), 1, spread=spread)
    s = pkg.Solver(model, g, None)
    E = s.energy()[0]
    G, h = s.pair_matrices()
    _, lam = s.get_state()
    health = s.health()
    s.close()
    Eo, lo = orc.solve_amplitudes(G, h)
    w = np.linalg.eigvalsh(G)
    if spread > 1e-3:
        assert w[0] > 1e-7 * w[-1]                  # the direct route's premise
        # both solvers are backward stable: (G, h) moves by a few M u, which a solve amplifies by cond(G) and
        # the eigenvector by the gap; u = 2^-53, 16 M for the constants of the two reductions
        e = scipy.linalg.eigh(h, G, eigvals_only=True)
        bar = 16 * M * 2.0 ** -53 * (w[-1] / w[0])
        scale = np.abs(e).max()
        assert abs(E - Eo) <= bar * scale
        assert np.linalg.norm(lam.conj() @ G @ lam - 1.0) <= bar
        gap = e[1] - e[0] if M > 1 else 1.0
        assert np.linalg.norm(lam - lo) <= (2 * bar * scale / gap + bar) * np.linalg.norm(lo)
        assert abs(health["gram_eig_ratio"] - w[0] / w[-1]) <= bar
    else:
        assert w[0] < 1e-12 * w[-1]
        assert abs(E - Eo) <= 1e-9 * abs(Eo)


def test_random_states_keep_exact_zeros():
    """States whose overlaps are below rounding: the solve leaves the other amplitudes exactly zero (frozen states),
    and a step runs."""
    model = pkg.build_anderson(63, 2.0, -1.0, 0.5)
    g, lam = pkg.seeded_states(model.n_modes, 6, 3)
    s = pkg.Solver(model, g, lam, dtau=0.05)
    s.step(3)
    _, lam = s.get_state()
    G, _ = s.pair_matrices()
    s.close()
    assert np.abs(G - np.eye(6)).max() < 1e-9
    assert np.isfinite(lam).all() and np.sort(np.abs(lam))[-1] > 0.99
