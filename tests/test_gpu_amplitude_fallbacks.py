"""Where the amplitude solve leaves the direct route for Jacobi, whose exact zeros freeze a state (c_mu = 1 / (lambda_mu
conj(lt_mu)) is set to 0 there): states whose overlaps are below rounding, and overlapping states beside one that
is coupled to none, which the direct route's normwise errors would give an amplitude of 1e-45 and c_mu of 1e90."""
import numpy as np
import pytest

from test_gpu_amplitude_failures import shard_solve

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def test_frozen_states_stay():
    model = sgs.build_anderson(63, 2.0, -1.0, 0.5)
    g, lam = sgs.seeded_states(model.n_modes, 6, 3)
    s = sgs.Solver(model, g, lam, dtau=0.05)
    s.step(3)
    after, lam = s.get_state()
    G, _ = s.pair_matrices()
    s.close()
    assert 0.0 < np.abs(G - np.eye(6)).max() < 1e-9
    assert np.count_nonzero(lam) == 1 and np.abs(lam).max() > 0.99
    # R = 1 exactly; R Gamma R^T and one purification a step, 4 n u each
    for mu in np.flatnonzero(lam == 0.0):
        assert np.abs(after[mu] - g[mu]).max() <= 3 * 8 * model.n * 2.0 ** -53


@pytest.mark.parametrize("M,alone", [(3, 0), (3, 1), (3, 2), (9, 8), (34, 17)])
def test_a_state_coupled_to_none(M, alone):
    def edit(G, h):
        rng = np.random.default_rng(M + alone)
        X = rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))
        G[:] = np.eye(M) + 0.05 / M * (X + X.conj().T)
        X = rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))
        h[:] = X + X.conj().T
        for A, d in ((G, 1.0), (h, 50.0)):          # its energy well above the lowest
            A[alone, :] = A[:, alone] = 0.0
            A[alone, alone] = d
    E, lam, G, h = shard_solve(M, edit)
    import scipy.linalg
    e, v = scipy.linalg.eigh(h, G)
    assert lam[alone] == 0.0
    # both backward stable; cond(G) below 2, |h| below 50 beside the gap
    bar = 64 * M * 2.0 ** -53 * 50.0
    assert abs(E - e[0]) <= bar
    j = np.argmax(np.abs(lam))
    ref = v[:, 0] * (abs(v[j, 0]) / v[j, 0])
    assert np.linalg.norm(lam - ref) <= bar / (e[1] - e[0]) * 2.0
