"""Renyi-2 entropies around the sizes where the Pfaffian kernel changes: the smallest subsystem, one and several
warps of live rows, the last shared-memory size (impurity + 18 sites) and the blocked Pfaffian beyond it, against
the oracle; the whole system has S_2 = 0."""
import numpy as np
import pytest

import sgs_inputs as inp
from oracle import sgs_oracle as orc

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M,ls", [(3, 3, [0, 1, 3]), (10, 2, [4, 6, 9]), (20, 2, [13, 17, 18, 19, 20])])
def test_renyi2_sizes(n_bath, M, ls):
    model = sgs.build_anderson(n_bath, 3.0, -1.5, 0.6)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(n_bath), 1, spread=1.0)
    s = sgs.Solver(model, g, None)
    got = s.correlator(sgs.SGS_CORR_RENYI2, ls)
    s.close()
    E, lam, G, h = orc.energy(orc.anderson_model(n_bath, 3.0, -1.5, 0.6), list(g))
    ref = np.array([orc.renyi2(list(g), lam, G, 2 * (1 + l)) for l in ls])
    assert np.abs(got - ref).max() <= 1e-10 * max(1.0, np.abs(ref).max())
    if ls[-1] == n_bath:
        assert abs(got[-1]) < 1e-10
