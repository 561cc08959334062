"""The phase Pfaffians on both sides of the line between one CTA per matrix and the blocked panels (few matrices
of many rows), the smallest system and a matrix that fills shared memory, against the oracle's Gram matrix."""
import numpy as np
import pytest

import sgs_inputs as inp
from oracle import sgs_oracle as orc

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M", [(1, 3), (2, 4), (10, 3), (11, 5), (15, 4), (26, 3), (27, 3), (27, 4), (31, 7), (37, 11),
                                      (38, 11)])
def test_gram(n_bath, M):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(n_bath), 1, spread=1.0)
    s = sgs.Solver(model, g, None, cmode=sgs.SGS_C_PHASE)
    E = s.energy()[0]
    G = s.pair_matrices()[0]
    s.close()
    e, lam, ref, h = orc.energy(orc.anderson_model(n_bath, 2.0, -1.0, 0.5), list(g))
    assert np.abs(G - ref).max() <= 1e-10       # |G_ab| <= 1; the step tests' bar
    assert abs(np.ravel(E)[0] - e) <= 1e-10 * abs(e)
