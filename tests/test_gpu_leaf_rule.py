"""Default Gauss-Jordan widths by the number of pairs: both sides of each line of the rule (the widths do not depend on
which form the panels of a batch take), with the energy of another blocking."""
import numpy as np
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M,width", [(15, 19, 32), (15, 23, 32), (15, 24, 16), (63, 23, 32), (64, 13, 32),
                                            (64, 14, 16), (64, 23, 16)])
def test_width_by_pairs(n_bath, M, width):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g, lam = sgs.seeded_states(model.n_modes, M, 5)
    s = sgs.Solver(model, g, lam)
    assert s.tuning(0) == (width, 16, -1)
    E = s.energy()
    s.set_panel_widths(8, 16)
    assert np.abs(s.energy() - E).max() <= 1e-10 * np.abs(E).max()
    s.close()
