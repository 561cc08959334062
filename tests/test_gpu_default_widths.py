"""Default widths of the Gauss-Jordan panels: on both sides of each line of the rule, the inverse and the energy agree with
a solver at width 8 (another blocking of the same elimination: rounding only), tuning() reports the width in use,
and that width can be set again."""
import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M,prec,width", [
    (14, 3, "fp64", 16), (15, 3, "fp64", 32), (40, 6, "fp64", 32), (127, 4, "fp64", 32), (128, 3, "fp64", 16),
    (40, 6, "tf32", 16), (449, 2, "fp64", 16), (449, 2, "tf32", 12)])
def test_default_width(n_bath, M, prec, width):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(n_bath), 1, spread=1.0)
    kind = sgs.SGS_FP64 if prec == "fp64" else sgs.SGS_MIXED_TF32
    a = sgs.Solver(model, g, None, precision=kind, cmode=sgs.SGS_C_PHASE)
    assert a.tuning(0)[0] == width and a.tuning(0)[2] == -1
    E = a.energy()
    a.set_panel_widths(*a.tuning(0)[:2])
    assert np.array_equal(a.energy(), E)
    a.set_panel_widths(8, 8)
    # the amplitudes and S^{-1} of clustered states are well conditioned: the step tests' bar
    assert np.abs(a.energy() - E).max() <= 1e-10 * np.abs(E).max()
    a.close()
