"""Steps whose products run on the FP64 pipe because they are small (single tiles, ragged tiles and K slabs, both
sides of the line for parts of a step), against the oracle: every form a step uses (general, antisymmetric,
transposed, Gauss-Jordan and Pfaffian updates, the exponential's addends), both integrators, both
arithmetics.  Clustered states keep the amplitudes' conditioning out of the bar (1e-10 of the largest
entry, as the step tests)."""
import numpy as np
import pytest

import sgs_inputs as inp
from oracle import sgs_oracle as orc

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M", [(1, 1), (1, 2), (2, 3), (4, 5), (6, 4), (8, 4), (15, 4), (16, 5), (20, 3), (32, 4)])
@pytest.mark.parametrize("integrator", [sgs.SGS_INTEGRATOR_EXP, sgs.SGS_INTEGRATOR_EULER])
@pytest.mark.parametrize("path", [sgs.FP64_EMULATED, sgs.FP64_FMA])
def test_small_step(n_bath, M, integrator, path):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    om = orc.anderson_model(n_bath, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(10 * n_bath + M), 1, spread=1.0)
    s = sgs.Solver(model, g, None, dtau=0.05, cmode=sgs.SGS_C_PHASE, integrator=integrator, fp64_path=path)
    E = s.step(2)[0]
    got, _ = s.get_state()
    s.close()
    ref, Es = list(g), []
    for _ in range(2):
        e, lam, G, h = orc.energy(om, ref)
        d = orc.eom(om, ref, G, h, e, lam, orc.C_PHASE)
        step = orc.euler_step if integrator == sgs.SGS_INTEGRATOR_EULER else (
            lambda x, y, ds: orc.purify(orc.orthogonal_step(x, y, ds)))
        ref = [step(x, y, 0.05) for x, y in zip(ref, d)]
        Es.append(e)
    assert np.abs(E - Es).max() <= 1e-10 * np.abs(Es).max()
    assert np.abs(got - np.stack(ref)).max() <= 1e-10
