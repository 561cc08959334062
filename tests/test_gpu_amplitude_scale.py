"""The amplitude solve of a Hamiltonian given in other units: H times a power of two has that multiple of the energy and
the same amplitudes, bit for bit (every operation of the solve scales exactly), up to magnitudes whose fourth
power over- or underflows.  Both sides of the line at 2^150 from which the tridiagonal is scaled."""
import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 6, 33])
@pytest.mark.parametrize("power", [-300, -160, -140, 1, 140, 160, 300])
def test_energy_scales_exactly(M, power):
    m = sgs.build_anderson(5, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(m.n_modes, M, np.random.default_rng(M), 1, spread=1.0)
    out = []
    for f in (1.0, 2.0 ** power):
        s = sgs.Solver(sgs.MajoranaModel(m.A * f, m.quartic_idx, m.quartic_val * f, m.e_const * f), g, None)
        out.append((s.energy() / f, s.get_state()[1]))
        s.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])
