"""What the amplitude solve does with (G, h) that have no solution: entries that are not finite, wherever they stand,
end the call with SGS_ENOTCONV (4), also where every pivot of the reduction up to them is finite (the last
diagonal entry of h, the last row's coupling), on the direct route (overlapping states)."""
import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def shard_solve(M, edit):
    """(energy, lambda) from the shard interface's second stage on (G, h) edited by the caller."""
    import torch
    model = sgs.build_anderson(5, 2.0, -1.0, 0.5)
    g = inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(M), 1, spread=1.0)
    whole = sgs.Solver(model, g, None)
    whole.energy()
    G, h = whole.pair_matrices()
    whole.close()
    edit(G, h)
    s = sgs.Solver()
    s.admit(model, g, None, 0.05, shard=(0, 2))
    try:
        gh = torch.empty(2, M, M, 2, dtype=torch.float64, device="cuda")
        dg = torch.empty(M, model.n, model.n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        s.shard_pairs(gh.data_ptr())
        gh.copy_(torch.from_numpy(np.stack([np.stack([x.real, x.imag], -1) for x in (G, h)])))
        torch.cuda.synchronize()
        E = s.shard_eom(gh.data_ptr(), dg.data_ptr())
        return E, s.get_state()[1], G, h
    finally:
        s.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("M", [1, 2, 3, 8, 33])
@pytest.mark.parametrize("where", ["h_last", "h_first", "h_coupling", "G_coupling"])
def test_non_finite_is_reported(M, where, bad):
    def edit(G, h):
        X, i, j = {"h_last": (h, M - 1, M - 1), "h_first": (h, 0, 0), "h_coupling": (h, M - 1, 0),
                   "G_coupling": (G, 0, M - 1)}[where]
        X[i, j] = bad
        X[j, i] = bad
    if M == 1 and "coupling" in where:
        pytest.skip("no coupling")
    with pytest.raises(sgs.SGSError) as e:
        shard_solve(M, edit)
    assert e.value.status == 4
