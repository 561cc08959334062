"""The last stage of a pair-sharded step takes dGamma/ds as the caller gives it: with a symmetric part (a sum over ranks
that rounds entry (k, l) otherwise than (l, k), here exaggerated) both FP64 paths apply the same update, on
products of either side of the small-product line."""
import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bath,M", [(5, 2), (40, 2), (31, 3)])      # n = 24: 3e4 FMAs; 164 and 128: 9e6 and 6e6
def test_update_of_a_callers_derivative(n_bath, M):
    import torch
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    n = model.n
    rng = np.random.default_rng(n)
    g = inp.clustered_pure_gammas(model.n_modes, M, rng, 1, spread=1.0)
    d = rng.standard_normal((M, n, n)) / np.sqrt(n)
    d = d - np.swapaxes(d, 1, 2)
    d += 1e-3 * rng.standard_normal((M, n, n)) / np.sqrt(n)
    out = []
    for path in (sgs.FP64_EMULATED, sgs.FP64_FMA):
        s = sgs.Solver(fp64_path=path)
        s.admit(model, g, None, 0.05, shard=(0, 2))
        dg = torch.from_numpy(d).cuda()
        torch.cuda.synchronize()
        s.shard_update(dg.data_ptr())
        out.append(s.get_state()[0])
        s.close()
    # rounding of a dozen products of matrices with norms of order one: 12 n u each way
    assert np.abs(out[0] - out[1]).max() <= 24 * n * 2.0 ** -53
