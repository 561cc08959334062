"""What the autotuner's cache distinguishes: a shape is timed once, also where the width chosen is one that only the
cluster form of the panels can run (n above about 1700); an instance of the same n, rank and precision whose
launches hold fewer pairs (chunks, a rank's share) is timed on its own."""
import numpy as np
import pytest

import sgs_inputs as inp

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def states(model, M):
    if model.n < 500:
        return inp.clustered_pure_gammas(model.n_modes, M, np.random.default_rng(M), 1, spread=1.0)
    return sgs.seeded_states(model.n_modes, M, 3)[0]


@pytest.mark.parametrize("n_bath,M", [(424, 2), (13, 5)])        # n = 1700 and 56
def test_timed_once(n_bath, M):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = states(model, M)
    got = []
    for _ in range(2):
        s = sgs.Solver(model, g, None, autotune=True)
        got.append(s.tuning(0))
        s.close()
    assert got[0][2] == 0 and got[1] == got[0][:2] + (1,)


def test_fewer_pairs_are_timed_on_their_own():
    model = sgs.build_anderson(16, 2.0, -1.0, 0.5)
    g = states(model, 6)
    s = sgs.Solver(autotune=True)
    assert s.tuning(s.admit(model, g))[2] == 0
    assert s.tuning(s.admit(model, g))[2] == 1
    assert s.tuning(s.admit(model, g, pair_chunk=7))[2] == 0
    assert s.tuning(s.admit(model, g, shard=(0, 2)))[2] == 0
    assert s.tuning(s.admit(model, g, pair_chunk=7))[2] == 1
    s.close()


@pytest.mark.parametrize("n_bath,chunk", [(16, 5), (30, 3)])     # n = 68 and 124: the chunk of state 0's pairs first
def test_chunks_without_phase_pfaffians(n_bath, chunk):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = states(model, 6)
    s = sgs.Solver(model, g, None, autotune=True, pair_chunk=chunk)
    E = s.energy()
    s.close()
    s = sgs.Solver(model, g, None)
    # other panel widths: rounding of well-conditioned (G, h)
    assert np.abs(s.energy() - E).max() <= 1e-10 * np.abs(E).max()
    s.close()


@pytest.mark.parametrize("n_bath,M", [(7, 3), (9, 4), (15, 4), (21, 5), (26, 6)])       # n = 32 .. 108
def test_no_width_is_chosen_where_there_is_no_panel(n_bath, M):
    """Phase Pfaffians of a CTA each: the tuner leaves the width as a solver without tuning has it (timing them told
    five widths of one kernel apart by noise)."""
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g = states(model, M)
    s = sgs.Solver(model, g, None)
    want = s.tuning(0)[1]
    s.close()
    for chunk in (0, 2):
        s = sgs.Solver(model, g, None, autotune=True, pair_chunk=chunk)
        assert s.tuning(0)[1] == want
        s.close()
