"""Device memory of an instance: tuning adds room for wider Pfaffian panels and nothing for the Gauss-Jordan panels, which
stay in shared memory, and the admission estimate covers what an instance holds."""
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def test_tuned_instance_holds_no_panel_rows():
    model = sgs.build_anderson(60, 2.0, -1.0, 0.5)
    g, lam = sgs.seeded_states(model.n_modes, 2, 3)
    held = []
    for tune in (False, True):
        s = sgs.Solver(model, g, lam, autotune=tune)
        held.append(s.bytes_in_use())
        s.close()
    wider = 20 * model.n * (32 - 16) * 8             # T, U vectors and packed operands, 16 more column pairs
    assert held[1] - held[0] <= wider + 8192


@pytest.mark.parametrize("n_bath,M,tune", [(15, 4, False), (60, 6, False), (60, 6, True), (127, 5, False)])
def test_estimate_covers_the_instance(n_bath, M, tune):
    model = sgs.build_anderson(n_bath, 2.0, -1.0, 0.5)
    g, lam = sgs.seeded_states(model.n_modes, M, 3)
    s = sgs.Solver(model, g, lam, autotune=tune)
    held = s.bytes_in_use()
    s.close()
    s = sgs.Solver(hbm_budget=held - 1, autotune=tune)
    with pytest.raises(sgs.SGSError) as e:
        s.admit(model, g, lam)
    assert e.value.status == 2
    s.close()
