"""Every kernel that needs more dynamic shared memory than the default has its limit raised, and the largest request that
the library makes of it fits (bytes: the cluster panels' own bounds, a packed Pfaffian of 152 rows, the amplitude
solve and the Gram matrix at rank 64, the 64-column product tile)."""
import pytest

sgs = pytest.importorskip("paper_2105_01088_gb300")
pytestmark = pytest.mark.gpu


def test_limits():
    lim = sgs.smem_limits()
    assert len(lim) == 16
    packed = 152 * 151 // 2 * 18 + 4 * 152 * 8 + 16
    need = {2: packed, 9: 200 * 1024, 10: 220 * 1024, 11: packed, 12: 3 * 64 * 65 * 16, 13: 64 * 65 * 16,
            14: 2 * 8 * 64 * 128 + 3 * 2 * 128 * 128 + 1024}
    for i, (in_force, expected) in enumerate(lim):
        assert in_force == expected >= need.get(i, 0), i
