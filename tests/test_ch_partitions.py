"""One rule for the line solver's partitions: what a plan is created with (cs_ch_partition) is what the host
replay (cs_ch_solver_check) takes, solved to rounding level (no GPU needed)."""
import pytest


@pytest.fixture(scope="module")
def cs():
    import paper_1902_09931_gb300 as cs
    cs.load()
    return cs


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n", [64, 320, 448, 1472, 2368, 4096])
def test_default_partition_is_replayed(cs, boundary, n):
    P, m = cs.cs_ch_partition(cs.CHDesc(n=n, storage=0, D=1.0, gamma=0.01, dt=0.01, boundary=boundary))
    assert P * m == n
    for a in (0.7, 2885.8, 1.85e5):
        assert cs.cs_ch_solver_check(n, P, a, boundary) <= 64 * 2.0 ** -52  # the bound of every other partition
