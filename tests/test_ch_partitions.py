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


def test_tune_files_of_the_former_solver_are_not_read(tmp_path):
    """Its chunk counts (16 at 4096^2) are not this solver's; what the autotuner saves now is (own process:
    the tuning table is process-wide)."""
    import subprocess
    import sys
    old, new = tmp_path / "old.json", tmp_path / "new.json"
    keys = [f"{{}}|f64|n4096|sm{sms}" for sms in (148, 152, 160)]
    old.write_text("{" + ", ".join(f'"{k.format("ch")}": 16' for k in keys) + "}")
    new.write_text("{" + ", ".join(f'"{k.format("chlines")}": 32' for k in keys) + "}")
    code = ("import sys, paper_1902_09931_gb300 as cs; cs.load(); d = cs.CHDesc(n=4096, storage=0, D=1.0, gamma=0.01, dt=0.01)\n"
            "print(cs.cs_ch_partition(d)[0]); cs.cs_tune_load(sys.argv[1]); print(cs.cs_ch_partition(d)[0])\n"
            "cs.cs_tune_load(sys.argv[2]); print(cs.cs_ch_partition(d)[0])")
    got = subprocess.run([sys.executable, "-c", code, str(old), str(new)], capture_output=True, text=True, check=True).stdout.split()
    assert got == ["64", "64", "32"]


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("a", [1e24, 1e25, 1e60, 1e200, 1e300, 1e301, 1e304, 1e307, 1.7e308])
def test_every_finite_coefficient(cs, a, boundary):
    for n, P in ((64, 1), (64, 4), (1024, 32)):
        assert cs.cs_ch_solver_check(n, P, a, boundary) <= 64 * 2.0 ** -52
