"""The Cahn-Hilliard autotuner on a grid of 64 times an odd number: the plan's own partition is among the
candidates (chunks of 46 points, three times as fast as the longest in whole batches of 8)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1])
def test_autotune_times_the_default_partition(storage):
    import torch
    import paper_1902_09931_gb300 as cs
    n = 1472
    dt = torch.float64 if storage == 0 else torch.float32
    f = [0.1 * torch.rand(n, n, device="cuda", dtype=dt) for _ in range(2)] + [torch.zeros(n, n, device="cuda", dtype=dt)]
    plan = cs.cs_ch_create(cs.CHDesc(n=n, storage=storage, D=1.0, gamma=0.01, dt=0.2 * np.pi / n), *f)
    before = cs.cs_ch_config(plan)
    cs.cs_autotune(plan)
    after = cs.cs_ch_config(plan)
    cs.cs_destroy(plan)
    assert before == (32, 46)
    assert after[0] >= 16, after  # 8 chunks are the most that have whole batches
