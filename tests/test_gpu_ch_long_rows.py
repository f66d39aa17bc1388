"""Rows too long for shared memory: the 32-byte accesses of aligned rows give the bits of the word-by-word ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n", [26624, 26688, 32768])  # chunks of 416, 417 (never wide) and 512 points
def test_aligned_and_unaligned_rows_agree(n, boundary):
    import torch
    import paper_1902_09931_gb300 as cs
    rows = 32
    plan = cs.cs_ch_band_create(cs.CHDesc(n=n, storage=0, D=1.0, gamma=0.01, dt=0.2 * np.pi / n, boundary=boundary), rows)
    g = torch.Generator(device="cuda").manual_seed(n)
    b = torch.rand(rows, n, generator=g, device="cuda", dtype=torch.float64) - 0.5
    b[3, 5] = float("nan")
    x = torch.empty_like(b)
    cs.cs_ch_band_solve(plan, b, x)
    pool = torch.empty(rows * n + 1, device="cuda", dtype=torch.float64)
    y = pool[1:].view(rows, n)
    y.copy_(b)
    cs.cs_ch_band_solve(plan, y, y)
    torch.cuda.synchronize()
    cs.cs_destroy(plan)
    assert torch.isnan(x[3]).all() and torch.isnan(y[3]).all()
    keep = [r for r in range(rows) if r != 3]
    assert torch.equal(x[keep], y[keep]) and bool(torch.isfinite(x[keep]).all())
