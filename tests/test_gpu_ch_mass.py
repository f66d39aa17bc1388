"""The line solves conserve the sum of a periodic line exactly but for rounding, and the rounding has no bias:
the mean of x - b over many random lines stays within its own statistical error (a bias is a steady drift of the
Cahn-Hilliard mass)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, dt, lines", [(64, 0.1 * 2 * np.pi / 64, 20480), (64, 1e-5, 20480), (128, 0.1 * 2 * np.pi / 128, 20480),
                                          (512, 0.1 * 2 * np.pi / 512, 40960)])
def test_sums_of_random_lines_are_unbiased(n, dt, lines):
    import torch
    import paper_1902_09931_gb300 as cs
    rows = min(n, 512)
    plan = cs.cs_ch_band_create(cs.CHDesc(n=n, storage=0, D=1.0, gamma=0.01, dt=dt), rows)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.empty(rows, n, device="cuda", dtype=torch.float64)
    means = []
    for _ in range(lines // rows):
        b = torch.rand(rows, n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
        cs.cs_ch_band_solve(plan, b, x)
        hi, total = [], 0.0
        for v in (x, -b):  # parts on a grid of 2^-30, whose sums are exact, and the rest
            top = (v * 2.0 ** 30).round() * 2.0 ** -30
            hi.append(top.sum(1))
            total = total + (v - top).sum(1)
        means.append((hi[0] + hi[1] + total) / n)
    cs.cs_destroy(plan)
    d = torch.cat(means).cpu().numpy()
    error = d.std() / np.sqrt(d.size)
    assert abs(d.mean()) <= 5 * error, (d.mean(), error)  # 5 standard errors of the mean
