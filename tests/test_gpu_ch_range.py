"""The line solves at the ends of FP64's range: right-hand sides near the largest finite value (where c times
the result would overflow), and coefficients up to the largest finite one (where a line becomes its mean)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


def _solve(n, dt, boundary, b):
    import torch
    import paper_1902_09931_gb300 as cs
    plan = cs.cs_ch_band_create(cs.CHDesc(n=n, storage=0, D=1.0, gamma=0.01, dt=dt, boundary=boundary), b.shape[0])
    d = torch.from_numpy(b).cuda()
    cs.cs_ch_band_solve(plan, d, d)
    torch.cuda.synchronize()
    cs.cs_destroy(plan)
    return d.cpu().numpy()


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n", [64, 4096])
def test_right_hand_sides_near_the_largest_value(n, boundary):
    """Backward error of rows scaled by 2^1020, to the bound of every other scale (the solver's own replay's)."""
    dt = 0.1 * 2 * np.pi / n
    a = (2.0 / 3.0) * 0.01 * dt / (2 * np.pi / n) ** 4
    rng = np.random.Generator(np.random.PCG64(n))
    b = rng.uniform(-1, 1, (32, n))
    x = _solve(n, dt, boundary, b * 2.0 ** 1020) / 2.0 ** 1020
    p = np.pad(x.astype(np.longdouble), ((0, 0), (2, 2)), mode="symmetric" if boundary else "wrap")
    d4 = p[:, :n] - 4 * p[:, 1:n + 1] + 6 * p[:, 2:n + 2] - 4 * p[:, 3:n + 3] + p[:, 4:]
    r = np.abs(x + a * d4 - b).max(axis=1)
    assert (r <= 64 * EPS * (1 + 16 * a) * np.abs(x).max(axis=1)).all()


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("dt", [1e40, 1e100, 1e250, 1e303])
def test_lines_become_their_means(dt, boundary):
    n = 256
    rng = np.random.Generator(np.random.PCG64(3))
    b = rng.uniform(0.5, 1.5, (32, n)) * np.exp2(np.array([0, 900, -900, 1000] * 8))[:, None]
    x = _solve(n, dt, boundary, b)
    mean = b.astype(np.longdouble).mean(axis=1)[:, None]
    assert (np.abs(x - mean) <= 64 * EPS * mean).all(), float((np.abs(x - mean) / mean).max())
