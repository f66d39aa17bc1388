"""The fixed-point line solver of the Cahn-Hilliard step (Sec. 5.1's pentadiagonal solves), through the
row-band entry points: backward error along rows for every kernel shape (one to 64 chunks' worth of
lengths, lines that do not fit in shared memory), values over the whole exponent range, rows with
infinities and NaN, and the column kernels against the row kernels bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1902_09931_gb300 as cs
    cs.load()
    return cs, torch


def _plan(cs, n, rows, boundary, dt):
    return cs.cs_ch_band_create(cs.CHDesc(n=n, storage=0, D=1.0, gamma=0.01, dt=dt, boundary=boundary), rows)


def _coefficient(n, dt):
    h = 2 * np.pi / n
    return (2.0 / 3.0) * 0.01 * dt / h ** 4


def _residual(x, b, a, boundary):
    """max |x + a D4 x - b| per row, in extended precision where the host has it."""
    x, b = x.astype(np.longdouble), b.astype(np.longdouble)
    p = np.pad(x, ((0, 0), (2, 2)), mode="symmetric" if boundary else "wrap")
    n = x.shape[1]
    d4 = p[:, :n] - 4 * p[:, 1:n + 1] + 6 * p[:, 2:n + 2] - 4 * p[:, 3:n + 3] + p[:, 4:]
    return np.abs(x + a * d4 - b).max(axis=1)


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n, rows", [(64, 64), (128, 32), (320, 32), (512, 64), (1024, 32), (1472, 32), (2368, 32), (4096, 32), (8192, 32),
                                     (16384, 32), (32768, 32)])
def test_rows_backward_error(env, n, rows, boundary):
    """|L x - b| <= 64 eps (1 + 16 a) max|x| per row (the bound the solver's host replay is held to), for
    white and smooth right-hand sides and rows scaled by 1e-200, 1e200 and (outside fixed point) 1e270."""
    cs, torch = env
    dt = 0.1 * 2 * np.pi / n
    a = _coefficient(n, dt)
    rng = np.random.Generator(np.random.PCG64(n + boundary))
    b = rng.uniform(-1, 1, (rows, n))
    b[1::4] = np.sin(2 * np.pi * (np.arange(n) + 0.5) * 3 / n) + 1e-3 * b[1::4]
    scale = np.ones((rows, 1))
    scale[2], scale[3], scale[6], scale[7] = 1e-200, 1e200, 1e270, 2.0 ** -1000
    b *= scale
    b[4, : n // 2] = 0.0
    b[5] = 0.0
    d = torch.from_numpy(b).cuda()
    x = torch.full_like(d, 7.0)
    plan = _plan(cs, n, rows, boundary, dt)
    cs.cs_ch_band_solve(plan, d, x)
    cs.cs_ch_band_solve(plan, d, d)  # in place
    torch.cuda.synchronize()
    cs.cs_destroy(plan)
    got = x.cpu().numpy()
    assert np.array_equal(got, d.cpu().numpy())
    assert np.array_equal(got[5], np.zeros(n))
    r = _residual(got / scale, b / scale, a, boundary)
    lim = 64 * EPS * (1 + 16 * a) * np.maximum(np.abs(got / scale).max(axis=1), 1e-300)
    assert (r <= lim).all(), (r / lim).max()


@pytest.mark.parametrize("n", [64, 1024, 32768])
def test_rows_with_non_finite_values(env, n):
    """A row holding an infinity or a NaN gives no finite value where the solver couples it in, and the
    other rows are bit for bit what they are without it."""
    cs, torch = env
    dt = 0.1 * 2 * np.pi / n
    rng = np.random.Generator(np.random.PCG64(5))
    b = rng.uniform(-1, 1, (32, n))
    bad = b.copy()
    bad[3, n // 3], bad[9, 0], bad[10, n - 1] = np.nan, np.inf, -np.inf
    plan = _plan(cs, n, 32, 0, dt)
    out = []
    for v in (b, bad):
        d = torch.from_numpy(v).cuda()
        cs.cs_ch_band_solve(plan, d, d)
        torch.cuda.synchronize()
        out.append(d.cpu().numpy())
    cs.cs_destroy(plan)
    rows = [r for r in range(32) if r not in (3, 9, 10)]
    assert np.array_equal(out[0][rows], out[1][rows])
    for r in (3, 9, 10):
        assert not np.isfinite(out[1][r]).any()


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n", [64, 512, 1472, 2048, 2368])
def test_column_kernels_equal_row_kernels(env, n, boundary, storage):
    """One full-grid step (columns by clusters of blocks) against its pieces on a band of all rows: the
    y lines by chunks through global memory, and through transposes as rows; fields bit for bit."""
    cs, torch = env
    dt = 0.1 * 2 * np.pi / n
    tdt = torch.float64 if storage == 0 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n + boundary)
    prev = ((torch.rand(n, n, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.2).to(tdt)
    cur = ((torch.rand(n, n, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.2).to(tdt)
    desc = cs.CHDesc(n=n, storage=storage, D=1.0, gamma=0.01, dt=dt, boundary=boundary)
    nxt = torch.zeros_like(cur)
    full = cs.cs_ch_create(desc, prev.clone(), cur.clone(), nxt)
    cs.cs_ch_step(full, 1)
    torch.cuda.synchronize()
    cs.cs_destroy(full)

    def padded(f):
        top, low = (f[:2].flip(0), f[-2:].flip(0)) if boundary else (f[-2:], f[:2])
        return torch.cat([top, f, low]).contiguous()

    pp, pc = padded(prev), padded(cur)
    out = torch.zeros_like(pc)
    rhs = torch.empty(n, n, device="cuda", dtype=torch.float64)
    band = cs.cs_ch_band_create(desc, n)
    cs.cs_ch_band_rhs(band, pp, pc, rhs)
    cs.cs_ch_band_solve(band, rhs, rhs)
    chunks, _ = cs.cs_ch_partition(desc)
    ends = torch.empty(4 * chunks * n, device="cuda", dtype=torch.float64)
    v = torch.empty_like(rhs)
    cs.cs_ch_band_ycols_local(band, 0, rhs, ends)
    cs.cs_ch_band_ycols_correct(band, 0, ends, v)
    vt = rhs.T.contiguous()
    cs.cs_ch_band_solve(band, vt, vt)
    cs.cs_ch_band_update(band, pp, pc, v, out)
    torch.cuda.synchronize()
    cs.cs_destroy(band)
    assert torch.equal(v, vt.T)
    assert torch.equal(out[2:n + 2], nxt)
