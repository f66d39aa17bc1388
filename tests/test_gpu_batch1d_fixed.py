"""The fixed-point form of the batched FP64 lines (weights c n_k): against extended-precision sums on
ragged lines with segment and line ends in every position, over values of every magnitude, with infinities
and NaN, and for weights that are c n_k only to rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

D2 = [-1 / 12, 16 / 12, -30 / 12, 16 / 12, -1 / 12]


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1902_09931_gb300 as cs
    cs.load()
    return cs, torch


def _run(cs, torch, x, off, w, left, right, bc):
    d = torch.from_numpy(x).cuda()
    out = torch.full_like(d, 5.0)
    o = torch.from_numpy(off).cuda()
    desc = cs.StencilDesc(dir=cs.CS_DIR_X, bc=bc, dtype=cs.CS_F64, left=left, right=right, weights=list(w))
    plan = cs.cs_plan_create_1d_batch(desc, off.size - 1, o, x.size, d, out)
    cs.cs_compute(plan)
    torch.cuda.synchronize()
    cs.cs_destroy(plan)
    return out.cpu().numpy()


def _reference(x, off, w, left, right, bc):
    ref = np.full(x.size, 5.0, dtype=np.longdouble)
    xl = x.astype(np.longdouble)
    for a, b in zip(off[:-1], off[1:]):
        n = b - a
        if n == 0:
            continue
        k = np.arange(n)
        s = sum(np.longdouble(w[p]) * xl[a + (k + p - left) % n] for p in range(left + right + 1))
        if bc:
            ref[a:b] = s
        else:
            ok = (k >= left) & (k < n - right)
            ref[a:b][ok] = s[ok]
    return ref


def _offsets(lengths):
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("left, right, w", [(2, 2, D2), (2, 2, np.array(D2) * 1.7e7), (1, 1, [1.0, -2.0, 1.0]), (1, 2, [1.0, 3.0, -9.0, 2.0]),
                                            (2, 0, [0.5, -2.0, 1.5]), (0, 0, [0.3]), (2, 2, np.array([1, -4, 6, -4, 1]) / 0.31 ** 4)])
def test_against_extended_precision(env, left, right, w, bc):
    """|error| <= 2^-54 sum|w| max|x| (inputs cut at 2^-55 of a segment's largest, up to rho's last bits) plus
    2^-52 of the result (its two roundings)."""
    cs, torch = env
    rng = np.random.Generator(np.random.PCG64(left * 7 + right + bc))
    off = _offsets(np.concatenate([rng.integers(1, 9, 40), [0, 0, 255, 256, 257, 1, 300], rng.integers(64, 900, 60), [4096, 3, 5000]]))
    n = int(off[-1])
    k = np.arange(n)
    for x in (np.sin(0.013 * k) + 1e-3 * rng.uniform(-1, 1, n), rng.uniform(-1, 1, n) * 1e-150, rng.uniform(-1, 1, n) * 3e120,
              rng.integers(-1024, 1025, n).astype(np.float64)):
        got = _run(cs, torch, x, off, w, left, right, bc)
        ref = _reference(x, off, w, left, right, bc)
        lim = 2.0 ** -54 * np.abs(w).sum() * np.abs(x).max() + 2.0 ** -52 * np.abs(ref)
        assert (np.abs(got - ref) <= lim).all(), (np.abs(got - ref) / lim).max()


def test_integer_sums_are_exact(env):
    cs, torch = env
    rng = np.random.Generator(np.random.PCG64(3))
    off = _offsets(rng.integers(1, 700, 50))
    x = rng.integers(-2 ** 20, 2 ** 20, int(off[-1])).astype(np.float64)
    w = [3.0, -5.0, 7.0, 2.0, -1.0]
    assert np.array_equal(_run(cs, torch, x, off, w, 2, 2, 1), _reference(x, off, w, 2, 2, 1).astype(np.float64))


def test_wide_range_zeros_and_non_finite(env):
    """Segments whose values span the exponent range, zero segments, and non-finite values: each output is
    finite exactly where its five inputs are, and correct to the chain's own bound there."""
    cs, torch = env
    rng = np.random.Generator(np.random.PCG64(4))
    off = _offsets([1500, 700, 2000])
    n = int(off[-1])
    x = rng.uniform(-1, 1, n)
    x[256:512] = 0.0
    x[600:900] *= 2.0 ** rng.integers(-1000, -900, 300)
    x[1024:1100] *= 1e300
    x[1300], x[1600], x[2300] = np.nan, np.inf, -np.inf
    with np.errstate(invalid="ignore", over="ignore"):
        got = _run(cs, torch, x, off, D2, 2, 2, 1)
        ref = _reference(x, off, D2, 2, 2, 1)
    fine = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fine) and (~fine).sum() == 15
    seg = np.maximum.reduceat(np.where(np.isfinite(x), np.abs(x), 0), np.arange(0, n, 256))
    near = np.maximum.reduce([np.roll(seg, j) for j in (-1, 0, 1)]).repeat(256)[:n]
    lim = 2.0 ** -51 * np.abs(D2).sum() * near + 2.0 ** -52 * np.abs(np.where(fine, ref, 0)).astype(np.float64)
    assert (np.abs(got - ref)[fine] <= lim[fine]).all()
