"""Batched FP64 lines whose weights are c n_k (the fixed-point kernel): each output against its own five
inputs' magnitude, so that lines of any scale may lie side by side."""
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


def _run(env, x, off, w, left, right, bc):
    cs, torch = env
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
    """(sums, sums of magnitudes) in extended precision; untouched outputs 5 and 0."""
    ref, size = np.full(x.size, 5.0, dtype=np.longdouble), np.zeros(x.size, dtype=np.longdouble)
    xl = x.astype(np.longdouble)
    for a, b in zip(off[:-1], off[1:]):
        n = b - a
        if n == 0:
            continue
        k = np.arange(n)
        t = [np.longdouble(w[p]) * xl[a + (k + p - left) % n] for p in range(left + right + 1)]
        ok = np.ones(n, bool) if bc else (k >= left) & (k < n - right)
        ref[a:b][ok], size[a:b][ok] = sum(t)[ok], sum(abs(v) for v in t)[ok]
    return ref, size


def _offsets(lengths):
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)


# at most five roundings, each at most 2^-53 of a partial sum of the five products
LIMIT = 5 * 2.0 ** -53


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("w", [[1.0, -2.0, 1.0], [1.0, -2.0 * (1 + 2.0 ** -50), 1.0], [1.0, -2.0 - 2.0 ** -45, 1.0],
                               [-1 / 12, 16 / 12, -30 / 12 * (1 + 2.0 ** -46), 16 / 12, -1 / 12], D2, [1.0, -1.0, 0.0], [3.0]])
def test_values_just_below_a_power_of_two(env, w, sign):
    """The weighted sum at the end of its range: values of the weights' signs (and their opposites) as near
    to 1 as there are, with weights that are c n_k exactly and to 2^-45."""
    r = len(w) // 2
    s = np.sign(w)
    s[s == 0] = 1.0
    for top in (1 - 2.0 ** -53, 1 - 2.0 ** -48, 1 - 2.0 ** -21, 1 - 2.0 ** -20, 1.0):
        x = sign * top * np.tile(s, 400)
        off = _offsets([x.size])
        ref, size = _reference(x, off, w, r, r, 1)
        got = _run(env, x, off, w, r, r, 1)
        assert (np.abs(got - ref) <= LIMIT * size).all(), (got[:6], ref[:6])


SCALES = [1.0, 1e-18, 1e20, 1e-8, 3e-100, 1.0, 1e150, 1e-12]


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("left, right, w", [(2, 2, D2), (2, 2, np.array(D2) * 1.7e7), (1, 1, [1.0, -2.0, 1.0]), (1, 2, [1.0, 3.0, -9.0, 2.0]),
                                            (2, 0, [0.5, -2.0, 1.5]), (0, 0, [0.3])])
def test_lines_of_different_scale_side_by_side(env, left, right, w, bc):
    """Short and long lines of amplitudes 1e-100 to 1e150 packed next to one another, smooth and random, and
    lines that decay over their length: every output to the bound of the multiply-add chain on its own inputs."""
    rng = np.random.Generator(np.random.PCG64(left * 7 + right + bc))
    off = _offsets(np.concatenate([rng.integers(1, 60, 200), [0, 256, 255, 0, 1, 8, 16, 300], rng.integers(64, 900, 60)]))
    n = int(off[-1])
    line = np.repeat(np.arange(off.size - 1), np.diff(off))
    k = np.arange(n) - off[line]
    scale = np.array(SCALES)[line % len(SCALES)]
    decay = np.where(line % 3 == 0, np.exp2(-0.7 * np.minimum(k, 400)), 1.0)
    for x in (scale * np.sin(0.1 * k + line), scale * rng.uniform(-1, 1, n), scale * decay * (1 + 0.3 * np.sin(0.05 * k)),
              scale * np.where(rng.uniform(0, 1, n) < 0.7, 0.0, rng.uniform(-1, 1, n))):
        ref, size = _reference(x, off, w, left, right, bc)
        got = _run(env, x, off, w, left, right, bc)
        assert (np.abs(got - ref) <= LIMIT * size).all(), float((np.abs(got - ref) / np.maximum(size, 1e-300)).max())


def test_a_line_does_not_depend_on_its_neighbours(env):
    """The same bits in a line whatever the other lines hold: other values, zeros, NaN."""
    rng = np.random.Generator(np.random.PCG64(9))
    off = _offsets(np.concatenate([rng.integers(1, 60, 100), rng.integers(200, 900, 30)]))
    n = int(off[-1])
    line = np.repeat(np.arange(off.size - 1), np.diff(off))
    x = np.sin(0.07 * np.arange(n)) + 1e-3 * rng.uniform(-1, 1, n)
    for w in (D2, [0.0, 1.0, -2.0, 1.0, 0.0], np.array(D2) * 0.37):
        for bc in (0, 1):
            ref = _run(env, x, off, w, 2, 2, bc)
            for other in (1e20, 0.0, np.nan):
                for keep in (0, 1):
                    with np.errstate(invalid="ignore"):
                        y = np.where(line % 2 == keep, x, other * x)
                    assert np.array_equal(_run(env, y, off, w, 2, 2, bc)[line % 2 == keep], ref[line % 2 == keep])


def test_nothing_to_tune_in_fixed_point(env):
    """The fixed-point kernel has one launch shape: the autotuner launches nothing for it and leaves the
    tuning key, which plans with other weights share, alone."""
    cs, torch = env
    off = torch.arange(0, 6401, 64, device="cuda")
    x = torch.rand(6400, device="cuda", dtype=torch.float64)
    out = torch.zeros_like(x)
    for w, tuned in ((D2, False), ([0.1, 0.7, -1.3, 0.9, 0.25], True)):
        plan = cs.cs_plan_create_1d_batch(cs.StencilDesc(dir=cs.CS_DIR_X, bc=1, dtype=cs.CS_F64, left=2, right=2, weights=w), 100, off, 6400, x, out)
        before = cs.cs_launch_count()
        cs.cs_autotune(plan)
        assert (cs.cs_launch_count() > before) == tuned
        cs.cs_destroy(plan)
