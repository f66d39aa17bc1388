"""FP64 sweeps of plans for which nobody chose a tile shape: the digit grid is that of 64-row tiles whatever shape
runs, so alone, grouped and with tile choice 1 they give the same bits (other weights: the same bits too where
the tile's values allow the double-float path)."""
import numpy as np
import pytest

from gpu_helpers import stencil_cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1902_09931_gb300 as cs
    cs.load()
    return cs, torch


# weights with small integer ratios, which groups evaluate as digits too
DIGITS = {"lap5", "lap9", "biharm13", "ddx4", "ddy4", "d2x4", "d2y4", "x1", "y1", "cubic"}
SIZES = [(1, 5), (31, 517), (32, 64), (33, 64), (64, 64), (65, 66), (95, 130), (96, 128), (100, 260), (127, 63), (192, 320), (257, 129), (256, 256),
         (1025, 1027), (1536, 512), (2097089, 2), (2097120, 2)]  # the last: the most rows a launch has


def _field(ny, nx, seed):
    """Values whose scale changes from row to row and from tile to tile, so that the digit grid shows."""
    rng = np.random.Generator(np.random.PCG64(seed))
    y, x = np.mgrid[0:ny, 0:nx]
    return np.exp2(6 * np.sin(0.11 * y) + 3 * np.sin(0.05 * x)) * rng.uniform(-1, 1, (ny, nx))


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("special", ["finite", "nan", "zeros"])
def test_default_shape_gives_the_bits_of_64_row_tiles(env, bc, special):
    cs, torch = env
    for ny, nx in SIZES:
        u = _field(ny, nx, ny + nx)
        if special == "nan":  # one half of a 64-row tile only
            u[min(ny - 1, 40), nx // 2] = np.nan
            u[ny // 3, 0] = np.inf
        elif special == "zeros":
            u[min(ny - 1, 20):] = 0.0
        d = torch.from_numpy(u).cuda()
        cases = [(n, dict(dir=dr, left=L, right=R, top=T, bottom=B, weights=w)) for n, L, R, T, B, dr, w in stencil_cases(2 * np.pi / nx)]
        cases.append(("cubic", dict(dir=2, left=1, right=1, top=1, bottom=1, fn=3, coe=[40.0])))
        for name, kw in cases:
            if nx <= kw["left"] + kw["right"] or ny <= kw["top"] + kw["bottom"]:
                continue
            if special == "nan" and name not in DIGITS:
                continue
            desc = cs.StencilDesc(nx=nx, ny=ny, bc=bc, dtype=0, **kw)
            outs = [torch.full_like(d, 7.0) for _ in range(3)]
            plans = [cs.cs_plan_create_2d(desc, d, o) for o in outs]
            cs.cs_compute(plans[0])
            cs.cs_plan_set_tile_choice(plans[1], 1)
            cs.cs_compute(plans[1])
            try:
                cs.cs_compute_group([plans[2]])
                grouped = name in DIGITS
            except cs.CSError as e:
                assert e.code == cs.CS_EUNSUPPORTED
                grouped = False
            torch.cuda.synchronize()
            for p in plans:
                cs.cs_destroy(p)
            bits = [o.view(torch.int64) for o in outs]
            nan = torch.isnan(outs[1])
            for k in (0, 2) if grouped else (0,):
                same = (bits[k] == bits[1]) | (nan & torch.isnan(outs[k]))
                assert bool(same.all()), (name, ny, nx, k, int((~same).sum()))
