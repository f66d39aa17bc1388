"""The calls whose speed this framework is judged by, as a user's program makes them.

A case is a dict of plain values; ``kind`` says which entry points it goes through:

``sweep``    one 2D stencil sweep (``cs_plan_create_2d``, ``cs_compute``),
``group``    many small grids of one stencil in one call (``cs_compute_group``), as the serving loop sends them,
``batch1d``  one sweep over a ragged batch of 1D lines (``cs_plan_create_1d_batch``, ``cs_compute``),
``ch``       Cahn-Hilliard ADI steps (``cs_ch_create``, ``cs_ch_step``), the fields staying on the device,
``weno``     one evaluation of the WENO advection term (``cs_plan_create_weno_adv``, ``cs_compute``).

Plans keep their default tile and partition choices.  Everything is made from the seed on the GPU.
``exact`` restates each case with plain torch operations in 64 bits.
"""
from __future__ import annotations

import math

import torch

import paper_1902_09931_gb300 as cs

TWO_PI = 2.0 * math.pi

# name: (direction, left, right, top, bottom, weights in units of 1 / h^order, order).  The weights
# are those of the tests and of the benchmark's suite; d2x8 / d2y8 are the 8th-order second
# derivatives of the worked example.
_D1 = [1 / 12, -8 / 12, 0.0, 8 / 12, -1 / 12]
_D2 = [-1 / 12, 16 / 12, -30 / 12, 16 / 12, -1 / 12]
_D2_8 = [-1 / 560, 8 / 315, -1 / 5, 8 / 5, -205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560]
_STENCILS = {
    "lap5": (cs.CS_DIR_XY, 1, 1, 1, 1, [0, 1, 0, 1, -4, 1, 0, 1, 0], 2),
    "lap9": (cs.CS_DIR_XY, 1, 1, 1, 1, [v / 6 for v in (1, 4, 1, 4, -20, 4, 1, 4, 1)], 2),
    "biharm13": (cs.CS_DIR_XY, 2, 2, 2, 2,
                 [0, 0, 1, 0, 0, 0, 2, -8, 2, 0, 1, -8, 20, -8, 1, 0, 2, -8, 2, 0, 0, 0, 1, 0, 0], 4),
    "ddx4": (cs.CS_DIR_X, 2, 2, 0, 0, _D1, 1),
    "ddy4": (cs.CS_DIR_Y, 0, 0, 2, 2, _D1, 1),
    "d2x8": (cs.CS_DIR_X, 4, 4, 0, 0, _D2_8, 2),
    "d2y8": (cs.CS_DIR_Y, 0, 0, 4, 4, _D2_8, 2),
    # u^3 - u - Laplacian(u), the compiled-in user function
    "cubic": (cs.CS_DIR_XY, 1, 1, 1, 1, [0, -1, 0, -1, 4, -1, 0, -1, 0], 2),
}
_GROUP_SIZES = (32, 64, 128, 256, 512)
_CH_D, _CH_GAMMA = 1.0, 0.01


def listed():
    return [
        # the smallest call: one 5-point Laplacian of a grid that sits in L2, where latency and launches count
        dict(name="lap5 f64 256", kind="sweep", stencil="lap5", nx=256, ny=256, f32=False, periodic=True),
        # the sweeps of the suite: FP32 storage with untouched boundary cells, and the two that
        # take the most arithmetic in FP64 storage, the second one at the largest grid
        dict(name="lap9 np f32 4096", kind="sweep", stencil="lap9", nx=4096, ny=4096, f32=True, periodic=False),
        dict(name="cubic f64 4096", kind="sweep", stencil="cubic", nx=4096, ny=4096, f32=False, periodic=True),
        dict(name="biharm13 f64 8192", kind="sweep", stencil="biharm13", nx=8192, ny=8192, f32=False, periodic=True),
        # the worked example's 8th-order second derivative on a grid with both end points: odd rows,
        # weights without small integer ratios
        dict(name="d2x8 np f64 4097x2049", kind="sweep", stencil="d2x8", nx=4097, ny=2049, f32=False, periodic=False),
        # what the serving loop sends: a batch of small resident grids in one call
        dict(name="group f32 64", kind="group", grids=64, mix=64, f32=True),
        # the full ragged batch, both storage types
        dict(name="batch1d f32 65536", kind="batch1d", lines=65536, radius=2, f32=True, periodic=True),
        dict(name="batch1d f64 65536", kind="batch1d", lines=65536, radius=2, f32=False, periodic=True),
        # a Cahn-Hilliard run's inner loop at the two benchmark sizes, and one with the other boundary and storage
        dict(name="ch f64 1024", kind="ch", n=1024, f32=False, noflux=False, steps=10),
        dict(name="ch f64 4096", kind="ch", n=4096, f32=False, noflux=False, steps=3),
        dict(name="ch noflux f32 2048", kind="ch", n=2048, f32=True, noflux=True, steps=10),
        # the advection term of a time stepper
        dict(name="weno f64 2048", kind="weno", nx=2048, ny=2048, f32=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("sweep", "sweep", "sweep", "group", "batch1d", "ch", "ch", "weno"))
    f32 = rng.random() < 0.5
    if kind == "sweep":
        return dict(kind=kind, stencil=rng.choice(sorted(_STENCILS)), nx=_log_int(rng, 64, 8192),
                    ny=_log_int(rng, 64, 8192), f32=f32, periodic=rng.random() < 0.5)
    if kind == "group":
        return dict(kind=kind, grids=_log_int(rng, 4, 64), mix=rng.randrange(1 << 20), f32=f32)
    if kind == "batch1d":
        return dict(kind=kind, lines=_log_int(rng, 512, 65536), radius=rng.choice((1, 2, 2, 4)), f32=f32,
                    periodic=rng.random() < 0.5)
    if kind == "ch":
        return dict(kind=kind, n=64 * _log_int(rng, 1, 48), f32=f32, noflux=rng.random() < 0.5,
                    steps=rng.randint(1, 5))
    return dict(kind=kind, nx=_log_int(rng, 64, 3000), ny=_log_int(rng, 64, 3000), f32=f32)


class _Plan:
    """A plan handle, destroyed with the state that holds it."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        try:
            cs.cs_destroy(self.handle)
        except Exception:
            pass


def _dt(case):
    return torch.float32 if case["f32"] else torch.float64


def _cs_dt(case):
    return cs.CS_F32 if case["f32"] else cs.CS_F64


def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _sines(ny, nx, seed, modes=8, kmax=32, noise=1e-3):
    """Sum of random-phase plane waves plus noise, FP64 (the recipe of workloads.sines_field)."""
    g = _rng(seed)
    top = max(1, min(kmax, min(nx, ny) // 4))
    k = torch.randint(1, top + 1, (2, modes), generator=g, device="cuda").double()
    phi = torch.rand(modes, generator=g, device="cuda", dtype=torch.float64) * TWO_PI
    x = torch.arange(nx, device="cuda", dtype=torch.float64) * (TWO_PI / nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64) * (TWO_PI / ny)
    ax, by = k[0][:, None] * x, k[1][:, None] * y + phi[:, None]
    u = (by.cos().T @ ax.sin() + by.sin().T @ ax.cos()) / modes
    return u + (torch.rand(ny, nx, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * noise


def _sweep_desc(case, stencil, nx, ny, periodic):
    d, left, right, top, bottom, w, order = _STENCILS[stencil]
    h = TWO_PI / nx
    kw = dict(weights=[v / h ** order for v in w])
    if stencil == "cubic":
        kw = dict(fn=cs.CS_FN_CUBIC_MINUS_LAP, coe=[1.0 / h ** order])
    return cs.StencilDesc(nx=nx, ny=ny, dir=d, bc=cs.CS_BC_PERIODIC if periodic else cs.CS_BC_NONPERIODIC,
                          dtype=_cs_dt(case), left=left, right=right, top=top, bottom=bottom, **kw)


def _group_sizes(case):
    # a small linear congruential sequence of the case alone, so that every seed has the same sizes
    s, got = case["mix"] * 2 + 1, []
    for _ in range(case["grids"]):
        s = (s * 6364136223846793005 + 1442695040888963407) % (1 << 64)
        got.append(_GROUP_SIZES[(s >> 33) % len(_GROUP_SIZES)])
    return got


def _lines(case, seed):
    """(offsets, packed values): lengths log-uniform in 64..4096 (the case's own, whatever the seed), a
    sine sum and noise on each line."""
    m = case["lines"]
    u = torch.rand(m, generator=_rng(m), device="cuda", dtype=torch.float64)
    g = _rng(seed)
    n = (u * (math.log(4097) - math.log(64)) + math.log(64)).exp().floor().clamp(64, 4096).long()
    off = torch.zeros(m + 1, device="cuda", dtype=torch.int64)
    off[1:] = n.cumsum(0)
    total = int(off[-1])
    line = torch.repeat_interleave(torch.arange(m, device="cuda"), n)
    theta = (torch.arange(total, device="cuda") - off[line]).double() * (TWO_PI / n.double())[line]
    x = torch.zeros(total, device="cuda", dtype=torch.float64)
    for _ in range(4):
        k = torch.minimum(torch.randint(1, 33, (m,), generator=g, device="cuda"), n // 4).double()
        phi = torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * TWO_PI
        x += (theta * k[line] + phi[line]).sin() / 4
    x += (torch.rand(total, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * 1e-3
    return off, x


def _line_weights(case):
    return {1: [1.0, -2.0, 1.0], 2: _D2, 4: _D2_8}[case["radius"]]


def _ch_start(case, seed):
    n = case["n"]
    c = torch.rand(n, n, generator=_rng(seed), device="cuda", dtype=torch.float64) * 0.2 - 0.1
    return (c - c.mean()).to(_dt(case))


def _ch_numbers(case):
    h = TWO_PI / case["n"]
    return h, 0.1 * h


def prepare(case, seed):
    kind, dt = case["kind"], _dt(case)
    if kind == "sweep":
        x = _sines(case["ny"], case["nx"], seed).to(dt)
        y = torch.zeros_like(x)
        desc = _sweep_desc(case, case["stencil"], case["nx"], case["ny"], case["periodic"])
        return dict(kind=kind, x=x, out=y, plan=_Plan(cs.cs_plan_create_2d(desc, x, y)))
    if kind == "group":
        xs = [_sines(n, n, seed * 1000 + k).to(dt) for k, n in enumerate(_group_sizes(case))]
        ys = [torch.zeros_like(x) for x in xs]
        plans = [_Plan(cs.cs_plan_create_2d(_sweep_desc(case, "lap9", x.shape[1], x.shape[0], True), x, y))
                 for x, y in zip(xs, ys)]
        return dict(kind=kind, x=xs, out=ys, plans=plans, handles=[p.handle for p in plans])
    if kind == "batch1d":
        off, x = _lines(case, seed)
        x = x.to(dt)
        y = torch.zeros_like(x)
        bc = cs.CS_BC_PERIODIC if case["periodic"] else cs.CS_BC_NONPERIODIC
        desc = cs.StencilDesc(dir=cs.CS_DIR_X, bc=bc, dtype=_cs_dt(case), left=case["radius"], right=case["radius"],
                              weights=_line_weights(case))
        plan = _Plan(cs.cs_plan_create_1d_batch(desc, case["lines"], off, x.numel(), x, y))
        return dict(kind=kind, x=x, out=y, offsets=off, plan=plan)
    if kind == "ch":
        c = _ch_start(case, seed)
        fields = [c, c.clone(), torch.zeros_like(c)]
        _, step = _ch_numbers(case)
        desc = cs.CHDesc(n=case["n"], storage=_cs_dt(case), D=_CH_D, gamma=_CH_GAMMA, dt=step,
                         boundary=cs.CS_CH_NOFLUX if case["noflux"] else cs.CS_CH_PERIODIC)
        return dict(kind=kind, at={f.data_ptr(): f for f in fields}, steps=case["steps"],
                    plan=_Plan(cs.cs_ch_create(desc, *fields)))
    c, u, v = (_sines(case["ny"], case["nx"], seed * 3 + k).to(dt) for k in range(3))
    y = torch.zeros_like(c)
    plan = cs.cs_plan_create_weno_adv(case["nx"], case["ny"], _cs_dt(case), TWO_PI / case["nx"], TWO_PI / case["ny"],
                                      c, u, v, y)
    return dict(kind=kind, x=(c, u, v), out=y, plan=_Plan(plan))


def run(state):
    kind = state["kind"]
    if kind == "group":
        cs.cs_compute_group(state["handles"])
        return state["out"]
    if kind == "ch":
        handle = state["plan"].handle
        cs.cs_ch_step(handle, state["steps"])
        prev, cur, _ = cs.cs_ch_fields(handle)
        return [state["at"][prev], state["at"][cur]]
    cs.cs_compute(state["plan"].handle)
    return state["out"]


def work(case):
    size = 4 if case["f32"] else 8
    kind = case["kind"]
    if kind == "sweep":
        n = case["nx"] * case["ny"]
        taps = sum(1 for w in _STENCILS[case["stencil"]][5] if w)
        return {"bytes": 2 * size * n, "flops": (2 * taps + (4 if case["stencil"] == "cubic" else 0)) * n}
    if kind == "group":
        n = sum(k * k for k in _group_sizes(case))
        return {"bytes": 2 * size * n, "flops": 18 * n}
    if kind == "batch1d":
        n = int(case["lines"] * (4096 - 64) / math.log(4096 / 64))  # the mean length of a log-uniform draw
        return {"bytes": 2 * size * n + 8 * case["lines"], "flops": 2 * (2 * case["radius"] + 1) * n}
    if kind == "ch":
        # each step reads C^n and C^(n-1) and writes C^(n+1); right-hand side about 30 operations a
        # point, two pentadiagonal solves of 9 each
        n = case["n"] ** 2 * case["steps"]
        return {"bytes": 3 * size * n, "flops": 48 * n}
    n = case["nx"] * case["ny"]
    return {"bytes": 4 * size * n, "flops": 180 * n}


# ---- the same results from plain torch operations in 64 bits ------------------------------------


def _apply(u, stencil, h):
    _, left, _, top, _, w, order = _STENCILS[stencil]
    width = left + _STENCILS[stencil][2] + 1
    acc = torch.zeros_like(u)
    for k, v in enumerate(w):
        if v:
            acc += (v / h ** order) * u.roll((top - k // width, left - k % width), (0, 1))
    return acc + u ** 3 - u if stencil == "cubic" else acc


def _lap(u, noflux):
    """Unscaled 5-point Laplacian, periodic or with reflected ghost cells."""
    if not noflux:
        return u.roll(1, 0) + u.roll(-1, 0) + u.roll(1, 1) + u.roll(-1, 1) - 4 * u
    p = torch.nn.functional.pad(u[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    return p[:-2, 1:-1] + p[2:, 1:-1] + p[1:-1, :-2] + p[1:-1, 2:] - 4 * u


def _ch_exact(case, seed):
    n, noflux = case["n"], case["noflux"]
    h, dt = _ch_numbers(case)
    a = (2 / 3) * _CH_D * _CH_GAMMA * dt / h ** 4
    alpha = (2 / 3) * _CH_D * dt / h ** 2
    prev = _ch_start(case, seed).double()
    cur = prev.clone()
    size = 2 * n if noflux else n  # a reflected line is half of an even periodic one
    s = 1 + a * (2 - 2 * torch.cos(torch.arange(size, device="cuda", dtype=torch.float64) * (TWO_PI / size))) ** 2
    lines = s[:, None] * s[None, : size // 2 + 1]
    for _ in range(case["steps"]):
        cbar = 2 * cur - prev
        rhs = -(2 / 3) * (cur - prev) + _lap(alpha * (cur ** 3 - cur) - a * _lap(cbar, noflux), noflux)
        if noflux:
            rhs = torch.cat([rhs, rhs.flip(0)], 0)
            rhs = torch.cat([rhs, rhs.flip(1)], 1)
        v = torch.fft.irfft2(torch.fft.rfft2(rhs) / lines, s=(size, size))[:n, :n]
        prev, cur = cur, cbar + v
    return [prev, cur]


def _weno5(v1, v2, v3, v4, v5):
    s1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + (v1 - 4 * v2 + 3 * v3) ** 2 / 4
    s2 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + (v2 - v4) ** 2 / 4
    s3 = 13 / 12 * (v3 - 2 * v4 + v5) ** 2 + (3 * v3 - 4 * v4 + v5) ** 2 / 4
    big = torch.stack([v1, v2, v3, v4, v5]).square().amax(0)
    eps = 1e-6 * big + 1e-99
    a1, a2, a3 = 0.1 / (s1 + eps) ** 2, 0.6 / (s2 + eps) ** 2, 0.3 / (s3 + eps) ** 2
    p1, p2, p3 = v1 / 3 - 7 * v2 / 6 + 11 * v3 / 6, -v2 / 6 + 5 * v3 / 6 + v4 / 3, v3 / 3 + 5 * v4 / 6 - v5 / 6
    return (a1 * p1 + a2 * p2 + a3 * p3) / (a1 + a2 + a3)


def _weno_term(c, vel, h, axis):
    d = (c.roll(-1, axis) - c) / h
    at = {k: d.roll(-k, axis) for k in (-3, -2, -1, 0, 1, 2)}
    minus = _weno5(at[-3], at[-2], at[-1], at[0], at[1])
    plus = _weno5(at[2], at[1], at[0], at[-1], at[-2])
    return vel * torch.where(vel > 0, minus, plus)


def exact(case, seed):
    kind, dt = case["kind"], _dt(case)
    if kind == "sweep":
        u = _sines(case["ny"], case["nx"], seed).to(dt).double()
        r = _apply(u, case["stencil"], TWO_PI / case["nx"])
        if case["periodic"]:
            return r
        _, left, right, top, bottom, _, _ = _STENCILS[case["stencil"]]
        out = torch.zeros_like(r)
        rows, cols = slice(top, case["ny"] - bottom), slice(left, case["nx"] - right)
        out[rows, cols] = r[rows, cols]
        return out
    if kind == "group":
        return [_apply(_sines(n, n, seed * 1000 + k).to(dt).double(), "lap9", TWO_PI / n)
                for k, n in enumerate(_group_sizes(case))]
    if kind == "batch1d":
        off, x = _lines(case, seed)
        x = x.to(dt).double()
        n, m, r = off.diff(), case["lines"], case["radius"]
        line = torch.repeat_interleave(torch.arange(m, device="cuda"), n)
        start, length = off[:-1][line], n[line]
        rel = torch.arange(x.numel(), device="cuda") - start
        acc = torch.zeros_like(x)
        for p, w in enumerate(_line_weights(case)):
            acc += w * x[start + (rel + p - r) % length]
        if not case["periodic"]:
            acc[(rel < r) | (rel >= length - r)] = 0
        return acc
    if kind == "ch":
        return _ch_exact(case, seed)
    c, u, v = (_sines(case["ny"], case["nx"], seed * 3 + k).to(dt).double() for k in range(3))
    return _weno_term(c, u, TWO_PI / case["nx"], 1) + _weno_term(c, v, TWO_PI / case["ny"], 0)
