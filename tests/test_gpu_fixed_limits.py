"""Limits of the fixed-point marches: what ends a segment, and what its values may be.

Bounds as in test_gpu_fixed.py: |gpu - ref| <= 2^-46 sum|terms| at every point, unless a test says
otherwise.
"""
import numpy as np
import pytest

import oracle
from paper_2306_13002_gb300 import binding, inputs
from _parity import padded_dev, to_dev
from test_gpu_fixed import RHS_TILES, TAYLOR, TILES, _check_rhs, _field, _rhs, _rhs_scale, _star, _star_scale

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 1.5, 1.25)])
@pytest.mark.parametrize("dims", [(48, 32, 120), (41, 37, 120)])
@pytest.mark.parametrize("tile", RHS_TILES + [(16, 16, 60, 2), (16, 16, 60, 0)])
@pytest.mark.parametrize("signs", ["cells", "random"])
def test_rhs_values_that_double_within_a_segment(signs, tile, dims, h):
    """Momenta of one sign per cell (the largest dissipation a bound on |m| allows) that grow by just under
    a factor of two behind the planes a segment's scale was taken from, at several heights: twelve times
    the larger value in the smaller one's scale is more than 63 bits."""
    nx, ny, nz = dims
    U = inputs.rhs_field(nx, ny, nz, halo=2, seed=31)
    z, y, x = np.meshgrid(*(np.arange(n) for n in U.shape[1:]), indexing="ij")
    s = np.where((x + y + z) % 2, 1.0, -1.0) if signs == "cells" else np.random.default_rng(32).choice([-1.0, 1.0], x.shape)
    U[0], U[4] = 1.0, 8.0
    U[1:4] = s * np.where(z % 40 < 13, 0.95, 1.9)
    _check_rhs(U, tile, (signs, dims, h), h=h)


@pytest.mark.parametrize("tile", TILES)
def test_star_negative_zeros(tile):
    """A field of zeros of both signs gives zeros."""
    u = np.where(np.random.default_rng(33).random((29, 33, 45)) < 0.5, 0.0, -0.0)
    a = np.random.default_rng(34).uniform(0.5, 1.5, u.shape)
    assert not np.any(_star(u, a, TAYLOR, tile))
    assert not np.any(_star(np.full(u.shape, -0.0), a, TAYLOR, tile))


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 0.5, 2.0)])
@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("kchunk", [1, 2, 3, 4, 5, 6, 7, 9, 14])
def test_rhs_fp64_rest_from_the_scanned_planes(kchunk, flags, h):
    """Values the scan refuses (a weak dissipation), in chunks as short as the planes it leaves in the ring and
    longer, on whole and cut tiles."""
    U = inputs.rhs_field(75, 50, 43, halo=2, seed=35)
    _check_rhs(U, (16, 16, kchunk, flags), (kchunk, flags, h), eps=0.004, h=h)


@pytest.mark.parametrize("flags", [1, 3])
@pytest.mark.parametrize("every", [1, 7, 40])
def test_rhs_fp64_rest_of_many_columns(every, flags):
    """A balanced launch on a thin grid: 17 columns and more per block, all of them, most or a few with values
    that do not fit."""
    nx, ny, nz = 1150, 1144, 2
    U = inputs.rhs_field(nx, ny, nz, halo=2, seed=36)
    y, x = np.meshgrid(np.arange(ny + 4), np.arange(nx + 4), indexing="ij")
    odd = ((x // 16) + 72 * (y // 16)) % every == 0
    U[:, :, odd & (x % 16 == 3) & (y % 16 == 5)] *= 2.0 ** 11
    _check_rhs(U, (16, 16, 0, flags), (every, flags))


@pytest.mark.parametrize("eps,spiked", [(0.25, 0), (0.25, 3), (0.25, 8), (0.004, 0)])
def test_rhs_batch_fp64_rest(eps, spiked):
    """A batch with work for the fixed-point march, some or all of whose grids hold values that do not fit."""
    host, grids = [], []
    for q, (nx, ny, nz) in enumerate([(64, 48, 50), (49, 47, 61), (33, 70, 40), (80, 31, 45), (48, 48, 48), (65, 50, 37),
                                      (40, 40, 60), (51, 62, 30), (17, 90, 50), (60, 60, 60)]):
        U = inputs.rhs_field(nx, ny, nz, halo=2, seed=3700 + q)
        if q < spiked:
            U[:, 20:24, 10:15, 9:18] *= 2.0 ** 12
        host.append(U)
        grids.append((to_dev(U), None, torch.full((5, nz, ny, nx), float("nan"), dtype=torch.float64, device="cuda")))
    ws = torch.zeros(binding.acs_batch_workspace_bytes(len(grids)) // 8 + 2, dtype=torch.float64, device="cuda")
    plan = binding.acs_batch_prepare(binding.KIND_RHS, grids, ws)
    for _ in range(2):
        binding.acs_batch_launch(plan, {"eps": eps})
    torch.cuda.synchronize()
    for U, (_, _, R) in zip(host, grids):
        bad = ~(np.abs(R.cpu().numpy() - oracle.rhs(U, eps=eps, threads=8)) <= 2.0 ** -46 * _rhs_scale(U, 1.4, eps, (1.0,) * 3))
        assert not bad.any(), (U.shape, np.argwhere(bad)[:3])


@pytest.mark.parametrize("bxy", [(16, 8), (32, 8), (64, 4), (16, 16)])
@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("kind", ["lumps", "growing", "pulse", "tiny"])
@pytest.mark.parametrize("kchunk", [1, 2, 3, 5, 6, 7, 8, 9, 20])
def test_star_fp64_rest(kchunk, kind, flags, bxy):
    """Planes left for FP64: by the scan (mostly small values, values below the scales' range), by several
    short segments, by a full list; chunks as short as the planes a scan leaves in the ring and longer."""
    nx, ny, nz = 75, 34, 41
    u = _field("plain" if kind == "tiny" else kind, (nz + 8, ny + 8, nx + 8), 38)
    a = np.random.default_rng(39).uniform(-1.0, 1.0, u.shape)
    s = 2.0 ** -900 if kind == "tiny" else 1.0
    got, ref = _star(u * s, a, TAYLOR, (*bxy, kchunk, flags)) / s, oracle.stencil(u, a, TAYLOR, threads=4)
    bad = ~(np.abs(got - ref) <= 2.0 ** -46 * _star_scale(u, a, TAYLOR))
    assert not bad.any(), (int(bad.sum()), np.argwhere(bad)[:3])


@pytest.mark.parametrize("flags", [1, 3])
@pytest.mark.parametrize("every", [1, 7, 50])
def test_star_fp64_rest_of_many_columns(every, flags):
    """A balanced launch on a thin grid: 17 columns and more per block, all of them, some or a few with values
    that do not suit a scale."""
    nx, ny, nz = 2310, 1150, 2
    rng = np.random.default_rng(40)
    shape = (nz + 8, ny + 8, nx + 8)
    u = rng.uniform(-1.0, 1.0, shape)
    y, x = np.meshgrid(np.arange(shape[1]), np.arange(shape[2]), indexing="ij")
    odd = ((x // 16) + 145 * (y // 8)) % every == 0
    u[:, odd] *= 2.0 ** rng.integers(-60, 1, (shape[0], int(odd.sum())))
    a = rng.uniform(-1.0, 1.0, shape)
    got, ref = _star(u, a, TAYLOR, (16, 8, 0, flags)), oracle.stencil(u, a, TAYLOR, threads=8)
    bad = ~(np.abs(got - ref) <= 2.0 ** -46 * _star_scale(u, a, TAYLOR))
    assert not bad.any(), (int(bad.sum()), np.argwhere(bad)[:3])


@pytest.mark.parametrize("pitch", [0, 1])
def test_star_batch_fp64_rest(pitch):
    """A batch of which some grids are pulses, some uniform and some values far apart; both stagings."""
    host, grids = [], []
    for q, (nx, ny, nz) in enumerate([(64, 48, 50), (50, 46, 61), (34, 70, 40), (80, 31, 45), (48, 48, 48), (16, 90, 50)]):
        shape = (nz + 8, ny + 8, nx + 8)
        u = _field(("plain", "pulse", "lumps", "zeros", "growing", "wave")[q], shape, 41 + q)
        a = np.random.default_rng(50 + q).uniform(-1.0, 1.0, shape)
        ud, ad = padded_dev(u, nx + 8 + pitch), padded_dev(a, nx + 8 + pitch)
        host.append((u, a))
        grids.append((ud, ad, torch.full((nz, ny, nx), float("nan"), dtype=torch.float64, device="cuda")))
    ws = torch.zeros(binding.acs_batch_workspace_bytes(len(grids)) // 8 + 2, dtype=torch.float64, device="cuda")
    for c in (None, [[w / (h * h) for w in binding.TAYLOR8] for h in (1.0, 0.8, 1.25)]):
        plan = binding.acs_batch_prepare(binding.KIND_STENCIL, grids, ws)
        binding.acs_batch_launch(plan, c)
        torch.cuda.synchronize()
        cn = TAYLOR if c is None else np.array(c)
        for (u, a), (_, _, out) in zip(host, grids):
            bad = ~(np.abs(out.cpu().numpy() - oracle.stencil(u, a, cn, threads=4)) <= 2.0 ** -46 * _star_scale(u, a, cn))
            assert not bad.any(), (u.shape, int(bad.sum()), np.argwhere(bad)[:3])


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 0.8, 1.25), (1.0, 1.0, 0.4)])
def test_star_points_far_below_the_scale_are_as_exact_as_fp64(tile, h):
    """Single values of 1 to 2^-12 among values of 2^-20, no two in reach of one point: a point's error, relative
    to its sum of |terms|, whatever the block's largest value is. An FP64 sum of one such value in any place
    has 1.3e-16 to 1.7e-16 (root mean square; emulated), at most 8.1e-16. 2.2e-16 and 1.3e-15 leave room for
    weights that share the bound to the nearest power of two (a factor of 1.4)."""
    nz, ny, nx = 68, 62, 70
    rng = np.random.default_rng(42)
    u = rng.uniform(-1.0, 1.0, (nz + 8, ny + 8, nx + 8)) * 2.0 ** -20
    z, y, x = np.meshgrid(*(np.arange(0, n, 9) for n in u.shape), indexing="ij")
    big = rng.uniform(1.0, 2.0, z.shape) * 2.0 ** -rng.integers(1, 13, z.shape) * rng.choice([-1.0, 1.0], z.shape)
    u[z, y, x] = np.where(rng.random(z.shape) < 0.25, 1.0, big)
    a = np.ones(u.shape)
    c = np.array([[w / (s * s) for w in binding.TAYLOR8] for s in h])
    got = _star(u, a, c, tile)
    L = np.longdouble
    v, ref, scale = u.astype(L), np.zeros(got.shape, L), np.zeros(got.shape)
    for d in range(3):
        for o in range(1, 5):
            s = [slice(4, -4)] * 3
            p, m = list(s), list(s)
            n = u.shape[2 - d]
            p[2 - d], m[2 - d] = slice(4 + o, n - 4 + o), slice(4 - o, n - 4 - o)
            ref += L(c[d][o - 1]) * (v[tuple(p)] - 2 * v[tuple(s)] + v[tuple(m)])
            scale += abs(c[d][o - 1]) * (np.abs(u[tuple(p)]) + 2 * np.abs(u[tuple(s)]) + np.abs(u[tuple(m)]))
    err = (np.abs(got.astype(L) - ref) / scale).astype(np.float64)
    octave = np.floor(np.log2(scale / np.abs(c).max())).astype(int)
    for k in range(-12, 1):
        e = err[octave == k]
        assert e.size > 50 and np.sqrt(np.mean(e * e)) <= 2.2e-16 and e.max() <= 1.3e-15, (k, e.size, np.sqrt(np.mean(e * e)), e.max())


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 0.8, 1.25)])
def test_star_points_near_the_small_value_bound(tile, h):
    """Values of 2^-9 to 2^-3 alone in small balls of a field of ordinary ones, so that the block keeps its
    scale: the points whose only large term is their own value or their +x, +y or +z neighbour's. Bounds
    as above."""
    n, L = 96, np.longdouble
    c = np.array([[w / (s * s) for w in binding.TAYLOR8] for s in h])
    got, errs = None, []
    for seed in range(4):
        rng = np.random.default_rng(4300 + seed)
        u = rng.uniform(-1.001, 1.001, (n + 8,) * 3)
        i = 16 + 24 * np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij")).reshape(3, -1) + rng.integers(-3, 4, (3, 64))
        z, y, x = np.meshgrid(*[np.arange(n + 8)] * 3, indexing="ij", sparse=True)
        for k, j, m in i.T:
            ball = (z - k) ** 2 + (y - j) ** 2 + (x - m) ** 2 <= 36
            u[ball] *= 2.0 ** -20
        u[tuple(i)] = rng.uniform(1.0, 2.0, 64) * 2.0 ** -rng.integers(4, 10, 64) * rng.choice([-1.0, 1.0], 64)
        got = _star(u, np.ones(u.shape), c, tile)
        for off in ((0, 0, 0), (0, 0, -1), (0, -1, 0), (-1, 0, 0)):
            p = i + np.array(off)[:, None]
            ref, scale = np.zeros(64, L), np.zeros(64)
            for d in range(3):
                for o in range(1, 5):
                    s = np.zeros((3, 1), int)
                    s[2 - d] = o
                    a, b, m = u[tuple(p + s)], u[tuple(p)], u[tuple(p - s)]
                    ref += L(c[d][o - 1]) * (a.astype(L) - 2 * b.astype(L) + m.astype(L))
                    scale += abs(c[d][o - 1]) * (np.abs(a) + 2 * np.abs(b) + np.abs(m))
            e = (np.abs(got[tuple(p - 4)].astype(L) - ref) / scale).astype(np.float64)
            errs.append(np.stack([np.floor(np.log2(np.abs(u[tuple(i)]))), e]))
    octave, e = np.concatenate(errs, axis=1)
    for k in range(-9, -3):
        v = e[octave == k]
        assert v.size > 50 and np.sqrt(np.mean(v * v)) <= 2.2e-16 and v.max() <= 1.3e-15, (k, np.sqrt(np.mean(v * v)), v.max())


@pytest.mark.parametrize("kchunk,flags", [(0, 1), (5, 0), (17, 0), (64, 0)])
@pytest.mark.parametrize("kind", ["wave", "slope", "pulse", "growing", "corner"])
def test_stagings_agree_bitwise_where_scales_differ(kind, kchunk, flags):
    """Tensor copies and element-wise staging take the same scales, also where a block's largest value is in a
    corner of its halo, which no point reads."""
    def fields(n, halo):
        shape = tuple(v + 2 * halo for v in (60, 66, 104))
        z, y, x = np.meshgrid(*(np.arange(v) for v in shape), indexing="ij")
        base = np.random.default_rng(44).uniform(0.6, 1.0, (n,) + shape)
        if kind == "slope":
            return base * 2.0 ** (0.11 * (x + 1.7 * y) - 0.05 * z)
        if kind == "corner":    # larger values at the crossings of every second tile's edges
            return base * np.where((((x - halo) % 16) // 2 == 0) & (((y - halo) % 8) // 2 == 0), 5.0, 1.0)
        return np.stack([_field(kind, shape, 45 + q) for q in range(n)]) if kind != "wave" else base * _field("wave", shape, 0)

    u = fields(1, 4)[0]
    a = np.random.default_rng(46).uniform(-1.0, 1.0, u.shape)
    for bx, by in ((16, 8), (32, 8), (16, 16)):
        for c in (TAYLOR, np.array([[w * s for w in binding.TAYLOR8] for s in (1.0, 1.5, 0.7)])):
            t, e = (_star(u, a, c, (bx, by, kchunk, flags | f)) for f in (binding.TILE_TMA, 0))
            assert np.array_equal(t, e), (bx, by, int((t != e).sum()))
    U = fields(5, 2)
    U[0] = np.abs(U[0]) + 0.5
    U[4] = np.abs(U[4]) + 1.0
    for h in ((1.0, 1.0, 1.0), (1.0, 1.5, 2.0)):
        t, e = (_rhs(U, (16, 16, kchunk, flags | f), 1.4, 0.25, h) for f in (binding.TILE_TMA, 0))
        assert np.array_equal(t, e), (h, int((t != e).sum()))


def _rhs_grids(sides, seed):
    out = []
    for q, (nx, ny, nz) in enumerate(sides):
        U = inputs.rhs_field(nx, ny, nz, halo=2, seed=seed + q)
        out.append((to_dev(U), None, torch.full((5, nz, ny, nx), float("nan"), dtype=torch.float64, device="cuda")))
    return out


@pytest.mark.parametrize("sides", [[(16, 16, 16), (20, 18, 5)], [(64, 48, 50)] * 6])
@pytest.mark.parametrize("tile", [None, (32, 8, 12), (16, 16, 32)])
def test_rhs_batch_plan_tile_prepares_the_same_plan(tile, sides):
    """A prepared plan's tile is the shape that runs, and prepares it again: batches with little work, which
    run the FP64 march, and others."""
    grids = _rhs_grids(sides, 4700)
    ws = torch.zeros(binding.acs_batch_workspace_bytes(len(grids)) // 8 + 2, dtype=torch.float64, device="cuda")

    def run(t):
        plan = binding.acs_batch_prepare(binding.KIND_RHS, grids, ws, tile=t)
        binding.acs_batch_launch(plan)
        torch.cuda.synchronize()
        return plan, [R.clone() for _, _, R in grids]

    p, first = run(tile)
    assert (p.tile.bx, p.tile.by, p.tile.flags) == (16, 16, 0)
    again, second = run((p.tile.bx, p.tile.by, p.tile.kchunk, p.tile.flags))
    assert again.total_units == p.total_units
    assert all(torch.equal(x, y) for x, y in zip(first, second))
    binding.acs_batch_run_static(binding.KIND_RHS, grids, tile=(p.tile.bx, p.tile.by, p.tile.kchunk, p.tile.flags))
    torch.cuda.synchronize()
    assert all(torch.equal(x, R) for x, (_, _, R) in zip(first, grids))


def test_autotuners_name_the_columns_that_run():
    """Grids and batches the fixed-point RHS takes run in 16 x 16 columns: so do the tuners' winners."""
    try:
        (U, _, R), = _rhs_grids([(96, 64, 48)], 4800)
        assert tuple(binding.acs_autotune_rhs(U, R)[0])[:2] == (16, 16)
        grids = _rhs_grids([(64, 48, 50)] * 4, 4900)
        ws = torch.zeros(binding.acs_batch_workspace_bytes(len(grids)) // 8 + 2, dtype=torch.float64, device="cuda")
        assert tuple(binding.acs_autotune_batch(binding.KIND_RHS, grids, ws)[0])[:2] == (16, 16)
    finally:
        binding.acs_tune_cache_clear()


@pytest.mark.parametrize("fixed,prm", [
    (True, {}), (True, {"eps": 0.03}), (True, {"eps": 0.1, "h": (0.37, 0.37, 0.37)}), (True, {"h": (0.1, 0.1, 0.1)}),
    (True, {"h": (1.0, 0.5, 2.0)}), (True, {"h": (1.0, 1.0, 8.0)}), (True, {"gamma": 5.0 / 3.0}), (True, {"gamma": 0.5}),
    (False, {"eps": 0.01}), (False, {"h": (1.0 / 64,) * 3}), (False, {"h": (1.0, 1.0, 16.0)}), (False, {"gamma": 1.0}),
    (False, {"eps": 1e-9}), (False, {"h": (1e-5, 1.0, 1.0)}),
])
def test_rhs_which_march_ran(fixed, prm):
    """A grid too small for the fixed-point march runs in FP64, and what a block leaves runs the same operations in
    the same order: a slab of a larger grid, taken alone, has the larger one's bits if and only if that ran in FP64.
    Both within the bound of the exact value."""
    U = inputs.rhs_field(83, 70, 61, halo=2, seed=60)
    args = (prm.get("gamma", 1.4), prm.get("eps", 0.25), prm.get("h", (1.0, 1.0, 1.0)))
    for tile in (None, (16, 16, 20, 2), (16, 16, 20, 0)):
        whole, slab = _rhs(U, tile, *args), _rhs(U[:, 20:44], None, *args)
        same = whole[:, 20:40] == slab
        assert same.mean() < 0.9 if fixed else same.all(), (tile, same.mean())
        _check_rhs(U, tile, str(prm), *args)
