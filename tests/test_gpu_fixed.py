"""The fixed-point marches of the saturated kernels at the edges of their range: values far below the
block's scale, values that outgrow it on the way, zeros, infinities and NaN, unset halo corners,
every staging and tile edge. Compared point by point with the FP64 oracle,

    |gpu - ref| <= 2^-46 sum|terms|,

sum|terms| being the point's condition scale (every addend of the as-written sums): the bound of the
saturated RHS's range test, which covers the roundings of about 40 additions in any order, each
at most 2^-53 of the scale.
"""
import numpy as np
import pytest

import oracle
from paper_2306_13002_gb300 import binding, inputs
from _parity import padded_dev, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILES = [None, (16, 8, 5, 2), (32, 16, 0, 0), (64, 4, 3, 2), (16, 16, 0, 3), (32, 4, 7, 0)]
TAYLOR = np.array([binding.TAYLOR8] * 3)


def _star_scale(u, a, c, halo=4):
    nz, ny, nx = (s - 2 * halo for s in u.shape)

    def at(d, o):
        s = [halo, halo, halo]
        s[2 - d] += o
        return np.abs(u[s[0]:s[0] + nz, s[1]:s[1] + ny, s[2]:s[2] + nx])

    tot = np.zeros((nz, ny, nx))
    for d in range(3):
        for o in range(1, 5):
            tot += abs(c[d][o - 1]) * (at(d, o) + 2 * at(d, 0) + at(d, -o))
    return tot * np.abs(a[halo:halo + nz, halo:halo + ny, halo:halo + nx])


def _star(u, a, c, tile, ud=None):
    nz, ny, nx = (s - 8 for s in u.shape)
    out = torch.full((nz, ny, nx), float("nan"), dtype=torch.float64, device="cuda")
    binding.acs_stencil_saturated(to_dev(u) if ud is None else ud, to_dev(a) if ud is None else padded_dev(a, ud.stride(1)),
                                  out, c, tile=tile)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _check_star(u, a, c, tile, what, ud=None):
    got, ref = _star(u, a, c, tile, ud), oracle.stencil(u, a, c, threads=4)
    bad = ~(np.abs(got - ref) <= 2.0 ** -46 * _star_scale(u, a, c))
    assert not bad.any(), (what, tile, int(bad.sum()), np.argwhere(bad)[:3], got[bad][:3], ref[bad][:3])


def _field(kind, shape, seed):
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
    base = rng.uniform(-1.0, 1.0, shape)
    if kind == "pulse":       # a Gaussian falling by 2^-150 within a few tiles
        r2 = sum((v - n / 3.0) ** 2 for v, n in zip((z, y, x), shape))
        return base * np.exp(-r2 / 9.0)
    if kind == "growing":     # the scale is outgrown every few planes
        return base * 2.0 ** (0.7 * z)
    if kind == "decaying":
        return base * 2.0 ** (-1.3 * z)
    if kind == "lumps":       # neighbouring cells 2^80 apart
        return base * 2.0 ** rng.integers(-60, 20, shape)
    if kind == "zeros":       # empty but for a slab near the end
        return np.where(z > 2 * shape[0] // 3, base, 0.0)
    if kind == "wave":
        return np.sin(0.61 * x + 0.1) * np.sin(0.57 * y + 0.2) * np.sin(0.7 * z + 0.3)
    return base


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("kind", ["plain", "pulse", "growing", "decaying", "lumps", "zeros", "wave"])
def test_star_fixed_ranges(kind, tile):
    nx, ny, nz = 45, 37, 41
    u = _field(kind, (nz + 8, ny + 8, nx + 8), 11)
    a = np.random.default_rng(12).uniform(-1.0, 1.0, u.shape)
    _check_star(u, a, TAYLOR, tile, kind)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("scale", [-1000, -700, 700, 1000])
def test_star_fixed_extreme_scales(scale, tile):
    """Inputs near both ends of the exponent range (the fixed-point scale covers 2^-500 .. 2^570)."""
    u, a = inputs.stencil_fields(33, 18, 13, seed=77)
    c = TAYLOR
    got = _star(u * 2.0 ** scale, a, c, tile) * 2.0 ** -scale
    ref = oracle.stencil(u, a, c)
    assert np.all(np.abs(got - ref) <= 2.0 ** -46 * _star_scale(u, a, c))


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 3), (17, 9, 2), (31, 16, 33), (65, 17, 6), (64, 32, 8)])
def test_star_fixed_tile_edges(dims, tile):
    nx, ny, nz = dims
    u, a = inputs.stencil_fields(nx, ny, nz, seed=500 + nx)
    for pitch in (nx + 8, nx + 9 + nx % 2, nx + 10 + nx % 2):   # odd and even row pitches
        _check_star(u, a, TAYLOR, tile, f"{dims} pitch {pitch}", padded_dev(u, pitch))


@pytest.mark.parametrize("tile", TILES)
def test_star_fixed_non_finite_and_unset_corners(tile):
    """NaN and infinities spread to the same points as in the as-written form and leave the others
    alone; halo corners, which no point reads, may hold anything."""
    nx, ny, nz = 50, 27, 22
    u, a = inputs.stencil_fields(nx, ny, nz, seed=81)
    z, y, x = np.meshgrid(*(np.arange(n) for n in u.shape), indexing="ij")
    outside = sum(((v < 4) | (v >= n - 4)).astype(int) for v, n in zip((z, y, x), u.shape))
    u[outside >= 2] = np.nan
    _check_star(np.where(outside >= 2, 0.0, u), a, TAYLOR, tile, "corners", None)
    got = _star(u, a, TAYLOR, tile)
    clean = np.where(outside >= 2, 0.0, u)
    assert np.all(np.abs(got - oracle.stencil(clean, a)) <= 2.0 ** -46 * _star_scale(clean, a, TAYLOR))
    u[12, 13, 30], u[20, 9, 8], u[4, 20, 44] = np.nan, np.inf, -np.inf
    got, ref = _star(u, a, TAYLOR, tile), oracle.stencil(u, a)
    fine = np.isfinite(ref)
    assert 0 < np.count_nonzero(~fine) < ref.size // 10 and np.array_equal(fine, np.isfinite(got))
    zero = np.where(np.isfinite(u), u, 0.0)
    assert np.all((np.abs(got - ref) <= 2.0 ** -46 * _star_scale(zero, a, TAYLOR))[fine])


@pytest.mark.parametrize("tile", [None, (16, 16, 0, 0)])
@pytest.mark.parametrize("c", [
    [[-w for w in binding.TAYLOR8]] * 3,                                  # the negative operator
    [[4.0 / 3.0, -1.0 / 12.0, 0.0, 0.0]] * 3,                             # fourth order
    [[w * s for w in binding.TAYLOR8] for s in (1.0, 7.0, 0.2)],          # a stretched grid
    [[1.0, 0.0, 0.0, 0.0], [2.0, 0.0, 0.0, 0.0], [0.5, 0.0, 0.0, 0.0]],   # second order
    [[w * 2.0 ** 90 for w in binding.TAYLOR8]] * 3,
    [[0.25, 0.25, 0.25, 0.25]] * 3,                                       # no alternating signs: FP64
    [[1.0, -1.0, 1.0, -1.0]] * 3,                                         # no centre: FP64
])
def test_star_fixed_weights(c, tile):
    u, a = inputs.stencil_fields(37, 21, 19, seed=91)
    _check_star(u - 0.5, a, np.array(c), tile, "weights")
