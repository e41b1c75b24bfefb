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
    with np.errstate(all="ignore"):
        near = np.abs(got - ref) <= 2.0 ** -46 * _star_scale(zero, a, TAYLOR)
    assert np.all(near[fine])


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


# ------------------------------------------------------------------------------------------ RHS

RHS_TILES = [None, (16, 16, 6, 2), (32, 8, 0, 1), (16, 8, 0, 3), (16, 8, 5, 0)]


def _rhs_scale(U, gamma, eps, h):
    """sum|terms| of every component: fluxes with every addend's magnitude, and the dissipation's."""
    g1 = abs(gamma - 1.0)
    A = np.abs(U)
    with np.errstate(all="ignore"):
        v = A[1:4] / A[0]
        P = g1 * (A[4] + 0.5 * (A[1:4] * v).sum(0))
        F = [np.stack([A[1 + d]] + [A[1 + c] * v[d] + (P if c == d else 0.0) for c in range(3)] + [(A[4] + P) * v[d]])
             for d in range(3)]
    inner = (slice(None),) + (slice(2, -2),) * 3
    tot = np.zeros_like(U[inner])
    for d in range(3):
        ax = 3 - d

        def at(x, o):
            return np.roll(x, -o, axis=ax)[inner]

        tot += (at(F[d], 1) + at(F[d], -1)) / (2 * abs(h[d]))
        tot += abs(eps) * (at(A, 2) + 4 * at(A, 1) + 6 * at(A, 0) + 4 * at(A, -1) + at(A, -2))
    return tot


def _rhs(U, tile, gamma, eps, h):
    _, Z, Y, X = U.shape
    R = torch.full((5, Z - 4, Y - 4, X - 4), float("nan"), dtype=torch.float64, device="cuda")
    binding.acs_rhs_saturated(to_dev(U), R, gamma, eps, h, tile=tile)
    torch.cuda.synchronize()
    return R.cpu().numpy()


def _check_rhs(U, tile, what, gamma=1.4, eps=0.25, h=(1.0, 1.0, 1.0)):
    got, ref = _rhs(U, tile, gamma, eps, h), oracle.rhs(U, gamma=gamma, eps=eps, h=h, threads=8)
    bad = ~(np.abs(got - ref) <= 2.0 ** -46 * _rhs_scale(U, gamma, eps, h))
    assert not bad.any(), (what, tile, int(bad.sum()), np.argwhere(bad)[:3], got[bad][:3], ref[bad][:3])


def _flow(kind, nx, ny, nz, seed):
    U = inputs.rhs_field(nx, ny, nz, halo=2, seed=seed)
    z, y, x = np.meshgrid(*(np.arange(n) for n in U.shape[1:]), indexing="ij")
    rng = np.random.default_rng(seed)
    if kind == "shock":             # a jump of 2^12 in density and energy
        jump = np.where(x + y + z > (nx + ny + nz) // 2, 2.0 ** 12, 1.0)
        U = U * jump
    elif kind == "ramp":            # outgrows the scale every other plane
        U = U * 2.0 ** (0.5 * z)
    elif kind == "fall":
        U = U * 2.0 ** (-0.5 * z)
    elif kind == "rest":
        U[1:4] = 0.0
    elif kind == "slow":            # momenta far below the other components
        U[1:4] *= 2.0 ** -70
    elif kind == "fast":            # momenta far above
        U[1:4] *= 2.0 ** 20
    elif kind == "lumps":
        U[1:4] *= 2.0 ** rng.integers(-60, 1, U[1:4].shape)
        U[0] *= 2.0 ** rng.integers(-4, 4, U[0].shape)
    elif kind == "negative":        # nothing keeps the signs of a state apart
        U = U * rng.choice([-1.0, 1.0], U.shape)
    elif kind == "large":
        U = U * 2.0 ** 150
    elif kind == "small":
        U = U * 2.0 ** -190
    return U


@pytest.mark.parametrize("tile", RHS_TILES)
@pytest.mark.parametrize("kind", ["plain", "shock", "ramp", "fall", "rest", "slow", "fast", "lumps", "negative", "large",
                                  "small"])
def test_rhs_fixed_ranges(kind, tile):
    """Grids large enough for the fixed-point march (two planes per resident block)."""
    _check_rhs(_flow(kind, 83, 70, 37, 21), tile, kind)


@pytest.mark.parametrize("tile", RHS_TILES)
@pytest.mark.parametrize("prm", [
    {"gamma": 5.0 / 3.0, "eps": 0.03, "h": (0.37, 0.37, 0.37)}, {"gamma": 1.1, "eps": 0.25, "h": (0.2, 1.0, 3.0)},
    {"eps": 1e-9}, {"eps": 0.0}, {"eps": -0.25}, {"h": (-1.0, 1.0, 1.0)}, {"gamma": 1.0}, {"gamma": 0.5},
    {"eps": 40.0}, {"h": (2.0 ** -80,) * 3, "eps": 2.0 ** 78}, {"h": (1e-5, 1.0, 1.0)},
])
def test_rhs_fixed_parameters(prm, tile):
    _check_rhs(_flow("plain", 67, 50, 49, 22), tile, str(prm), **prm)


@pytest.mark.parametrize("tile", RHS_TILES)
@pytest.mark.parametrize("dims", [(17, 16, 400), (31, 33, 160), (64, 48, 60), (1, 1, 700), (15, 90, 120), (160, 2, 70)])
def test_rhs_fixed_tile_edges(dims, tile):
    """One, all but one and all columns and rows of the last tile."""
    _check_rhs(_flow("plain", *dims, 23), tile, dims, h=(1.0, 0.5, 2.0))
    _check_rhs(_flow("plain", *dims, 24), tile, dims)


@pytest.mark.parametrize("tile", RHS_TILES)
def test_rhs_fixed_non_finite_and_unset_corners(tile):
    U = _flow("plain", 70, 61, 40, 25)
    z, y, x = np.meshgrid(*(np.arange(n) for n in U.shape[1:]), indexing="ij")
    outside = sum(((v < 2) | (v >= n - 2)).astype(int) for v, n in zip((z, y, x), U.shape[1:]))
    clean = U.copy()
    U[:, outside >= 2] = np.nan
    got, ref = _rhs(U, tile, 1.4, 0.25, (1.0,) * 3), oracle.rhs(clean, threads=8)
    scale = _rhs_scale(clean, 1.4, 0.25, (1.0,) * 3)
    assert np.all(np.abs(got - ref) <= 2.0 ** -46 * scale)
    U[0, 20, 30, 33], U[4, 9, 50, 60], U[2, 38, 12, 7] = np.nan, np.inf, -np.inf
    U[0, 30, 10, 50] = 0.0
    got, ref = _rhs(U, tile, 1.4, 0.25, (1.0,) * 3), oracle.rhs(U, threads=8)
    fine = np.isfinite(ref)
    assert 0 < np.count_nonzero(~fine) < ref.size // 10 and np.array_equal(fine, np.isfinite(got))
    with np.errstate(all="ignore"):
        far = np.abs(got - ref) <= 2.0 ** -46 * scale * 4.0   # neighbours of the changed cells have larger terms
    assert np.all(far[fine & (scale < 30.0)])


# --------------------------------------------------------------------------- ranker training

@pytest.mark.parametrize("n,F", [(8, 1), (9, 5), (63, 20), (64, 20), (65, 20), (400, 20), (430, 7), (100, 92), (57, 93),
                                 (1200, 20)])
def test_ranker_one_launch_training(n, F):
    """The one-launch training (64 hidden units, what fits shared memory; the last two sizes are past its
    limits) against Adam steps formed here from acs_ranker_gradient at the same parameters. Each update
    is lr times a ratio of moments computed in about ten FP32 roundings (below 1e-6 of it), and each
    parameter is rounded once per epoch; 1e-5 lr and 2^-22 |p| per epoch bound both, with room for the
    later gradients, which see the differences of earlier steps."""
    rng = np.random.default_rng(n)
    H, lr, epochs, FW = 64, 3e-3, 6, 1.0
    X = to_dev(rng.uniform(0.0, 100.0, (n, F)).astype(np.float32))
    T = to_dev((2.0 + rng.uniform(0.0, 1.0, n)).astype(np.float32))
    P = binding.acs_ranker_param_count(F, H)
    ws = torch.empty(binding.acs_ranker_workspace_bytes(n, F, H) // 4 + 4, dtype=torch.float32, device="cuda")

    def train(e):
        params = torch.full((P,), float("nan"), dtype=torch.float32, device="cuda")
        binding.acs_ranker_train(X, T, params, ws, hidden=H, epochs=e, lr=lr, fast_weight=FW)
        return params

    p = train(0)
    m = np.zeros(P)
    v = np.zeros(P)
    g = torch.empty(P, dtype=torch.float32, device="cuda")
    fixed = 2 * F + 2   # the statistics are not trained
    for e in range(1, epochs + 1):
        binding.acs_ranker_gradient(X, T, p, g, ws, hidden=H, fast_weight=FW)
        gn = g.cpu().numpy().astype(np.float64)
        m, v = 0.9 * m + 0.1 * gn, 0.999 * v + 0.001 * gn * gn
        step = lr * (m / (1 - 0.9 ** e)) / (np.sqrt(v / (1 - 0.999 ** e)) + 1e-8)
        step[:fixed] = 0.0
        p = train(e)
        want = (train(e - 1).cpu().numpy().astype(np.float64) - step)
        got = p.cpu().numpy()
        assert np.all(np.abs(got - want) <= e * (1e-5 * lr + 2.0 ** -22 * np.abs(want))), (e, np.abs(got - want).max())
    assert torch.equal(p, train(epochs))
