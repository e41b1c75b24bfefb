"""Limits of the fixed-point marches: what ends a segment, and what its values may be.

Bounds as in test_gpu_fixed.py: |gpu - ref| <= 2^-46 sum|terms| at every point, unless a test says
otherwise.
"""
import numpy as np
import pytest

from paper_2306_13002_gb300 import inputs
from test_gpu_fixed import RHS_TILES, TAYLOR, TILES, _check_rhs, _star

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
