"""The single-precision tile spread's integer words (variant 1): tiles at the
limits of their scales and of the rule that takes compensated sums instead,
charges far from one and far from each other, several x-slabs a tile.

Tolerance 2e-5 of the grid, as for the other single-precision grids: a position
in grid units carries a rounding of M 2^-25 (1.4e-6 at M = 48), which the window's
slope multiplies by up to about ten; the words add 2^-44."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1712_04718_gb300 import se, systems
from parity import assert_close

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _grid(x, q, L, xi, M, P, tile=8):
    plan = se.Plan(len(q), L, xi, M, P, precision="fp32", spread_variant=1, tile=tile)
    xd, qd = torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda")
    plan.spread(xd, qd)
    H = plan.copy_grid(0).double().cpu().numpy()
    plan.close()
    return H


def _check(x, q, M, P, tile=8, scale=1.0, L=2.0):
    xi = min(4.0, math.sqrt(0.7 * 0.95 ** 2 * math.pi * M * M / (P * L * L)))
    x, q = x.astype(np.float32), q.astype(np.float32)
    H = _grid(x, q * np.float32(scale), L, xi, M, P, tile)
    r = oracle.se_kspace(x.astype(np.float64), q.astype(np.float64), L, xi, M, P, cell_mode=32,
                         grids=True)
    assert_close(H / float(np.float32(scale)), r["H"], TOL, label="spread grid")


@pytest.mark.parametrize("P", [4, 8, 16])
@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 472, 473, 700])
def test_crowded_tile(P, n):
    """n charges of one sign in one cell and 40 around them in the same tile
    (512 and 513 particles among the counts)."""
    rng = np.random.default_rng(n)
    L, M = 2.0, 24
    xc = 0.31 + 1e-3 * rng.random((n, 3))
    xr = 8 * L / M * rng.random((40, 3))
    q = np.concatenate([np.ones(n), np.full(40, -n / 40.0)])
    _check(np.vstack([xc, xr]), q, M, P)


@pytest.mark.parametrize("scale", [1e-24, 1e-18, 2.0 ** -40, 3.0, 1e18, 1e24])
def test_charge_scale(scale):
    x, q = systems.uniform_charges(200, 2.0, seed=5)
    _check(x, q, 24, 8, scale=scale)


@pytest.mark.parametrize("M,P,tile", [(33, 8, 2), (33, 8, 16), (40, 24, 5), (40, 24, 16), (48, 32, 32)])
def test_tile_edges(M, P, tile):
    x, q = systems.uniform_charges(400, 2.0, seed=tile)
    _check(x, q, M, P, tile=tile)


def test_unlike_charges():
    """The words' scale is the tile's own: what a tile of charges of 1e-6 adds
    does not depend on charges elsewhere, to the last bit."""
    rng = np.random.default_rng(3)
    L, M, P = 2.0, 40, 4
    x = np.vstack([0.35 * rng.random((60, 3)) + 0.02, 1.2 + 0.35 * rng.random((60, 3))])
    q = 1e-6 * rng.standard_normal(120)
    x, q = x.astype(np.float32), q.astype(np.float32)
    H = _grid(x, q, L, 3.0, M, P)
    q[60:] *= 1e6
    H2 = _grid(x, q, L, 3.0, M, P)
    assert np.array_equal(H[:12, :12, :12], H2[:12, :12, :12])
    assert not np.array_equal(H, H2)


def test_nonfinite_charge_gives_nan():
    x, q = systems.uniform_charges(200, 2.0, seed=5, dtype=np.float32)
    q[7] = np.nan
    assert np.isnan(_grid(x, q, 2.0, 3.0, 24, 8)).any()
