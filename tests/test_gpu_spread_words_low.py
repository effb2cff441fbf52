"""The low word of the single-precision tile spread (variant 1).  Unit charges of
both signs at the same positions cancel to the last bit in either word; what
small charges in the same tile leave on the grid lies far below one unit of the
high word (2^-22 to 2^-21 of the largest weight) and is the low word's alone.

Tolerance 1e-3 of the small charges' grid: a weight is kept to 2^-44 of the
largest charge's (2^-43 and a factor of two for the power of two above 256
particles), ten small charges meet in a point, and their mean weight is 0.05
2^-26: 10^(1/2) 2^-43 / (0.05 2^-26) = 5e-4."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1712_04718_gb300 import se
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("P", [4, 8, 16])
@pytest.mark.parametrize("pairs", [1, 60, 123, 124, 251])    # 256 | 258 and 512 particles
def test_small_charges_under_cancelling_ones(P, pairs):
    L, M, n = 2.0, 24, 10
    rng = np.random.default_rng(pairs)
    cell = 8 * L / M                                         # one tile
    xp = (cell * (0.02 + 0.9 * rng.random((pairs, 3)))).astype(np.float32)
    xs = (cell * (0.3 + 0.4 * rng.random((n, 3)))).astype(np.float32)
    qs = np.full(n, 2.0 ** -26, np.float32)
    x = np.vstack([xp, xp, xs])
    q = np.concatenate([np.ones(pairs), -np.ones(pairs), qs]).astype(np.float32)
    xi = min(4.0, math.sqrt(0.7 * 0.95 ** 2 * math.pi * M * M / (P * L * L)))
    plan = se.Plan(len(q), L, xi, M, P, precision="fp32", spread_variant=1)
    plan.spread(torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda"))
    H = plan.copy_grid(0).double().cpu().numpy()
    plan.close()
    r = oracle.se_kspace(xs.astype(np.float64), qs.astype(np.float64), L, xi, M, P, cell_mode=32,
                         grids=True)["H"]
    assert_close(H, r, 1e-3, label="spread grid")
