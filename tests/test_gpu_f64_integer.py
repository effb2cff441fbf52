"""The double-precision spread and gather (integer arithmetic on split numbers)
where they can go wrong: every support, tile edges that do and do not divide the
grid, tiles and cells with more particles than the integer grid has bits for,
few particles, charges far from one, flat windows (the gather's scales), several
ranges of particles, and input beyond the range or not finite.

Tolerances as the other FP64 comparisons: 1e-12 for the grid (weights are
multiples of 2^-54 or less of the largest charge's, or FP64 numbers), 5e-12 for
particle outputs."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1712_04718_gb300 import se, systems
from parity import assert_close

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _check(x, q, L, xi, M, P, tile=0, scale=1.0, eta=None):
    plan = se.Plan(len(q), L, xi, M, P, precision="fp64", tile=tile, eta=eta)
    xd, qd = torch.tensor(x, device="cuda"), torch.tensor(q * scale, device="cuda")
    plan.spread(xd, qd)
    H = plan.copy_grid(0).cpu().numpy()
    E, F, phi = plan.energy_force(xd, qd)
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    gx, gq = torch.empty_like(xd), torch.empty_like(qd)
    plan.adjoint(xd, qd, one, gx, gq)
    torch.cuda.synchronize()
    plan.close()
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64, grids=True,
                         **({} if eta is None else {"eta": eta}))
    assert_close(H / scale, r["H"], TOL, label="spread grid")
    assert_close(phi.cpu().numpy() / scale, r["phi"], 5 * TOL, label="phi")
    assert_close(F.cpu().numpy() / scale / scale, r["F"], 5 * TOL, label="F")
    assert abs(E / scale / scale - r["E"]) < 5 * TOL * abs(r["E"])
    assert torch.equal(gx, -F) and torch.equal(gq, phi)


def _xi(L, M, P, most=0.7):
    return min(4.0, math.sqrt(most * 0.95 ** 2 * math.pi * M * M / (P * L * L)))


@pytest.mark.parametrize("P", list(range(2, 34, 2)))
def test_every_support(P):
    """A grid that is no multiple of the tile, 301 charges (neutral)."""
    L, M = 2.0, max(19, P + 3)
    x, q = systems.uniform_charges(301, L, seed=P)
    q[-1] = -q[:-1].sum()
    _check(x, q, L, _xi(L, M, P), M, P)


@pytest.mark.parametrize("M,P,tile", [(33, 8, 2), (33, 8, 3), (33, 8, 9), (33, 8, 16), (40, 24, 5),
                                      (40, 24, 16), (48, 32, 8), (48, 32, 32), (12, 12, 8)])
def test_tile_edges(M, P, tile):
    x, q = systems.uniform_charges(400, 2.0, seed=tile)
    _check(x, q, 2.0, _xi(2.0, M, P), M, P, tile=tile)


@pytest.mark.parametrize("P", [4, 8, 10, 16, 24])
@pytest.mark.parametrize("n", [1, 2, 27, 28, 29, 57, 700])
def test_crowded_cell(P, n):
    """n charges of one sign in one cell (the words' sums are largest where
    weights coincide), the opposite charge spread over the box."""
    rng = np.random.default_rng(n)
    L, M = 2.0, 26
    xc = 0.31 + 1e-3 * rng.random((n, 3))
    xr = L * rng.random((40, 3))
    q = np.concatenate([np.ones(n), np.full(40, -n / 40.0)])
    _check(np.vstack([xc, xr]), q, L, _xi(L, M, P), M, P)


@pytest.mark.parametrize("scale", [1e-80, 2.0 ** -40, 3.0, 1e70])
def test_charge_scale(scale):
    x, q = systems.uniform_charges(200, 2.0, seed=5)
    _check(x, q, 2.0, 3.0, 24, 8, scale=scale)


@pytest.mark.parametrize("P,eta", [(8, 0.97), (32, 0.9), (16, 0.05)])
def test_window_shapes(P, eta):
    """Wide and narrow windows: the bounds of the factors' sums change."""
    x, q = systems.uniform_charges(200, 2.0, seed=6)
    _check(x, q, 2.0, 1.5, 40, P, eta=eta)


def test_unlike_charges():
    """Charges from 1e-6 to 1."""
    x, q = systems.uniform_charges(300, 2.0, seed=7)
    q *= 10.0 ** -np.random.default_rng(7).uniform(0, 6, 300)
    q[-1] -= q.sum()
    _check(x, q, 2.0, 3.0, 28, 10)


def test_several_ranges():
    """More particles than one range of window factors holds (4 GB at 1792
    bytes a particle): the grid is the sum of the halves' grids, and 1/2 sum
    q phi over all of them is the energy of the grid (Parseval)."""
    L, M, P, N = 3.0, 40, 32, 2_500_000
    g = torch.Generator(device="cuda").manual_seed(1)
    x = L * torch.rand(N, 3, generator=g, device="cuda", dtype=torch.float64)
    q = torch.where(torch.arange(N, device="cuda") % 2 == 0, 1.0, -1.0).double()
    xi, half = _xi(L, M, P), N // 2
    whole = se.Plan(N, L, xi, M, P, precision="fp64")
    part = se.Plan(half, L, xi, M, P, precision="fp64")
    whole.spread(x, q)
    H = whole.copy_grid(0)
    S = torch.zeros_like(H)
    for s in (slice(0, half), slice(half, N)):
        part.spread(x[s].contiguous(), q[s].contiguous())
        S += part.copy_grid(0)
    assert float((H - S).norm() / S.norm()) < TOL
    E, F, phi = whole.energy_force(x, q)
    e = 0.5 * float((q * phi).sum())
    assert abs(E - e) < 5 * TOL * abs(E)
    Eg = torch.zeros(1, dtype=torch.float64, device="cuda")
    whole.spread(x, q)
    whole.scale(Eg)
    assert abs(E - Eg.item()) < 5 * TOL * abs(E)
    whole.close()
    part.close()


@pytest.mark.parametrize("scale", [1e-200, 1e-150, 1e150, 1e200])
def test_potential_beyond_the_energys_range(scale):
    """Charges whose energy underflows or overflows still have a potential."""
    L, xi, M, P = 2.0, 3.0, 24, 8
    x, q = systems.uniform_charges(200, L, seed=5)
    plan = se.Plan(len(q), L, xi, M, P, precision="fp64")
    xd, qd = torch.tensor(x, device="cuda"), torch.tensor(q * scale, device="cuda")
    F, phi = torch.empty_like(xd), torch.empty_like(qd)
    plan.evaluate(xd, qd, F, phi)
    torch.cuda.synchronize()
    plan.close()
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64)
    assert_close(phi.cpu().numpy() / scale, r["phi"], 5 * TOL, label="phi")


@pytest.mark.parametrize("where,value", [("x", float("nan")), ("x", float("inf")),
                                         ("q", float("nan")), ("q", float("-inf"))])
def test_nonfinite_input_gives_nan(where, value):
    """A call that does not read the status sees it in the results, and the
    next call with finite input is as any other."""
    L, xi, M, P = 2.0, 3.0, 24, 8
    x, q = systems.uniform_charges(200, L, seed=5)
    plan = se.Plan(len(q), L, xi, M, P, precision="fp64")
    xd, qd = torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda")
    F, phi = torch.empty_like(xd), torch.empty_like(qd)
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    xb, qb = xd.clone(), qd.clone()
    if where == "x":
        xb[7, 1] = value
    else:
        qb[7] = value
    plan.evaluate(xb, qb, F, phi, E)
    assert bool(F.isnan().all()) and bool(phi.isnan().all()) and bool(E.isnan())
    plan.evaluate(xd, qd, F, phi, E)
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64)
    assert_close(phi.cpu().numpy(), r["phi"], 5 * TOL, label="phi")
    plan.close()
