"""Limits of the double-precision integer spread and gather: what one grid
point can receive where the last tile is narrow, charges near the ends of the
FP64 range, systems whose charges crowd or differ so much that the integer
grid's quantum would show, rounding without a preferred sign, ranges of
particles, and the memory that a plan takes.

Tolerances as the other FP64 comparisons (1e-12 for grids, 5e-12 for particle
outputs) unless a test says otherwise."""
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


def _xi(L, M, P, most=0.7):
    return min(4.0, math.sqrt(most * 0.95 ** 2 * math.pi * M * M / (P * L * L)))


def _dev(a):
    return torch.tensor(a, device="cuda", dtype=torch.float64)


def _evaluate(x, q, L, xi, M, P, **kw):
    plan = se.Plan(len(q), L, xi, M, P, precision="fp64", **kw)
    xd, qd = _dev(x), _dev(q)
    plan.spread(xd, qd)
    H = plan.copy_grid(0).cpu().numpy()
    F, phi = torch.empty_like(xd), torch.empty_like(qd)
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.evaluate(xd, qd, F, phi, E)
    torch.cuda.synchronize()
    plan.close()
    return H, F.cpu().numpy(), phi.cpu().numpy(), E.item()


@pytest.mark.parametrize("M,P,tile,c", [(33, 24, 8, 10), (33, 8, 8, 14), (41, 8, 8, 60),
                                        (57, 16, 8, 30), (34, 8, 8, 15), (26, 24, 5, 10),
                                        (32, 8, 8, 60)])
def test_cluster_at_the_narrow_last_tile(M, P, tile, c):
    """c equal charges in each of the 27 tiles round the box's corner, within a
    cell of it where the last tile is one cell wide: every one of them reaches
    the corner's grid point with nearly its whole weight."""
    L = 2.0
    h = L / M
    a = np.array([1e-3, M - 1e-3, (M - M % tile if M % tile else M - 1) - 1e-3]) * h
    x = np.stack(np.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3).repeat(c, axis=0)
    q = np.ones(27 * c)      # not neutral: the k = 0 mode is dropped
    xi = _xi(L, M, P)
    H, F, phi, E = _evaluate(x, q, L, xi, M, P, tile=tile)
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64, grids=True)
    assert_close(H, r["H"], TOL, label="spread grid")
    assert_close(phi, r["phi"], 5 * TOL, label="phi")
    assert_close(F, r["F"], 5 * TOL, label="F", q=q)
    assert abs(E - r["E"]) < 5 * TOL * abs(r["E"])


def test_grid_beyond_the_range_gives_nan():
    """Finite charges whose grid or transform overflows: no finite number."""
    L, xi, M, P = 2.0, 3.0, 24, 8
    x, q = systems.uniform_charges(200, L, seed=5)
    plan = se.Plan(len(q), L, xi, M, P, precision="fp64")
    xd = _dev(x)
    F, phi = torch.empty_like(xd), torch.empty(len(q), dtype=torch.float64, device="cuda")
    for scale in (1e306, 1e307):
        plan.evaluate(xd, _dev(q * scale), F, phi)
        assert not phi.isfinite().any() and not F.isfinite().any()
    plan.evaluate(xd, _dev(q), F, phi)   # and the next call is as any other
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64)
    assert_close(phi.cpu().numpy(), r["phi"], 5 * TOL, label="phi")
    plan.close()


@pytest.mark.parametrize("scale", [1e-300, 1e-295, 1e295, 1e300])
def test_charges_near_the_ends_of_the_range(scale):
    """Results keep their digits where products of two scales would be
    subnormal or overflow."""
    L, xi, M, P = 2.0, 3.0, 24, 8
    x, q = systems.uniform_charges(200, L, seed=5)
    H, F, phi, _ = _evaluate(x, q * scale, L, xi, M, P)
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64, grids=True)
    assert_close(H / scale, r["H"], TOL, label="spread grid")
    assert_close(phi / scale, r["phi"], 5 * TOL, label="phi")


@pytest.mark.parametrize("n,P", [(20000, 8), (20000, 16)])
def test_many_charges_of_both_signs_in_one_place(n, P):
    """20 000 unit charges of alternating sign in eight cells.  The potential is
    what their weights' cancellation leaves: rounding each weight to 2^-53 of
    itself leaves sqrt(n sum w^2) 2^-53 of net charge, below 1e-13 of the
    potential here; rounding it to 2^-45 of the largest weight, 1e-12."""
    L, M = 2.0, 24
    rng = np.random.default_rng(1)
    x = np.vstack([0.31 + 2 * L / M * rng.random((n, 3)), L * rng.random((200, 3))])
    q = np.where(np.arange(n + 200) % 2 == 0, 1.0, -1.0)
    xi = _xi(L, M, P)
    H, F, phi, E = _evaluate(x, q, L, xi, M, P)
    r = oracle.se_kspace(x, q, L, xi, M, P, cell_mode=64, grids=True)
    assert np.linalg.norm(phi - r["phi"]) < 1e-13 * np.linalg.norm(r["phi"])
    assert np.linalg.norm(F - r["F"]) < 1e-13 * np.linalg.norm(r["F"])
    assert abs(E - r["E"]) < 1e-13 * abs(r["E"])


@pytest.mark.parametrize("big", [1.0, 30.0, 1e4, 1e8, 1e15])
@pytest.mark.parametrize("P", [4, 8, 24])
def test_grid_of_small_charges_beside_a_large_one(big, P):
    """Grid points that only the small charges reach keep their digits."""
    L, M = 2.0, 64
    rng = np.random.default_rng(3)
    x = np.vstack([[[0.05 * L] * 3], L * (0.45 + 0.2 * rng.random((400, 3)))])
    q = np.concatenate([[big], rng.uniform(-1, 1, 400)])
    H, _, _, _ = _evaluate(x, q, L, _xi(L, M, P), M, P)
    r = oracle.se_kspace(x, q, L, _xi(L, M, P), M, P, cell_mode=64, grids=True)["H"]
    s = slice(M // 3, 5 * M // 6)    # beyond the large charge's support
    assert_close(H[s, s, s], r[s, s, s], TOL, label="spread grid")


@pytest.mark.parametrize("P", [4, 8])
def test_gather_errors_have_no_preferred_sign(P):
    """The sums' intermediate results are rounded, not cut: over 500 particles
    the mean error of a field component stays below its spread (cutting makes
    it 2.6 times as large at P = 4).  Reference: the sums over the plan's own
    grid in extended precision."""
    L, M, n = 2.0, 24, 500
    x, q = systems.uniform_charges(n, L, seed=7)
    q = np.sign(q)
    xi = _xi(L, M, P)
    plan = se.Plan(n, L, xi, M, P, precision="fp64")
    xd, qd = _dev(x), _dev(q)
    F = torch.empty_like(xd)
    plan.evaluate(xd, qd, F)
    Ht = plan.copy_grid(1).cpu().numpy()
    p = plan.params()
    plan.close()
    ld = np.longdouble
    beta = ld(p["alpha"]) * ld(p["h"]) ** 2
    c = np.floor(x * M / L).astype(int)
    a = np.arange(P)
    dz = (a - ld(P - 1) / 2)[None, :, None] - (x.astype(ld) * M / ld(L) - c - ld(0.5))[:, None, :]
    g = np.exp(-beta * dz ** 2)
    gd = g * dz
    idx = (c[:, None, :] - P // 2 + 1 + a[None, :, None]) % M
    err = np.empty((n, 3))
    for i in range(n):
        V = Ht[np.ix_(*idx[i].T)].astype(ld)
        for d in range(3):
            w = [gd[i, :, k] if k == d else g[i, :, k] for k in range(3)]
            ref = (((V * w[2]).sum(2) * w[1]).sum(1) * w[0]).sum()
            ref *= ld(-2.0) * ld(p["alpha"]) * ld(p["h"]) ** 4 * ld(p["cg"]) * ld(q[i])
            err[i, d] = float((ld(F[i, d].item()) - ref) * ld(q[i]))
    assert (np.abs(err.mean(0)) < err.std(0)).all(), (err.mean(0), err.std(0))


def test_ranges_gather_from_the_plans_copies():
    """More particles than one range of window factors holds (4 GB at 1792
    bytes a particle).  Results of a second range are those of any other
    particle, and the gather needs the positions and charges of the spread no
    more: writing the potential over the charges, or changing the positions
    between the steps, changes nothing."""
    L, M, P, N = 3.0, 40, 32, 2_500_000
    g = torch.Generator(device="cuda").manual_seed(1)
    x = L * torch.rand(N, 3, generator=g, device="cuda", dtype=torch.float64)
    q = torch.where(torch.arange(N, device="cuda") % 2 == 0, 1.0, -1.0).double()
    plan = se.Plan(N, L, _xi(L, M, P), M, P, precision="fp64")
    F, phi = torch.empty_like(x), torch.empty_like(q)
    plan.evaluate(x, q, F, phi)
    # the same grid seen by particles of both ends of the tile order, as a
    # system of test charges too small to change it
    Ht = plan.copy_grid(1)
    p = plan.params()
    beta = p["alpha"] * p["h"] ** 2
    s = torch.randperm(N, generator=torch.Generator().manual_seed(2))[:4000].cuda()
    c = torch.floor(x[s] * (M / L)).long()
    a = torch.arange(P, device="cuda")
    dz = (a - (P - 1) / 2)[None, :, None] - (x[s] * (M / L) - c - 0.5)[:, None, :]
    w = torch.exp(-beta * dz ** 2)
    idx = (c[:, None, :] - P // 2 + 1 + a[None, :, None]) % M
    ref, refF = torch.empty(4000, device="cuda").double(), torch.empty(4000, 3, device="cuda").double()
    for k in range(0, 4000, 100):
        i, v = idx[k:k + 100], w[k:k + 100]
        V = Ht[i[:, :, None, None, 0], i[:, None, :, None, 1], i[:, None, None, :, 2]]
        ref[k:k + 100] = torch.einsum("nabc,na,nb,nc->n", V, v[..., 0], v[..., 1], v[..., 2])
        for d in range(3):
            u = [v[..., e] * dz[k:k + 100, :, e] if e == d else v[..., e] for e in range(3)]
            refF[k:k + 100, d] = torch.einsum("nabc,na,nb,nc->n", V, *u)
    ref *= p["h"] ** 3 * p["cg"]
    refF *= -2 * p["alpha"] * p["h"] ** 4 * p["cg"] * q[s][:, None]
    assert_close(phi[s].cpu().numpy(), ref.cpu().numpy(), 5 * TOL, label="phi")
    assert_close(F[s].cpu().numpy(), refF.cpu().numpy(), 5 * TOL, label="F", q=q[s].cpu().numpy())
    q2, F2 = q.clone(), torch.empty_like(x)
    plan.set_graph(False)
    plan.evaluate(x, q2, F2, q2)      # phi over q
    assert torch.equal(q2, phi) or float((q2 - phi).norm() / phi.norm()) < TOL
    assert float((F2 - F).norm() / F.norm()) < TOL
    plan.spread(x, q)
    plan.scale()
    x2 = x.clone().roll(1, 0)
    plan.gather(x2, q, phi=q2, F=F2)
    assert float((q2 - phi).norm() / phi.norm()) < TOL
    assert float((F2 - F).norm() / F.norm()) < TOL
    plan.close()


def test_memory_of_a_plan():
    """Only the integer spread has a padded integer grid, and the gather's copy
    of the grid shares the spectrum's memory."""
    M, N = 256, 10

    def used(P, **kw):
        plan = se.Plan(N, 3.0, 1.0, M, P, precision="fp64", **kw)
        x = 3.0 * torch.rand(N, 3, device="cuda", dtype=torch.float64)
        q = torch.rand(N, device="cuda", dtype=torch.float64) - 0.5
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        plan.spread(x, q)
        torch.cuda.synchronize()
        free -= torch.cuda.mem_get_info()[0]
        plan.close()
        return free

    used(8)                    # loads the kernels
    mb = 1 << 20
    grid, pad = 8 * M ** 3, 8 * (M + 31) ** 3
    direct = used(32, spread_variant=2)
    assert abs(used(32, spread_variant=1) - direct - pad) < 8 * mb
    assert direct - used(2, spread_variant=2) < pad - grid + 8 * mb


@pytest.mark.parametrize("N,M,P,few", [(0, 128, 4, True), (2, 129, 2, True), (100, 128, 4, True),
                                       (700, 160, 8, True), (700, 128, 8, False),
                                       (10, 33, 16, False)])
def test_few_particles_on_a_large_grid(N, M, P, few):
    """The FP64 path that few particles take gives what the integer one (variant
    1) gives, in every mode of evaluation."""
    L = 2.0
    x, q = systems.uniform_charges(max(N, 1), L, seed=N + M)
    xd, qd = _dev(x[:N].reshape(N, 3)), _dev(q[:N])
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    out = {}
    for variant in (0, 1):
        plan = se.Plan(N, L, _xi(L, M, P), M, P, precision="fp64", spread_variant=variant)
        assert plan.params()["spread_variant"] == (2 if few and variant == 0 else 1)
        r = []
        for mode in ("analytic", "ik"):
            plan.set_force_mode(mode)
            F, phi, E = torch.empty_like(xd), torch.empty_like(qd), torch.zeros_like(one)
            plan.evaluate(xd, qd, F, phi, E)
            phi1, E0 = torch.empty_like(qd), torch.zeros_like(one)
            plan.evaluate(xd, qd, None, phi1, None)
            plan.evaluate(xd, qd, None, None, E0)
            gx, gq = torch.empty_like(xd), torch.empty_like(qd)
            plan.adjoint(xd, qd, one, gx, gq)
            r += [F, phi, E, phi1, E0, gx, gq, plan.copy_grid(1)]
            plan.spread(xd, qd)
            r.append(plan.copy_grid(0))
        out[variant] = [t.cpu().numpy() for t in r]
        plan.close()
    for a, b in zip(out[0], out[1]):
        assert np.linalg.norm(a - b) <= 5 * TOL * np.linalg.norm(b)
