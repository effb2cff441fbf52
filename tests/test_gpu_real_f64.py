"""The double-precision real-space kernel where its pair table and its
single-precision distance test can go wrong: pairs at the edges of the
table's octaves and beyond its ends (v = xi^2 r^2 below 2^-5 and above 2^6),
pairs at the cut-off, across the box's faces, and cells whose particle counts
leave a warp or a chunk of candidates partly filled.

Tolerance: rounding only.  A pair's terms carry the relative error of v
(a few 2^-53) times their sensitivity, at most v + 1 (e^{-v}): 1e-12 up to v
of 1000; sums as the other FP64 comparisons, 1e-12."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1712_04718_gb300 import se
from parity import assert_close

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _run(x, q, L, xi, rc):
    rs = se.RealSpace(len(q), L, xi, rc, precision="fp64")
    xd, qd = torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda")
    F, phi = torch.empty_like(xd), torch.empty_like(qd)
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    rs.evaluate(xd, qd, F, phi, E)
    torch.cuda.synchronize()
    rs.close()
    return F.cpu().numpy(), phi.cpu().numpy(), E.item()


EDGES = [2.0 ** -5, 0.5, 1.0, 8.0, 16.0, 32.0, 64.0]


@pytest.mark.parametrize("v", [1e-6, 1e-3, 3.0, 11.6, 24.0, 48.0, 80.0]
                         + [e * (1 + s * 1e-9) for e in EDGES for s in (-1, 1)])
def test_one_pair(v):
    L, rc, xi = 3.0, 1.0, 9.5     # v at the cut-off: 90
    r = math.sqrt(v) / xi
    d = np.array([0.36, -0.48, 0.8])   # a unit vector
    for a in ([1.5, 1.5, 1.5], [0.01, 2.99, 1.0]):   # inside, and across two faces
        x = np.stack([np.array(a), np.array(a) + r * d])
        x -= L * np.floor(x / L)
        q = np.array([1.0, -0.7])
        F, phi, E = _run(x, q, L, xi, rc)
        w = oracle.ewald_real(x, q, L, xi, rc)
        assert np.abs(F - w["F_real"]).max() < TOL * np.abs(w["F_real"]).max()
        self_phi = 2 * xi / math.sqrt(math.pi) * np.abs(q).max()
        assert np.abs(phi - w["phi_real"] - w["phi_self"]).max() < TOL * self_phi
        assert abs(E - w["E_real"] - w["E_self"]) < TOL * (abs(w["E_self"]) + abs(w["E_real"]))


def test_pairs_at_the_cut_off():
    """Distances a rounding of single precision away from r_c on both sides:
    the sum takes exactly the pairs with r < r_c."""
    L, rc, xi = 3.0, 1.0, 1.0     # erfc(xi rc) = 0.16: a pair taken or missed shows
    for k in (-30, -3, -1, 1, 3, 30):
        r = rc * (1 + k * 2.0 ** -26)
        x = np.array([[2.5, 0.3, 1.7], [2.5 + r - L, 0.3, 1.7]])
        q = np.array([1.0, 1.0])
        F, _, _ = _run(x, q, L, xi, rc)
        w = oracle.ewald_real(x, q, L, xi, rc)
        assert (np.abs(w["F_real"]).max() > 0.1) == (k < 0)
        assert np.abs(F - w["F_real"]).max() <= TOL


@pytest.mark.parametrize("N,L,rc", [(1, 2.0, 0.6), (5, 2.0, 0.6), (7, 1.5, 0.5), (129, 1.5, 0.5),
                                    (3000, 3.0, 1.0), (2600, 2.4, 0.3)])
def test_counts(N, L, rc):
    """Few and many particles a cell, more candidates than one chunk holds
    (half of the charges in one corner), a last charge that makes it neutral."""
    rng = np.random.default_rng(N)
    x = L * rng.random((N, 3))
    x[: N // 2] *= 0.3
    q = rng.uniform(0.5, 1.0, N)      # one sign: no cancellation in the sums
    xi = 3.1 / rc
    F, phi, E = _run(x, q, L, xi, rc)
    w = oracle.ewald_real(x, q, L, xi, rc)
    assert_close(phi, w["phi_real"] + w["phi_self"], TOL, label="phi")
    if N > 1 and np.abs(w["F_real"]).max() > 0:
        assert_close(F, w["F_real"], 10 * TOL, q=q, label="F")   # forces of one sign's shell cancel
    assert abs(E - w["E_real"] - w["E_self"]) < TOL * (abs(w["E_self"]) + abs(w["E_real"]))
