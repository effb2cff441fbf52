"""The double-precision real-space sum in boxes and with splitting parameters
far from one: lengths whose squares leave the single-precision range (the
distance test's), and xi r so small that powers of it leave the FP64 range.

Tolerance: rounding only, 1e-12 as in the other tests of this kernel."""
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


def _check(x, q, L, xi, rc, s=1.0):
    """The system scaled by s: phi s, F s^2 and E s do not depend on it."""
    F, phi, E = _run(x * s, q, L * s, xi / s, rc * s)
    w = oracle.ewald_real(x, q, L, xi, rc)
    assert_close(F * s * s, w["F_real"], 10 * TOL, q=q, label="F")
    assert_close(phi * s, w["phi_real"] + w["phi_self"], TOL, label="phi")
    assert abs(E * s - w["E_real"] - w["E_self"]) < TOL * (abs(w["E_self"]) + abs(w["E_real"]))


@pytest.mark.parametrize("s", [1e-90, 1e-30, 1e-25, 1e-21, 1e-19, 1e-15, 1.0, 1e15, 1e19, 1e25, 1e90])
@pytest.mark.parametrize("N", [2, 300])
def test_units_of_length(s, N):
    L, rc, xi = 3.0, 1.0, 3.1
    rng = np.random.default_rng(N)
    x = L * rng.random((N, 3))
    if N == 2:
        x = np.array([[0.01, 2.9, 1.0], [2.8, 0.2, 1.1]])
    _check(x, rng.uniform(0.5, 1.0, N), L, xi, rc, s)


def test_positions_that_differ_by_a_rounding_of_the_test():
    """Pairs at r_c (1 +- 2^-23 k) in a box where the cut-off is a small part of
    the side: the single-precision test must not lose any."""
    L, rc, xi = 64.0, 1.0, 1.0
    rng = np.random.default_rng(5)
    x = []
    for k in (-40, -7, -2, -1, 1, 2, 7, 40):
        a = np.floor(3 + 58 * rng.random(3)) + rng.random(3)
        d = rng.standard_normal(3)
        x += [a, a + rc * (1 + k * 2.0 ** -23) * d / np.linalg.norm(d)]
    x = np.array(x)
    _check(x, np.ones(len(x)), L, xi, rc)


@pytest.mark.parametrize("xi", [1e-8, 1e-60, 1e-103, 1e-110, 1e-155, 1e-200])
def test_bare_coulomb_limit(xi):
    """xi r far below one: erfc(xi r)/r is 1/r."""
    L, rc = 3.0, 1.0
    rng = np.random.default_rng(9)
    x = L * rng.random((200, 3))
    _check(x, rng.uniform(0.5, 1.0, 200), L, xi, rc)
