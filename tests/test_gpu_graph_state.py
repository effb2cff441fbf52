"""A spread that no scaling step follows leaves weights on the plan's grid; the
evaluations after it, captured before or not, start from a clean one.
Tolerances as test_gpu_parity: 1e-12 (FP64), 2e-5 (FP32), between two runs of
the same code."""
import numpy as np
import pytest
import torch

from paper_1712_04718_gb300 import se, systems

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("prec,variant", [("fp64", 1), ("fp64", 2), ("fp32", 1), ("fp32", 3),
                                          ("fp32", 4), ("fp32plain", 2)])
@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("captured", [False, True])
def test_evaluate_after_a_spread_alone(prec, variant, host, captured):
    L, xi, M, P, N = 2.0, 3.0, 24, 8, 200
    x, q = systems.uniform_charges(N, L, seed=5)
    x2, q2 = systems.uniform_charges(N, L, seed=6)
    plan = se.Plan(N, L, xi, M, P, precision=prec, spread_variant=variant)
    dt = plan.dtype

    def buffers(x, q):
        t = [torch.tensor(x, dtype=dt), torch.tensor(q, dtype=dt),
             torch.empty(N, 3, dtype=dt), torch.empty(N, dtype=dt)]
        return [b.pin_memory() if host else b.cuda() for b in t]

    a = buffers(x, q)

    def evaluate():
        if host:
            plan.energy_force_host_ptrs(*[t.data_ptr() for t in a])
        else:
            plan.evaluate(*a)
        torch.cuda.synchronize()
        return a[2].double().cpu().numpy().copy(), a[3].double().cpu().numpy().copy()

    ref = evaluate()
    if not captured:
        plan.set_graph(False)      # drops the graph
        plan.set_graph(True)
    plan.spread(torch.tensor(x2, dtype=dt, device="cuda"), torch.tensor(q2, dtype=dt, device="cuda"))
    tol = 1e-12 if prec == "fp64" else 2e-5
    for _ in range(2):
        for got, want in zip(evaluate(), ref):
            assert np.linalg.norm(got - want) < tol * np.linalg.norm(want)
    plan.close()
