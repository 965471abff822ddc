"""The top operator (level 1 and above in one product) and the sparse solute pass built on it, where they can go
wrong: the shallowest trees, the counts at which the sparse pass starts and stops, solute charges that share a
cell at every level or none, kappa changed after creation -- against the FP64 oracle at the tolerances of the
other solute tests (FP64 1e-10, mixed 1e-5 of |A| + |C| + |E_uv|; energies 1e-12 and 1e-6)."""
import numpy as np
import pytest

import oracle
from paper_2003_13218_gb300 import boxes

pytestmark = pytest.mark.gpu


def _cuda(*xs):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in xs]


def _solute(pos, n, how):
    sol = np.zeros(len(pos), np.uint8)
    if how == "near":  # neighbours of one point: shared cells on most levels
        sol[np.argsort(((pos - pos[0]) ** 2).sum(1), kind="stable")[:n]] = 1
    else:
        sol[np.linspace(0, len(pos) - 1, n).astype(int)] = 1
    return sol


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("d,p,ws,n,how", [(2, 4, 1, 1, "near"), (2, 9, 1, 64, "spread"), (2, 6, 1, 65, "near"),
                                          (3, 8, 1, 2, "near"), (3, 5, 1, 64, "near"), (3, 4, 2, 40, "spread"),
                                          (4, 4, 1, 64, "spread"), (4, 3, 2, 64, "near")])
def test_solute_energy(precision, tol, d, p, ws, n, how):
    from paper_2003_13218_gb300.fmm import FMMPlan
    pos, q = boxes.random_charges(400, 10.0, seed=n + d)
    sol = _solute(pos, n, how)
    ref = oracle.solute_solvent(pos, q, sol, 10.0, d, p, ws=ws)
    plan = FMMPlan(10.0, len(q), d, p, precision=precision, ws=ws)
    for _ in range(2):
        e, uv = plan.solute_solvent_energy(*_cuda(pos, q, sol))
        scale = abs(ref["A"]) + abs(ref["C"]) + abs(ref["e_uv"])
        for k in ("e_uv", "W", "A", "B", "C"):
            assert abs(uv[k] - ref[k]) <= tol * scale, k
    plan.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-6)])
@pytest.mark.parametrize("d,ws", [(2, 1), (3, 1), (3, 2)])
def test_kappa_after_creation(precision, tol, d, ws):
    from paper_2003_13218_gb300.fmm import FMM_OPT_KAPPA, FMMPlan
    pos, q = boxes.random_charges(300, 10.0, seed=d)
    plan = FMMPlan(10.0, len(q), d, 6, precision=precision, ws=ws)
    for kappa in (0.13, 0.45):
        plan.set_option(FMM_OPT_KAPPA, 0, kappa)
        e, _ = plan.energy(*_cuda(pos, q))
        ref = oracle.fmm(pos, q, 10.0, d, 6, ws=ws, kappa=kappa, forces=False)
        assert abs(e - ref["total"]) <= tol * (abs(ref["total"]) + abs(ref["near"]))
    plan.close()
