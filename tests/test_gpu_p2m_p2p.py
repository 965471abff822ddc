"""P2M with one charge per lane and the FP64 near field by rows, where they can go wrong: counts of lanes per target on
both sides of each line (N below and above 4,864, 9,728, 19,456 and 38,912), a lone charge, leaves below, at and above
the 32 charges of one round, all charges in one corner, orders without a kernel of their own.  Against the FP64 oracle:
both sides differ only in rounding (FP64 1e-12 of the total, forces 1e-10 of their RMS; mixed 1e-5 and 5e-5)."""
import numpy as np
import pytest

import oracle
from paper_2003_13218_gb300 import boxes

pytestmark = pytest.mark.gpu


def _check(pos, q, L, d, p, precision="fp64", ws=1):
    import torch
    from paper_2003_13218_gb300.fmm import FMMPlan
    tol, ftol = (1e-12, 1e-10) if precision == "fp64" else (1e-5, 5e-5)
    plan = FMMPlan(L, len(q), d, p, precision=precision, ws=ws)
    F = torch.empty((len(q), 3), dtype=torch.float64, device="cuda")
    terms, _ = plan.evaluate(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), forces=F)
    plan.close()
    ref = oracle.fmm(pos, q, L, d, p, ws=ws)
    scale = abs(ref["total"]) + abs(ref["near"]) + abs(ref["far"])
    for k in ("near", "far", "total"):
        assert abs(terms[k] - ref[k]) <= tol * scale, k
    rms = np.sqrt(np.mean(ref["forces"] ** 2))
    assert np.sqrt(np.mean((F.cpu().numpy() - ref["forces"]) ** 2)) <= ftol * rms + (rms == 0) * 1e-12


@pytest.mark.parametrize("n,d,ws", [(1, 2, 1), (33, 2, 1), (4863, 3, 1), (4865, 3, 2), (9727, 3, 1), (9729, 4, 1),
                                    (19457, 4, 2), (38911, 4, 1), (38913, 4, 1)])
def test_near_field_lanes_per_target(n, d, ws):
    pos, q = boxes.random_charges(n, 12.0, seed=n)
    _check(pos, q, 12.0, d, 2, ws=ws)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,d,p", [(40, 3, 0), (300, 3, 1), (1800, 2, 5), (2048, 2, 7), (2600, 2, 9), (500, 4, 11),
                                   (9000, 2, 8)])
def test_leaf_counts_and_orders(n, d, p, precision):
    pos, q = boxes.random_charges(n, 12.0, seed=n + p)
    _check(pos, q, 12.0, d, p, precision)


@pytest.mark.parametrize("n,p", [(700, 3), (97, 6)])
def test_all_charges_in_one_corner(n, p):
    pos, q = boxes.random_charges(n, 12.0, seed=n)
    _check(pos * 0.2, q, 12.0, 3, p)
