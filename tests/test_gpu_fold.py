"""M2M and L2L folded over the mirror images of the child octants, where they can go wrong: levels on both sides of
the line between one and four parents per block, the smallest and largest orders, and four parents at an order whose
shared memory exceeds the default limit.  Against the FP64 oracle: both sides differ only in rounding (FP64 1e-12 of
the total, mixed 1e-5, most of the energy being far field; forces 1e-10 and 5e-5 of their RMS).  The last case is too large for it and is held to the
Ewald energy within the expansion's own error at that order (below 3e-6 from p = 12 on for a few charges per leaf;
1e-4 here)."""
import numpy as np
import pytest

import oracle
from paper_2003_13218_gb300 import boxes

pytestmark = pytest.mark.gpu


def _evaluate(pos, q, L, d, p, precision, ws=1):
    import torch
    from paper_2003_13218_gb300.fmm import FMMPlan
    plan = FMMPlan(L, len(q), d, p, precision=precision, ws=ws)
    F = torch.empty((len(q), 3), dtype=torch.float64, device="cuda")
    terms, _ = plan.evaluate(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), forces=F)
    plan.close()
    return terms, F.cpu().numpy()


@pytest.mark.parametrize("precision,tol,ftol", [("fp64", 1e-12, 1e-10), ("mixed", 1e-5, 5e-5)])
@pytest.mark.parametrize("d,p,ws", [(5, 0, 1), (5, 3, 1), (5, 2, 2), (3, 13, 1), (2, 17, 1)])
def test_against_oracle(d, p, ws, precision, tol, ftol):
    pos, q = boxes.random_charges(900, 10.0, seed=d + p)
    terms, F = _evaluate(pos, q, 10.0, d, p, precision, ws)
    ref = oracle.fmm(pos, q, 10.0, d, p, ws=ws)
    scale = abs(ref["total"]) + abs(ref["near"])
    assert abs(terms["far"] - ref["far"]) <= tol * (scale + abs(ref["far"]))
    assert abs(terms["total"] - ref["total"]) <= tol * scale
    rms = np.sqrt(np.mean(ref["forces"] ** 2))
    assert np.sqrt(np.mean((F - ref["forces"]) ** 2)) <= ftol * rms


def test_wide_blocks_at_a_high_order():
    pos, q = boxes.random_charges(2000, 10.0, seed=4)
    terms, _ = _evaluate(pos, q, 10.0, 5, 15, "fp64")
    e = oracle.ewald(pos, q, 10.0)["energy"]
    assert abs(terms["total"] - e) <= 1e-4 * abs(e)
