"""FP64 M2L by residue products on the tensor cores: every column width and number of moduli it takes (orders up
to 15), the CUDA-core orders above, both interaction-list widths, charges over many orders of magnitude, a level
whose moduli take several launches -- against the FP64 oracle at the FP64 path's tolerances (both sides differ
only in rounding: 1e-12 of the total energy, 1e-10 of the RMS force)."""
import numpy as np
import pytest

import oracle
from paper_2003_13218_gb300 import boxes

pytestmark = pytest.mark.gpu


def _plan(*a, **kw):
    from paper_2003_13218_gb300.fmm import FMMPlan
    return FMMPlan(*a, **kw)


def _check(pos, q, L, d, p, ws=1):
    import torch
    plan = _plan(L, len(q), d, p, ws=ws)
    F = torch.empty((len(q), 3), dtype=torch.float64, device="cuda")
    terms, _ = plan.evaluate(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), forces=F)
    plan.close()
    ref = oracle.fmm(pos, q, L, d, p, ws=ws)
    scale = abs(ref["total"]) + abs(ref["near"])
    assert abs(terms["total"] - ref["total"]) <= 1e-12 * scale
    assert abs(terms["far"] - ref["far"]) <= 1e-12 * scale
    rms = np.sqrt(np.mean(ref["forces"] ** 2))
    assert np.sqrt(np.mean((F.cpu().numpy() - ref["forces"]) ** 2)) <= 1e-10 * rms


@pytest.mark.parametrize("p", [0, 1, 2, 3, 5, 6, 7, 9, 11, 13, 14, 15, 16])
def test_orders(p):
    pos, q = boxes.random_charges(311, 9.0, seed=p)
    _check(pos, q, 9.0, 2 if p > 11 else 3, p)


@pytest.mark.parametrize("d,p,ws", [(4, 4, 1), (3, 5, 2), (4, 3, 2)])
def test_levels_and_interaction_lists(d, p, ws):
    pos, q = boxes.random_charges(700, 11.0, seed=d + p)
    _check(pos, q, 11.0, d, p, ws)


@pytest.mark.parametrize("scale", [1e-60, 1e-5, 1e5, 1e60])
def test_charge_scales(scale):
    pos, q = boxes.random_charges(300, 9.0, seed=5)
    q = q * scale
    q[7] *= 1e4  # one charge far above the rest of its level
    _check(pos, q, 9.0, 3, 6)


def test_no_charge_at_all():
    pos, q = boxes.random_charges(50, 9.0, seed=5)
    import torch
    plan = _plan(9.0, 50, 3, 6)
    terms, _ = plan.evaluate(torch.from_numpy(pos).cuda(), torch.zeros(50, dtype=torch.float64, device="cuda"))
    plan.close()
    assert terms["total"] == 0.0


def test_moduli_in_several_launches():
    """Depth 7: the operand planes of all moduli exceed what a launch holds at once."""
    import torch
    pos, q = boxes.random_charges(3000, 40.0, seed=3)
    idx = np.arange(0, 3000, 300)
    plan = _plan(40.0, 3000, 7, 4)
    F = torch.empty((3000, 3), dtype=torch.float64, device="cuda")
    plan.evaluate(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), forces=F)
    plan.close()
    ref = oracle.fmm_sampled(pos, q, 40.0, 7, 4, idx)
    got = F.cpu().numpy()[idx]
    assert np.sqrt(np.mean((got - ref["forces"]) ** 2)) <= 1e-10 * np.sqrt(np.mean(ref["forces"] ** 2))
