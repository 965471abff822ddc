"""FP64 M2L in whole numbers: values far from 1, where the gain that turns moments into whole numbers meets the ends
of the range of a double, and levels with one charge far above the others, whose exponent is the level's."""
import numpy as np
import pytest

import oracle
from paper_2003_13218_gb300 import boxes

pytestmark = pytest.mark.gpu


def _potentials(pos, q, L, d, p, ws=1):
    import torch
    from paper_2003_13218_gb300.fmm import FMMPlan
    plan = FMMPlan(L, len(q), d, p, ws=ws)
    phi, _ = plan.potentials(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), with_energy=False)
    phi = phi.cpu().numpy()
    plan.close()
    return phi


@pytest.mark.parametrize("exponent", [-990, -960, 960, 1000])
def test_charges_at_the_ends_of_the_range(exponent):
    """The potentials are linear in the charges, and a power of two commutes with every FP64 operation as long as
    nothing leaves the normal range.  At 2^-990 and order 4 the smallest moments do, which costs them 2^-84 of the
    charges; 1e-13 of the RMS potential is asked for."""
    pos, q = boxes.random_charges(300, 9.0, seed=6)
    ref = _potentials(pos, q, 9.0, 3, 4)
    phi = _potentials(pos, q * 2.0 ** exponent, 9.0, 3, 4) / 2.0 ** exponent
    assert np.sqrt(np.mean((phi - ref) ** 2)) <= 1e-13 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("n,d,p,ws", [(200_000, 7, 3, 1), (60_000, 6, 4, 1), (60_000, 6, 3, 2)])
def test_field_far_from_a_dominant_charge(n, d, p, ws):
    """The field at charges a quarter box and more from one 1e8 times as large.  It is that charge's, (h / r)^2 of what
    it does to its own cell's neighbours, so a rounding relative to the level's largest moment is 2^12 to 2^14 times
    too coarse here at depth 6 or 7 (measured in the whole numbers alone: above 1e-13).  FP64 sums of some forty
    sources err by 3e-15 (both sides); 2e-14 of the RMS field is asked for."""
    import torch
    from paper_2003_13218_gb300.fmm import FMMPlan
    L = 40.0
    pos, q = boxes.random_charges(n, L, seed=d + ws)
    q[0] *= 1e8
    r = np.abs(pos - pos[0])
    far = np.flatnonzero((np.minimum(r, L - r) ** 2).sum(1) > (L / 4) ** 2)
    idx = far[:: len(far) // 24][:24]
    ref = oracle.fmm_sampled(pos, q, L, d, p, idx, ws=ws)
    plan = FMMPlan(L, n, d, p, ws=ws)
    F, _ = plan.forces(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), with_energy=False)
    F = F.cpu().numpy()[idx]
    plan.close()
    E, E_ref = F / q[idx, None], ref["forces"] / q[idx, None]
    assert np.sqrt(np.mean((E - E_ref) ** 2)) <= 2e-14 * np.sqrt(np.mean(E_ref ** 2))


@pytest.mark.parametrize("d,p,ws", [(2, 0, 1), (2, 8, 1), (2, 15, 1), (3, 5, 1), (3, 11, 1), (3, 4, 2), (4, 2, 1)])
def test_targets_of_floating_point_sums(d, p, ws):
    """A charge 1e4 times as large as the others: at level 2 the 27 cells around it take floating-point sums, each
    spread over several blocks; at the deeper levels most cells do, a block each.  Forces and potentials of the other charges against the oracle, rounding on both
    sides: 1e-12 of their RMS, which the small charges' part exceeds by 1e8."""
    import torch
    from paper_2003_13218_gb300.fmm import FMMPlan
    pos, q = boxes.random_charges(1500, 9.0, seed=10 * d + p)
    q[0] *= 1e4
    ref = oracle.fmm(pos, q, 9.0, d, p, ws=ws)
    plan = FMMPlan(9.0, len(q), d, p, ws=ws)
    F = torch.empty((len(q), 3), dtype=torch.float64, device="cuda")
    terms, _ = plan.evaluate(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda(), forces=F)
    plan.close()
    assert abs(terms["far"] - ref["far"]) <= 1e-12 * (abs(ref["total"]) + abs(ref["near"]) + abs(ref["far"]))
    E, E_ref = F.cpu().numpy()[1:] / q[1:, None], ref["forces"][1:] / q[1:, None]
    assert np.sqrt(np.mean((E - E_ref) ** 2)) <= 1e-12 * np.sqrt(np.mean(E_ref ** 2))
