"""FP64 M2L in whole numbers: values far from 1, where the gain that turns moments into whole numbers meets the ends
of the range of a double."""
import numpy as np
import pytest

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
