"""The bounded waits of the FP64 path's tensor-core M2L: its levels follow the same three options as the mixed path's
(wait budget, the stall hook of the single-CTA kernels, CTA pairs), and the plan stays usable after a timeout.  A
budget below the default keeps every level of both paths on single CTAs, which wait for their copies before they end,
also where pairs are on."""
import numpy as np
import pytest

from paper_2003_13218_gb300 import boxes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _inputs(b):
    return torch.from_numpy(b.pos).cuda(), torch.from_numpy(b.q).cuda()


@pytest.mark.parametrize("d,pair,precision", [(3, True, "fp64"), (4, True, "fp64"), (4, False, "fp64"),
                                              (4, True, "mixed")])
def test_wait_budget_runs_out_and_the_plan_recovers(d, pair, precision):
    from paper_2003_13218_gb300.fmm import FMMError, FMMPlan, FMM_OPT_INJECT_STALL, FMM_OPT_WAIT_BUDGET_NS
    b = boxes.ion_in_water(1500, "Na", seed=31)
    pos, q = _inputs(b)
    plan = FMMPlan(b.L, b.N, d, 8, m2l_pair=pair, precision=precision)
    plan.set_option(FMM_OPT_WAIT_BUDGET_NS, 1_000_000)  # 1 ms
    e_ok, _ = plan.energy(pos, q)
    plan.set_option(FMM_OPT_INJECT_STALL, 1)
    for _ in range(2):
        with pytest.raises(FMMError) as e:
            plan.energy(pos, q)
        assert e.value.code == 5  # FMM_ERR_TIMEOUT
    plan.set_option(FMM_OPT_INJECT_STALL, 0)
    assert plan.energy(pos, q)[0] == e_ok
    plan.close()


def test_pairs_and_single_ctas_agree():
    """The sums are whole numbers: the same results bit for bit, on levels 4 and 5."""
    from paper_2003_13218_gb300.fmm import FMMPlan
    b = boxes.ion_in_water(2000, "Mg", seed=3)
    pos, q = _inputs(b)
    out = []
    for pair in (True, False):
        plan = FMMPlan(b.L, b.N, 5, 7, m2l_pair=pair)
        out.append(plan.forces(pos, q)[0].cpu().numpy())
        plan.close()
    assert np.array_equal(out[0], out[1])
