"""Which M2L an FP64 plan runs: residue products on the tensor cores up to order 15 once the first evaluation has built
their operands, CUDA cores above; accuracy alone does not tell the two apart."""
import pytest

from paper_2003_13218_gb300 import boxes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,name", [(0, "fp64-residues"), (8, "fp64-residues"), (15, "fp64-residues"), (16, "fp64-simt")])
def test_backend_after_the_first_evaluation(p, name):
    from paper_2003_13218_gb300.fmm import FMMPlan
    pos, q = boxes.random_charges(100, 9.0, seed=1)
    plan = FMMPlan(9.0, 100, 3, p)
    assert [plan.m2l_backend(l) for l in (1, 2, 3)] == ["fp64-simt"] * 3
    plan.energy(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda())
    assert [plan.m2l_backend(l) for l in (1, 2, 3)] == ["fp64-simt", name, name]
    plan.close()
    plan = FMMPlan(9.0, 100, 3, p, precision="mixed")
    plan.energy(torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda())
    assert plan.m2l_backend(3) == ("tcgen05" if p <= 15 else "fp32-simt")
    plan.close()
