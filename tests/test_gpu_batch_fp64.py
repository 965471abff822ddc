"""Batches in FP64: the depth tuner has to time the M2L that the boxes then run (residue products on the tensor cores;
on the CUDA cores the M2L costs hundreds of times as much and the shallowest tree wins)."""
import pytest

from paper_2003_13218_gb300.fmm import FMMBatch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _boxes(n, k, L):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    pos = [torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64) * L for _ in range(k)]
    q = [torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1 for _ in range(k)]
    sol = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in range(k)]
    for s in sol:
        s[0] = 1
    return pos, q, sol


@pytest.mark.parametrize("n,k,p", [(3001, 2, 8), (40000, 1, 12)])
def test_tuned_depth_is_near_the_fastest(n, k, p):
    """Within 1.5 times the fastest of the depths next to it (one level off costs 2 to 10 times here)."""
    L = 40.0
    data = _boxes(n, k, L)

    def best_ms(depths):
        b = FMMBatch([L] * k, [n] * k, depths, [p] * k, precision="fp64")
        d, ts = b.info(0)["depth"], []
        for i in range(8):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            torch.cuda.synchronize()
            e0.record()
            b.lambda_energies(*data)
            e1.record()
            torch.cuda.synchronize()
            if i >= 3:
                ts.append(e0.elapsed_time(e1))
        b.close()
        return d, min(ts)

    d, tuned = best_ms(None)
    assert tuned <= 1.5 * min(best_ms([x] * k)[1] for x in range(max(2, d - 1), d + 2))


def test_operators_are_built_once_for_all_boxes():
    """Ten boxes at p = 12: the operator residues take 0.32 GB, so building them per box would hold 2.9 GB more while
    the batch is created than afterwards.  The results are those of the same boxes alone, bit for bit."""
    import threading
    from paper_2003_13218_gb300.fmm import FMMPlan
    k, n, L, d, p = 10, 501, 20.0, 3, 12
    pos, q, sol = _boxes(n, k, L)
    used, stop = [], threading.Event()

    def watch():
        while not stop.is_set():
            free, total = torch.cuda.mem_get_info()
            used.append(total - free)

    plan = FMMPlan(L, n, d, p)
    ref = [plan.energy(pos[i], q[i])[0] for i in range(k)]
    plan.close()
    t = threading.Thread(target=watch)
    t.start()
    batch = FMMBatch([L] * k, [n] * k, [d] * k, [p] * k, precision="fp64")
    stop.set()
    t.join()
    free, total = torch.cuda.mem_get_info()
    assert len(used) > 20
    assert max(used) - (total - free) <= 0.5e9
    out = batch.lambda_energies(pos, q, sol)
    batch.close()
    assert list(out["e_total"]) == ref
