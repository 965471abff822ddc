"""The first evaluation of an FP64 plan builds its residue operands: it must neither wait for the stream (a call that
only enqueues returns at once, the first time as well) nor disturb a capture in another thread, and under capture it
runs without them."""
import threading

import numpy as np
import pytest

from paper_2003_13218_gb300 import boxes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup():
    from paper_2003_13218_gb300.fmm import FMMPlan
    pos, q = boxes.random_charges(800, 9.0, seed=2)
    pos, q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    warm = FMMPlan(9.0, 800, 3, 6)  # the kernels are loaded
    ref = warm.forces(pos, q)[0]
    warm.close()
    torch.cuda.synchronize()
    return FMMPlan(9.0, 800, 3, 6), pos, q, torch.empty_like(ref), ref


def test_first_call_only_enqueues():
    plan, pos, q, F, ref = _setup()
    busy = torch.cuda.Event()
    torch.cuda._sleep(1_000_000_000)  # some 0.5 s
    busy.record()
    plan.forces(pos, q, out=F, with_energy=False)
    assert not busy.query()
    torch.cuda.synchronize()
    assert torch.equal(F, ref)
    plan.close()


def test_first_call_beside_a_capture():
    plan, pos, q, F, ref = _setup()
    x = torch.zeros(16, device="cuda")
    failed = []

    def call():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                plan.forces(pos, q, out=F, with_energy=False)
        except Exception as e:  # seen by the main thread
            failed.append(e)

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="global"):
        x.add_(1.0)
        t = threading.Thread(target=call)
        t.start()
        t.join()
        x.add_(1.0)
    torch.cuda.synchronize()
    assert not failed, failed
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 32.0
    assert torch.equal(F, ref)
    plan.close()


def test_first_call_under_capture():
    """No operands then: the CUDA cores' sums, the same forces to rounding (1e-10 of their RMS)."""
    plan, pos, q, F, ref = _setup()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        plan.forces(pos, q, out=F, with_energy=False)
    for _ in range(2):
        F.zero_()
        g.replay()
        torch.cuda.synchronize()
        rms = np.sqrt(np.mean(ref.cpu().numpy() ** 2))
        assert np.sqrt(np.mean((F - ref).cpu().numpy() ** 2)) <= 1e-10 * rms
    plan.close()
