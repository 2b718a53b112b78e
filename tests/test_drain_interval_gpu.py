"""laph_plan_set_chunk_sites on a plan whose timeslices are cut into drains changes host values only.

An execute that is queued on a non-blocking stream, and a CUDA graph captured before the call, keep the interval and
the tile tables they were launched with: same bits as before the call.  Executes after the call give the bits of a plan
made with the new interval."""
import numpy as np
import pytest

from helpers import ensure_built
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [[(16, 2, 14, synth.momentum_shell(1))], [(16, 1, 20, synth.momentum_shell(2)), (9, 1, 11, synth.momentum_shell(0))]]


@pytest.mark.parametrize("insts", CASES)
def test_interval_changed_under_queued_executes_and_a_captured_graph(insts):
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    phis = [torch.from_numpy(synth.random_phi(L, N, T=T, instance=800 + n)).cuda()
            for n, (L, T, N, _) in enumerate(insts)]

    def fresh(chunk):
        plan = laph.Plan(insts, mode="f16x3", chunk_sites=chunk)
        Bs, Ms = plan.alloc_outputs()
        return plan, Bs + Ms, (phis, Bs, Ms, plan.alloc_workspace())

    def host(outs):
        torch.cuda.synchronize()
        return [o.cpu().numpy() for o in outs]

    want = {}
    for chunk in (0, 64):
        plan, outs, args = fresh(chunk)
        plan.execute(*args)
        want[chunk] = host(outs)
        plan.close()

    plan, outs, args = fresh(0)
    s = torch.cuda.Stream()   # non-blocking: not ordered with the default stream
    s.wait_stream(torch.cuda.current_stream())
    cut = plan.describe()["n_tiles"]
    with torch.cuda.stream(s):
        plan.execute(*args, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        plan.execute(*args, stream=s)
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    for _ in range(8):
        plan.execute(*args, stream=s)
    assert laph.lib().laph_plan_set_chunk_sites(plan.handle, 64) == laph.LAPH_OK   # with executes queued
    assert plan.describe()["n_tiles"] < cut
    for a, b in zip(host(outs), want[0]):
        assert np.array_equal(a, b)
    for replay, chunk in ((True, 0), (False, 64), (True, 0), (False, 64)):
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        if replay:
            g.replay()
        else:
            plan.execute(*args, stream=s)
        for a, b in zip(host(outs), want[chunk]):
            assert np.array_equal(a, b)
    assert plan.device_status() == laph.LAPH_OK
    plan.close()
