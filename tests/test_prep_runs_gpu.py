"""Scale and blocking passes of batches of very different sizes: a launch covers units of similar size only, so that the
small ones do not each take the largest one's blocks; the outputs are the bits of a plan of every instance alone, from
device and from host buffers."""
import numpy as np
import pytest

from helpers import ensure_built
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("specs,runs", [([(32, 1, 4)] + [(2, 40, 5)] * 3, 2),            # one large, many of one site block
                                        ([(2, 50, 5), (28, 1, 6), (3, 60, 4), (28, 2, 5)], 2),
                                        ([(8, 2, 5), (5, 3, 8)], 1)])                     # alike: one launch
def test_batches_of_mixed_sizes(specs, runs):
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    mom = synth.momentum_shell(0)
    insts = [(L, T, N, mom) for L, T, N in specs]
    host = [synth.random_phi(L, N, T=T, instance=970 + n) for n, (L, T, N) in enumerate(specs)]
    phis = [torch.from_numpy(h).cuda() for h in host]
    plan = laph.Plan(insts, mode="f16x3")
    Bs, Ms = plan.alloc_outputs()
    ws = plan.alloc_workspace()
    plan.execute(phis, Bs, Ms, ws)
    Bh, Mh = [np.zeros(b.shape, np.complex128) for b in Bs], [np.zeros(m.shape, np.complex128) for m in Ms]
    plan.execute_host(host, Bh, Mh, torch.empty(plan.host_workspace_size(), dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    assert plan.device_status() == laph.LAPH_OK
    n_chunks = plan.schedule()["n_chunks"]
    launches = plan.launches_per_execute() - 1 - 3 * n_chunks
    assert launches in (2 * runs, 2 * runs + 1), launches   # + 1: a reduction for units cut into drains and whole ones
    plan.close()
    for n, inst in enumerate(insts):
        one = laph.Plan([inst], mode="f16x3")
        B, M = one.alloc_outputs()
        one.execute([phis[n]], B, M, one.alloc_workspace())
        torch.cuda.synchronize()
        one.close()
        for got, goth, want in ((Bs[n], Bh[n], B[0]), (Ms[n], Mh[n], M[0])):
            assert np.array_equal(got.cpu().numpy(), want.cpu().numpy())
            assert np.array_equal(goth, want.cpu().numpy())
