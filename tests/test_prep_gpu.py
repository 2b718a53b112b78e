"""The scale and site-blocking passes: fields that start 8 but not 16 bytes into an allocation take the 8-byte loads,
aligned ones of an even site count the 16-byte ones; both are the same exact copies, so every output has the same
bits.  Odd and even site counts, ragged last site blocks, several instances in one launch, one to three fields."""
import numpy as np
import pytest

from helpers import ensure_built
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [([(4, 1, 5), (5, 3, 8), (6, 2, 11)], 1), ([(6, 1, 7), (3, 2, 9)], 3), ([(7, 1, 6), (4, 2, 13)], 2)]


@pytest.mark.parametrize("specs,nf", CASES)
def test_alignment_of_the_fields_does_not_change_the_results(specs, nf):
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    mom = synth.momentum_shell(1)
    flags = 0 if nf == 1 else laph.PLAN_FIELDS | (laph.PLAN_SKIP_M if nf == 3 else laph.PLAN_SKIP_B)
    plan = laph.Plan([(L, T, N, mom) for L, T, N in specs], mode="f16x3", flags=flags)
    results = []
    for shift in (0, 1):
        fields = []
        for n, (L, T, N) in enumerate(specs):
            fs = []
            for f in range(nf):
                h = torch.from_numpy(synth.random_phi(L, N, T=T, instance=500 + 10 * n + f))
                buf = torch.empty(h.numel() + shift, dtype=torch.complex64, device="cuda")
                fs.append(buf[shift:].view(h.shape).copy_(h))
            assert all(f.data_ptr() % 16 == 8 * shift for f in fs)
            fields.append(fs)
        Bs, Ms = plan.alloc_outputs()
        ws = plan.alloc_workspace()
        if nf == 1:
            plan.execute([f[0] for f in fields], Bs, Ms, ws)
        else:
            plan.execute_fields(fields, Bs if nf == 3 else Ms, ws)
        torch.cuda.synchronize()
        assert plan.device_status() == laph.LAPH_OK
        results.append([o.cpu().numpy() for o in Bs + Ms if o is not None])
    plan.close()
    for a, b in zip(*results):
        assert np.array_equal(a, b)
