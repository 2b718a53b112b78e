"""Tiles worked by pairs of CTAs (many row vectors per tile), against single CTAs.

The pair's MMAs add the same products in the same order as the row-doubled layout's, so the outputs are the same
bits.  Shapes: several row and column tiles with ragged ends and skipped leading columns, odd and even site counts, one
and several site blocks, three fields, every term count and split type; the timeout of a stalled producer."""
import numpy as np
import pytest

from helpers import ensure_built
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def laph():
    ensure_built()
    import torch
    torch.cuda.set_device(0)
    from paper_2510_26313_gb300 import binding
    return binding


CASES = [
    # (L, T, N, momenta, options, fields)
    (9, 1, 128, synth.momentum_shell(4), {}, 1),
    (7, 3, 120, synth.momentum_shell(4), {"sum_sites": 200}, 1),
    (12, 1, 100, synth.momentum_shell(4), {"chunk_sites_b": 64}, 1),
    (4, 1, 150, synth.momentum_shell(2), {}, 3),
]


def run(laph, case, mode, **opts):
    import torch
    L, T, N, mom, o, nf = case
    flags = laph.PLAN_FIELDS | laph.PLAN_SKIP_M if nf == 3 else 0
    plan = laph.Plan([(L, T, N, mom)], mode=mode, flags=flags, **o, **opts)
    phis = [torch.from_numpy(synth.random_phi(L, N, T=T, instance=600 + f)).cuda() for f in range(nf)]
    Bs, Ms = plan.alloc_outputs()
    ws = plan.alloc_workspace()
    for _ in range(2):   # back to back: the barriers' phases of a second launch
        plan.execute_fields([phis], Bs, ws) if nf == 3 else plan.execute(phis, Bs, Ms, ws)
    torch.cuda.synchronize()
    assert plan.device_status() == laph.LAPH_OK
    d = plan.describe()
    plan.close()
    return d, [x.cpu().numpy() for x in Bs + Ms if x is not None]


@pytest.mark.parametrize("mode", ["f16x3", "bf16x3", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_pairs_give_the_bits_of_single_ctas(laph, case, mode):
    d, got = run(laph, CASES[case], mode)
    assert (d["tile_rows"], d["tile_cols"]) == (128, 208), d
    _, ref = run(laph, CASES[case], mode, layout=1, tile_cols=128)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)


def test_a_stalled_producer_of_a_pair_times_out(laph):
    import torch
    L, T, N, mom = 9, 1, 128, synth.momentum_shell(4)
    phi = torch.from_numpy(synth.random_phi(L, N, T=T, instance=700)).cuda()
    plan = laph.Plan([(L, T, N, mom)], mode="f16x3", flags=laph.PLAN_DEBUG_STALL)
    assert plan.describe()["tile_cols"] == 208
    Bs, Ms = plan.alloc_outputs()
    plan.execute([phi], Bs, Ms, plan.alloc_workspace())
    torch.cuda.synchronize()
    assert plan.device_status() == laph.LAPH_ERR_TIMEOUT
    plan.close()
    _, got = run(laph, CASES[0], "f16x3")
    assert np.isfinite(got[0]).all()
