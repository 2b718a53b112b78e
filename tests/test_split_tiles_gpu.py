"""Units cut into tiles of one drain interval, against the same plan with whole site blocks.

A plan cuts the trailing timeslices of a small batch into drains; the reduction then makes the FP32 additions a
whole tile's epilogue makes, so the outputs are the same bits.  laph_plan_set_chunk_sites takes the cut back
(another interval, then the first one again), which gives the reference.
"""
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
    # (instances, options, fields): one drain and a bit; the last site block and its last drain ragged; three site blocks
    # whose size is no multiple of the drain interval; a ragged batch whose trailing units alone are cut
    ([(11, 1, 9, synth.momentum_shell(1))], {}, 0),
    ([(23, 1, 20, synth.momentum_shell(1))], {}, 0),
    ([(17, 2, 13, synth.momentum_shell(2))], {"sum_sites": 1800}, 0),
    ([(16, 1, 20, synth.momentum_shell(2)), (9, 1, 11, synth.momentum_shell(0))], {"layout": 1}, 0),
    ([(16, 1, 12, synth.momentum_shell(1))], {}, 3),
    ([(14, 2, 21, synth.momentum_shell(0))], {"layout": 1, "tile_cols": 128}, 2),
]


@pytest.mark.parametrize("c64", [False, True])
@pytest.mark.parametrize("mode", ["f16x3", "bf16x3", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_cut_units_give_the_bits_of_whole_site_blocks(laph, case, mode, c64):
    import torch
    insts, opts, nf = CASES[case]
    flags = laph.PLAN_OUT_C64 if c64 else 0
    if nf:
        flags |= laph.PLAN_FIELDS | (laph.PLAN_SKIP_M if nf == 3 else laph.PLAN_SKIP_B)
    phis = [[torch.from_numpy(synth.random_phi(L, N, T=T, instance=300 + 10 * n + f)).cuda() for f in range(max(nf, 1))]
            for n, (L, T, N, _) in enumerate(insts)]
    outs, tiles = [], []
    for whole in (False, True):
        plan = laph.Plan(insts, mode=mode, flags=flags, **opts)
        ws = plan.alloc_workspace()
        if whole:
            for cs in (64, 0):
                assert laph.lib().laph_plan_set_chunk_sites(plan.handle, cs) == laph.LAPH_OK
            assert plan.workspace_size() <= ws.numel()
        Bs, Ms = plan.alloc_outputs()
        if nf:
            plan.execute_fields(phis, Bs if nf == 3 else Ms, ws)
        else:
            plan.execute([p[0] for p in phis], Bs, Ms, ws)
        torch.cuda.synchronize()
        assert plan.device_status() == laph.LAPH_OK
        outs.append([o.cpu().numpy() for o in Bs + Ms if o is not None])
        tiles.append((plan.describe()["n_tiles"], plan.tensor_flops()))
        plan.close()
    assert tiles[0][0] > tiles[1][0] and np.isclose(tiles[0][1], tiles[1][1])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
