"""The tile shape a plan takes changes no bit of its outputs (with one drain interval for all tiles).

In the imaginary parts the layouts hand the two products of a K entry to the tensor core in exchanged slots, so equality
rests on its sum over a k-step not depending on the order within it; the layouts also cut rows and columns
differently.  Every compiled shape against layout 0 with 104 (pairs: 96) columns, meson and baryon rows, several drains
and site blocks, and the automatic choice for one to three fields; the pairs also replayed from a CUDA graph."""
import numpy as np
import pytest

from helpers import ensure_built
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(0, 96), (0, 80), (0, 64), (1, 208), (1, 192), (1, 176), (1, 128), (0, 0)]


@pytest.fixture(scope="module")
def laph():
    ensure_built()
    import torch
    torch.cuda.set_device(0)
    from paper_2510_26313_gb300 import binding
    return binding


def outputs(laph, inst, mode, nf=1, flags=0, graph=False, **opts):
    import torch
    L, T, N, mom = inst
    if nf > 1:
        flags |= laph.PLAN_FIELDS | (laph.PLAN_SKIP_M if nf == 3 else laph.PLAN_SKIP_B)
    phis = [torch.from_numpy(synth.random_phi(L, N, T=T, instance=900 + f)).cuda() for f in range(nf)]
    plan = laph.Plan([inst], mode=mode, flags=flags, **opts)
    Bs, Ms = plan.alloc_outputs()
    ws = plan.alloc_workspace()

    def execute(stream=None):
        if nf > 1:
            plan.execute_fields([phis], Bs if nf == 3 else Ms, ws, stream=stream)
        else:
            plan.execute(phis, Bs, Ms, ws, stream=stream)

    if graph:
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            execute(s)
        g.replay()
    else:
        execute()
    torch.cuda.synchronize()
    assert plan.device_status() == laph.LAPH_OK
    d = plan.describe()
    out = [o.cpu().numpy() for o in Bs + Ms if o is not None]
    plan.close()
    return (d["tile_rows"], d["tile_cols"]), out


@pytest.mark.parametrize("mode", ["f16x3", "bf16x3", "f16"])
@pytest.mark.parametrize("inst,opts", [((11, 2, 21, synth.momentum_shell(1)), {}),
                                       ((10, 1, 33, synth.momentum_shell(2)), {"sum_sites": 400, "chunk_sites": 56})])
def test_every_shape_gives_the_same_bits(laph, inst, opts, mode):
    _, want = outputs(laph, inst, mode, layout=0, tile_cols=104, **opts)
    for layout, cols in SHAPES:
        shape, got = outputs(laph, inst, mode, layout=layout, tile_cols=cols, **opts)
        for a, b in zip(got, want):
            assert np.array_equal(a, b), (layout, cols, shape)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("mode", ["f16x3", "bf16x3"])
def test_pairs_of_ctas_give_the_bits_of_layout_0(laph, mode, graph):
    inst = (9, 1, 128, synth.momentum_shell(4))
    shape, got = outputs(laph, inst, mode, graph=graph)
    assert shape == (128, 208)
    _, want = outputs(laph, inst, mode, layout=0, tile_cols=96)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("inst,nf,skip", [((16, 4, 64, synth.momentum_shell(2)), 1, "B"),     # meson rows alone
                                          ((12, 4, 90, synth.momentum_shell(1)), 2, None),    # projection
                                          ((16, 8, 32, synth.momentum_shell(1)), 1, None),    # 224 columns
                                          ((12, 1, 24, synth.momentum_shell(2)), 3, None)])   # triplets
def test_the_automatic_shape_gives_the_bits_of_layout_0(laph, inst, nf, skip):
    flags = laph.PLAN_SKIP_B if skip else 0
    shape, got = outputs(laph, inst, "f16x3", nf, flags)
    print(inst[:3], nf, shape)
    _, want = outputs(laph, inst, "f16x3", nf, flags, layout=0, tile_cols=64)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
