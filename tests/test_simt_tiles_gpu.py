"""The FP32 path at the edges of its tiles against the FP64 oracle: rows and columns that fill a 64 x 64 tile, fall one
short of it or one over, warps whose column groups are left out below the triangle, site counts that are no multiple
of the 8-site chunk, and drain intervals that are no multiple of 16 sites.  The sums are FP32 over at most an
interval and FP64 beyond, so the suite's 1e-5 bound for the FP32 path holds with room."""
import numpy as np
import pytest

from helpers import ensure_built, rel_frob, tol_for
from oracle import oracle as O
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [0, 20])
@pytest.mark.parametrize("L,N,P", [(4, 16, 4), (5, 13, 5), (3, 33, 2), (7, 21, 3), (6, 65, 1), (3, 11, 7)])
def test_fp32_blocks_at_tile_edges(L, N, P, chunk):
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    mom = synth.momentum_shell(1)[:P]
    phi_h = synth.random_phi(L, N, T=2, instance=400 + N)
    plan = laph.Plan([(L, 2, N, mom)], mode="fp32", chunk_sites=chunk)
    Bs, Ms = plan.alloc_outputs()
    plan.execute([torch.from_numpy(phi_h).cuda()], Bs, Ms, None)
    torch.cuda.synchronize()
    for t in range(2):
        assert rel_frob(Bs[0][t].cpu().numpy(), O.baryon_blocks(phi_h[t], L, mom)) <= tol_for("fp32")
        assert rel_frob(Ms[0][t].cpu().numpy(), O.meson_blocks(phi_h[t], L, mom)) <= tol_for("fp32")
    plan.close()
