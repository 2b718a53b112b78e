"""The choice of the tile shape where a plan's tiles stay whole: an interval of its own for tiles without meson rows, or one
timeslice per chunk, and a short drain interval, whose cut tiles carry more overhead.  The estimate must not count on
cutting a thin last wave evenly there: it takes a shape with more tiles than the one it would take otherwise, and the
outputs stay within the suite's bound of the oracle."""
import pytest

from helpers import ensure_built, rel_frob, tol_for
from oracle import oracle as O
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,T,N,P,per_ts,opts", [
    (18, 1, 40, 27, False, {"chunk_sites_b": 192}), (20, 3, 48, 7, False, {"chunk_sites_b": 192}),
    (20, 3, 48, 7, False, {"chunk_sites": 32}), (14, 4, 40, 33, True, {})])
def test_shapes_of_plans_whose_tiles_stay_whole(L, T, N, P, per_ts, opts):
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    inst = (L, T, N, synth.momentum_shell(4)[:P])
    flags = laph.PLAN_CHUNK_PER_TIMESLICE if per_ts else 0
    base = laph.Plan([inst], mode="f16x3", flags=flags, tile_cols=96, **opts)
    plan = laph.Plan([inst], mode="f16x3", flags=flags, **opts)
    d, d0 = plan.describe(), base.describe()
    base.close()
    print(inst[:3], P, opts, (d["tile_rows"], d["tile_cols"]), d["n_tiles"], d0["n_tiles"])
    if not opts.get("chunk_sites"):   # (cut into drains otherwise)
        assert d["n_tiles"] >= 1.25 * d0["n_tiles"]
    assert (d["tile_rows"], d["tile_cols"]) == (64, 128)
    phi = synth.random_phi(L, N, T=T, instance=950)
    Bs, Ms = plan.alloc_outputs()
    plan.execute([torch.from_numpy(phi).cuda()], Bs, Ms, plan.alloc_workspace())
    torch.cuda.synchronize()
    assert plan.device_status() == laph.LAPH_OK
    assert rel_frob(Ms[0][T - 1].cpu().numpy(), O.meson_blocks(phi[T - 1], L, inst[3])) <= tol_for("f16x3")
    plan.close()
