"""Gram-Schmidt launches of a batch of many small timeslices: blocks between one wave and many (two rows at a time in the
update, the inner products' rows shared out), a last block of a few elements, an odd number of rows."""
import numpy as np
import pytest

from helpers import ensure_built
from oracle import oracle as O
from paper_2510_26313_gb300 import synth

pytestmark = pytest.mark.gpu


def test_lanczos_batch_between_one_and_many_waves_of_blocks():
    """L=7 (1029 elements a vector: two blocks of the update, the second of 5 elements), T=400: 800 blocks on 152 SMs.
    Eigenvalues at the suite's 5e-5 and residuals at its 1e-3 (FP32 vectors; spectral radius 12)."""
    ensure_built()
    import torch
    from paper_2510_26313_gb300 import binding as laph
    L, T, n_ev, m, d, lo = 7, 400, 12, 61, 8, 1.6
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = -(-3 * L ** 3 // 1024) * T
    assert 4 * sms < blocks < 16 * sms
    U = synth.random_links(L, T, instance=77, eps=0.6)
    vecs, ev, res = laph.lanczos(torch.from_numpy(U).cuda(), L, n_ev, m, cheb_degree=d, cheb_lo=lo)
    assert res.max() <= 1e-3 * 12
    for t in (0, 199, 399):
        lam = O.lowest_eigenpairs(U[t], L, n_ev)[0]
        assert np.abs(ev[t] - lam).max() <= 5e-5
        v = vecs[t].cpu().numpy().astype(np.complex128).reshape(n_ev, -1)
        assert np.abs(v.conj() @ v.T - np.eye(n_ev)).max() <= 1e-4
