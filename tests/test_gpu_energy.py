"""Energies and virial of every molecule of a batch whose molecules share warps
and blocks: the per-warp and per-block sums must not mix them."""
import numpy as np
import pytest

import oracle as O
from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("threads", [64, 256])
def test_energy_per_molecule_of_a_ragged_batch(prec, threads):
    lengths = [1, 1, 2, 3, 1, 16, 15, 17, 33, 1, 300, 129, 5, 1, 1, 1, 640, 8]
    cfg = I.ragged_batch(lengths, seed=3, spread=0.02)
    kw = dict(seed=4)
    ctx = D.Context(D.dsdna_default_params(precision=prec, block_threads=threads, **kw), cfg.n_bp, X=cfg.X, V=cfg.V,
                    u=cfg.u, Om=cfg.Om)
    X, V, u, Om = ctx.get_state()
    Eo, Wo = O.energy(O.params(**kw), cfg.n_bp, X, V, u, Om, 0)
    # the bounds of the energies: 1e-9 of the terms' magnitude in FP64, 2e-5 in mixed precision
    rel = 1e-9 if prec == D.PREC_FP64 else 2e-5
    tot_E, tot_W = ctx.energy_virial(-1)
    sum_E, sum_W = np.zeros_like(tot_E), np.zeros_like(tot_W)
    for m in range(len(lengths)):
        E, W = ctx.energy_virial(m)
        assert (np.abs(E - Eo[m]) <= rel * (np.abs(Eo[m]) + np.abs(Eo[m]).sum())).all(), (m, E, Eo[m])
        assert (np.abs(W - Wo[m]) <= rel * (np.abs(Wo[m]).max() + np.abs(Eo[m]).sum()) * 10).all(), (m, W, Wo[m])
        sum_E += E
        sum_W += W
    assert np.allclose(sum_E, tot_E, rtol=1e-12) and np.allclose(sum_W, tot_W, rtol=1e-9, atol=1e-9)
    ctx.close()
