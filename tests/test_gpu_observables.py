"""Observable kernels at the edges of their blocks: one warp holds 31 base-pair
steps, one block of the linking-number kernel 124 segments and runs of up to
64, and short or circular molecules wrap or clamp their neighbours."""
import numpy as np
import pytest

import oracle as O
from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FLAGS = D.OBS_EXT | D.OBS_DENAT | D.OBS_TW | D.OBS_LK


def _check(n_bp, X, u, ring):
    kw = {} if ring is None else dict(ring=ring)
    ctx = D.Context(D.dsdna_default_params(precision=D.PREC_FP64), n_bp, X=X, u=u, circular=ring)
    Xs, _, us, _ = ctx.get_state()
    for m in range(len(n_bp)):
        o = ctx.observables(m, FLAGS)
        r = O.observables(O.params(**kw), n_bp, Xs, us, mol=m, with_lk=True)
        # the bound of the observables (1e-6); the closed curves' linking number is
        # an integer, here to 1e-9: some 1e5 pairs, a rounding of 2^-53 each
        for k in ("rz", "denat", "tw", "tw_ideal", "lk", "wr"):
            assert abs(o[k] - r[k]) < 1e-6, (n_bp[m], k, o[k], r[k])
        assert abs(o["lk"] - round(o["lk"])) < 1e-9, (n_bp[m], o["lk"])
        assert o == ctx.observables(m, FLAGS)       # sums in a fixed order
    ctx.close()


def test_linear_molecules_at_block_edges():
    rng = np.random.default_rng(11)
    n_bp = [2, 3, 30, 31, 32, 33, 61, 62, 63, 93, 119, 120, 121, 124, 125, 187, 249]
    parts = [I.perturb(*I.straight_helix(n), rng, dx=0.02, dtheta=0.1) for n in n_bp]
    _check(n_bp, np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), None)


def test_rings_at_block_edges():
    n_bp = [6, 31, 32, 62, 124, 125, 311]
    rng = np.random.default_rng(12)
    parts = [I.perturb(*I.ring_helix(n, max(1, round(n / 10)), center=(0, 0, 9.0 * m)), rng, dx=0.01, dtheta=0.05)
             for m, n in enumerate(n_bp)]
    _check(n_bp, np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]),
           np.ones(len(n_bp), np.int32))
