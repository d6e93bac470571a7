"""Strip step kernel with the list rebuilt inside it (lists by the cell walk, boxes of few segment-grid cells, systems too
long for the resident kernel): bitwise the trajectories of the same steps with separate rebuild kernels.  CTAs of 96
threads, a size the resident kernel never takes, show which kernel steps."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PRECS = [D.PREC_MIXED, D.PREC_FP64]


def _both(n_bp, X, u, V, Om, steps, rebuilds, modes=(1, 2), tether=None, ring=None, loads=None, **kw):
    out = []
    for mode in modes:
        ctx = D.Context(D.dsdna_default_params(rebuild_mode=mode, block_threads=96, **kw), n_bp, X=X, u=u, V=V, Om=Om,
                        tether=tether, circular=ring)
        for m, (f, t) in enumerate(loads or []):
            ctx.set_external_force_torque(m, f, t)
        for k in (1, 50, steps - 51):
            ctx.step(k)
        info = ctx.info()
        assert info["rebuild_in_step"] == (mode != 1) and info["block_threads"] == 96 and info["rebuilds"] >= rebuilds
        out.append([*ctx.get_state(), ctx.get_bubble_mask()])
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", PRECS)
def test_cell_walk_open_box(prec):
    """Loaded molecules of several lengths, tiles that span two of them; hashed cell table."""
    cfg = I.c4_batch(n_mol=7, lo=100, hi=900, seed=8, random_pose=True)
    _both(cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om, 300, 8, tether=cfg.tether, loads=list(zip(cfg.ext_f, cfg.ext_t)),
          precision=prec, list_build=1, skin=0.1, seed=3)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n_bp,list_build", [(2500, 1), (400, 0)])
def test_periodic_box(prec, n_bp, list_build):
    """Linear cell table; 400 base pairs in a box of two segment-grid cells per edge, where the chain window does not apply."""
    cfg = I.random_walk_helix(n_bp=n_bp, phi=0.15, clearance=1.7, seed=4)
    _both(cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om, 300, 8, precision=prec, box=cfg.box, list_build=list_build, skin=0.1, seed=3)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("rule", [0, 1, 2])
def test_rings_and_bubbles(prec, rule):
    """A junction barrier each step besides the rebuild's; weak hydrogen bonds so that bubbles open."""
    rng = np.random.default_rng(5)
    n_bp, ring = [60, 37, 40, 700, 45, 36], [1, 1, 0, 1, 1, 1]
    parts = [I.ring_helix(n, round(n / 10), center=(0, 0, 15.0 * m)) if c else I.straight_helix(n, (0, 0, 15.0 * m))
             for m, (n, c) in enumerate(zip(n_bp, ring))]
    X, u = I.perturb(np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), rng, dx=0.005, dtheta=0.01)
    V, Om = I.maxwell(u, rng)
    _both(n_bp, X, u, V, Om, 400, 8, ring=ring, precision=prec, list_build=1, skin=0.1, seed=7, dt=0.002,
          K2=1.0 if rule else 6.0, bubble_rule=rule)


@pytest.mark.parametrize("prec", PRECS)
def test_just_above_the_resident_limit(prec):
    """The default choice of path for the shortest system that no longer fits a stretch per SM."""
    import torch
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    n = nsm * (256 if prec == D.PREC_MIXED else 128) + 8
    cfg = I.c1_linear(n)
    X, u = I.perturb(cfg.X, cfg.u, np.random.default_rng(1), dx=0.01, dtheta=0.02)
    _both(cfg.n_bp, X, u, cfg.V, cfg.Om, 100, 5, modes=(1, 0), precision=prec, skin=0.1, seed=6)
