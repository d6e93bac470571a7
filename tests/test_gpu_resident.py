"""Step kernel of small systems (stretches of the chain kept in shared memory):
bitwise the trajectories of the strip kernel with separate rebuild kernels, at
the edges of its stretches and tables."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PRECS = [D.PREC_MIXED, D.PREC_FP64]


def _both(n_bp, X, u, V, Om, steps=120, tether=None, ring=None, loads=None, **kw):
    out = []
    for mode in (1, 2):
        ctx = D.Context(D.dsdna_default_params(rebuild_mode=mode, **kw), n_bp, X=X, u=u, V=V, Om=Om, tether=tether,
                        circular=ring)
        for m, (f, t) in enumerate(loads or []):
            ctx.set_external_force_torque(m, f, t)
        assert ctx.info()["rebuild_in_step"] == (mode == 2)
        done = 0
        for k in (1, 50, steps - 51):        # chunk edges: one step, a whole graph, a remainder
            ctx.step(k)
            done += k
        mask = ctx.get_bubble_mask()
        assert ctx.info()["rebuilds"] >= 1
        out.append([*ctx.get_state(), mask])
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def _ragged(lengths, seed):
    cfg = I.ragged_batch(lengths, seed=seed, spread=0.01)
    return cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("lengths", [[1], [7], [8], [9], [1] * 5 + [30, 2, 3], [8 * 152], [8 * 152 + 1], [2431, 3, 1700]])
def test_stretch_edges(prec, lengths):
    _both(*_ragged(lengths, len(lengths)), precision=prec, skin=0.1, seed=3)


@pytest.mark.parametrize("prec", PRECS)
def test_largest_stretch(prec):
    """The most nucleotides a CTA per SM holds on 152 SMs (512 per CTA, 256 in FP64)."""
    import torch
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    n_bp = nsm * (256 if prec == D.PREC_MIXED else 128)
    cfg = I.c1_linear(n_bp)
    X, u = I.perturb(cfg.X, cfg.u, np.random.default_rng(1), dx=0.01, dtheta=0.02)
    _both(cfg.n_bp, X, u, cfg.V, cfg.Om, precision=prec, skin=0.15, seed=6)


@pytest.mark.parametrize("prec", PRECS)
def test_more_list_entries_than_the_table(prec):
    """Skin 1 nm: over four partners per nucleotide, so the lists are walked in memory."""
    cfg = I.c1_linear(500)
    ctx = D.Context(D.dsdna_default_params(skin=1.0), cfg.n_bp, X=cfg.X, u=cfg.u, V=cfg.V, Om=cfg.Om)
    assert 2 * len(ctx.neighbor_pairs()) > 4.2 * cfg.n_nt
    ctx.close()
    _both(cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om, precision=prec, skin=1.0, seed=2)


@pytest.mark.parametrize("prec", PRECS)
def test_loads_and_dense_periodic_walk(prec):
    cfg = I.c4_batch(n_mol=5, lo=100, hi=900, seed=8, random_pose=True)
    _both(cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om, tether=cfg.tether, loads=list(zip(cfg.ext_f, cfg.ext_t)),
          precision=prec, skin=0.1, seed=3)
    cfg = I.random_walk_helix(n_bp=2500, phi=0.15, clearance=1.7, seed=4)
    _both(cfg.n_bp, cfg.X, cfg.u, cfg.V, cfg.Om, precision=prec, box=cfg.box, skin=0.1, seed=3)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("rule", [0, 2])
def test_rings_and_bubbles(prec, rule):
    """Rings down to 6 base pairs (several junctions per stretch), one longer than a stretch, a linear molecule
    between them, weak hydrogen bonds so that bubbles cross stretches and junctions."""
    rng = np.random.default_rng(5)
    n_bp = [60, 37, 40, 700, 45, 36]
    ring = [1, 1, 0, 1, 1, 1]
    parts = [I.ring_helix(n, round(n / 10), center=(0, 0, 15.0 * m)) if c else I.straight_helix(n, (0, 0, 15.0 * m))
             for m, (n, c) in enumerate(zip(n_bp, ring))]
    X, u = I.perturb(np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), rng, dx=0.005,
                     dtheta=0.01)
    V, Om = I.maxwell(u, rng)
    _both(n_bp, X, u, V, Om, ring=ring, precision=prec, skin=0.15, seed=7, dt=0.002, K2=1.0 if rule else 6.0,
          bubble_rule=rule, steps=400)


@pytest.mark.parametrize("lengths", [[1], [8], [9, 1, 7], [1] * 9, [16, 16, 16], [1216, 1217], [8192], [300] * 27])
@pytest.mark.parametrize("rule", [0, 1])
def test_single_launch_forces(lengths, rule):
    """dsdna_forces_noalloc in one launch: the forces of the context's separate
    rebuild and force kernels bit for bit, at stretch edges, at its size limit
    and with open base pairs."""
    import ctypes as C
    import torch
    cfg = I.ragged_batch(lengths, seed=len(lengths), spread=0.02)
    X = cfg.X.copy()
    kw = dict(bubble_rule=rule)
    if rule:
        for k in range(0, len(X) // 2 - 5, 40):          # runs of four open pairs
            for q in range(k, k + 4):
                r = X[2 * q + 1] - X[2 * q]
                X[2 * q + 1] += 0.5 * r / np.linalg.norm(r)
        kw["R0"] = 3.0
    p = D.dsdna_default_params(**kw)
    ctx = D.Context(p, cfg.n_bp, X=X, u=cfg.u, V=cfg.V, Om=cfg.Om)
    want = ctx.compute_forces()
    ctx.close()
    nb = cfg.n_bp.astype(np.int32)
    d = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (X, cfg.u)]
    F = [torch.full((len(X), 3), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
    for _ in range(3):
        rc = D.load().dsdna_forces_noalloc(C.byref(p), len(nb), nb.ctypes.data_as(C.POINTER(C.c_int)),
                                           *[C.c_void_p(t.data_ptr()) for t in (*d, *F)],
                                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        for a, b in zip(F, want):
            assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("rings,n_bp", [(30, 300), (250, 36), (40, 191)])
def test_rings_in_long_stretches(prec, rings, n_bp):
    """Stretches of more than 96 slots (FP64: up to 128), where junction owners have warps of their own: one or
    more junctions per stretch, molecules that end inside a segment."""
    parts = [I.ring_helix(n_bp, round(n_bp / 10), center=(0, 0, 0.5 * n_bp * m)) for m in range(rings)]
    rng = np.random.default_rng(9)
    X, u = I.perturb(np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), rng, dx=0.005, dtheta=0.01)
    V, Om = I.maxwell(u, rng)
    _both([n_bp] * rings, X, u, V, Om, ring=[1] * rings, precision=prec, skin=0.15, seed=4, dt=0.002, steps=80)
