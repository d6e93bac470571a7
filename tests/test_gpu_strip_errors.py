"""Errors that single threads of the strip kernels find before a grid barrier: the closing bond of a ring (junction owners)
and lists beyond their capacity in the rebuild inside the step kernel are reported whichever thread meets them."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PRECS = [D.PREC_MIXED, D.PREC_FP64]


def _status(call):
    try:
        call()
    except D.DsdnaError as e:
        return e.status
    return "OK"


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("mode,list_build", [(1, 0), (2, 0), (2, 1)])
def test_broken_closing_bond(prec, mode, list_build):
    """60 of the 66 base pairs of a planar ring: only the bonds across the junction are beyond their limit."""
    X, u = I.ring_helix(66, 7)
    X, u = X[:120], u[:120]
    for what in ("forces", "energy", "step"):
        ctx = D.Context(D.dsdna_default_params(precision=prec, rebuild_mode=mode, list_build=list_build, R0=1.5), [60], X=X, u=u,
                        circular=[1])
        call = {"forces": ctx.compute_forces, "energy": ctx.energy_virial,
                "step": lambda: (ctx.step(5), ctx.synchronize())}[what]
        assert _status(call) == "EFENE", what
        ctx.close()
    ctx = D.Context(D.dsdna_default_params(precision=prec, R0=1.5), [60], X=X, u=u)      # the same base pairs, open
    assert _status(ctx.compute_forces) == "OK"
    ctx.close()


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("mode,list_build", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_overflow_in_a_rebuild(prec, mode, list_build):
    """A melting molecule whose beads first have at most two listed partners, then three (the separate rebuild kernels
    say so, mode 1)."""
    cfg = I.c1_linear(120)
    X, u = I.perturb(cfg.X, cfg.u, np.random.default_rng(1), dx=0.02, dtheta=0.05)
    ctx = D.Context(D.dsdna_default_params(precision=prec, rebuild_mode=mode, list_build=list_build, max_neighbors=2,
                                           skin=0.05, seed=5, K2=0.5), cfg.n_bp, X=X, u=u, V=cfg.V, Om=cfg.Om)
    ctx.step(20)
    assert _status(ctx.synchronize) == "OK"
    ctx.step(380)
    assert _status(ctx.synchronize) == "EOVERFLOW"
    ctx.close()
