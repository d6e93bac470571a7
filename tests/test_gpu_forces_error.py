"""dsdna_compute_forces after a device-side error (a backbone bond beyond its limit): the caller's arrays stay as they
were, the context is poisoned, and a new state brings the forces back."""
import ctypes as C

import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("n_bp", [40, 3000])
def test_arrays_untouched_after_an_error(prec, n_bp):
    cfg = I.c1_linear(n_bp)
    X = cfg.X.copy()
    X[:2] += 50.0
    ctx = D.Context(D.dsdna_default_params(precision=prec), cfg.n_bp, X=X, V=cfg.V, u=cfg.u, Om=cfg.Om)
    F = [np.full(3 * cfg.n_nt, 7.0) for _ in range(2)]
    ptr = [f.ctypes.data_as(C.POINTER(C.c_double)) for f in F]
    L = D.load()
    assert D.STATUS[L.dsdna_compute_forces(ctx.h, *ptr)] == "EFENE"
    assert (F[0] == 7.0).all() and (F[1] == 7.0).all()
    assert D.STATUS[L.dsdna_compute_forces(ctx.h, *ptr)] == "ESTATE"
    ctx.set_state(-1, cfg.X, cfg.V, cfg.u, cfg.Om)
    assert L.dsdna_compute_forces(ctx.h, *ptr) == 0
    want = ctx.compute_forces()
    assert np.array_equal(F[0].reshape(-1, 3), want[0]) and np.array_equal(F[1].reshape(-1, 3), want[1])
    assert L.dsdna_compute_forces(ctx.h, None, ptr[1]) == 0
    ctx.close()
