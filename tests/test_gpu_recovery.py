"""A context after an error during steps: the state read is that of one step, the step counter is the device's, and a new
state goes on exactly as it does on a context that took the same number of steps without an error."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("mode,list_build", [(1, 0), (2, 0), (2, 1)])
@pytest.mark.parametrize("first,sync", [(1, True), (2, True), (1, False)])
def test_overflow_and_a_new_state(prec, mode, list_build, first, sync):
    cfg = I.c1_linear(120)
    X, u = I.perturb(cfg.X, cfg.u, np.random.default_rng(1), dx=0.02, dtheta=0.05)
    kw = dict(precision=prec, skin=0.05, seed=5, K2=0.5)

    def make(**more):
        return D.Context(D.dsdna_default_params(**kw, **more), cfg.n_bp, X=X, u=u, V=cfg.V, Om=cfg.Om)

    ctx, ref = make(max_neighbors=2, rebuild_mode=mode, list_build=list_build), make()
    ctx.step(first)                                  # the error at either parity of the step the call ends at
    ctx.step(200 - first)
    if sync:
        with pytest.raises(D.DsdnaError) as e:
            ctx.synchronize()
        assert e.value.status == "EOVERFLOW"
        got = ctx.get_state()
        for t in range(200):
            want = ref.get_state()
            if np.array_equal(got[1], want[1]):
                break
            ref.step(1)
        for a, b in zip(got, want):
            assert np.array_equal(a, b), t
        assert ctx.step_counter == t
    ctx.set_state(-1, cfg.X, cfg.V, cfg.u, cfg.Om)
    t = ctx.step_counter
    assert 0 < t < 200
    if not sync:
        ref.step(t)
    ref.set_state(-1, cfg.X, cfg.V, cfg.u, cfg.Om)
    for k in (0, 1, 9):
        for c in (ctx, ref):
            c.step(k)
        for a, b in zip(ctx.get_state(), ref.get_state()):
            assert np.array_equal(a, b), k
    assert ctx.observables(0, D.OBS_EXT | D.OBS_TW) == ref.observables(0, D.OBS_EXT | D.OBS_TW)
    assert ctx.step_counter == t + 10
    ctx.close()
    ref.close()


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("mode,list_build", [(1, 0), (2, 0), (2, 1)])
@pytest.mark.parametrize("steps", [4, 5])
def test_state_after_a_broken_bond(prec, mode, list_build, steps):
    """An error of a step's forces: the state shows that step taken (it is not counted), positions and orientations of the
    same step."""
    cfg = I.c1_linear(40)
    X = cfg.X.copy()
    X[2 * 20:, 2] += 0.25                            # a bond close to its limit: no error yet
    V = cfg.V.copy()
    V[2 * 20:, 2] += 20.0                            # within a few steps beyond it
    out = []
    for k in (0, 1):
        ctx = D.Context(D.dsdna_default_params(precision=prec, rebuild_mode=mode, list_build=list_build, seed=5), cfg.n_bp,
                        X=X, u=cfg.u, V=V, Om=cfg.Om)
        ctx.step(steps + k)
        with pytest.raises(D.DsdnaError) as e:
            ctx.synchronize()
        assert e.value.status == "EFENE"
        out.append([*ctx.get_state(), np.array([ctx.step_counter])])
        ctx.close()
    for a, b in zip(*out):                           # whatever the parity of the step the call would have ended at
        assert np.array_equal(a, b)
