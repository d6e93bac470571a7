"""A list overflow during steps in the resident kernel: the state read afterwards is that of the step whose list did not
fit, not of a step taken with the pairs left out, and the run can go on from it with a larger capacity."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("skin,first", [(0.05, 1), (0.02, 1), (0.05, 2)])
def test_state_after_an_overflow(prec, skin, first):
    cfg = I.c1_linear(120)
    X, u = I.perturb(cfg.X, cfg.u, np.random.default_rng(1), dx=0.02, dtheta=0.05)
    kw = dict(precision=prec, skin=skin, seed=5, K2=0.5)

    def make(**more):
        return D.Context(D.dsdna_default_params(**kw, **more), cfg.n_bp, X=X, u=u, V=cfg.V, Om=cfg.Om)

    def overflow(mode):
        ctx = make(max_neighbors=2, rebuild_mode=mode)
        assert ctx.info()["rebuild_in_step"] == (mode == 2) and ctx.info()["chain_list"]
        ctx.step(first)                              # the overflow at either parity of the step the call ends at
        ctx.step(400 - first)
        with pytest.raises(D.DsdnaError) as e:
            ctx.synchronize()
        assert e.value.status == "EOVERFLOW"
        state = ctx.get_state()
        ctx.close()
        return state

    got, stopped = overflow(2), overflow(1)          # the separate rebuild kernels stop at the build
    assert np.array_equal(got[1], stopped[1])
    ref = make()
    for t in range(400):
        want = ref.get_state()
        if np.array_equal(got[1], want[1]):
            break
        ref.step(1)
    for a, b in zip(got, want):
        assert np.array_equal(a, b), t
    assert np.bincount(ref.neighbor_pairs().ravel()).max() == 3      # and that list does not fit
    ref.close()
