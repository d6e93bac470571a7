"""Contexts and networks on a caller's allocator whose blocks start 4 or 8 bytes past a 16-byte boundary: the same results
bit for bit as on aligned ones, and every block released."""
import numpy as np
import pytest

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I
from paper_1608_03722_gb300 import surrogate as S

pytestmark = pytest.mark.gpu


class Offset(D._TorchAllocator):
    offset, live_blocks = 0, 0

    def __init__(self, stream):
        import torch
        super().__init__(stream)
        self.base = {}

        def alloc(nbytes, user):
            p = torch.cuda.caching_allocator_alloc(int(nbytes) + 256, self.device, self.stream)
            self.base[p + Offset.offset] = p
            Offset.live_blocks += 1
            return p + Offset.offset

        def release(ptr, user):
            torch.cuda.caching_allocator_delete(self.base.pop(int(ptr)))
            Offset.live_blocks -= 1

        self.alloc_cb, self.release_cb = D.ALLOC_FN(alloc), D.RELEASE_FN(release)
        self.struct = D.dsdna_allocator(self.alloc_cb, self.release_cb, None)


def _each_offset(monkeypatch, run):
    monkeypatch.setattr(D, "_TorchAllocator", Offset)
    out = []
    for off in (0, 4, 8):
        Offset.offset = off
        out.append(run())
        assert Offset.live_blocks == 0
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", [D.PREC_MIXED, D.PREC_FP64])
@pytest.mark.parametrize("mode", [1, 2])
def test_context(monkeypatch, prec, mode):
    cfg = I.ragged_batch([300, 40, 129], seed=2, spread=0.01)

    def run():
        ctx = D.Context(D.dsdna_default_params(precision=prec, rebuild_mode=mode, skin=0.15), cfg.n_bp, X=cfg.X, V=cfg.V,
                        u=cfg.u, Om=cfg.Om)
        ctx.step(60)
        o = ctx.observables(0, D.OBS_EXT | D.OBS_DENAT | D.OBS_TW | D.OBS_LK)
        out = [*ctx.get_state(), *ctx.compute_forces(), np.array([o[k] for k in sorted(o)])]
        ctx.close()
        return out
    _each_offset(monkeypatch, run)


def test_network(monkeypatch):
    import torch
    rng = np.random.default_rng(1)
    X = torch.tensor(rng.uniform(-1, 1, (30, 4)), dtype=torch.float32, device="cuda")
    T = torch.tensor(rng.normal(0, 1, (30, 3)), dtype=torch.float32, device="cuda")
    p = S._he_init(3)

    def run():
        net = S.Mlp(max_batch=30)
        net.set_params(p)
        Y = torch.empty((30, 3), device="cuda")
        net.forward(X, Y)
        net.backward(T)
        g = net.get_params()[1]
        net.adam()
        net.close()
        return [Y.cpu().numpy(), g]      # one tile of rows: no gradient is a sum in any order
    _each_offset(monkeypatch, run)
