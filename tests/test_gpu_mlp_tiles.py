"""Surrogate kernels at the edges of their 32-row batch tiles."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1608_03722_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

N = dict(in_mean=np.array([5.0, 0.0, 1e4, 1.1]), in_scale=np.array([5.0, 5.0, 1e4, 0.3]),
         out_mean=np.array([0.8, 0.0, 0.02]), out_scale=np.array([0.1, 0.03, 0.02]))


def _net(p, B):
    net = S.Mlp(max_batch=B)
    net.set_params(p, N["in_mean"], N["in_scale"], N["out_mean"], N["out_scale"])
    return net


@pytest.mark.parametrize("B", [1, 31, 32, 33, 63, 129, 2047])
def test_partial_tiles(B):
    """A row's outputs do not depend on the batch it is in (bit for bit), rows
    past the batch stay as they are, and the gradients hold the bound of the
    gradient test (1e-2 of each block's norm)."""
    import torch
    rng = np.random.default_rng(5)
    p = (M.init_params(3) + rng.normal(0, 0.05, M.NP)).astype(np.float32)
    n = 2048
    X = np.stack([rng.uniform(0.1, 10, n), rng.uniform(-5, 5, n), rng.uniform(500, 2e4, n), rng.uniform(0.8, 1.4, n)],
                 1).astype(np.float32)
    T = (N["out_mean"] + N["out_scale"] * rng.normal(0, 1, (n, 3))).astype(np.float32)
    Xd, Td = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    whole = torch.empty((n, 3), device="cuda")
    net = _net(p, n)
    net.forward(Xd, whole)
    net.close()
    net = _net(p, B)
    Y = torch.full((n, 3), 7.0, device="cuda")
    net.forward(Xd[:B], Y)
    loss = net.backward(Td[:B])
    _, g = net.get_params()
    net.close()
    assert torch.equal(Y[:B], whole[:B]) and bool((Y[B:] == 7.0).all())
    d = M.unpack(p.astype(np.float64))
    for k in ("W1", "W2", "W3"):
        d[k] = M.bf16(d[k])
    lo, go = M.loss_and_grad(M.pack(d), X[:B].astype(np.float64), T[:B].astype(np.float64), N)
    assert abs(loss - lo) < 1e-2 * lo
    gd, god = M.unpack(g.astype(np.float64)), M.unpack(go)
    for k, _ in M.SHAPES:
        rel = np.linalg.norm(gd[k] - god[k]) / max(np.linalg.norm(god[k]), 1e-30)
        assert rel < 1e-2, (k, rel)
