"""The single-launch force call over many clears of its device words (a build that clears them every fourth call), with
grids that grow and shrink from call to call and a failed call in between: always the context's forces, bit for bit."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1608_03722_gb300 import _build
from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch
    D.load()
    d = tmp_path_factory.mktemp("calls")
    obj, so = str(d / "noalloc.o"), str(d / "calls.so")
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-DDSDNA_ONCE_CALLS=4", "-c",
                           os.path.join(_build.CSRC, "noalloc.cu"), "-o", obj])
    others = [os.path.join(_build.BUILD, f.replace(".cu", ".o")) for f in _build.SOURCES if f != "noalloc.cu"]
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-shared", "-o", so, obj, *others])
    lib = C.CDLL(so, mode=os.RTLD_LOCAL)

    def f(p, n_bp, X, u):
        nb = np.ascontiguousarray(n_bp, np.int32)
        ins = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (X, u)]
        F = [torch.full((len(X), 3), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
        rc = lib.dsdna_forces_noalloc(C.byref(p), len(nb), nb.ctypes.data_as(C.POINTER(C.c_int)),
                                      *[C.c_void_p(t.data_ptr()) for t in (*ins, *F)],
                                      C.c_void_p(torch.cuda.current_stream().cuda_stream))
        return rc, [a.cpu().numpy() for a in F]
    return f


def test_forces_across_clears(call):
    p = D.dsdna_default_params()
    systems = []
    for k, lengths in enumerate([[3], [700, 1, 129], [8192], [40] * 5, [1216]]):
        cfg = I.ragged_batch(lengths, seed=k, spread=0.02)
        ctx = D.Context(p, cfg.n_bp, X=cfg.X, V=cfg.V, u=cfg.u, Om=cfg.Om)
        systems.append((cfg, ctx.compute_forces()))
        ctx.close()
    rng = np.random.default_rng(2)
    for k in range(40):
        cfg, want = systems[rng.integers(len(systems))]
        if k % 11 == 6:                              # a broken bond: the call fails and the next one starts over
            X = cfg.X.copy()
            X[:2] += 50.0
            rc, _ = call(p, cfg.n_bp, X, cfg.u)
            assert D.STATUS[rc] == "EFENE"
        rc, got = call(p, cfg.n_bp, cfg.X, cfg.u)
        assert rc == 0, k
        for a, b in zip(got, want):
            assert np.array_equal(a, b), k
