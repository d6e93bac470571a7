"""Performance cases of the dsDNA engine: the calls that users of this package make, at the sizes its
configurations, experiments and benchmark use.

Every case is one pass through the public entry points (``dsdna.Context``, ``dsdna_forces_noalloc``,
``surrogate.Surrogate``, ``surrogate.Mlp``).  ``prepare`` builds what a program holds before the call
(a context with its initial state, host buffers, a network), ``run`` makes the call, and ``exact`` says
what the call returns in plain 64-bit torch arithmetic (App. A and Sec. 2-5 of arXiv:1608.03722).
"""
from __future__ import annotations

import ctypes as C
import functools
import math
import random

import numpy as np
import torch

from paper_1608_03722_gb300 import dsdna as D
from paper_1608_03722_gb300 import inputs as I
from paper_1608_03722_gb300 import surrogate as S


# ---------------------------------------------------------------- the cases
def listed() -> list[dict]:
    return [
        # the paper's 200 bp molecule on the all-FP64 path: the shortest run, all latency
        dict(name="linear_200bp_fp64", kind="steps", layout="linear", n_mol=1, n_bp=200, precision="fp64", steps=50),
        # one anchored 10 kbp molecule pulled and twisted (Sec. 4), the ordinary single-molecule run
        dict(name="tethered_10kbp", kind="steps", layout="tethered", n_mol=1, n_bp=10_000, precision="mixed", steps=100),
        # a confined self-avoiding chain of middle size in a periodic box
        dict(name="walk_30kbp", kind="steps", layout="walk", n_mol=1, n_bp=30_000, precision="mixed", steps=100),
        # 1 Mbp in a periodic box, the size of the throughput benchmark
        dict(name="confined_1mbp", kind="steps", layout="rows", n_mol=1, n_bp=1_000_000, precision="mixed", steps=100),
        # 256 ragged molecules, each with its own load, in one context: the sweep generator's batch, the largest call
        dict(name="batch_256", kind="steps", layout="batch", n_mol=256, n_bp=20_000, precision="mixed", steps=50),
        # supercoiled rings (Sec. 6): circular molecules, an odd length that steric typing does not divide
        dict(name="rings_64x500bp", kind="steps", layout="rings", n_mol=64, n_bp=500, precision="mixed", steps=100),
        # melting below the H-bond threshold (Sec. 5): bubble rule 2, weak hydrogen bonds
        dict(name="melt_16x1000bp", kind="steps", layout="melt", n_mol=16, n_bp=1000, precision="mixed", steps=100),
        # one sampling point of the twist experiment (Sec. 4.2): extension, twist and linking number of 7 x 16 molecules
        dict(name="sample_112x600bp", kind="observe", n_mol=112, n_bp=600, lk=True),
        # energies, virial and site forces of a confined chain: monitoring and analysis of a run
        dict(name="energy_forces_30kbp", kind="energy", layout="walk", n_mol=1, n_bp=30_000, precision="mixed"),
        # forces on device arrays for a caller that may not allocate, a ragged number of odd molecules
        dict(name="noalloc_5x1339bp", kind="noalloc", n_mol=5, n_bp=1339, periodic=False),
        # committee prediction of 2000 sweep points (candidate scoring)
        dict(name="predict_2000", kind="predict", rows=2000, members=4),
        # one Adam iteration of the surrogate on a minibatch
        dict(name="train_256", kind="train", rows=256),
    ]


def _log(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["steps"] * 6 + ["observe", "energy", "noalloc", "predict", "train", "train"])
    if kind == "steps":
        layout = rng.choice(["linear", "tethered", "walk", "rows", "batch", "rings", "melt"])
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        c = dict(kind=kind, layout=layout, n_mol=1, precision=prec, steps=rng.choice([20, 50, 73, 100]))
        if layout in ("linear", "tethered"):
            c["n_bp"] = _log(rng, 60, 20_000)
        elif layout == "walk":
            c["n_bp"] = _log(rng, 1500, 30_000)
        elif layout == "rows":
            c["n_bp"] = _log(rng, 40_000, 1_000_000)
        elif layout == "batch":
            c["n_mol"] = _log(rng, 8, 256)
            c["n_bp"] = _log(rng, 1000, 20_000)
            c["steps"] = rng.choice([20, 33, 50])
        elif layout == "rings":
            c["n_mol"] = _log(rng, 1, 256)
            c["n_bp"] = _log(rng, 100, 1000)
        else:
            c["n_mol"] = _log(rng, 2, 64)
            c["n_bp"] = _log(rng, 100, 2000)
        if prec == "fp64":        # the FP64 path is some twenty times slower per step
            c["steps"] = 20
            c["n_mol"] = min(c["n_mol"], 32)
            c["n_bp"] = min(c["n_bp"], 100_000)
        return c
    if kind == "observe":
        n_mol = _log(rng, 4, 128)
        return dict(kind=kind, n_mol=n_mol, n_bp=_log(rng, 100, min(3000, math.sqrt(4e7 / n_mol))), lk=rng.random() < 0.7)
    if kind == "energy":
        layout, n_mol = rng.choice(["walk", "linear", "batch"]), rng.choice([1, 17, 40])
        return dict(kind=kind, layout=layout, n_mol=1 if layout == "walk" else n_mol,
                    n_bp=_log(rng, 500, 30_000 if layout == "walk" or n_mol == 1 else 60_000 / n_mol),
                    precision=rng.choice(["mixed", "mixed", "fp64"]))
    if kind == "noalloc":
        periodic = rng.random() < 0.3
        n_mol = 1 if periodic else _log(rng, 1, 32)
        return dict(kind=kind, n_mol=n_mol, n_bp=_log(rng, 200 if periodic else 40, 8000 / n_mol), periodic=periodic)
    if kind == "predict":
        return dict(kind=kind, rows=_log(rng, 16, 4096), members=rng.choice([1, 4]))
    return dict(kind=kind, rows=_log(rng, 16, 2048))


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=4)
def _geometry(layout: str, n_mol: int, n_bp: int):
    """Molecule lengths, relaxed positions and orientations, box and loads of a layout (no seed: the
    jitter, the velocities and the noise are what differs from run to run)."""
    rng = np.random.default_rng(n_mol * 1_000_003 + n_bp)
    box, tether, ring, ef, et = (0.0, 0.0, 0.0), None, None, None, None
    if layout == "walk":
        n_mol = 1
        cfg = I.random_walk_helix(n_bp=n_bp, phi=0.05, max_joint_deg=30.0, clearance=2.2)
        lengths, X, u, box = cfg.n_bp, cfg.X, cfg.u, cfg.box
    elif layout == "rows":
        n_mol = 1
        cfg = I.c3_confined(n_bp=n_bp, phi=0.05)
        lengths, X, u, box = cfg.n_bp, cfg.X, cfg.u, cfg.box
    elif layout == "batch":
        cfg = I.c4_batch(n_mol, lo=max(20, n_bp // 40), hi=n_bp)
        lengths, X, u, tether, ef, et = cfg.n_bp, cfg.X, cfg.u, cfg.tether, cfg.ext_f, cfg.ext_t
    elif layout == "rings":
        Xs, us = zip(*[I.ring_helix(n_bp, round(n_bp / 10) - 3 * (n_bp >= 400), center=(0.0, 0.0, 40.0 * m))
                       for m in range(n_mol)])
        lengths, X, u = np.full(n_mol, n_bp, np.int32), np.concatenate(Xs), np.concatenate(us)
        ring = np.ones(n_mol, np.int32)
    elif layout == "bent":        # worm-like molecules, eight shapes
        parts = [I.wlc_helix(n_bp, 150.0, rng) for _ in range(min(8, n_mol))]
        X = np.concatenate([parts[m % len(parts)][0] for m in range(n_mol)])
        u = np.concatenate([parts[m % len(parts)][1] for m in range(n_mol)])
        lengths = np.full(n_mol, n_bp, np.int32)
        tether = np.ones(n_mol, np.int32)
    else:                          # linear, tethered, melt: straight relaxed helices
        X, u = I.straight_helix(n_bp)
        X, u = np.concatenate([X] * n_mol), np.concatenate([u] * n_mol)
        lengths = np.full(n_mol, n_bp, np.int32)
        if layout == "tethered":
            tether = np.ones(n_mol, np.int32)
            ef, et = np.tile([0.0, 0.0, 5.0], (n_mol, 1)), np.tile([0.0, 0.0, 2.0], (n_mol, 1))
    return lengths, X, u, box, tether, ring, ef, et


def _system(layout: str, n_mol: int, n_bp: int, seed: int) -> dict:
    """One seeded thermal-like configuration of the layout, with velocities and engine parameters."""
    lengths, X0, u0, box, tether, ring, ef, et = _geometry(layout, n_mol, n_bp)
    rng = np.random.default_rng(seed)
    X, u = I.perturb(X0, u0, rng, dx=0.01, dtheta=0.03)
    V, Om = I.maxwell(u, rng)
    if tether is not None:
        first = 2 * np.concatenate([[0], np.cumsum(lengths)[:-1]])
        for a in (V, Om):
            a[first] = 0.0
            a[first + 1] = 0.0
    kw = dict(box=box, seed=seed & 0xFFFFFFFF)
    if layout == "melt":
        kw.update(K2=1.4, bubble_rule=2, dt=0.002)
    return dict(lengths=lengths, X=X, u=u, V=V, Om=Om, tether=tether, ring=ring, ef=ef, et=et, kw=kw)


def _context(s: dict, precision: str):
    p = D.dsdna_default_params(precision=D.PREC_FP64 if precision == "fp64" else D.PREC_MIXED, **s["kw"])
    ctx = D.Context(p, s["lengths"], X=s["X"], V=s["V"], u=s["u"], Om=s["Om"], tether=s["tether"], circular=s["ring"])
    if s["ef"] is not None:
        for m in range(len(s["lengths"])):
            ctx.set_external_force_torque(m, s["ef"][m], s["et"][m])
    return ctx


def _noalloc_system(case: dict, seed: int) -> dict:
    if case["periodic"]:
        return _system("walk", 1, case["n_bp"], seed)
    s = _system("linear", case["n_mol"], case["n_bp"], seed)
    return s


def _network(seed: int, rows: int):
    """Sweep points, plausible labels, their scales and He-style weights W1 b1 W2 b2 W3 b3."""
    pts = S.sample_points(rows, seed)
    lab = np.stack([1.0 - 0.5 / np.sqrt(pts[:, 0] + 0.5), 0.01 * pts[:, 1], 0.05 * np.exp(-pts[:, 0] / 3)], 1)
    lab = lab + np.random.default_rng(seed + 1).normal(0, 0.01, lab.shape)
    m, sc = S.input_norm(pts)
    return pts.astype(np.float32), lab.astype(np.float32), [np.asarray(a, np.float32) for a in
                                                            (m, sc, lab.mean(0), lab.std(0) + 1e-6)]


def _weights(seed: int) -> np.ndarray:
    r = np.random.default_rng(seed)
    return np.concatenate([r.normal(0, math.sqrt(0.5), 256), r.normal(0, 0.1, 64), r.normal(0, math.sqrt(1 / 32), 4096),
                           r.normal(0, 0.1, 64), r.normal(0, 0.125, 192), r.normal(0, 0.1, 3)]).astype(np.float32)


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind in ("steps", "energy"):
        s = _system(case["layout"], case["n_mol"], case["n_bp"], seed)
        n = len(s["X"])
        out = tuple(torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy() for _ in range(4))
        return dict(case=case, ctx=_context(s, case["precision"]), out=out)
    if kind == "observe":
        s = _system("bent", case["n_mol"], case["n_bp"], seed)
        flags = D.OBS_EXT | D.OBS_DENAT | D.OBS_TW | (D.OBS_LK if case["lk"] else 0)
        return dict(case=case, ctx=_context(s, "mixed"), flags=flags, n_mol=case["n_mol"])
    if kind == "noalloc":
        s = _noalloc_system(case, seed)
        n = len(s["X"])
        dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
        return dict(case=case, lib=D.load(), p=D.dsdna_default_params(**s["kw"]), n_bp=s["lengths"].astype(np.int32),
                    X=dev(s["X"]), u=dev(s["u"]), Fb=torch.empty((n, 3), dtype=torch.float64, device="cuda"),
                    Fp=torch.empty((n, 3), dtype=torch.float64, device="cuda"),
                    stream=torch.cuda.current_stream().cuda_stream)
    pts, lab, norm = _network(seed, case["rows"])
    if kind == "predict":
        sur = S.Surrogate(case["members"], max_batch=max(4096, case["rows"]), seed=seed)
        for k, m in enumerate(sur.models):
            m.set_params(_weights(seed + 10 + k), *norm)
        sur.norm = tuple(norm)
        return dict(case=case, sur=sur, pts=pts)
    net = S.Mlp(max_batch=max(256, case["rows"]))
    net.set_params(_weights(seed + 10), *norm)
    return dict(case=case, net=net, X=torch.tensor(pts, device="cuda"), T=torch.tensor(lab, device="cuda"),
                Y=torch.empty((case["rows"], S.NO), dtype=torch.float32, device="cuda"))


# ---------------------------------------------------------------- the calls
def run(state: dict):
    case = state["case"]
    kind = case["kind"]
    if kind == "steps":                     # a stretch of a production run, then the state for the caller's own analysis
        ctx = state["ctx"]
        ctx.step(case["steps"])
        X, V, u, Om = ctx.get_state(out=state["out"])
        return dict(X=X, V=V, u=u, Om=Om)
    if kind == "energy":
        E, W = state["ctx"].energy_virial()
        Fb, Fp = state["ctx"].compute_forces()
        return dict(E=E, W=W, Fb=Fb, Fp=Fp)
    if kind == "observe":
        obs = [state["ctx"].observables(m, state["flags"]) for m in range(state["n_mol"])]
        keys = ("rz", "denat", "tw", "tw_ideal") + (("lk",) if case["lk"] else ())   # wr is lk - tw
        return {k: np.array([o[k] for o in obs]) for k in keys}
    if kind == "noalloc":
        rc = state["lib"].dsdna_forces_noalloc(
            C.byref(state["p"]), len(state["n_bp"]), state["n_bp"].ctypes.data_as(C.POINTER(C.c_int)),
            C.c_void_p(state["X"].data_ptr()), C.c_void_p(state["u"].data_ptr()), C.c_void_p(state["Fb"].data_ptr()),
            C.c_void_p(state["Fp"].data_ptr()), C.c_void_p(state["stream"]))
        if rc != 0:
            raise D.DsdnaError(rc, "dsdna_forces_noalloc")
        return dict(Fb=state["Fb"], Fp=state["Fp"])
    if kind == "predict":
        mean, spread = state["sur"].predict(state["pts"])
        return dict(mean=mean, spread=spread)
    net = state["net"]
    net.forward(state["X"], state["Y"])
    loss = net.backward(state["T"])
    net.adam(lr=3e-3, weight_decay=1e-2)
    params, grads = net.get_params()
    return dict(Y=state["Y"], loss=loss, params=params, grads=grads)


def work(case: dict) -> dict:
    """Bytes: a step reads and writes the integrator's state (mixed: X, V in 8 bytes, u, Omega in 4; FP64: all
    in 8) once, the caller's arrays move once.  Operations: about 700 per nucleotide and force evaluation."""
    kind = case["kind"]
    if kind in ("predict", "train"):
        net = 2 * (4 * 64 + 64 * 64 + 64 * 3)
        f = (case["members"] if kind == "predict" else 3) * net * case["rows"]
        return dict(bytes=4 * case["rows"] * 7 + 4 * 4675 * (case["members"] if kind == "predict" else 8), flops=f)
    if case.get("layout") == "batch":
        n = 2 * int(_geometry("batch", case["n_mol"], case["n_bp"])[0].sum())
    elif case.get("layout") in ("walk", "rows") or case.get("periodic"):
        n = 2 * case["n_bp"]
    else:
        n = 2 * case["n_mol"] * case["n_bp"]
    if kind == "steps":
        per = 2 * (96 if case["precision"] == "fp64" else 72)
        return dict(bytes=n * (case["steps"] * per + 96), flops=700 * n * case["steps"])
    if kind == "energy":
        return dict(bytes=n * (96 + 48), flops=1400 * n)
    if kind == "noalloc":
        return dict(bytes=n * (48 + 48), flops=700 * n)
    lk = 60 * (case["n_bp"] + 4) ** 2 * case["n_mol"] if case["lk"] else 0
    return dict(bytes=48 * n, flops=50 * n + lk)


# ---------------------------------------------------------------- 64-bit evaluation
# The model of Sec. 2 and App. A (Table 1) in plain torch: every term vectorised over the nucleotides.
_RC6 = 2.0 ** (1.0 / 6.0)


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


class _Model:
    def __init__(self, s: dict, dev: str):
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.dev = dev
        kw = s["kw"]
        self.K2, self.dt, self.seed = kw.get("K2", 6.0), kw.get("dt", 0.005), kw["seed"]
        self.rule2 = kw.get("bubble_rule", 0) == 2
        self.L = t(kw["box"]) if kw["box"][0] > 0 else None
        lengths = np.asarray(s["lengths"], np.int64)
        off = np.concatenate([[0], np.cumsum(lengths)])
        n = 2 * int(off[-1])
        g = np.arange(n)
        k = g // 2
        mol = np.repeat(np.arange(len(lengths)), 2 * lengths)
        N, kk, sB = lengths[mol], k - off[mol], g % 2
        q = np.where(sB == 0, kk, N - 1 - kk)
        ring = np.zeros(len(lengths), bool) if s["ring"] is None else np.asarray(s["ring"], bool)
        rg = ring[mol]
        self.steric = torch.tensor((q % 3 == 0) & ~(rg & (q > N - 3)), device=dev)

        def neighbour(d):     # strand neighbour d steps towards the 3' end, -1 outside a linear molecule
            k2 = kk + np.where(sB == 0, d, -d)
            out = (k2 < 0) | (k2 >= N)
            j = 2 * (off[mol] + k2 % N) + sB
            return torch.tensor(np.where(out & ~rg, -1, j), device=dev)

        self.n, self.mol = n, torch.tensor(mol, device=dev)
        self.local = torch.tensor(g - 2 * off[mol], device=dev)
        self.nxt, self.prv, self.nx2 = neighbour(1), neighbour(-1), neighbour(2)
        self.o = torch.nonzero(self.nxt >= 0).flatten()
        self.q = self.nxt[self.o]
        self.b = torch.nonzero((self.nxt >= 0) & (self.prv >= 0)).flatten()
        frozen = np.zeros(n, bool)
        if s["tether"] is not None:
            for m in np.flatnonzero(s["tether"]):
                frozen[2 * off[m]:2 * off[m] + 2] = True
        self.mobile = torch.tensor(~frozen, device=dev)[:, None].double()
        self.last = torch.tensor(2 * (off[1:] - 1), device=dev)
        self.ef = None if s["ef"] is None else t(s["ef"])
        self.et = None if s["et"] is None else t(s["et"])
        self.removed = torch.zeros((2, n), dtype=torch.bool, device=dev)
        self.X, self.u, self.V, self.Om = t(s["X"]), t(s["u"]), t(s["V"]), t(s["Om"])
        self.step = 0
        self.pairs_at = None

    def _delta(self, d):
        return d if self.L is None else d - self.L * torch.round(d / self.L)

    def pairs(self, beads, skin=0.5):
        """Typed bead pairs i < j of one molecule within range + skin; rebuilt when a bead moved skin / 2."""
        if self.pairs_at is not None and (beads - self.pairs_at).norm(dim=1).max() < 0.5 * skin:
            return self.pi, self.pj
        r = _RC6 + skin
        if self.L is not None:
            nc = torch.floor(self.L / r).long()
            w = beads - self.L * torch.floor(beads / self.L)
            c = torch.minimum(torch.floor(w / (self.L / nc)).long(), nc - 1)
        else:
            c = torch.floor((beads - beads.min(0).values) / r).long() + 1
            nc = c.max(0).values + 2
        if self.L is not None and int(nc.min()) < 3:     # a small box: every pair
            i, j = torch.triu_indices(self.n, self.n, 1, device=self.dev)
            cand = [(i, j)]
        else:
            def key(x):
                return ((self.mol * nc[2] + x[:, 2]) * nc[1] + x[:, 1]) * nc[0] + x[:, 0]
            ks, order = torch.sort(key(c))
            idx = torch.arange(self.n, device=self.dev)
            cand = []
            for dx in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    for dz in (-1, 0, 1):
                        x = c + torch.tensor([dx, dy, dz], device=self.dev)
                        x = x % nc if self.L is not None else x
                        kk = key(x)
                        lo, hi = torch.searchsorted(ks, kk), torch.searchsorted(ks, kk, right=True)
                        cnt = hi - lo
                        i = torch.repeat_interleave(idx, cnt)
                        at = torch.arange(len(i), device=self.dev) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt - lo, cnt)
                        j = order[at]
                        keep = i < j
                        cand.append(self._in_range(beads, i[keep], j[keep], skin))
            i, j = torch.cat([a for a, _ in cand]), torch.cat([b for _, b in cand])
            cand = [(i, j)]
        self.pi, self.pj = self._in_range(beads, *cand[0], skin)
        self.pairs_at = beads.clone()
        return self.pi, self.pj

    def _in_range(self, beads, i, j, skin):
        cut = self._sigma(i, j) * _RC6
        d = self._delta(beads[j] - beads[i])
        keep = (cut > 0) & (self.mol[i] == self.mol[j]) & ((d * d).sum(1) < (cut + skin) ** 2)
        return i[keep], j[keep]

    def _sigma(self, i, j):
        """Two steric beads 1 nm, any other pair across strands 0.5 nm, else none (0)."""
        both = self.steric[i] & self.steric[j]
        across = ((i ^ j) & 1) == 1
        one = torch.ones((), dtype=torch.float64, device=self.dev)
        return torch.where(both, one, torch.where(across, 0.5 * one, 0.0 * one))

    def forces(self):
        """Site forces (bead, patch), energies of the eight interaction terms, virial (xx yy zz xy xz yz)."""
        X, u = self.X, self.u
        bead, patch = X - 0.25 * u, X + 0.25 * u
        Fb, Fp = torch.zeros_like(X), torch.zeros_like(X)
        E = torch.zeros(10, dtype=torch.float64, device=self.dev)
        W = torch.zeros((3, 3), dtype=torch.float64, device=self.dev)

        def add(F, i, f):
            F.index_add_(0, i, f)

        def vir(r, f):
            W.add_(r.T @ f)

        o, q = self.o, self.q
        # FENE and backbone WCA (Eq. 9)
        d = bead[q] - bead[o]
        r2 = _dot(d, d)
        w = 1.0 - r2 / 0.6825 ** 2
        E[0] = (-0.5 * 30.0 * 0.6825 ** 2 * torch.log(w)).sum()
        fr = -30.0 / w
        s6 = (0.443 ** 2 / r2) ** 3
        inside = (r2 < (_RC6 * 0.443) ** 2).double()
        fr = fr + inside * 24.0 * s6 * (2.0 * s6 - 1.0) / r2
        E[1] = (inside * 4.0 * (s6 * s6 - s6 + 0.25)).sum()
        f = fr * d
        add(Fb, q, f); add(Fb, o, -f); vir(d, f)
        # Morse (Eq. 13)
        d = patch[q] - patch[o]
        r = _dot(d, d).sqrt()
        x = torch.exp(-8.0 * (r - 0.34))
        E[5] = (30.0 * (1.0 - x) ** 2).sum()
        f = (-480.0 * x * (1.0 - x) / r) * d
        add(Fp, q, f); add(Fp, o, -f); vir(d, f)
        # bubble rule 2 (Sec. 5): terms removed for good inside runs of three open pairs
        keep_dih = torch.ones(len(o), dtype=torch.float64, device=self.dev)[:, None]
        keep_bend = torch.ones(len(self.b), dtype=torch.float64, device=self.dev)[:, None]
        dh = patch[1::2] - patch[0::2]
        r2h = _dot(dh, dh)
        if self.rule2:
            op = (r2h > 0.09).flatten().repeat_interleave(2)
            at = lambda j: op[j.clamp(min=0)] & (j >= 0)  # noqa: E731
            here, nxt, prv, far = op, at(self.nxt), at(self.prv), at(self.nx2)
            self.removed[0] |= here & nxt & (prv | far)
            self.removed[1] |= here & nxt & prv & (self.prv >= 0)
            keep_dih = (~self.removed[0][o]).double()[:, None]
            keep_bend = (~self.removed[1][self.b]).double()[:, None]
        # dihedral bead-patch-patch-bead (Eq. 12)
        A, B2, B3, Q = bead[o], patch[o], patch[q], bead[q]
        b1, b2, b3 = B2 - A, B3 - B2, Q - B3
        n1, n2 = _cross(b1, b2), _cross(b2, b3)
        l2 = _dot(b2, b2)
        lb = l2.sqrt()
        phi = torch.atan2(lb * _dot(b1, n2), _dot(n1, n2))
        dd = -144.0 * math.pi / 180.0
        E[4] = (keep_dih * 50.0 * (1.0 + torch.cos(phi - dd))).sum()
        dU = -50.0 * torch.sin(phi - dd) * keep_dih
        fA, fQ = (dU * lb / _dot(n1, n1)) * n1, (-dU * lb / _dot(n2, n2)) * n2
        p, qq = _dot(b1, b2) / l2, _dot(b3, b2) / l2
        fE, fF = (-1.0 - p) * fA + qq * fQ, p * fA - (1.0 + qq) * fQ
        add(Fb, o, fA); add(Fp, o, fE); add(Fp, q, fF); add(Fb, q, fQ)
        ref = X[o]
        vir(A - ref, fA); vir(B2 - ref, fE); vir(B3 - ref, fF); vir(Q - ref, fQ)
        # planarity, vertex patch q (Eq. 14)
        f1, f2, e = self._angle(B2 - B3, Q - B3, lambda cs, al, sn: (200.0 * (al - 0.5 * math.pi) / sn, 100.0 * (al - 0.5 * math.pi) ** 2))
        E[6] = e.sum()
        add(Fp, o, f1); add(Fb, q, f2); add(Fp, q, -(f1 + f2))
        vir(B2 - B3, f1); vir(Q - B3, f2)
        # bending of three patches (Eq. 15)
        b, bp, bn = self.b, self.prv[self.b], self.nxt[self.b]
        v1, v2 = patch[bp] - patch[b], patch[bn] - patch[b]
        f1, f2, e = self._angle(v1, v2, lambda cs, al, sn: (-52.0 * torch.ones_like(cs), 52.0 * (1.0 + cs)))
        f1, f2 = keep_bend * f1, keep_bend * f2
        E[7] = (keep_bend * e).sum()
        add(Fp, bp, f1); add(Fp, bn, f2); add(Fp, b, -(f1 + f2))
        vir(v1, f1); vir(v2, f2)
        # hydrogen bond (Eq. 10)
        kh = self.K2 / (2.0 * 0.09)
        closed = (r2h <= 0.09).double()
        f = closed * 2.0 * kh * dh
        Fp[0::2] += f
        Fp[1::2] -= f
        E[2] = (closed * kh * (r2h - 0.09)).sum()
        vir(dh, -f)
        # typed WCA (Eq. 11)
        i, j = self.pairs(bead)
        d = self._delta(bead[j] - bead[i])
        sg = self._sigma(i, j)[:, None]
        r2 = _dot(d, d)
        inside = (r2 < (_RC6 * sg) ** 2).double()
        s6 = (sg * sg / r2) ** 3
        E[3] = (inside * 4.0 * (s6 * s6 - s6 + 0.25)).sum()
        f = inside * 24.0 * s6 * (2.0 * s6 - 1.0) / r2 * d
        add(Fb, j, f); add(Fb, i, -f); vir(d, f)
        # loads on the last base pair (Sec. 4)
        if self.ef is not None:
            a, c = self.last, self.last + 1
            th = self.et / self.et.norm(dim=1, keepdim=True).clamp(min=1e-300)
            rho = 0.5 * (X[a] - X[c])
            rho = rho - _dot(rho, th) * th
            S2 = 2.0 * _dot(rho, rho)
            couple = torch.where(S2 > 1e-12, _cross(self.et, rho) / S2, torch.zeros_like(rho))
            for at, sign in ((a, 1.0), (c, -1.0)):
                f = 0.5 * (0.5 * self.ef + sign * couple)
                add(Fb, at, f); add(Fp, at, f)
        return Fb, Fp, E, torch.stack([W[0, 0], W[1, 1], W[2, 2], W[0, 1], W[0, 2], W[1, 2]])

    @staticmethod
    def _angle(v1, v2, law):
        i1, i2 = 1.0 / _dot(v1, v1).sqrt(), 1.0 / _dot(v2, v2).sqrt()
        e1, e2 = i1 * v1, i2 * v2
        cs = _dot(e1, e2).clamp(-1.0, 1.0)
        sn = (1.0 - cs * cs).sqrt().clamp(min=1e-6)
        k, e = law(cs, torch.acos(cs), sn)
        return (k * i1) * (e2 - cs * e1), (k * i2) * (e1 - cs * e2), e

    def total(self):
        """Force and torque on each nucleotide with friction and noise (App. A Eq. 8); energies, virial."""
        Fb, Fp, E, W = self.forces()
        eb, ep = self._noise()
        Ft = Fb + Fp - 2.0 * self.V + eb + ep
        Tt = 0.25 * _cross(self.u, Fp - Fb) - 0.125 * self.Om + 0.25 * _cross(self.u, ep - eb)
        return Ft * self.mobile, Tt * self.mobile, E, W

    def energy(self):
        Ft, Tt, E, W = self.total()
        Vf = self.V + 0.25 * self.dt * Ft
        Of = self.Om + 4.0 * self.dt * Tt
        Of = Of - _dot(Of, self.u) * self.u
        E[8] = (self.mobile * Vf * Vf).sum()
        E[9] = (self.mobile * 0.0625 * Of * Of).sum()
        return E, W

    def advance(self, steps):
        for _ in range(steps):
            Ft, Tt, _, _ = self.total()
            self.V = self.V + 0.5 * self.dt * Ft
            Om = self.Om + 8.0 * self.dt * Tt
            self.Om = Om - _dot(Om, self.u) * self.u
            self.X = self.X + self.dt * self.V * self.mobile
            w = self.Om.norm(dim=1, keepdim=True)
            ax = self.Om / w.clamp(min=1e-300)
            un = torch.cos(w * self.dt) * self.u + torch.sin(w * self.dt) * _cross(ax, self.u)
            self.u = un / un.norm(dim=1, keepdim=True)
            self.step += 1
        return self.X, self.V, self.u, self.Om

    def _noise(self):
        """Variance-matched uniform noise of both sites from one Philox4x32-10 draw per nucleotide and step."""
        mask = 0xFFFFFFFF
        z = torch.zeros_like(self.local)
        c = [self.local, z + self.step, z, self.mol]
        k0, k1 = self.seed & mask, 0

        def mulhilo(m, a):
            lo = (a & 0xFFFF) * m
            t = (a >> 16) * m + (lo >> 16)
            return (t >> 16) & mask, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

        for _ in range(10):
            h0, l0 = mulhilo(0xD2511F53, c[0])
            h1, l1 = mulhilo(0xCD9E8D57, c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        x, y, v, w = c
        k = torch.stack([x >> 11, y >> 11, v >> 11, w >> 11, (x & 0x7FF) | ((y & 0x3FF) << 11),
                         (v & 0x7FF) | ((w & 0x3FF) << 11)], 1)
        e = (k.double() - 1048575.5) * (math.sqrt(24.0 / self.dt) * 2.0 ** -21)
        return e[:, :3], e[:, 3:]


def _observables(X, u, n_bp: int, lk: bool):
    """R_z, denatured fraction, twist and linking number of one linear molecule (Sec. 3.2, 4.1, 5, App. B, C)."""
    patch, bead = X + 0.25 * u, X - 0.25 * u
    mid = 0.5 * (patch[0::2] + patch[1::2])
    ca, cb = bead[0::2], bead[1::2]
    unit = lambda a: a / a.norm(dim=-1, keepdim=True)  # noqa: E731
    t = unit(mid[1:] - mid[:-1])
    w = (cb - ca)[:-1]
    f = unit(w - _dot(w, t) * t)
    v = _cross(t, f)
    f0, v0, f1, v1 = f[:-1], v[:-1], f[1:], v[1:]
    tw = torch.atan2((_dot(v0, f1) - _dot(f0, v1)), (_dot(f0, f1) + _dot(v0, v1))).sum() / (2.0 * math.pi)
    opened = ((patch[1::2] - patch[0::2]).norm(dim=1) > 0.3).double().mean()
    out = [float(mid[-1, 2] - mid[0, 2]), float(opened), float(tw), (n_bp - 2) * 0.1]
    if lk:
        ext = max(float((ca - mid[0]).norm(dim=1).max()), float((cb - mid[0]).norm(dim=1).max()))
        e = unit(mid[-1] - mid[0])
        axis = torch.tensor([0.0, 1.0, 0.0] if abs(float(e[0])) > 0.9 else [1.0, 0.0, 0.0], dtype=torch.float64, device=X.device)
        side = unit(_cross(e, axis))
        far, step = ext + 5.0, 2.0 * ext + 10.0
        close = lambda p: torch.cat([p, torch.stack([p[-1] + far * e, p[-1] + far * e + step * side,  # noqa: E731
                                                     p[0] - far * e + step * side, p[0] - far * e])])
        a, b = close(ca), close(cb)
        a2, b2 = a.roll(-1, 0), b.roll(-1, 0)
        total = 0.0
        for i in range(0, len(a), 256):   # solid angle of each segment pair's quadrilateral as two triangles
            p, q = a[i:i + 256, None], a2[i:i + 256, None]
            r13, r14, r23, r24 = b - p, b2 - p, b - q, b2 - q
            l13, l14, l23, l24 = [x.norm(dim=-1) for x in (r13, r14, r23, r24)]
            d = lambda x, y: (x * y).sum(-1)  # noqa: E731
            t1, t2 = d(r13, _cross(r14, r24)), d(r13, _cross(r24, r23))
            w1 = torch.atan2(t1, l13 * l14 * l24 + d(r13, r14) * l24 + d(r14, r24) * l13 + d(r24, r13) * l14)
            w2 = torch.atan2(t2, l13 * l24 * l23 + d(r13, r24) * l23 + d(r24, r23) * l13 + d(r23, r13) * l24)
            total += float((w1 + w2).sum())
        out.append(-2.0 * total / (4.0 * math.pi))
    return out


def _network_exact(P, x, norm):
    """The 4-64-64-3 GELU network in 64 bits: normalised input, activations, normalised and scaled output."""
    W1, b1, W2, b2, W3, b3 = torch.split(P, [256, 64, 4096, 64, 192, 3])
    xn = (x - norm[0]) / norm[1]
    z1 = xn @ W1.view(64, 4).T + b1
    z2 = torch.nn.functional.gelu(z1) @ W2.view(64, 64).T + b2
    yn = torch.nn.functional.gelu(z2) @ W3.view(3, 64).T + b3
    return yn, norm[2] + norm[3] * yn


def exact(case: dict, seed: int):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    num = lambda a: a.cpu().numpy()  # noqa: E731
    if kind == "steps":
        m = _Model(_system(case["layout"], case["n_mol"], case["n_bp"], seed), dev)
        if m.n * case["steps"] > 220_000_000:
            return None
        X, V, u, Om = m.advance(case["steps"])
        return dict(X=num(X), V=num(V), u=num(u), Om=num(Om))
    if kind == "energy":
        m = _Model(_system(case["layout"], case["n_mol"], case["n_bp"], seed), dev)
        Fb, Fp, _, _ = m.forces()
        E, W = m.energy()
        return dict(E=num(E), W=num(W), Fb=num(Fb), Fp=num(Fp))
    if kind == "noalloc":
        m = _Model(_noalloc_system(case, seed), dev)
        Fb, Fp, _, _ = m.forces()
        return dict(Fb=Fb, Fp=Fp)
    if kind == "observe":
        s = _system("bent", case["n_mol"], case["n_bp"], seed)
        # the mixed path keeps the orientation in 32 bits: the observables are those of that state
        X, u = torch.tensor(s["X"], device=dev), torch.tensor(s["u"], device=dev).float().double()
        n = 2 * case["n_bp"]
        rows = np.array([_observables(X[k * n:(k + 1) * n], u[k * n:(k + 1) * n], case["n_bp"], case["lk"])
                         for k in range(case["n_mol"])])
        keys = ("rz", "denat", "tw", "tw_ideal") + (("lk",) if case["lk"] else ())
        return {k: rows[:, i].copy() for i, k in enumerate(keys)}
    pts, lab, norm = _network(seed, case["rows"])
    t = lambda a: torch.tensor(a, dtype=torch.float64)  # noqa: E731
    nd = [t(a) for a in norm]
    if kind == "predict":
        Y = torch.stack([_network_exact(t(_weights(seed + 10 + k)), t(pts), nd)[1] for k in range(case["members"])])
        return dict(mean=num(Y.mean(0)), spread=num(Y.std(0, correction=0)))
    P = t(_weights(seed + 10)).requires_grad_(True)
    yn, Y = _network_exact(P, t(pts), nd)
    loss = ((yn - (t(lab) - nd[2]) / nd[3]) ** 2).mean()
    loss.backward()
    g, p = P.grad, P.detach()
    decay = torch.ones_like(p)
    for lo, hi in ((256, 320), (4416, 4480), (4672, 4675)):
        decay[lo:hi] = 0.0
    new = p - 3e-3 * (g / (g.abs() + 1e-8) + 1e-2 * decay * p)      # the first Adam step, bias-corrected
    return dict(Y=num(Y.detach()), loss=float(loss.detach()), params=num(new), grads=num(g))
