"""Performance cases: what a run of the model has the library do.

Every case goes through the Python binding (``icarus.Icarus``) as a run
driver does: a grid is set up with its inner boundary, cone CME and state
(``prepare``), then ``run`` makes one pass of calls and takes the results to
the host.  Kinds:

* ``step``  — a stretch of steps between two outputs, then the state of every
  member (and the tracer, and a probe series at Earth where the case asks for
  them) read back.  Single level or a refined tree.
* ``cycle`` — an AMR cycle: steps, refinement flags, regrid, state.
* ``regrid`` — flags and regrid of a tree whose state was just set.
* ``train`` — the refinement pre-flagger trained from its initial weights.
* ``leaves`` — the pre-flagger's features and probabilities of every leaf.

The FP32 mode holds its state in float32, and the binding hands it out as
float64: a pass stores it, as a snapshot writer does, in the type it has.
Inputs are made from the seed alone: an expanding wind with a sector boundary
and a cone of fast plasma behind a steep front, evaluated at the cell centres.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_12867_gb300 import inputs as I
from paper_2211_12867_gb300.icarus import FP32_MIXED, FP64, MLP_PARAMS, Icarus, IcarusError

R_IN = 0.1
X_MIN = (R_IN, math.pi / 6, 0.0)
X_MAX = (2.0, 5 * math.pi / 6, 2 * math.pi)
GAMMA, CFL, CD, FLOOR = 1.5, 0.8, 0.8, 1e-8
CRIT = dict(e_refine=0.1, e_coarsen=0.0125, eps=0.01, dv=I.kms(50.0))
CAPACITY = 7


# ---------------------------------------------------------------- the cases
def _grid(name, kind, n, b, prec, steps=0, levels=1, stretch=1, members=1, tracer=0, probe=0, pool=0):
    return dict(name=name, kind=kind, n0=n[0], n1=n[1], n2=n[2], b0=b[0], b1=b[1], b2=b[2], prec=prec, steps=steps,
                levels=levels, stretch=stretch, members=members, tracer=tracer, probe=probe, pool=pool)


def listed():
    return [
        # the Low stretched grid of the resolution ladder, a probe series at Earth after every stretch of steps
        _grid("low_grid", "step", (60, 32, 96), (12, 8, 12), "fp32", steps=10, probe=16),
        # the smallest grid in use, in the mode that is checked against the oracle
        _grid("small_fp64", "step", (60, 16, 32), (12, 8, 8), "fp64", steps=10, stretch=0),
        # the ladder's Middle equidistant grid
        _grid("middle_grid", "step", (600, 64, 192), (24, 16, 48), "fp32", steps=10, stretch=0),
        # the headline single-level wedge
        _grid("wedge", "step", (512, 60, 180), (64, 60, 180), "fp32", steps=40, stretch=0),
        # one block of the wedge in FP64
        _grid("wedge_fp64", "step", (64, 60, 180), (64, 60, 180), "fp64", steps=6, stretch=0),
        # three levels around the CME's front on the stretched AMR grid, between two regrids
        _grid("amr3", "step", (264, 36, 96), (12, 12, 12), "fp32", steps=10, levels=3, pool=16000),
        # the same criterion-driven cycle in FP64: steps, flags, regrid
        _grid("amr2_cycle_fp64", "cycle", (60, 36, 96), (12, 12, 12), "fp64", steps=2, levels=2, pool=4000),
        # the density-tracer runs of the ladder on the Low grid
        _grid("tracer3", "step", (60, 32, 96), (12, 8, 12), "fp32", steps=10, levels=3, tracer=1, pool=8000),
        # an ensemble of CME draws that shares every launch
        _grid("ensemble", "step", (264, 36, 96), (12, 12, 12), "fp32", steps=10, members=6),
        # refinement flags and regrid of the stretched AMR grid
        _grid("regrid3", "regrid", (264, 36, 96), (12, 12, 12), "fp32", levels=3, pool=16000),
        # the pre-flagger: training, and the features and probabilities that replace the flags of a regrid
        dict(name="train", kind="train", samples=16384, batch=1024, epochs=1),
        _grid("leaves3", "leaves", (264, 36, 96), (12, 12, 12), "fp32", levels=3, pool=16000),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "amr", "amr", "cycle", "regrid", "train", "leaves"])
    if kind == "train":
        batch = rng.randint(96, 2048)
        return dict(kind=kind, samples=int(_log(rng, 1000, 16384)), batch=batch, epochs=1)
    if kind == "step":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        big = rng.random() < 0.4
        b = [2 * rng.randint(6, 32 if big else 12), 2 * rng.randint(3, 30 if big else 10),
             2 * rng.randint(4, 90 if big else 12)]
        cells = _log(rng, 4e4, 5e6 if prec == "fp32" else 4e5)
        n = [b[0], b[1] * max(1, round(36 / b[1])), b[2] * max(1, round(96 / b[2]))]
        n[0] *= max(1, round(cells / (n[0] * n[1] * n[2])))
        n[0] = min(n[0], b[0] * max(1, 700 // b[0]))
        members = rng.choice([1, 1, 1, 2, 3]) if n[0] * n[1] * n[2] < 1.5e6 else 1
        tracer = int(prec == "fp32" and rng.random() < 0.2)
        c = _grid("", kind, n, b, prec, steps=rng.randint(3, 12) if prec == "fp32" else rng.randint(1, 6),
                  stretch=int(n[0] < 350), members=members, tracer=tracer, probe=rng.choice([0, 0, 1, 33]))
    else:
        # refined trees: the 12^3 blocks of the AMR grid and the ladder's 12 x 8 x 12 ones, base grids of both sizes
        b = rng.choice([(12, 12, 12), (12, 12, 12), (12, 8, 12), (8, 8, 8), (16, 12, 16)])
        fp64 = kind == "cycle" or rng.random() < 0.15
        n = (b[0] * (rng.randint(4, 6) if fp64 else rng.randint(5, 22)), b[1] * round(36 / b[1]),
             b[2] * round(96 / b[2]))
        if kind == "leaves":
            b = (12, 12, 12) if b == (16, 12, 16) else b
            n = (b[0] * (n[0] // b[0]), b[1] * round(36 / b[1]), b[2] * round(96 / b[2]))
        levels = 2 if fp64 else rng.choice([2, 3, 3])
        c = _grid("", "step" if kind == "amr" else kind, n, b, "fp64" if fp64 else "fp32",
                  steps={"amr": rng.randint(2, 10), "cycle": rng.randint(1, 2)}.get(kind, 0), levels=levels,
                  tracer=int(kind == "amr" and not fp64 and rng.random() < 0.3), pool=16000)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _cmes(case, seed):
    """one cone CME per member, and the phase of its wind"""
    out = []
    for m in range(case["members"]):
        rng = np.random.default_rng(1000 * int(seed) + m)
        out.append((dict(t_start=0.0, t_max=I.hours(6.0), colat=0.5 * math.pi + math.radians(rng.uniform(-10, 10)),
                         lon=math.pi + math.radians(rng.uniform(-10, 10)), half_width=math.radians(rng.uniform(20, 30)),
                         v=I.kms(rng.uniform(800, 1200)), rho=rng.uniform(700, 1400),
                         p=I.pressure(1000.0, 8.0e5)), rng.uniform(0, 2 * math.pi, 3), rng.uniform(0.48, 0.55)))
    return out


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _wind(r, th, ph, phase):
    """Wind primitives at broadcastable centres (FP64 tensors), a list of 8."""
    lat = 0.5 * math.pi - th
    deg = math.pi / 180.0
    v_kms = 350.0 + 200.0 * (1.0 + torch.tanh((lat.abs() - 15 * deg) / (5 * deg)))
    n_cc = 300.0 * (v_kms / 450.0) ** -2
    sgn = torch.where(lat - 10 * deg * torch.sin(ph - phase[0]) >= 0.0, 1.0, -1.0).to(torch.float64)
    x = R_IN / r
    one = torch.ones_like(r + th + ph)
    vr, br0 = v_kms / 100.0, I.bfield(200.0) * sgn
    bp0 = -br0 * I.OMEGA * R_IN * torch.sin(th) / vr
    return [n_cc * x ** 2 * one, vr * one, 0.0 * one, -I.OMEGA * r * torch.sin(th) * one,
            I.pressure(1.0, 1.5e6) * n_cc * x ** 3 * one, br0 * x ** 2 * one, 0.0 * one, bp0 * x * one]


def _state(r, th, ph, cme, phase, front):
    """The wind with waves on it and a cone of fast plasma behind a front."""
    W = _wind(r, th, ph, phase)
    a = torch.sin(th) * math.sin(cme["colat"]) * torch.cos(ph - cme["lon"]) + torch.cos(th) * math.cos(cme["colat"])
    ang = torch.acos(a.clamp(-1.0, 1.0))
    s = 0.25 * (1 + torch.tanh((cme["half_width"] - ang) / 0.05)) * (1 + torch.tanh((front - r) / 0.01))
    s = s * 0.5 * (1 + torch.tanh((r - 0.6 * front) / 0.05))
    wave = torch.sin(3 * ph + phase[1]) * torch.sin(2 * th + 9 * r + phase[2])
    W[0] = W[0] * (1 + 1.5 * s) * (1 + 0.03 * wave)
    W[1] = W[1] + s * (cme["v"] - W[1])
    W[2] = 0.1 * wave * torch.sin(th)
    W[3] = W[3] + 0.1 * wave * torch.cos(2 * th)
    W[4] = W[4] * (1 + 4.0 * s)
    W[6] = 0.02 * W[5].abs() * wave
    return W


def _faces(n, d, stretch, levels=1):
    n = n << (levels - 1)
    x = np.arange(-2, n + 3) / n
    if d == 0 and stretch:
        return X_MIN[0] * (X_MAX[0] / X_MIN[0]) ** x
    return X_MIN[d] + (X_MAX[d] - X_MIN[d]) * x


def _leaf_prims(case, tree, cme, phase, front):
    """[leaf][8][i][j][k] primitives at the centres of the leaves' cells"""
    dev, b = _device(), (case["b0"], case["b1"], case["b2"])
    cen = []
    for d in range(3):
        rows = np.empty((len(tree), b[d]))
        for lev in np.unique(tree[:, 0]):
            f = _faces((case["n0"], case["n1"], case["n2"])[d], d, case["stretch"], int(lev))
            c = 0.5 * (f[1:] + f[:-1])
            at = np.nonzero(tree[:, 0] == lev)[0]
            rows[at] = c[2 + tree[at, 1 + d][:, None] * b[d] + np.arange(b[d])[None, :]]
        cen.append(torch.from_numpy(rows).to(dev))
    r, th, ph = cen[0][:, :, None, None], cen[1][:, None, :, None], cen[2][:, None, None, :]
    out = torch.empty((len(tree), 8) + b, dtype=torch.float64, device=dev)
    for v, w in enumerate(_state(r, th, ph, cme, phase, front)):
        out[:, v] = w
    return out


def _map(case, phase):
    """inner-boundary primitives [8][n1][n2] at the base cells' angles"""
    f1, f2 = _faces(case["n1"], 1, 0), _faces(case["n2"], 2, 0)
    th = torch.from_numpy(0.5 * (f1[1:] + f1[:-1])[2:-2])[:, None]
    ph = torch.from_numpy(0.5 * (f2[1:] + f2[:-1])[2:-2])[None, :]
    r = torch.full((1, 1), R_IN, dtype=torch.float64)
    return torch.stack([w.expand(case["n1"], case["n2"]) for w in _wind(r, th, ph, phase)]).numpy()


def _front_flags(case, tree):
    """+1 on the finest leaves near the fronts that _cmes draws: a CME towards
    Earth, so that a case's tree does not depend on the seed"""
    flags = np.zeros(len(tree), dtype=np.int8)
    top = tree[:, 0].max()
    for i, (lev, a, b, c) in enumerate(tree):
        if lev != top:
            continue
        lo, hi = [], []
        for d, (ix, nb) in enumerate(((a, case["b0"]), (b, case["b1"]), (c, case["b2"]))):
            f = _faces((case["n0"], case["n1"], case["n2"])[d], d, case["stretch"], int(lev))
            lo.append(f[2 + ix * nb])
            hi.append(f[2 + (ix + 1) * nb])
        cosang = -math.sin(0.5 * (lo[1] + hi[1])) * math.cos(0.5 * (lo[2] + hi[2]))
        if math.acos(max(-1.0, min(1.0, cosang))) < math.radians(35.0) and lo[0] < 0.56 and hi[0] > 0.45:
            flags[i] = 1
    return flags


def _mlp_inputs(seed, n):
    """features of leaves and whether the next regrid refines them"""
    rng = np.random.default_rng(int(seed))
    X = np.abs(rng.normal(0.02, 0.03, (n, 64)) * rng.uniform(0.2, 4.0, (n, 1))).astype(np.float32)
    return X, (X.mean(axis=1) + rng.normal(0, 0.01, n) > 0.06).astype(np.float32)


# ---------------------------------------------------------------- one pass
def prepare(case, seed):
    st = dict(case)
    if case["kind"] == "train":
        st["g"] = Icarus(n_cells=(8, 8, 8), block=(8, 8, 8), x_min=X_MIN, x_max=X_MAX, precision=FP32_MIXED)
        st["theta"], st["seed"] = I.mlp_init(int(seed)).astype(np.float32), int(seed)
        st["g"].mlp_set_params(st["theta"])
        st["g"].mlp_dataset_add(*_mlp_inputs(seed, case["samples"]))
        return st
    n, b = (case["n0"], case["n1"], case["n2"]), (case["b0"], case["b1"], case["b2"])
    g = Icarus(n_cells=n, block=b, max_level=case["levels"], stretch=bool(case["stretch"]), x_min=X_MIN, x_max=X_MAX,
               gamma=GAMMA, omega=I.OMEGA, cfl=CFL, divb_cd=CD, p_floor=FLOOR, rho_floor=FLOOR,
               precision=FP32_MIXED if case["prec"] == "fp32" else FP64, n_members=case["members"],
               max_blocks=case["pool"], tracer=bool(case["tracer"]))
    # the floors behind the CME are counted, not budgeted, as in the resolution ladder
    g.set_floor_budget(0.0)
    for m, (cme, phase, front) in enumerate(_cmes(case, seed)):
        g.set_inner_boundary(m, _map(case, phase))
        # the background of the refinement criterion is the wind without the CME
        quiet = dict(cme, v=0.0, half_width=-10.0)
        g.set_state(m, _leaf_prims(case, g.tree(m), quiet, phase, front).cpu().numpy(), prim=True)
        g.inject_cone_cme(m, **cme)
    for _ in range(case["levels"] - 1):
        g.set_flags(np.concatenate([_front_flags(case, g.tree(m)) for m in range(case["members"])]))
        g.regrid()
    for m, (cme, phase, front) in enumerate(_cmes(case, seed)):
        W = _leaf_prims(case, g.tree(m), cme, phase, front)
        g.set_state(m, W.cpu().numpy(), prim=True)
        if case["tracer"]:
            X = 0.5 * (1 + torch.tanh((W[:, 1] - 7.6) * 4.0))
            g.set_tracer(m, (X * W[:, 0]).cpu().numpy())
    if case["levels"] > 1:
        g.set_earth(0, 0.5 * math.pi, math.pi, 0.0, I.OMEGA_SYN)
    if case["kind"] == "leaves":
        g.mlp_set_params(I.mlp_init(int(seed)).astype(np.float32))
    st["g"] = g
    # host buffers of a snapshot writer: room for a tree that a regrid has grown
    if case["kind"] != "leaves":
        leaves = g.n_leaves(0) * (4 if case["kind"] in ("cycle", "regrid") else 1)
        shape = (leaves, 8) + b
        st["f64"] = [torch.zeros(shape, dtype=torch.float64).pin_memory() for _ in range(case["members"])]
        if case["prec"] == "fp32":
            st["f32"] = [torch.zeros(shape, dtype=torch.float32) for _ in range(case["members"])]
        st["flags"], st["tree"] = np.zeros(leaves, dtype=np.int8), np.zeros((leaves, 4), dtype=np.int32)
    st["points"] = np.stack([I.earth_position(I.hours(float(k)), 0.0) for k in range(max(1, case["probe"]))])
    return st


def _snapshot(st, m=0):
    """the member's state in the writer's buffer; the buffer as it stands"""
    g = st["g"]
    n = g.n_leaves(m)
    if len(st["f64"][m]) < n:   # a tree that has outgrown the buffers
        for k in ("f64", "f32"):
            if k in st:
                st[k][m] = torch.zeros((2 * n,) + st[k][m].shape[1:], dtype=st[k][m].dtype)
    f64 = st["f64"][m]
    g.get_state(m, out=f64[:n].numpy())
    if "f32" not in st:
        return f64
    st["f32"][m][:n].copy_(f64[:n])
    return st["f32"][m]


def run(st):
    g, kind = st["g"], st["kind"]
    if kind == "train":
        g.mlp_set_params(st["theta"])
        loss = g.mlp_train(st["samples"], st["epochs"], batch=st["batch"], lr=1e-3, seed=st["seed"])
        return {"theta": g.mlp_get_params(), "loss": loss}
    if kind == "leaves":
        return {"features": g.mlp_features(), "probability": g.mlp_predict_leaves()}
    if kind == "regrid":
        return _flag_regrid(st)
    g.step(st["steps"], want_time=False)
    if kind == "cycle":
        return _flag_regrid(st)
    out = {"state": [_snapshot(st, m) for m in range(st["members"])]}
    real = np.float32 if st["prec"] == "fp32" else np.float64
    if st["tracer"]:
        out["tracer"] = [g.get_tracer(m).astype(real) for m in range(st["members"])]
    if st["probe"]:
        out["probe"] = [g.probe(m, st["points"]).astype(real) for m in range(st["members"])]
    return out


def _flag_regrid(st):
    """a regrid as the run driver makes it: a full block pool leaves the tree"""
    g = st["g"]
    flags = g.flag_refine(**CRIT)
    try:
        g.regrid()
    except IcarusError as e:
        if e.code != CAPACITY:
            raise
    tree = g.tree(0)
    if len(st["tree"]) < max(len(tree), len(flags)):
        n = 2 * max(len(tree), len(flags))
        st["flags"], st["tree"] = np.zeros(n, dtype=np.int8), np.zeros((n, 4), dtype=np.int32)
    st["flags"][:len(flags)], st["tree"][:len(tree)] = flags, tree
    return {"flags": st["flags"], "tree": st["tree"], "state": _snapshot(st)}


# ---------------------------------------------------------------- what a pass cannot do without
def _leaves_of(case):
    """leaves of a member: the base blocks, and on refined trees about a
    twelfth of the base and half of each finer level refined around the front"""
    n = (case["n0"] // case["b0"]) * (case["n1"] // case["b1"]) * (case["n2"] // case["b2"])
    new = n / 12.0
    for _ in range(case["levels"] - 1):
        n += 7 * new
        new *= 4
    return n


def work(case):
    if case["kind"] == "train":
        p, rows = MLP_PARAMS, case["samples"] * case["epochs"]
        batches = -(-case["samples"] // case["batch"]) * case["epochs"]
        # features once; parameters, moments and gradients once a batch; forward, and twice that backward
        return {"bytes": 4.0 * (65 * rows + 8 * p * batches), "flops": 6.0 * p * rows}
    real = 4 if case["prec"] == "fp32" else 8
    cells = _leaves_of(case) * case["b0"] * case["b1"] * case["b2"] * case["members"]
    state = (8 + case["tracer"]) * real
    if case["kind"] == "leaves":
        return {"bytes": cells * 7.0 * real, "flops": cells * 60.0}
    # per step: the state read once and written once, and the arithmetic of two stages (per stage three faces of 130
    # operations, 24 limited slopes, conversion, sources and balance); then the snapshot: the state read, FP64 written
    flops = case["steps"] * cells * 2 * (3 * 130 + 24 * 8 + 150)
    bytes_ = case["steps"] * cells * 2 * state + cells * (state + 64 + 8 * case["tracer"])
    if case["kind"] in ("cycle", "regrid"):
        flops += cells * 100
        bytes_ += cells * 3.0 * state   # read by the estimator, moved once
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---------------------------------------------------------------- 64-bit results
def exact(case, seed):
    """The pass in 64 bits.  Refined trees (prolongation, restriction and
    reflux over thousands of leaves) would take minutes in plain tensor
    operations and are left out."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["levels"] > 1 or case["kind"] != "step":
        return None
    cells = case["n0"] * case["n1"] * case["n2"] * case["members"]
    if cells * case["steps"] > (3e8 if torch.cuda.is_available() else 2e6):
        return None
    out = {"state": [], "tracer": [], "probe": []}
    for cme, phase, front in _cmes(case, seed):
        w = _Wedge(case, _map(case, phase), cme, _state_at(case, cme, phase, front))
        for _ in range(case["steps"]):
            w.step()
        out["state"].append(w.blocks(w.U[:8]))
        if case["tracer"]:
            out["tracer"].append(w.blocks(w.U[8:])[:, 0])
        if case["probe"]:
            out["probe"].append(None)   # a sample of the state above
    return {k: v for k, v in out.items() if v}


def _state_at(case, cme, phase, front):
    dev = _device()
    c = [torch.from_numpy(0.5 * (f[1:] + f[:-1])[2:-2]).to(dev)
         for f in (_faces(case["n0"], 0, case["stretch"]), _faces(case["n1"], 1, 0), _faces(case["n2"], 2, 0))]
    return torch.stack(_state(c[0][:, None, None], c[1][None, :, None], c[2][None, None, :], cme, phase, front))


class _Wedge:
    """The single-level wedge as dense arrays [variable][r][theta][phi] with
    two ghost layers, in 64 bits: midpoint predictor-corrector with TVDLF
    fluxes of MC-limited primitives, spherical and rotation sources, parabolic
    cleaning, and the CME tracer's upwind transport."""

    def __init__(self, case, bmap, cme, W):
        self.case, self.cme, self.t = case, cme, 0.0
        dev = W.device
        f = [torch.from_numpy(_faces(case[k], d, case["stretch"])).to(dev) for d, k in enumerate(("n0", "n1", "n2"))]
        shape = [(-1, 1, 1), (1, -1, 1), (1, 1, -1)]
        self.c = [(0.5 * (x[1:] + x[:-1])).view(s) for x, s in zip(f, shape)]
        self.dx = [(x[1:] - x[:-1]).view(s) for x, s in zip(f, shape)]
        r, th = f[0].view(shape[0]), f[1].view(shape[1])
        self.r2f, self.sinf = r ** 2, torch.sin(th)
        self.dr3, self.dr2 = (r[1:] ** 3 - r[:-1] ** 3) / 3, (r[1:] ** 2 - r[:-1] ** 2) / 2
        self.dcos = torch.cos(th)[:, :-1] - torch.cos(th)[:, 1:]
        self.dphi = (X_MAX[2] - X_MIN[2]) / case["n2"]
        self.st, self.ct = torch.sin(self.c[1]), torch.cos(self.c[1])
        self.bmap = torch.from_numpy(bmap).to(dev)
        self.nv = 9 if case["tracer"] else 8
        n = [case["n0"], case["n1"], case["n2"]]
        self.U = torch.zeros([self.nv] + [x + 4 for x in n], dtype=torch.float64, device=dev)
        self.U[:8, 2:-2, 2:-2, 2:-2] = self._cons(W)
        if case["tracer"]:
            self.U[8, 2:-2, 2:-2, 2:-2] = 0.5 * (1 + torch.tanh((W[1] - 7.6) * 4.0)) * W[0]
        self.dt = self._cfl()

    @staticmethod
    def _cons(W):
        ke = 0.5 * W[0] * (W[1] ** 2 + W[2] ** 2 + W[3] ** 2)
        e = W[4] / (GAMMA - 1) + ke + 0.5 * (W[5] ** 2 + W[6] ** 2 + W[7] ** 2)
        return torch.stack([W[0], W[0] * W[1], W[0] * W[2], W[0] * W[3], e, W[5], W[6], W[7]])

    @staticmethod
    def _prim(U):
        v = U[1:4] / U[0]
        p = (GAMMA - 1) * (U[4] - 0.5 * U[0] * (v ** 2).sum(0) - 0.5 * (U[5:8] ** 2).sum(0))
        return torch.cat([U[:1], v, p.clamp(min=FLOOR)[None], U[5:8]])

    def _fill(self, U, t):
        """two ghost layers: inner map with the cone, outflow, periodic"""
        c = self.cme
        W, X = self.bmap.clone(), torch.zeros_like(self.bmap[0])
        rh = R_IN * math.sin(c["half_width"])
        tau = t - c["t_start"]
        rc = tau * c["v"] + R_IN - rh
        arg = (rc * rc + R_IN * R_IN - rh * rh) / (2 * rc * R_IN)
        if 0.0 <= tau <= c["t_max"] and not arg > 1.0:
            th, ph = self.c[1][0, 2:-2], self.c[2][0, :, 2:-2]
            a = torch.sin(th) * math.sin(c["colat"]) * torch.cos(ph - c["lon"]) + torch.cos(th) * math.cos(c["colat"])
            on = torch.acos(a.clamp(-1, 1)) <= math.acos(arg)
            zero = torch.zeros_like(W[0])
            inside = [zero + c["rho"], zero + c["v"], zero, -I.OMEGA * R_IN * torch.sin(th) + zero, zero + c["p"],
                      zero, zero, zero]
            W = torch.where(on, torch.stack(inside), W)
            X = on.to(torch.float64)
        ring = self._cons(W)
        if self.nv > 8:
            ring = torch.cat([ring, (W[0] * X)[None]])
        U[:, :2, 2:-2, 2:-2] = ring[:, None]
        U[:, -2:] = U[:, -3:-2]
        U[:, :, :2] = U[:, :, 2:3]
        U[:, :, -2:] = U[:, :, -3:-2]
        U[..., :2] = U[..., -4:-2]
        U[..., -2:] = U[..., 2:4]

    @staticmethod
    def _fast(W, d):
        a2, b2, bn2 = GAMMA * W[4] / W[0], (W[5:8] ** 2).sum(0) / W[0], W[5 + d] ** 2 / W[0]
        return torch.sqrt(0.5 * (a2 + b2 + torch.sqrt(((a2 + b2) ** 2 - 4 * a2 * bn2).clamp(min=0.0))))

    def _face_flux(self, W, d):
        """fluxes of the faces normal to d of the interior cells"""
        sel = [slice(None)] + [slice(2, -2)] * 3
        sel[1 + d] = slice(None)
        w = W[tuple(sel)].movedim(1 + d, 1)
        dm = w[:, 1:-1] - w[:, :-2]
        dp = w[:, 2:] - w[:, 1:-1]
        lim = torch.minimum(torch.minimum(2 * dm.abs(), 2 * dp.abs()), 0.5 * (dm + dp).abs())
        h = 0.5 * torch.where(dm * dp > 0, torch.sign(dm) * lim, torch.zeros_like(lim))
        b, c = w[:, 1:-2], w[:, 2:-1]
        L, R = b + h[:, :-1], c - h[:, 1:]
        ok = (L[0] > 0) & (L[4] > 0) & (R[0] > 0) & (R[4] > 0)
        L, R = torch.where(ok, L, b), torch.where(ok, R, c)
        cm = torch.maximum(L[1 + d].abs() + self._fast(L, d), R[1 + d].abs() + self._fast(R, d))
        F = 0.5 * (self._flux(L, d) + self._flux(R, d)) - 0.5 * cm * (self._cons(R) - self._cons(L))
        F[5 + d] = 0.0
        return F.movedim(1, 1 + d)

    def _flux(self, W, d):
        vn, bn, e = W[1 + d], W[5 + d], self._cons(W)[4]
        pt = W[4] + 0.5 * (W[5:8] ** 2).sum(0)
        F = torch.empty_like(W)
        F[0] = W[0] * vn
        F[1:4] = W[0] * vn * W[1:4] - bn * W[5:8]
        F[1 + d] += pt
        F[4] = (e + pt) * vn - bn * (W[1:4] * W[5:8]).sum(0)
        F[5:8] = vn * W[5:8] - bn * W[1:4]
        return F

    def _rate(self, U):
        """L(U) of the interior cells, and its primitives"""
        W = self._prim(U[:8])
        i = slice(2, -2)
        dcos, dr2, dth = self.dcos[:, i], self.dr2[i], self.dx[1][:, i]
        area = [self.r2f[2:-2] * dcos * self.dphi, self.sinf[:, 2:-2] * dr2 * self.dphi, dr2 * dth]
        V = self.dr3[i] * dcos * self.dphi
        out = torch.zeros_like(U[:, i, i, i])
        X = U[8] / U[0] if self.nv > 8 else None
        for d in range(3):
            F = self._face_flux(W, d)
            n = F.shape[1 + d] - 1
            lo, hi = F.narrow(1 + d, 0, n), F.narrow(1 + d, 1, n)
            A = area[d]
            al = A.narrow(d, 0, n) if d < 2 else A
            ah = A.narrow(d, 1, n) if d < 2 else A
            out[:8] -= (ah * hi - al * lo) / V
            if X is not None:
                sel = [i, i, i]
                sel[d] = slice(1, -1)
                x = X[tuple(sel)]
                xf = torch.where(F[0] > 0, x.narrow(d, 0, n + 1), x.narrow(d, 1, n + 1))
                out[8] -= (ah * hi[0] * xf.narrow(d, 1, n) - al * lo[0] * xf.narrow(d, 0, n)) / V
        gr, gt = (area[0][1:] - area[0][:-1]) / V, (area[1][:, 1:] - area[1][:, :-1]) / V
        ir = 0.5 * gr
        w = W[:, i, i, i]
        rho, vr, vt, vp, p, br, bt, bp = w
        pt = p + 0.5 * (br ** 2 + bt ** 2 + bp ** 2)
        out[1] += (rho * (vt ** 2 + vp ** 2) - bt ** 2 - bp ** 2) * ir + pt * gr
        out[2] += (br * bt - rho * vr * vt) * ir + (rho * vp ** 2 - bp ** 2 + pt) * gt
        out[3] += (br * bp - rho * vr * vp) * ir - (rho * vt * vp - bt * bp) * gt
        out[6] += (vr * bt - vt * br) * ir
        out[7] += (vr * bp - vp * br) * ir + (vt * bp - vp * bt) * gt
        rc, st, ct, om = self.c[0][i], self.st[:, i], self.ct[:, i], I.OMEGA
        vs = vr * st + vt * ct
        out[1] += rho * (2 * om * vp * st + om ** 2 * rc * st ** 2)
        out[2] += rho * (2 * om * vp * ct + om ** 2 * rc * st * ct)
        out[3] -= 2 * om * rho * vs
        out[4] += rho * om ** 2 * rc * st * vs
        return out, w

    def _clean(self, U):
        """C_d h^2 grad(div B) of the interior cells"""
        rc, th, ph, st = self.c[0], self.c[1], self.c[2], self.st
        i = slice(1, -1)
        br, bt, bp = U[5], U[6], U[7]
        a = rc ** 2 * br
        div = (a[2:, i, i] - a[:-2, i, i]) / (rc[i] ** 2 * (rc[2:] - rc[:-2]))
        a = st * bt
        div = div + (a[i, 2:, i] - a[i, :-2, i]) / (rc[i] * st[:, i] * (th[:, 2:] - th[:, :-2]))
        div = div + (bp[i, i, 2:] - bp[i, i, :-2]) / (rc[i] * st[:, i] * (ph[..., 2:] - ph[..., :-2]))
        rc, th, ph, st = rc[i], th[:, i], ph[..., i], st[:, i]
        g = torch.stack([(div[2:, i, i] - div[:-2, i, i]) / (rc[2:] - rc[:-2]),
                         (div[i, 2:, i] - div[i, :-2, i]) / (rc[i] * (th[:, 2:] - th[:, :-2])),
                         (div[i, i, 2:] - div[i, i, :-2]) / (rc[i] * st[:, i] * (ph[..., 2:] - ph[..., :-2]))])
        return CD / sum(x ** -2 for x in self._widths()) * g

    def _widths(self):
        rc, st = self.c[0][2:-2], self.st[:, 2:-2]
        return self.dx[0][2:-2], rc * self.dx[1][:, 2:-2], rc * st * self.dphi

    @staticmethod
    def _floors(u):
        u[0].clamp_(min=FLOOR)
        rest = 0.5 * (u[1:4] ** 2).sum(0) / u[0] + 0.5 * (u[5:8] ** 2).sum(0)
        u[4] = torch.where((GAMMA - 1) * (u[4] - rest) < FLOOR, FLOOR / (GAMMA - 1) + rest, u[4])

    def _cfl(self):
        w = self._prim(self.U[:8, 2:-2, 2:-2, 2:-2])
        return CFL / float(sum((w[1 + d].abs() + self._fast(w, d)) / x for d, x in enumerate(self._widths())).max())

    def step(self):
        i = slice(2, -2)
        self._fill(self.U, self.t)
        rate, _ = self._rate(self.U)
        half = self.U.clone()
        half[:, i, i, i] += 0.5 * self.dt * rate
        self._floors(half[:, i, i, i])
        self._fill(half, self.t + 0.5 * self.dt)
        rate, w = self._rate(half)
        u = self.U[:, i, i, i]
        u += self.dt * rate
        dB = self._clean(half)
        u[5:8] += dB
        u[4] += (w[5:8] * dB).sum(0)
        self._floors(u)
        self.t += self.dt
        self.dt = self._cfl()

    def blocks(self, U):
        """[leaf][variable][i][j][k] of the interior, leaves in Morton order"""
        c = self.case
        n, b = (c["n0"], c["n1"], c["n2"]), (c["b0"], c["b1"], c["b2"])
        U = U[:, 2:-2, 2:-2, 2:-2]

        def key(x):
            return [(v >> bit) & 1 for bit in range(20, -1, -1) for v in x]

        order = sorted(np.ndindex(*(n[d] // b[d] for d in range(3))), key=key)
        return torch.stack([U[:, x[0] * b[0]:(x[0] + 1) * b[0], x[1] * b[1]:(x[1] + 1) * b[1],
                            x[2] * b[2]:(x[2] + 1) * b[2]] for x in order]).cpu()


def _exact_train(case, seed):
    """Adam on the 64-128-128-1 network in 64 bits, the library's documented
    seeded shuffle (splitmix64, Fisher-Yates)"""
    dev = _device()
    th = torch.from_numpy(I.mlp_init(int(seed)).astype(np.float32)).double().to(dev)
    X, T = (torch.from_numpy(x).double().to(dev) for x in _mlp_inputs(seed, case["samples"]))
    sizes = [128 * 64, 128, 128 * 128, 128, 128, 1]
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    lr, step, losses = float(np.float32(1e-3)), 0, []
    state, mask = int(seed) & (2 ** 64 - 1), 2 ** 64 - 1
    for _ in range(case["epochs"]):
        perm = list(range(case["samples"]))
        for i in range(case["samples"] - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        perm = torch.tensor(perm, device=dev)
        total = 0.0
        for at in range(0, case["samples"], case["batch"]):
            x, t = X[perm[at:at + case["batch"]]], T[perm[at:at + case["batch"]]]
            q = th.clone().requires_grad_(True)
            w1, b1, w2, b2, w3, b3 = torch.split(q, sizes)
            h = torch.relu(x @ w1.view(128, 64).T + b1)
            h = torch.relu(h @ w2.view(128, 128).T + b2)
            y = torch.sigmoid(h @ w3 + b3)
            loss = torch.nn.functional.binary_cross_entropy(y, t, reduction="sum")
            (loss / len(x)).backward()
            total += float(loss.detach())
            step += 1
            m = 0.9 * m + 0.1 * q.grad
            v = 0.999 * v + 0.001 * q.grad ** 2
            th = th - lr * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
        losses.append(total / case["samples"])
    return {"theta": th.cpu(), "loss": torch.tensor(losses, dtype=torch.float64)}
