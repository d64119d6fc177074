"""The work this library is used for, as cases that can be timed and compared.

A case is one whole call sequence of a user's program on a context that the program keeps:
build (or load) a filtration, reduce it, read the results. Sizes are those of the repository's
benchmark workloads (40 points on a circle, 120 Gaussian points in R^8, 400 points on a torus,
512 ragged clouds, 256 fp32 clouds with a diagram loss, the paper's 15-point ensembles) and the
sizes between them. Points are drawn here from the seed alone, so that inputs of another seed
are other points of the same kind.

The kinds:
  vr      one point cloud: build_filtration, reduce, pairs, essential
  scales  one cloud on the paper's grid of scales, up to dimension 5: the same four calls
  batch   many clouds of different sizes in one context: the same four calls, all clouds' results
  diff    fp32 clouds: diagram_loss and its gradient (one training step's topological term)
  early   a reduction stopped after a few passes: counters, the essential estimate, the lows
  grid    a cubical complex of an image, loaded as a boundary matrix from host arrays: reduce and
          read the reduced matrix (representative cycles)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1708_04710_gb300 import Context
from paper_1708_04710_gb300.diff import diagram_loss

GRID = 65536  # grid units per unit length
CUT16 = 16 * GRID * GRID  # squared diameter 16


def listed():
    return [
        # the smallest complex: a sensor's 40 readings on a noisy circle, called again and again;
        # results go to host code
        {"name": "circle40", "kind": "vr", "shape": "circle", "n": 40, "D": 2, "max_dim": 2,
         "max_diam2": -1, "host": True},
        # the paper's own experiments: 15 points, complete up to dimension 5, on 10 scales
        {"name": "ensemble15", "kind": "scales", "shape": "gauss", "n": 15, "D": 3, "max_dim": 5,
         "step": GRID // 2, "n_scales": 10},
        # higher-dimensional data with a cut: tetrahedra of 120 points in R^8
        {"name": "gauss8_120", "kind": "vr", "shape": "gauss", "n": 120, "D": 8, "max_dim": 3,
         "max_diam2": CUT16, "host": False},
        # an ordinary cloud, an odd size
        {"name": "torus151", "kind": "vr", "shape": "torus", "n": 151, "D": 3, "max_dim": 2,
         "max_diam2": -1, "host": False},
        # the benchmark's workload, results kept on the device
        {"name": "torus400", "kind": "vr", "shape": "torus", "n": 400, "D": 3, "max_dim": 2,
         "max_diam2": -1, "host": False},
        # a mini-batch of ragged clouds
        {"name": "batch24", "kind": "batch", "clouds": 24, "n_lo": 20, "n_hi": 120,
         "max_dim": 2},
        # a data set in one filtration: 47 million simplices
        {"name": "batch512", "kind": "batch", "clouds": 512, "n_lo": 20, "n_hi": 120,
         "max_dim": 2},
        # a topological loss on a small training batch, loops
        {"name": "diff8x32", "kind": "diff", "clouds": 8, "n": 32, "D": 3, "dim": 1},
        # ... connected components of larger clouds in the plane
        {"name": "diff16x100_h0", "kind": "diff", "clouds": 16, "n": 100, "D": 2, "dim": 0},
        # ... and on a large one: the benchmark's differentiable workload
        {"name": "diff256x64", "kind": "diff", "clouds": 256, "n": 64, "D": 3, "dim": 1},
        # early stopping after 8 passes, with the per-pass counters
        {"name": "early100", "kind": "early", "shape": "torus", "n": 100, "D": 3, "max_dim": 2,
         "passes": 8},
        # representative cycles of an image's sublevel sets
        {"name": "grid96x80", "kind": "grid", "w": 96, "h": 80},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vr", "vr", "vr", "cut", "scales", "batch", "batch", "diff", "diff",
                       "early", "grid"])
    if kind == "vr":
        shape = rng.choice(["circle", "torus", "sphere", "gauss"])
        return {"kind": "vr", "shape": shape, "n": _log_int(rng, 30, 400),
                "D": {"circle": 2, "torus": 3, "sphere": 3}.get(shape) or rng.randint(2, 8),
                "max_dim": 2, "max_diam2": -1, "host": rng.random() < 0.5}
    if kind == "cut":
        return {"kind": "vr", "shape": "gauss", "n": _log_int(rng, 30, 120),
                "D": rng.randint(6, 10), "max_dim": 3, "max_diam2": CUT16,
                "host": rng.random() < 0.5}
    if kind == "scales":
        return {"kind": "scales", "shape": rng.choice(["gauss", "torus", "sphere"]),
                "n": rng.randint(10, 17), "D": 3, "max_dim": rng.randint(3, 5),
                "step": GRID // 2, "n_scales": 10}
    if kind == "batch":
        lo = rng.randint(8, 40)
        return {"kind": "batch", "clouds": _log_int(rng, 4, 512), "n_lo": lo,
                "n_hi": rng.randint(lo + 20, 120), "max_dim": 2}
    if kind == "diff":
        dim = rng.choice([0, 1, 1])
        return {"kind": "diff", "clouds": _log_int(rng, 2, 256),
                "n": rng.randint(16, 64) if dim else _log_int(rng, 16, 128),
                "D": rng.randint(2, 4), "dim": dim}
    if kind == "early":
        return {"kind": "early", "shape": rng.choice(["torus", "sphere"]),
                "n": _log_int(rng, 60, 180), "D": 3, "max_dim": 2, "passes": rng.randint(2, 8)}
    return {"kind": "grid", "w": _log_int(rng, 24, 160), "h": _log_int(rng, 24, 120)}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _unit(x):
    return x / np.linalg.norm(x, axis=1, keepdims=True)


def _points(shape, n, D, rng):
    if shape == "circle":
        t = rng.uniform(0.0, 2.0 * np.pi, n)
        return np.stack([np.cos(t), np.sin(t)], axis=1) + rng.normal(0.0, 0.05, (n, 2))
    if shape == "torus":
        t, p = rng.uniform(0.0, 2.0 * np.pi, (2, n))
        return np.stack([(2 + np.cos(p)) * np.cos(t), (2 + np.cos(p)) * np.sin(t), np.sin(p)],
                        axis=1)
    if shape == "sphere":
        return _unit(rng.standard_normal((n, D)))
    return rng.standard_normal((n, D))


def _to_grid(x):
    return np.rint(x * GRID).astype(np.int32)


def _batch_points(case, rng):
    # the sizes belong to the case: a program's data set keeps them from call to call
    sizes = np.random.default_rng([case["clouds"], case["n_lo"], case["n_hi"]]).integers(
        case["n_lo"], case["n_hi"] + 1, case["clouds"])
    shapes = ("sphere", "torus", "gauss")
    pts = [_to_grid(_points(shapes[i % 3], int(n), 3, rng)) for i, n in enumerate(sizes)]
    return np.concatenate(pts), np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _diff_points(case, seed):
    rng = np.random.default_rng(seed)
    n = case["clouds"] * case["n"]
    x = _unit(rng.standard_normal((n, case["D"]))) + rng.normal(0.0, 0.02, (n, case["D"]))
    return x.astype(np.float32), np.arange(case["clouds"] + 1, dtype=np.int64) * case["n"]


def _image_complex(w, h, rng):
    """Sublevel filtration of a smooth random w x h image: pixels are vertices, a cell enters
    with its largest pixel. Returns (dims, colptr, rows), cells in filtration order."""
    f = rng.standard_normal((h, w))
    for _ in range(4):  # a few smoothing steps: features some pixels wide
        f = (f + np.roll(f, 1, 0) + np.roll(f, -1, 0) + np.roll(f, 1, 1) + np.roll(f, -1, 1)) / 5
    v = np.arange(w * h).reshape(h, w)
    e = np.concatenate([np.stack([v[:, :-1], v[:, 1:]], -1).reshape(-1, 2),
                        np.stack([v[:-1], v[1:]], -1).reshape(-1, 2)])
    nv, ne, nhor = w * h, len(e), h * (w - 1)
    hor = np.arange(nhor).reshape(h, w - 1)
    ver = nhor + np.arange(ne - nhor).reshape(h - 1, w)
    sq = np.stack([hor[:-1], hor[1:], ver[:, :-1], ver[:, 1:]], -1).reshape(-1, 4)
    fv = f.reshape(-1)
    fe = fv[e].max(1)
    fs = fe[sq].max(1)
    dims = np.repeat(np.arange(3, dtype=np.int32), [nv, ne, len(sq)])
    order = np.lexsort((dims, np.concatenate([fv, fe, fs])))
    pos = np.empty(len(order), np.int64)
    pos[order] = np.arange(len(order))
    cells = np.full((len(order), 4), np.iinfo(np.int64).max)
    cells[nv:nv + ne, :2] = pos[e]
    cells[nv + ne:] = pos[nv + sq]
    cells = np.sort(cells[order], axis=1)
    dims = dims[order]
    length = np.array([0, 2, 4])[dims]
    colptr = np.concatenate([[0], np.cumsum(length)]).astype(np.int64)
    rows = cells[np.arange(4)[None, :] < length[:, None]].astype(np.int32)
    return dims, colptr, rows


class State:
    def __init__(self, case):
        self.case = case
        self.context = Context(collect_stats=case["kind"] == "early")
        self.buffers = {}  # results whose number depends on the points: name -> (array, used)

    def keep(self, name, x, capacity):
        """x at the start of a buffer of fixed capacity that the program keeps, zeros after it."""
        buf, used = self.buffers.get(name, (None, 0))
        if buf is None:
            buf = (np.zeros(capacity, x.dtype) if isinstance(x, np.ndarray) else
                   torch.zeros(capacity, dtype=x.dtype, device=x.device))
        n = len(x)
        buf[:n] = x
        if n < used:
            buf[n:used] = 0
        self.buffers[name] = buf, n
        return buf


def prepare(case, seed):
    s = State(case)
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s.offsets = None
    if kind == "batch":
        x, s.offsets = _batch_points(case, rng)
        s.x = torch.from_numpy(x).cuda()
    elif kind == "diff":
        x, s.offsets = _diff_points(case, seed)
        s.x = torch.from_numpy(x).cuda().requires_grad_(True)
    elif kind == "grid":
        s.dims, s.colptr, s.rows = _image_complex(case["w"], case["h"], rng)
    else:
        s.x = torch.from_numpy(_to_grid(_points(case["shape"], case["n"], case["D"], rng))).cuda()
    return s


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def run(s):
    case, ctx = s.case, s.context
    kind = case["kind"]
    if kind == "diff":
        loss = diagram_loss(s.x, s.offsets, case["dim"], ctx)
        (grad,) = torch.autograd.grad(loss.sum(), s.x)
        return {"loss": loss.detach(), "grad": grad}
    if kind == "grid":
        ctx.load_boundary(s.dims, s.colptr, s.rows)
        st = ctx.reduce()
        colptr, rows = ctx.columns()
        return {"passes": st["passes"], "colptr": colptr,
                "rows": s.keep("rows", rows, 24 * len(s.dims))}
    if kind == "scales":
        ctx.build_filtration_scales(s.x, None, case["max_dim"], case["step"], case["n_scales"])
    else:
        ctx.build_filtration(s.x, s.offsets, case["max_dim"], case.get("max_diam2", -1))
    if kind == "early":
        st = ctx.reduce(max_passes=case["passes"])
        return {"passes": st["passes"], "counters": ctx.pass_stats(),
                "estimate": ctx.essential_estimate().astype(np.uint8),
                "low": ctx.filtration()["low"]}
    st = ctx.reduce()
    on_device = not case.get("host", False)
    cloud = -1 if kind == "batch" else 0
    pairs, ess = ctx.pairs(cloud, on_device), ctx.essential(cloud, on_device)
    if case.get("max_diam2", -1) >= 0:  # a cut complex: at most the complete one's counts
        cap = _complete_counts(case["n"], case["max_dim"])
        pairs = {k: s.keep(k, x, cap[0]) for k, x in pairs.items()}
        ess = {k: s.keep(k + "_ess", x, cap[1]) for k, x in ess.items()}
    return {"passes": st["passes"], "pairs": pairs, "essential": ess}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without: its inputs read once, its results written once
# ---------------------------------------------------------------------------------------------
def _complete_counts(n, max_dim):
    """Pairs and essential simplices of a complete complex on n points: C(n-1, d) pairs with
    deaths of dimension d, 1 + C(n-1, max_dim+1) essential simplices. A cut leaves some pairs'
    births essential instead, so its essentials are bounded by all simplices that give birth."""
    pairs = sum(math.comb(n - 1, d) for d in range(1, max_dim + 1))
    return pairs, pairs + 1 + math.comb(n - 1, max_dim + 1)


def _complete_bytes(n, max_dim):
    pairs, births = _complete_counts(n, max_dim)
    return 36 * pairs + 20 * (births - pairs)  # bytes per pair, per essential simplex


def work(case):
    kind = case["kind"]
    if kind == "grid":
        w, h = case["w"], case["h"]
        v, e, q = w * h, h * (w - 1) + w * (h - 1), (w - 1) * (h - 1)
        # dims, colptr and rows in; column pointers and about as many reduced rows out
        return {"bytes": 12 * (v + e + q) + 4 * (2 * e + 4 * q)
                + 8 * (v + e + q) + 4 * (2 * (v - 1) + 4 * q), "flops": 0}
    if kind == "batch":
        mid = range(case["n_lo"], case["n_hi"] + 1)
        per = sum(12 * n + _complete_bytes(n, case["max_dim"]) for n in mid) / len(mid)
        return {"bytes": int(case["clouds"] * per), "flops": 0}
    if kind == "diff":  # coordinates in, loss and gradient out; about 8 D flops per pair
        pairs = math.comb(case["n"] - 1, case["dim"] + 1)
        c = case["clouds"]
        return {"bytes": c * (8 * case["n"] * case["D"] + 4),
                "flops": 8 * case["D"] * pairs * c}
    n, D = case["n"], case["D"]
    if kind == "early":  # the estimate and the lows of every simplex, the counters
        m = sum(math.comb(n, k) for k in range(1, case["max_dim"] + 2))
        return {"bytes": 4 * n * D + 5 * m + 104 * (case["passes"] + 1), "flops": 0}
    out = _complete_bytes(n, case["max_dim"])
    if case.get("max_diam2", -1) >= 0:  # the cut keeps about an eighth of the complex
        out //= 8
    return {"bytes": 4 * n * D + out, "flops": 0}


# ---------------------------------------------------------------------------------------------
# losses and gradients in 64 bits (the other kinds' results are whole numbers)
# ---------------------------------------------------------------------------------------------
def _pairs_of_cloud(g, dim):
    """Pairs of one cloud (integer coordinates g) as realising edges: (birth edge or -1, death
    edge) indices into the edges sorted by (squared length, vertices)."""
    n = len(g)
    a, b = np.triu_indices(n, 1)
    d2 = ((g[a] - g[b]) ** 2).sum(1)
    order = np.lexsort((b, a, d2))
    a, b, d2 = a[order], b[order], d2[order]
    root = list(range(n))

    def find(x):
        while root[x] != x:
            root[x] = root[root[x]]
            x = root[x]
        return x

    tree = []
    for i in range(len(a)):
        x, y = find(a[i]), find(b[i])
        if x != y:
            root[x] = y
            tree.append(i)
    if dim == 0:
        return a, b, [(-1, i) for i in tree]
    idx = np.zeros((n, n), np.int64)
    idx[a, b] = idx[b, a] = np.arange(len(a))
    t = np.array([(i, j, k) for i in range(n) for j in range(i + 1, n)
                  for k in range(j + 1, n)]).reshape(-1, 3)
    e = np.sort(np.stack([idx[t[:, 0], t[:, 1]], idx[t[:, 0], t[:, 2]], idx[t[:, 1], t[:, 2]]],
                         axis=1), axis=1)
    rank = np.unique(d2, return_inverse=True)[1]  # equal lengths tie: then by vertices
    e = e[np.argsort(rank[e[:, 2]], kind="stable")]
    want = len(a) - len(tree)  # every cycle of a complete complex dies
    pivots, pairs = {}, []
    for x, y, z in e.tolist():
        col = (1 << x) | (1 << y) | (1 << z)
        while col:
            low = col.bit_length() - 1
            if low not in pivots:
                pivots[low] = col
                pairs.append((low, z))
                break
            col ^= pivots[low]
        if len(pairs) == want:
            break
    return a, b, pairs


def exact(case, seed):
    if case["kind"] != "diff":
        return None
    if case["clouds"] * math.comb(case["n"], case["dim"] + 2) > 600_000:
        return None  # minutes in plain Python
    x, off = _diff_points(case, seed)
    x = x.astype(np.float64)
    loss = np.zeros(case["clouds"])
    grad = np.zeros_like(x)
    for c in range(case["clouds"]):
        xs = x[off[c]:off[c + 1]]
        a, b, pairs = _pairs_of_cloud(np.rint(xs * GRID).astype(np.int64), case["dim"])
        for birth, death in pairs:
            r = xs[a[death]] - xs[b[death]]
            d = np.sqrt((r ** 2).sum())
            length = 0.0
            if birth >= 0:
                p = xs[a[birth]] - xs[b[birth]]
                length = np.sqrt((p ** 2).sum())
            loss[c] += (d - length) ** 2
            if d > 0:
                t = 2 * (d - length) / d * r
                grad[off[c] + a[death]] += t
                grad[off[c] + b[death]] -= t
            if length > 0:
                t = 2 * (d - length) / length * p
                grad[off[c] + a[birth]] -= t
                grad[off[c] + b[birth]] += t
    return {"loss": loss, "grad": grad}
