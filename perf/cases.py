"""The calls that this library is used for, at the sizes that it is used at.

Every case is one pass through a public entry point, as a program that holds
its points, output buffers and workspace on the GPU makes it:

* ``hull``     ``ch_hull``: Algorithm 1 end to end on one set;
* ``filter``   ``ch_extremes`` and then ``ch_filter``: the paper's filter
               stage, its two steps called one after the other;
* ``sweep``    ``ch_extremes_filter``: the same results from one call;
* ``batched``  ``ch_hull_batched``: many sets of uneven sizes in one call;
* ``kgon``     ``ch_hull_octagon_kgon``: the octagon and a K-direction
               polygon, the call that the learned proposal's labels time;
* ``kfilter``  ``ch_filter_kgon``: the K-direction polygon as the filter;
* ``learned``  ``Proposal.hull_on_device`` with the committed weights;
* ``train``    ``Proposal.train_step``: one Adam step of the proposal.

Points come from the study's distributions (standard normal, unit circle,
displaced circle with radius 1 - |N(0, 0.01)|) and the learned proposal's
families (mixtures of Gaussians, ellipses), drawn in binary64 and rounded
once.  Output buffers are zeroed once, so the unspecified entries beyond a
count compare equal.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2303_10581_gb300 as ch
from paper_2303_10581_gb300 import learned

DISTS = ("normal", "circle", "displaced", "gaussians", "ellipse")
CHUNK = 1 << 24
DEV = "cuda"


def listed():
    return [
        # a handful of points (one object's outline, one cluster): launches and latency
        {"name": "hull_normal_1k", "kind": "hull", "dist": "normal", "n": 1000, "shift": 0},
        # the smallest benchmark configuration: one set of 2^20 normal points
        {"name": "hull_normal_2p20", "kind": "hull", "dist": "normal", "n": 1 << 20, "shift": 0},
        # a medium set that the filter cannot thin out, odd size, 8-byte aligned
        {"name": "hull_circle_1m", "kind": "hull", "dist": "circle", "n": 1_000_003, "shift": 1},
        # the headline benchmark's three sets: favourable, worst and intermediate
        {"name": "hull_normal_1e8", "kind": "hull", "dist": "normal", "n": 100_000_000, "shift": 0},
        {"name": "hull_circle_1e8", "kind": "hull", "dist": "circle", "n": 100_000_000, "shift": 0},
        {"name": "hull_displaced_1e8", "kind": "hull", "dist": "displaced", "n": 100_000_000, "shift": 0},
        # the filter stage by itself at its largest: the bandwidth study
        {"name": "filter_normal_1e9", "kind": "filter", "dist": "normal", "n": 1_000_000_000, "shift": 0},
        # the filter as a pre-pass for another hull code: most points survive and are written, odd size
        {"name": "sweep_displaced_1e7", "kind": "sweep", "dist": "displaced", "n": 10_000_019, "shift": 0},
        # the batched benchmark: 4096 sets of 10^2 to 10^6 points
        {"name": "batched_4096", "kind": "batched", "sets": 4096, "min_n": 100, "max_n": 1_000_000},
        # a batch of small sets (outlines, clusters)
        {"name": "batched_small", "kind": "batched", "sets": 1000, "min_n": 100, "max_n": 10_000},
        # the learned proposal's evaluation: one large set of a training family
        {"name": "learned_ellipse_1e8", "kind": "learned", "dist": "ellipse", "n": 100_000_000, "shift": 0},
        # the learned proposal's training step at its default batch
        {"name": "train_b64", "kind": "train", "batch": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("hull", "hull", "hull", "filter", "sweep", "batched", "batched", "kgon", "kfilter", "learned",
                       "train"))
    if kind == "batched":
        return {"kind": kind, "sets": _log_int(rng, 16, 4096), "min_n": 100, "max_n": _log_int(rng, 1000, 900_000)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 8, 256)}
    # a K-direction polygon as the only filter costs several sweeps' time
    n = _log_int(rng, 100, {"filter": 300_000_000, "kgon": 30_000_000, "kfilter": 30_000_000}.get(kind, 90_000_000))
    case = {"kind": kind, "dist": rng.choice(DISTS), "n": n, "shift": rng.choice((0, 0, 0, 1))}
    if kind in ("kgon", "kfilter"):
        case["K"] = rng.choice((16, 32, 64))
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, m, lo, hi):
    return torch.rand(m, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _normal(g, m):
    return torch.randn(m, generator=g, device=DEV, dtype=torch.float64)


def _family(dist, seed):
    """The parameters of one set of a training family."""
    r = np.random.Generator(np.random.PCG64(seed))
    f = {"scale": 1.0, "turn": 0.0, "ratio": 1.0}
    if dist in ("gaussians", "ellipse"):
        f = {"scale": r.uniform(0.1, 10.0), "turn": r.uniform(0.0, 2.0 * math.pi), "ratio": r.uniform(1.0, 20.0)}
    if dist == "gaussians":
        k = int(r.integers(1, 5))
        f |= {"mean": r.uniform(-3.0, 3.0, (k, 2)), "sig": r.uniform(0.1, 1.0, (k, 2)),
              "rot": r.uniform(0.0, 2.0 * math.pi, k)}
    return f


def _chunk(dist, f, g, m):
    """m points of one distribution in binary64."""
    if dist == "normal":
        return _normal(g, m), _normal(g, m)
    if dist == "gaussians":
        k = len(f["rot"])
        which = torch.randint(0, k, (m,), generator=g, device=DEV)
        t = [torch.as_tensor(a, device=DEV)[which] for a in
             (f["mean"][:, 0], f["mean"][:, 1], f["sig"][:, 0], f["sig"][:, 1], np.cos(f["rot"]), np.sin(f["rot"]))]
        a, b = _normal(g, m) * t[2], _normal(g, m) * t[3]
        x, y = t[0] + t[4] * a - t[5] * b, t[1] + t[5] * a + t[4] * b
    else:
        th = _uniform(g, m, 0.0, 2.0 * math.pi)
        x, y = torch.cos(th), torch.sin(th)
        if dist != "circle":
            r = 1.0 - 0.01 * _normal(g, m).abs()
            x, y = r * x, r * y
        if dist == "ellipse":
            c, s = math.cos(f["turn"]), math.sin(f["turn"])
            y = y / f["ratio"]
            x, y = c * x - s * y, s * x + c * y
    return f["scale"] * x, f["scale"] * y


def _points(dist, n, seed, shift=0):
    """(n, 2) float32 points; shift: 8 bytes past a 16-byte boundary."""
    g, f = _gen(seed), _family(dist, seed)
    buf = torch.zeros((n + shift, 2), dtype=torch.float32, device=DEV)
    pts = buf[shift:]
    for lo in range(0, n, CHUNK):
        m = min(CHUNK, n - lo)
        x, y = _chunk(dist, f, g, m)
        pts[lo:lo + m, 0] = x
        pts[lo:lo + m, 1] = y
    return pts


def _sizes(case, seed):
    """Sizes log-uniform in [min_n, max_n], the same ones for every seed in
    another order."""
    k = case["sets"]
    q = (np.arange(k) + 0.5) / k
    lo, hi = math.log(case["min_n"]), math.log(case["max_n"])
    sizes = np.rint(np.exp(lo + q * (hi - lo))).astype(np.int64)
    return sizes if seed is None else np.random.Generator(np.random.PCG64(seed)).permutation(sizes)


def _batch(case, seed):
    """(points, offsets): each set one of normal, circle and displaced circle,
    scaled by U[0.1, 10] and rotated by U[0, 2 pi)."""
    sizes = _sizes(case, seed)
    k = len(sizes)
    off = np.zeros(k + 1, np.int64)
    off[1:] = np.cumsum(sizes)
    n = int(off[-1])
    g = _gen(seed)
    offsets = torch.from_numpy(off).to(DEV)
    kind = torch.randint(0, 3, (k,), generator=g, device=DEV)
    scale, turn = _uniform(g, k, 0.1, 10.0), _uniform(g, k, 0.0, 2.0 * math.pi)
    pts = torch.empty((n, 2), dtype=torch.float32, device=DEV)
    for lo in range(0, n, CHUNK):
        m = min(CHUNK, n - lo)
        b = torch.searchsorted(offsets, torch.arange(lo, lo + m, device=DEV), right=True) - 1
        kb = kind[b]
        th = _uniform(g, m, 0.0, 2.0 * math.pi)
        r = torch.where(kb == 2, 1.0 - 0.01 * _normal(g, m).abs(), torch.ones((), dtype=torch.float64, device=DEV))
        x = torch.where(kb == 0, _normal(g, m), r * torch.cos(th))
        y = torch.where(kb == 0, _normal(g, m), r * torch.sin(th))
        c, s = (torch.cos(turn) * scale)[b], (torch.sin(turn) * scale)[b]
        pts[lo:lo + m, 0] = c * x - s * y
        pts[lo:lo + m, 1] = s * x + c * y
    return pts, offsets


GRID = 32


def _grid(x, y):
    """The 32 x 32 occupancy grids of samples (B, m) as fractions (B, 1024)."""
    x0, y0 = x.amin(1, keepdim=True), y.amin(1, keepdim=True)
    sx, sy = 32.0 / (x.amax(1, keepdim=True) - x0), 32.0 / (y.amax(1, keepdim=True) - y0)
    cell = ((y - y0) * sy).floor().clamp(max=31).long() * GRID + ((x - x0) * sx).floor().clamp(max=31).long()
    out = torch.zeros((x.shape[0], GRID * GRID), dtype=torch.float32, device=x.device)
    return out.scatter_add_(1, cell, torch.ones_like(x, dtype=torch.float32)) / x.shape[1]


SHAPES = ((64, 1024), (64,), (64, 64), (64,), (68, 64), (68,))


def _training(batch, seed):
    """A batch of the training families and the optimiser's state some way
    into the training."""
    g = _gen(seed)
    xs, ys = [], []
    for b in range(batch):
        dist = ("gaussians", "ellipse", "displaced")[b % 3]
        x, y = _chunk(dist, _family(dist, seed * 1000 + b), g, 4096)
        xs.append(x.float())
        ys.append(y.float())
    X = _grid(torch.stack(xs), torch.stack(ys)).contiguous()
    label = torch.randint(0, 4, (batch,), generator=g, device=DEV).int()
    off = _uniform(g, batch * 64, -0.45, 0.45).float().reshape(batch, 64)
    mask = torch.ones(batch, dtype=torch.float32, device=DEV)
    w = []
    for s in SHAPES:
        a = math.sqrt(6.0 / s[1]) if len(s) == 2 else 0.1
        w.append(_uniform(g, int(np.prod(s)), -a, a))
    w = torch.cat(w).float()
    m = (1e-3 * _normal(g, w.numel())).float()
    v = (1e-6 * (0.1 + _uniform(g, w.numel(), 0.0, 1.0))).float()
    return X, label, off, mask, w, m, v


TRAIN_STEP, LAM, LR = 100, 0.5, 3e-3


# ---------------------------------------------------------------- cases

def _ints(n):
    return torch.zeros(n, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "train":
        X, label, off, mask, w, m, v = _training(case["batch"], seed)
        p = learned.Proposal(DEV)
        p.master, p.params, p.m, p.v, p.step = w, w.to(torch.bfloat16), m, v, TRAIN_STEP - 1
        scratch = torch.empty(int(ch.load().ch_mlp_scratch_floats(case["batch"])), dtype=torch.float32, device=DEV)
        return s | {"prop": p, "batch": (X, label, off, mask), "scratch": scratch,
                    "loss": torch.zeros(case["batch"], dtype=torch.float32, device=DEV)}
    if kind == "batched":
        pts, offsets = _batch(case, seed)
        n, k = pts.shape[0], case["sets"]
        return s | {"pts": pts, "offsets": offsets, "idx": _ints(n), "ws": ch.Workspace(n, k),
                    "hoff": torch.zeros(k + 1, dtype=torch.int64, device=DEV)}
    n = case["n"]
    s |= {"pts": _points(case["dist"], n, seed, case["shift"]), "ws": ch.Workspace(n), "idx": _ints(n),
          "cnt": _ints(1)}
    if kind in ("filter", "sweep", "kfilter"):
        s["sp"] = torch.zeros((n, 2), dtype=torch.float32, device=DEV)
    if kind in ("filter", "sweep"):
        s["ext"] = _ints(8)
    if kind in ("kgon", "kfilter"):
        s["ext"] = _ints(case["K"])
        s["dirs"] = torch.from_numpy(learned.directions(case["K"])).to(DEV)
    if kind == "learned":
        s["prop"] = learned.load_params(learned.DEFAULT_WEIGHTS, DEV)[0]
        s["out"] = (s["idx"], s["cnt"], _ints(1), torch.zeros(128, dtype=torch.float32, device=DEV))
    return s


def run(s):
    kind = s["kind"]
    if kind == "hull":
        ch.ch_hull(s["pts"], s["idx"], s["cnt"], s["ws"].buf)
        return s["idx"], s["cnt"]
    if kind == "filter":
        ch.ch_extremes(s["pts"], s["ext"], s["ws"].buf)
        ch.ch_filter(s["pts"], s["ext"], s["idx"], s["sp"], s["cnt"], s["ws"].buf)
        return s["ext"], s["idx"], s["sp"], s["cnt"]
    if kind == "sweep":
        ch.ch_extremes_filter(s["pts"], s["ext"], s["idx"], s["sp"], s["cnt"], s["ws"].buf)
        return s["ext"], s["idx"], s["sp"], s["cnt"]
    if kind == "batched":
        ch.ch_hull_batched(s["pts"], s["offsets"], s["idx"], s["hoff"], s["ws"].buf)
        return s["idx"], s["hoff"]
    if kind == "kgon":
        ch.ch_hull_octagon_kgon(s["pts"], s["dirs"], s["dirs"].shape[0], None, s["idx"], s["cnt"], s["ws"].buf)
        return s["idx"], s["cnt"]
    if kind == "kfilter":
        ch.ch_filter_kgon(s["pts"], s["dirs"], s["ext"], s["idx"], s["sp"], s["cnt"], s["ws"].buf)
        return s["ext"], s["idx"], s["sp"], s["cnt"]
    if kind == "learned":
        return s["prop"].hull_on_device(s["pts"], s["ws"], sync=False, out=s["out"])
    p = s["prop"]
    p.train_step(*s["batch"], lam=LAM, lr=LR, scratch=s["scratch"], loss=s["loss"])
    return s["loss"], p.master, p.m, p.v, p.params


# the share of the points that the octagon leaves
KEPT = {"normal": 0.0, "circle": 1.0, "displaced": 0.95, "gaussians": 0.0, "ellipse": 0.95}


def work(case):
    kind = case["kind"]
    if kind == "train":
        b, p = case["batch"], sum(int(np.prod(s)) for s in SHAPES)
        # inputs and losses; weights, master and both moments read and written
        return {"bytes": b * (1024 + 64 + 3) * 4 + p * (2 * 2 + 3 * 8), "flops": 6 * b * p}
    if kind == "batched":   # (the hulls, a few hundredths of the points, are left out)
        return {"bytes": 8 * int(_sizes(case, None).sum()) + 16 * (case["sets"] + 1), "flops": 0}
    kept = 12 * KEPT[case["dist"]] if kind in ("filter", "sweep", "kfilter") else 0
    return {"bytes": int((8 + kept) * case["n"]), "flops": 0}


def _exact_learned(case, seed):
    """The direction table in binary64: the features by their definition, the
    network on the committed BF16 weights."""
    n = case["n"]
    pts = _points(case["dist"], n, seed, 0)
    m = min(n, 4096)
    p = pts[(torch.arange(m, device=DEV) * n) // m].cpu().numpy()
    del pts
    x, y = p[:, 0], p[:, 1]
    w, h = np.float32(x.max() - x.min()), np.float32(y.max() - y.min())
    sx = np.float32(32) / w if w > 0 else np.float32(0)
    sy = np.float32(32) / h if h > 0 else np.float32(0)
    cx = np.minimum(31, np.floor((x - x.min()) * sx).astype(np.int64))
    cy = np.minimum(31, np.floor((y - y.min()) * sy).astype(np.int64))
    a = np.bincount(cy * GRID + cx, minlength=GRID * GRID) / m
    bits = np.load(os.path.join(os.path.dirname(learned.__file__), "weights", "proposal.npz"))["params"]
    flat = (bits.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    at = 0
    for i in range(3):
        W = flat[at:at + int(np.prod(SHAPES[2 * i]))].reshape(SHAPES[2 * i])
        at += W.size
        a = W @ a + flat[at:at + W.shape[0]]
        at += W.shape[0]
        a = np.maximum(a, 0.0) if i < 2 else a
    K = 8 << int(np.argmax(a[:4]))
    th = 2.0 * math.pi * np.arange(K) / K + np.clip(a[4:4 + K], -0.45, 0.45) * math.pi / K
    dirs = np.zeros(128)
    dirs[0:2 * K:2], dirs[1:2 * K:2] = np.cos(th), np.sin(th)
    return None, None, None, dirs


def _exact_train(case, seed):
    X, label, off, mask, w, m, v = _training(case["batch"], seed)
    W = [t.reshape(s).requires_grad_() for t, s in
         zip(w.to(torch.bfloat16).double().split([int(np.prod(s)) for s in SHAPES]), SHAPES)]
    a = torch.relu(X.double() @ W[0].T + W[1])
    a = torch.relu(a @ W[2].T + W[3])
    o = a @ W[4].T + W[5]
    loss = torch.nn.functional.cross_entropy(o[:, :4], label.long(), reduction="none")
    loss = loss + LAM * mask.double() * ((o[:, 4:] - off.double()) ** 2).mean(1)
    g = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss.mean(), W)])
    m = 0.9 * m.double() + 0.1 * g
    v = 0.999 * v.double() + 0.001 * g * g
    w = w.double() - LR * (m / (1 - 0.9 ** TRAIN_STEP)) / ((v / (1 - 0.999 ** TRAIN_STEP)).sqrt() + 1e-8)
    return loss.detach(), w, m, v, w


def exact(case, seed):
    """Only the learned proposal computes numbers: the other outputs are
    indices, counts and copies of input points."""
    if case["kind"] == "learned":
        return _exact_learned(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    return None
