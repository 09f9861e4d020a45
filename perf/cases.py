"""The hull workloads that are timed, one pass each through the public calls.

A case is a dict of plain values:

    name     listed cases only
    form     'one'    one set, (x, y) rows         hull / hull_async
             'f32soa' one set, two float32 vectors hull_f32soa_async
             'batch'  many sets, (x, y) rows       hull_batched_async
    dtype    'i32' or 'f64' ('f32' for 'f32soa')
    kind     the distribution (see _points); 'mixed' for a batch: a square or
             a disk per set by a fair coin
    n        points of the set          (form 'one', 'f32soa')
    nsets, lo, hi    number of sets and the range of their log-uniform sizes
                     (form 'batch')
    wait     form 'one': the caller reads the hull's size back at once (the
             launch-to-answer time); otherwise it only enqueues the call

Points are drawn in device memory by a torch generator seeded with `seed`;
the set sizes of a batch belong to the case, not to the seed.  The output
buffers that a caller keeps are zero-filled once, so that the slots after the
hull compare equal.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

import paper_1508_05488_gb300 as cch

_TORCH = {"i32": torch.int32, "f64": torch.float64, "f32": torch.float32}
_BYTES = {"i32": 8, "f64": 16, "f32": 8}     # of one point
_SPAN = 2 ** 29                              # int32 coordinates lie in [0, 2^29)
_GRID = 2.0 ** -20                           # rounding grid of the degenerate sets


def listed():
    return [
        # The smallest request of a program that wants the hull's indices
        # before it goes on: launches and latency.
        {"name": "tiny_i32", "form": "one", "dtype": "i32", "kind": "square", "n": 1003, "wait": True},
        # An ordinary small set, waited for (a scanned outline, a cluster of detections).
        {"name": "small_disk", "form": "one", "dtype": "f64", "kind": "disk", "n": 60_001, "wait": True},
        # A million integer points in a square, the middle of the paper's size range.
        {"name": "square_i32_1M", "form": "one", "dtype": "i32", "kind": "square", "n": 1_000_000, "wait": False},
        # The headline sets: the paper's largest size, uniform in a square
        # (rbox) and in a disk (many more survivors).
        {"name": "square_20M", "form": "one", "dtype": "f64", "kind": "square", "n": 20_000_000, "wait": False},
        {"name": "disk_20M", "form": "one", "dtype": "f64", "kind": "disk", "n": 20_000_000, "wait": False},
        # A Gaussian cloud of a ragged mid size: hardly any point survives round 1.
        {"name": "gauss_5M", "form": "one", "dtype": "f64", "kind": "gauss", "n": 5_000_011, "wait": False},
        # A thin annulus (one of the serving stream's kinds): every point is
        # close to the hull, so far more survive than on the disk.
        {"name": "shell_2M", "form": "one", "dtype": "f64", "kind": "shell", "n": 2_000_003, "wait": False},
        # Collinear runs, coincident points and a fifth of the set on a circle.
        {"name": "degenerate_20M", "form": "one", "dtype": "f64", "kind": "degenerate", "n": 20_000_000,
         "wait": False},
        # Every point a hull vertex: the limit that the paper names in Sec. 4.3.
        {"name": "circle_2M", "form": "one", "dtype": "f64", "kind": "circle", "n": 2_000_000, "wait": False},
        # The paper's own input form, two float32 coordinate vectors, at its largest size.
        {"name": "f32_disk_20M", "form": "f32soa", "dtype": "f32", "kind": "disk", "n": 20_000_000},
        # Many independent integer sets of very different size in one call.
        {"name": "batch_i32", "form": "batch", "dtype": "i32", "kind": "mixed", "nsets": 1024, "lo": 256,
         "hi": 2 ** 18},
        # Thousands of small float64 sets in one call (the server's batches at high load).
        {"name": "batch_small_f64", "form": "batch", "dtype": "f64", "kind": "mixed", "nsets": 4096, "lo": 256,
         "hi": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["f64", "f64", "i32", "f32soa", "hard", "batch"])
    if form == "f64":
        return {"form": "one", "dtype": "f64", "kind": rng.choice(["square", "disk", "gauss", "shell"]),
                "n": _log_int(rng, 1_000, 20_000_000), "wait": rng.random() < 0.25}
    if form == "i32":
        return {"form": "one", "dtype": "i32", "kind": rng.choice(["square", "disk"]),
                "n": _log_int(rng, 1_000, 20_000_000), "wait": rng.random() < 0.25}
    if form == "f32soa":
        return {"form": "f32soa", "dtype": "f32", "kind": rng.choice(["square", "disk", "gauss"]),
                "n": _log_int(rng, 1_000, 20_000_000)}
    if form == "hard":
        kind = rng.choice(["circle", "degenerate"])
        return {"form": "one", "dtype": "f64", "kind": kind,
                "n": _log_int(rng, 1_000, 2_000_000 if kind == "circle" else 20_000_000), "wait": False}
    hi = _log_int(rng, 1_024, 2 ** 18)
    return {"form": "batch", "dtype": rng.choice(["i32", "f64"]), "kind": "mixed",
            "nsets": min(_log_int(rng, 16, 4096), (2 ** 28) // hi), "lo": 256, "hi": hi}


# ------------------------------------------------------------------- inputs

def _unit(kind, n, g):
    """n float64 points [n, 2] of a distribution around the unit square or circle."""
    dev = g.device
    f64 = torch.float64
    if kind == "square":
        return torch.rand((n, 2), dtype=f64, device=dev, generator=g)
    if kind == "gauss":
        return torch.randn((n, 2), dtype=f64, device=dev, generator=g)
    if kind == "circle":      # angles 2 pi (k + phase) / n, shuffled
        phase = torch.rand(1, dtype=f64, device=dev, generator=g)
        t = 2.0 * math.pi * (torch.randperm(n, device=dev, generator=g).to(f64) + phase) / n
        return torch.stack([torch.cos(t), torch.sin(t)], dim=1)
    if kind == "degenerate":
        nc, nd = n // 5, n // 100
        p = torch.cat([_unit("ring", nc, g), (1.0 - 2.0 ** -10) * _unit("disk", n - nc, g)])
        p = torch.round(p / _GRID) * _GRID
        dst = torch.randint(0, n, (nd,), device=dev, generator=g).unique()
        src = torch.randint(0, n, (dst.shape[0],), device=dev, generator=g)
        src[::2] %= max(nc, 1)          # half of the copies repeat circle points
        p[dst] = p[src]
        return p[torch.randperm(n, device=dev, generator=g)]
    u = torch.rand((n, 2), dtype=f64, device=dev, generator=g)
    t = 2.0 * math.pi * u[:, 1]
    if kind == "disk":
        r = torch.sqrt(u[:, 0])
    elif kind == "shell":     # 0.99 <= r <= 1
        r = torch.sqrt(0.99 ** 2 + u[:, 0] * (1.0 - 0.99 ** 2))
    elif kind == "ring":      # random angles on the circle
        r = torch.ones_like(t)
    else:
        raise ValueError(kind)
    return torch.stack([r * torch.cos(t), r * torch.sin(t)], dim=1)


def _as_i32(p, disk):
    """Float64 points of the unit square, or of the unit disk where `disk`, on [0, 2^29)^2."""
    half = _SPAN // 2
    q = torch.where(disk, p * (half - 1) + half, p * _SPAN)
    return q.floor().clamp(0, _SPAN - 1).to(torch.int32).contiguous()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _points(case, seed):
    """The points of a case: [n, 2], or the vectors (x, y) of an 'f32soa' case; and the offsets of a batch."""
    g = _generator(seed)
    if case["form"] == "batch":
        rng = np.random.default_rng([case["nsets"], case["lo"], case["hi"]])
        sizes = np.floor(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["nsets"])))
        off = np.zeros(case["nsets"] + 1, dtype=np.int64)
        off[1:] = np.cumsum(sizes.astype(np.int64))
        coin = torch.from_numpy(rng.random(case["nsets"]) < 0.5).cuda()
        disk = torch.repeat_interleave(coin, torch.from_numpy(np.diff(off)).cuda())[:, None]
        n = int(off[-1])
        p = torch.where(disk, _unit("disk", n, g), _unit("square", n, g))
        return (_as_i32(p, disk) if case["dtype"] == "i32" else p.contiguous()), off
    p = _unit(case["kind"], case["n"], g)
    if case["form"] == "f32soa":
        return (p[:, 0].float().contiguous(), p[:, 1].float().contiguous()), None
    if case["dtype"] == "i32":
        p = _as_i32(p, torch.tensor(case["kind"] == "disk", device=p.device))
    return p.contiguous(), None


# --------------------------------------------------------------------- pass

def prepare(case, seed):
    p, off = _points(case, seed)
    n = p[0].shape[0] if case["form"] == "f32soa" else p.shape[0]
    return {"form": case["form"], "wait": case.get("wait", False), "points": p, "offsets": off,
            "idx": torch.zeros(n, dtype=torch.int32, device="cuda"),
            "count": torch.zeros(case.get("nsets", 1), dtype=torch.int32, device="cuda")}


def run(state):
    if state["form"] == "f32soa":
        x, y = state["points"]
        return cch.hull_f32soa_async(x, y, state["idx"], state["count"])
    if state["form"] == "batch":
        return cch.hull_batched_async(state["points"], state["offsets"], state["idx"], state["count"])
    idx, count = cch.hull_async(state["points"], state["idx"], state["count"])
    return (idx, count.item()) if state["wait"] else (idx, count)


def work(case):
    """Every point read once and the hull's indices written once (only a
    circle's hull is of any size); per point the operations of one test
    against the quadrilateral's four edges (two products and two sums each)."""
    if case["form"] == "batch":
        lo, hi = case["lo"], case["hi"]
        n = int(case["nsets"] * (hi - lo) / math.log(hi / lo))    # mean of a log-uniform size
    else:
        n = case["n"]
    hull = 4 * n if case["kind"] == "circle" else 0
    return {"bytes": n * _BYTES[case["dtype"]] + hull, "flops": 16 * n}


# -------------------------------------------------------------------- exact

def _outside(x, y, idx, dirs):
    """The points that are not well inside the polygon of the extremes along `dirs` directions."""
    t = torch.arange(dirs, dtype=torch.float64) * (2.0 * math.pi / dirs)
    ext = []
    for c, s in zip(torch.cos(t).tolist(), torch.sin(t).tolist()):
        k = int(torch.argmax(c * x + s * y))
        ext.append((float(x[k]), float(y[k])))
    ext = [e for i, e in enumerate(ext) if e != ext[i - 1]]
    if len(ext) < 3:
        return x, y, idx
    inside = torch.ones_like(x, dtype=torch.bool)
    for (ax, ay), (bx, by) in zip(ext, ext[1:] + ext[:1]):
        dx, dy = bx - ax, by - ay
        margin = 1e-9 * (abs(dx) + abs(dy)) * max(abs(ax), abs(ay), abs(bx), abs(by))
        inside &= dx * (y - ay) - dy * (x - ax) > margin
    out = ~inside
    return x[out], y[out], idx[out]


def _cross(a, b, c):
    """A number of the exact sign of (b - a) x (c - a)."""
    lhs, rhs = (b[0] - a[0]) * (c[1] - a[1]), (b[1] - a[1]) * (c[0] - a[0])
    d = lhs - rhs
    if isinstance(d, int) or abs(d) > 1e-14 * (abs(lhs) + abs(rhs)):
        return d
    ax, ay, bx, by, cx, cy = (Fraction(v) for v in (*a[:2], *b[:2], *c[:2]))
    return (bx - ax) * (cy - ay) - (by - ay) * (cx - ax)


def _hull(p):
    """Indices of the strict hull of [n, 2] points, counter-clockwise from the
    smallest (x, y); the smallest index of coincident points."""
    x, y = p[:, 0].double(), p[:, 1].double()
    idx = torch.arange(p.shape[0], device=p.device)
    if p.shape[0] > 64:
        x, y, idx = _outside(x, y, idx, 8)
    if idx.shape[0] > 100_000:
        x, y, idx = _outside(x, y, idx, 128)
    cast = int if p.dtype == torch.int32 else float
    pts = sorted(zip(map(cast, x.tolist()), map(cast, y.tolist()), idx.tolist()))
    pts = [q for i, q in enumerate(pts) if i == 0 or q[:2] != pts[i - 1][:2]]
    if len(pts) < 3:
        return [q[2] for q in pts]

    def chain(seq):
        st = []
        for q in seq:
            while len(st) > 1 and _cross(st[-2], st[-1], q) <= 0:
                st.pop()
            st.append(q)
        return st

    return [q[2] for q in chain(pts)[:-1] + chain(reversed(pts))[:-1]]


def exact(case, seed):
    """The hull by Andrew's monotone chain with rational arithmetic where
    float64 leaves the sign open; None for large sets with most of their
    points on or beside the hull."""
    limit = {"circle": 20_000, "degenerate": 20_000, "shell": 4_000_000}.get(case["kind"])
    if limit is not None and case["n"] > limit:
        return None
    p, off = _points(case, seed)
    if case["form"] == "batch":
        idx = np.zeros(p.shape[0], dtype=np.int32)
        count = np.zeros(case["nsets"], dtype=np.int32)
        for s in range(case["nsets"]):
            h = _hull(p[int(off[s]):int(off[s + 1])])
            idx[int(off[s]):int(off[s]) + len(h)] = h
            count[s] = len(h)
        return idx, count
    if case["form"] == "f32soa":
        p = torch.stack(p, dim=1)
    h = np.array(_hull(p), dtype=np.int32)
    idx = np.zeros(p.shape[0], dtype=np.int32)
    idx[:h.shape[0]] = h
    if case.get("wait"):
        return idx, int(h.shape[0])
    return idx, np.array([h.shape[0]], dtype=np.int32)
