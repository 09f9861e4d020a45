"""CPU restatement of the sieve's bands (csrc/k_sieve.cu): every point that the
chords of a sample's polylines drop is strictly inside the exact hull of the
sample.  The model keeps the FP32 operations and their order; peeling is left
out or replaced by a coarser polyline, since any polyline through sample points
must do."""
from fractions import Fraction

import numpy as np
import pytest

import oracle

F = np.float32
U18, U20 = F(2.0 ** -18), F(2.0 ** -20)


def fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))


def view(v):
    """float64 truncated to FP32 (significands only: magnitudes here are normal)."""
    return ((v.view(np.uint64) >> np.uint64(29)) << np.uint64(29)).view(np.float64).astype(F)


def table(V, W, R, keep, E):
    """Bands of V with the chords in W: (s, o, [(a, m, a', m')])."""
    v0, v1 = V.min(), V.max()
    wm, vm = np.abs(W).max(), max(abs(v0), abs(v1))
    sb = F(R) / (v1 - v0)
    band = np.minimum(((V - v0) * sb).astype(np.int64), R - 1)
    lines = []
    for sign in (F(1), F(-1)):
        ext = {}
        for i in range(len(V)):
            b = band[i]
            if b not in ext or sign * W[i] < sign * W[ext[b]]:
                ext[b] = i
        ids = [int(V.argmin())] + [ext[b] for b in sorted(ext) if keep(b)] + [int(V.argmax())]
        lines.append((V[ids], W[ids]))

    def at(line, y):
        pv, pw = line
        l = max(0, min(int(np.searchsorted(pv, y, side="right")) - 1, len(pv) - 2))
        dy = pv[l + 1] - pv[l]
        f = min(max((y - pv[l]) / dy, F(0)), F(1)) if dy > 0 else F(0)
        return fma(f, pw[l + 1] - pw[l], pw[l])

    d = vm * U20
    va, vb = v0 + F(2) * d, v1 - F(2) * d
    if not vb > va:
        return None
    s = F(R) / (vb - va)
    o = fma(-va, s, F(1))
    rows = [None]
    for b in range(1, R + 1):
        l, h = (F(b) - o) / s - d, (F(b + 1) - o) / s + d
        if not (l >= v0 and h <= v1):
            rows.append(None)
            continue
        l0, l1, r0, r1 = at(lines[0], l), at(lines[0], h), at(lines[1], l), at(lines[1], h)
        ml, mr = (l1 - l0) / (h - l), (r1 - r0) / (h - l)
        rows.append((fma(-ml, l, l0) + E * fma(abs(ml), vm, wm), ml, fma(-mr, l, r0) - E * fma(abs(mr), vm, wm), mr))
    return s, o, rows + [None]


def dropped(t, Vp, Wp):
    s, o, rows = t
    out = np.zeros(len(Vp), bool)
    for i, (y, x) in enumerate(zip(Vp, Wp)):
        b = int(min(max(fma(y, s, o), F(0)), F(len(rows) - 1)))
        if rows[b] is not None:
            a, m, a2, m2 = rows[b]
            out[i] = x > fma(m, y, a) and x < fma(m2, y, a2)
    return out


def hull_points(p):
    return [(Fraction(x), Fraction(y)) for x, y in p[oracle.hull(p)].tolist()]


def strictly_inside(hull, x, y):
    x, y = Fraction(float(x)), Fraction(float(y))
    return all((bx - ax) * (y - ay) - (by - ay) * (x - ax) > 0
               for (ax, ay), (bx, by) in zip(hull, hull[1:] + hull[:1]))


def sets():
    rng = np.random.default_rng(11)
    disk = rng.normal(size=(600, 2))
    disk /= np.maximum(1, np.linalg.norm(disk, axis=1))[:, None]
    square = rng.random((600, 2))
    yield "disk", disk
    yield "square", square
    yield "offset", square + [1000.0, -37.0]
    yield "sliver", (disk * [1.0, 1e-4]) @ np.array([[0.8, 0.6], [-0.6, 0.8]])
    yield "scaled", disk * [2.0 ** 50, 2.0 ** -60]
    yield "grid", rng.integers(0, 9, (400, 2)).astype(np.float64)


def probes(p, rng):
    """Random points, and points on, just inside and just outside the hull's edges and vertices."""
    h = p[oracle.hull(p)]
    lo, hi = p.min(0), p.max(0)
    yield from lo + rng.random((400, 2)) * (hi - lo)
    for a, b in zip(h, np.roll(h, -1, axis=0)):
        for t in (0.0, 0.25, 0.5, rng.random()):
            q = a + t * (b - a)
            for e in (-8, -1, 0, 1, 8):
                yield q * (1 + e * 2.0 ** -52)
                yield q + (q - p.mean(0)) * e * 2.0 ** -24


@pytest.mark.parametrize("name,p", list(sets()), ids=[n for n, _ in sets()])
def test_dropped_points_are_inside(name, p):
    rng = np.random.default_rng(5)
    q = np.array(list(probes(p, rng)))
    hull = hull_points(p)
    X, Y, QX, QY = (view(np.ascontiguousarray(c)) for c in (p[:, 0], p[:, 1], q[:, 0], q[:, 1]))
    for R, keep in ((16, lambda b: True), (64, lambda b: True), (64, lambda b: b % 3 == 0)):
        for V, W, QV, QW in ((Y, X, QY, QX), (X, Y, QX, QY)):
            t = table(V, W, R, keep, U18)
            if t is None:
                continue
            drop = dropped(t, QV, QW)
            if name in ("disk", "square"):
                assert drop.sum() > 100          # the bands do drop the inside
            for i in np.flatnonzero(drop):
                assert strictly_inside(hull, *q[i]), (name, R, q[i])


def test_missing_margin_is_caught():
    """A margin of the wrong sign, on edges that run through many bands."""
    rng = np.random.default_rng(3)
    p = np.concatenate([[[-1.0, -0.9], [1.0, -0.2], [0.3, 1.0]], rng.random((50, 2)) * 0.1])
    q = np.array(list(probes(p, np.random.default_rng(5))))
    hull = hull_points(p)
    X, Y, QX, QY = (view(np.ascontiguousarray(c)) for c in (p[:, 0], p[:, 1], q[:, 0], q[:, 1]))
    drop = dropped(table(Y, X, 64, lambda b: True, F(-2.0 ** -18)), QY, QX)
    assert any(not strictly_inside(hull, *q[i]) for i in np.flatnonzero(drop))


def test_quantised_keys_are_monotone():
    """The multi-block sort's quantised key (csrc/k_big.cu) never decreases with the key and fits 30 bits."""
    rng = np.random.default_rng(2)
    mask = (1 << 64) - 1

    def key(v):
        b = 0 if v == 0 else int(np.float64(v).view(np.uint64))
        return (~b & mask) if b >> 63 else b | 1 << 63

    def fix(k, emax):
        b = k & ((1 << 63) - 1) if k >> 63 else ~k & mask
        e = (b >> 52) & 0x7FF
        sh = emax - e
        f = 0 if e == 0 or sh > 62 else (((b & ((1 << 52) - 1)) | 1 << 52) << 9) >> max(sh, 0)
        return (1 << 63) + f if k >> 63 else (1 << 63) - f

    for lo, hi in ((-1.0, 1.0), (-1.0, 0.0), (0.0, 2.0 ** 59), (3.0, 3.0 + 2.0 ** -50), (-2.0 ** -300, 2.0 ** -310), (5.0, 5.0)):
        v = np.concatenate([lo + (hi - lo) * rng.random(300), (hi - lo) * 2.0 ** -rng.uniform(0, 300, 300), [lo, hi, 0.0, -0.0]])
        v = np.sort(v[(v >= lo) & (v <= hi)])
        kl, kh = key(lo), key(hi)
        ex = [((k if k >> 63 else ~k & mask) >> 52) & 0x7FF for k in (kl, kh)]
        emax = max(ex)
        d = max(fix(kh, emax) - fix(kl, emax), 0)
        shift = max(0, d.bit_length() - 30)
        q = [min(max(fix(key(x), emax) - fix(kl, emax), 0) >> shift, (1 << 30) - 1) for x in v]
        assert all(a <= b for a, b in zip(q, q[1:])) and q[0] >= 0 and q[-1] < 1 << 30
        if hi - lo > 1e-3 * max(abs(lo), abs(hi)):
            assert q[-1] >= (1 << 29) - 1
