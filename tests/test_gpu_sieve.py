"""The one-pass sieve of large sets against the oracle, element by element: at
the sizes where its units, its sample and its lists change, and on inputs on
which its polygon is poor, empty or must not be trusted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SIZES = [12_288, 16_384, 20_011, 60_001, 262_145, 700_003]


def rot(p, t):
    c, s = np.cos(t), np.sin(t)
    return p @ np.array([[c, s], [-s, c]])


def grid(n, s):
    return np.random.default_rng(s).integers(-400, 401, (n, 2)).astype(np.float64)


def half_zero(n, s):
    p = inputs.disk_f64(n, s)
    p[::2, 0] = 0.0
    return p


def dupes(n, s):
    p = inputs.disk_f64(n, s)
    q = np.random.default_rng(s).integers(0, n, n // 2)
    p[: n // 2] = p[q]
    return p


KINDS = {
    "square": inputs.square_f64,
    "disk": inputs.disk_f64,
    "gauss": inputs.gauss_f64,
    "shell": inputs.shell_f64,
    "circle": inputs.circle_f64,
    "grid": grid,                                            # flat sides, equal coordinates, zeros
    "half_zero": half_zero,
    "dupes": dupes,
    "sorted_x": lambda n, s: np.sort(inputs.disk_f64(n, s).view("f8,f8"), axis=0).view("f8").reshape(-1, 2),
    "sorted_r": lambda n, s: (lambda p: p[np.argsort((p * p).sum(1))])(inputs.disk_f64(n, s)),
    "sliver": lambda n, s: rot(inputs.disk_f64(n, s) * [1.0, 1e-5], 0.7),
    "flat": lambda n, s: inputs.disk_f64(n, s) * [1.0, 1e-9] + [0.0, 1.0],
    "line": lambda n, s: np.outer(inputs.square_f64(n, s)[:, 0], [1.0, 2.0]),
    "level": lambda n, s: inputs.square_f64(n, s) * [1.0, 0.0],
    "far": lambda n, s: inputs.disk_f64(n, s) + [1e5, -1e7],
    "huge": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** 90,
    "edge60": lambda n, s: inputs.square_f64(n, s) * 2.0 ** 60.5,     # views end inside the set
    "tiny": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** -200,
    "edge126": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** -95,
    "idisk": inputs.disk_i32,
    "isquare": inputs.square_i32,
    "igrid": lambda n, s: np.random.default_rng(s).integers(-99, 100, (n, 2)).astype(np.int32),
    "iwide": lambda n, s: np.random.default_rng(s).integers(-2 ** 31, 2 ** 31, (n, 2)).astype(np.int32),
}


def run(p):
    return cch.hull(torch.from_numpy(np.ascontiguousarray(p)).to(DEV)).cpu().numpy()


@pytest.mark.parametrize("kind", list(KINDS))
def test_sizes(kind):
    for n in SIZES:
        p = np.ascontiguousarray(KINDS[kind](n, n % 97 + 1))
        assert np.array_equal(run(p), oracle.hull(p)), (kind, n)


def test_float32_vectors():
    for n in SIZES:
        for p in (inputs.disk_f64(n, n), inputs.gauss_f64(n, n) * 2.0 ** -140, grid(n, n)):
            q = p.astype(np.float32)
            buf = torch.zeros(2 * n + 3, device=DEV)             # vectors at every 4-byte alignment
            x, y = buf[1:n + 1], buf[n + 3:]
            x.copy_(torch.from_numpy(q[:, 0].copy()))
            y.copy_(torch.from_numpy(q[:, 1].copy()))
            assert np.array_equal(cch.hull_f32soa(x, y).cpu().numpy(), oracle.hull(q.astype(np.float64))), n


def test_int32_odd_base():
    n = 50_021
    p = inputs.disk_i32(n + 1, 3)
    t = torch.from_numpy(p).to(DEV)[1:]
    assert np.array_equal(cch.hull(t).cpu().numpy(), oracle.hull(np.ascontiguousarray(p[1:])))


@pytest.mark.parametrize("bad,name", [(np.nan, "NONFINITE"), (np.inf, "NONFINITE"), (2.0 ** 401, "RANGE"),
                                      (1e-200, "RANGE")])
def test_domain_errors_inside(bad, name):
    """One bad coordinate of a point that would lie deep inside."""
    n = 300_007
    for pos in (0, 151_111, n - 1):
        for col in (0, 1):
            p = inputs.disk_f64(n, 5)
            p[pos] = [0.01, 0.02]
            p[pos, col] = bad
            idx = torch.zeros(n, dtype=torch.int32, device=DEV)
            cnt = torch.zeros(1, dtype=torch.int32, device=DEV)
            cch.hull_async(torch.from_numpy(p).to(DEV), idx, cnt)
            assert int(cnt.item()) == {"NONFINITE": -3, "RANGE": -4}[name]


def test_larger_sets():
    for kind, n in (("square", 5_000_011), ("disk", 5_000_011), ("shell", 3_000_017), ("idisk", 4_000_037)):
        p = KINDS[kind](n, 11)
        assert np.array_equal(run(p), oracle.hull(p)), kind


def test_batches():
    """Sets of every route in one call: whole, sieved, refused (circles), over the sieve's unit limit."""
    rng = np.random.default_rng(3)
    sizes = [16_383, 16_384, 18_433, 40_000, 65_537, 131_072, 262_144, 700, 20_000, 0, 33_333]
    for kinds in (["square", "disk", "gauss"], ["disk", "circle", "shell", "dupes", "sliver"], ["idisk", "isquare", "igrid"],
                  ["iwide", "idisk"]):
        sets = [np.ascontiguousarray(KINDS[kinds[int(rng.integers(len(kinds)))]](max(n, 1), i + 1)[:n])
                for i, n in enumerate(sizes * 3)]
        off = np.concatenate([[0], np.cumsum([len(p) for p in sets])])
        for _ in range(2):
            got = cch.hull_batched(torch.from_numpy(np.concatenate(sets)).to(DEV), off)
            for i, (p, h) in enumerate(zip(sets, got)):
                assert np.array_equal(h.cpu().numpy(), oracle.hull(p)), (kinds, i, len(p))


def test_batch_bad_and_large():
    big, bad = inputs.disk_f64(2_200_000, 4), inputs.disk_f64(90_001, 5)
    bad[777] = [0.01, np.nan]
    sets = [inputs.disk_f64(50_000, 1), bad, big, inputs.circle_f64(30_000, 2), inputs.square_f64(400_001, 3)]
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])])
    idx = torch.zeros(int(off[-1]), dtype=torch.int32, device=DEV)
    cnt = torch.zeros(len(sets), dtype=torch.int32, device=DEV)
    cch.hull_batched_async(torch.from_numpy(np.concatenate(sets)).to(DEV), off, idx, cnt)
    c = cnt.cpu().numpy()
    assert c[1] == -3
    for i in (0, 2, 3, 4):
        assert np.array_equal(idx[int(off[i]):int(off[i]) + int(c[i])].cpu().numpy(), oracle.hull(sets[i])), i


def test_graph_capture():
    """A captured call (with its fork to the workspace's stream) replayed on other points."""
    n = 300_007
    s = torch.cuda.Stream()
    pts = torch.zeros((n, 2), dtype=torch.float64, device=DEV)
    idx = torch.zeros(n, dtype=torch.int32, device=DEV)
    cnt = torch.zeros(1, dtype=torch.int32, device=DEV)
    pts.copy_(torch.from_numpy(inputs.disk_f64(n, 1)))
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        cch.hull_async(pts, idx, cnt)                    # the workspace
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        cch.hull_async(pts, idx, cnt)
    for kind, seed in (("square", 2), ("disk", 3), ("gauss", 4), ("shell", 5)):
        p = KINDS[kind](n, seed)
        pts.copy_(torch.from_numpy(np.ascontiguousarray(p)))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(idx[:int(cnt.item())].cpu().numpy(), oracle.hull(p)), kind


def test_streams_at_once():
    """Sieved and refused sets on several streams, each with its own workspace and side stream."""
    sets = [KINDS[k](150_001 + 7 * i, i + 1) for i, k in enumerate(["disk", "circle", "square", "shell", "gauss", "circle"])]
    pts = [torch.from_numpy(np.ascontiguousarray(p)).to(DEV) for p in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    torch.cuda.synchronize()
    for _ in range(5):
        outs = []
        for p, s in zip(pts, streams):
            with torch.cuda.stream(s):
                outs.append(cch.hull_async(p))
        torch.cuda.synchronize()
        for p, (idx, cnt) in zip(sets, outs):
            assert np.array_equal(idx[:int(cnt.item())].cpu().numpy(), oracle.hull(p))
