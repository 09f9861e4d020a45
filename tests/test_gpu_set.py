"""Sets small enough for the one-CTA kernel (k_set), against the oracle:
element-by-element equality at the edges of its size classes, in batches that
mix them with larger sets, and on inputs that take its rare branches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EDGES = [1, 2, 5, 31, 127, 129, 1023, 1024, 1025, 2047, 2048, 4095, 4096, 4097, 12_287, 12_288, 16_382, 16_383, 16_384]
KINDS = {
    "square": inputs.square_f64,
    "disk": inputs.disk_f64,
    "gauss": inputs.gauss_f64,
    "shell": lambda n, s: inputs.shell_f64(n, s),
    "circle": inputs.circle_f64,
    "huge": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** 90,          # beyond the FP32 views
    "tiny": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** -200,
    "igrid": lambda n, s: np.random.default_rng(s).integers(-9, 10, (n, 2)).astype(np.int32),
    "idisk": inputs.disk_i32,
    "iwide": lambda n, s: np.random.default_rng(s).integers(-2 ** 31, 2 ** 31, (n, 2)).astype(np.int32),
}


def check(p):
    got = cch.hull(torch.from_numpy(np.ascontiguousarray(p)).to(DEV)).cpu().numpy()
    assert np.array_equal(got, oracle.hull(p)), (p.dtype, p.shape)
    return got


@pytest.mark.parametrize("kind", list(KINDS))
def test_class_edges(kind):
    sets = [KINDS[kind](n, n % 101 + 1) for n in EDGES]
    for p in sets:
        check(p)
    off = np.concatenate([[0], np.cumsum(EDGES)])
    got = cch.hull_batched(torch.from_numpy(np.concatenate(sets)).to(DEV), off)
    for p, h in zip(sets, got):
        assert np.array_equal(h.cpu().numpy(), oracle.hull(p)), (kind, len(p))


def test_float32_vectors():
    for n in EDGES:
        for p in (inputs.disk_f64(n, n), inputs.gauss_f64(n, n) * 2.0 ** -140):   # float32 subnormals too
            q = p.astype(np.float32)
            x, y = (torch.from_numpy(np.ascontiguousarray(q[:, k])).to(DEV) for k in (0, 1))
            w = q.astype(np.float64)
            assert np.array_equal(cch.hull_f32soa(x, y).cpu().numpy(), oracle.hull(w))


def test_crowded_sort_keys():
    """Hundreds of region points with one sort key: the bitonic sort."""
    rng = np.random.default_rng(5)
    for m in (65, 700, 3000, 12_000):
        col = np.stack([np.full(m, -0.9), -0.11 - 0.88 * rng.random(m)], 1)
        p = np.concatenate([[[-1.0, 0.0], [0.0, -1.0], [1.0, 0.0], [0.0, 1.0]], col, col[: m // 3],
                            -col, np.stack([col[:, 1], col[:, 0]], 1)[: m // 10]])
        check(p[rng.permutation(len(p))])


@pytest.mark.parametrize("m", [40, 200, 3000, 15_000])
def test_convex_run_undone_from_its_end(m):
    """A convex arc that one later point takes off the hull, one point per
    peeling round: the stack and bridge-walk branch."""
    t = np.linspace(0.0, 5.0, m)
    arc = np.stack([t, -0.15 * t + 0.0049 * t * t], 1)
    p = np.concatenate([arc, [[5.01, -0.99], [10.0, -1.0], [10.0, 5.0]]])
    rng = np.random.default_rng(m)
    for q in (p, -p, np.stack([-p[:, 1], p[:, 0]], 1)):
        check(q[rng.permutation(len(q))])


@pytest.mark.parametrize("dtype", [np.int32, np.float64])
def test_mixed_batch(dtype):
    rng = np.random.default_rng(3)
    sizes = [0, 1, 20_000, 900, 1024, 16_383, 0, 16_384, 70_000, 5, 4096, 3000] + list(rng.integers(0, 3000, 60))
    sets = []
    for k, n in enumerate(sizes):
        n = int(n)
        if dtype is np.int32:
            sets.append(inputs.square_i32(n, k) if k % 2 else inputs.disk_i32(n, k))
        else:
            sets.append([inputs.square_f64, inputs.disk_f64, inputs.circle_f64][k % 3](max(n, 1), k)[:n])
    bad = 13
    if dtype is np.float64:
        sets[bad] = sets[bad].copy()
        sets[bad][-1, 0] = np.nan
    off = np.concatenate([[0], np.cumsum([len(q) for q in sets])])
    pts = torch.from_numpy(np.concatenate(sets)).to(DEV)
    idx, cnt = cch.hull_batched_async(pts, off)
    idx, cnt = idx.cpu().numpy(), cnt.cpu().numpy()
    for k, q in enumerate(sets):
        if dtype is np.float64 and k == bad:
            assert cnt[k] == -3
            continue
        want = oracle.hull(q)
        assert cnt[k] == len(want), k
        assert np.array_equal(idx[off[k]:off[k] + cnt[k]], want), k


def test_domain_errors():
    for n in (3, 1000, 9000):
        for v, code in ((np.nan, -3), (np.inf, -3), (-np.inf, -3), (2.0 ** 401, -4), (2.0 ** -410, -4)):
            p = inputs.disk_f64(n, 4)
            p[n // 2, 1] = v
            _, cnt = cch.hull_async(torch.from_numpy(p).to(DEV))
            assert int(cnt.item()) == code, (n, v)
