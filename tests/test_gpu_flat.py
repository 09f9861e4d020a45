"""Sets with flat sides: many points of one sort key, and copies, in every
region, through the sort of k_set (whole sets, lists of the sieve, batches)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def grid(n, rng, w=40, h=40):
    return np.stack([rng.integers(-w, w + 1, n), rng.integers(-h, h + 1, n)], axis=1).astype(np.float64)


def cut_grid(n, rng):
    """Without its corners, so that whole sides lie outside the quadrilateral."""
    p = grid(n, rng)
    return p[(np.abs(p[:, 0]) < 40) | (np.abs(p[:, 1]) < 40)]


def near_equal(n, rng):
    """Sides whose keys differ by ulps: one bucket, no two keys equal."""
    p = cut_grid(n, rng)
    side = rng.integers(0, 4, len(p))
    eps = rng.integers(0, 2 ** 20, len(p)) * 2.0 ** -47
    p[side == 0, 0] = -40 + eps[side == 0]
    p[side == 1, 1] = -40 + eps[side == 1]
    p[side == 2, 0] = 40 - eps[side == 2]
    p[side == 3, 1] = 40 - eps[side == 3]
    return p


def columns(n, rng):
    p = rng.random((n, 2)) * [1.0, 2.0] - [0.5, 1.0]
    p[: n // 2, 0] = np.round(p[: n // 2, 0] * 4) / 4
    p[n // 4: n // 2, 1] = np.round(p[n // 4: n // 2, 1] * 3) / 3
    return p


def check(p):
    p = np.ascontiguousarray(p)
    for q in (p, p[:, ::-1].copy(), -p):
        got = cch.hull(torch.from_numpy(q).to(DEV)).cpu().numpy()
        assert np.array_equal(got, oracle.hull(q)), p.shape


@pytest.mark.parametrize("kind", [grid, cut_grid, near_equal, columns])
def test_sides(kind):
    for n in (900, 2500, 9000, 12_200, 100_003, 700_001):
        rng = np.random.default_rng(n)
        check(kind(n, rng))
        if kind is not near_equal and kind is not columns:
            check(kind(n, rng).astype(np.int32))


def test_batch_of_sides():
    rng = np.random.default_rng(4)
    for dtype, reps in ((np.float64, 1), (np.int32, 1), (np.float64, 12)):
        sets = [(grid if i % 2 else cut_grid)(n, rng, *(() if i % 2 == 0 else (60, 25))).astype(dtype)
                for i, n in enumerate([1500, 6000, 15_000, 50_000, 3000, 200_000, 9000] * reps)]
        off = np.concatenate([[0], np.cumsum([len(p) for p in sets])])
        got = cch.hull_batched(torch.from_numpy(np.concatenate(sets)).to(DEV), off)
        for i, (p, h) in enumerate(zip(sets, got)):
            assert np.array_equal(h.cpu().numpy(), oracle.hull(p)), (dtype, i)
