"""Sets on which every orientation is close to zero, so that the exact tests
decide: collinear points, and points an ulp beside a line, with coordinates of
very different magnitude."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def grid_line(n, rng):
    return np.outer(rng.random(n), [1.0, 2.0])                        # exactly collinear


def rounded_line(n, rng):
    t = rng.random(n)
    return np.stack([t, t / 3.0], axis=1)                             # within an ulp of a line


def spread_line(n, rng):
    t = rng.random(n) * 2.0 ** rng.integers(-70, 1, n)                # gaps beyond 63 bits too
    return np.stack([t, 3.0 * t], axis=1)


def two_lines(n, rng):
    p = rounded_line(n, rng)
    p[::2, 1] = -p[::2, 0] * 2.0 ** -40
    return p


def ulps(n, rng):
    p = grid_line(n, rng)
    k = rng.integers(0, n, n // 3)
    p[k, 1] = np.nextafter(p[k, 1], rng.choice([-9.0, 9.0], len(k)))
    return p


@pytest.mark.parametrize("kind", [grid_line, rounded_line, spread_line, two_lines, ulps])
@pytest.mark.parametrize("scale", [1.0, -2.0 ** 100, 2.0 ** -250])
def test_near_collinear(kind, scale):
    for n in (700, 3000, 12_000, 16_384, 70_001):
        p = kind(n, np.random.default_rng(n)) * scale
        got = cch.hull(torch.from_numpy(p).to(DEV)).cpu().numpy()
        assert np.array_equal(got, oracle.hull(p)), (kind.__name__, scale, n)
