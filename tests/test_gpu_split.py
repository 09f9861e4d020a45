"""Sets split over a cluster of four CTAs, one region each: single sets from
1024 points, batches of few sets, and the lists of a batch of few sets."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def degenerate_regions(n, s):
    """Extremes that coincide: regions without a chain."""
    p = inputs.disk_f64(n, s)
    p[:2] = [[-3.0, -3.0], [3.0, 3.0]]
    return p


KINDS = {
    "disk": inputs.disk_f64,
    "circle": inputs.circle_f64,
    "regions": degenerate_regions,
    "triangle": lambda n, s: (lambda p: np.where((p.sum(1) > 1.0)[:, None], 1.0 - p, p))(inputs.square_f64(n, s)),
    "huge": lambda n, s: inputs.circle_f64(n, s) * 2.0 ** 90,
    "huge_far": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** 330 + 2.0 ** 200,
    "huge_spread": lambda n, s: inputs.disk_f64(n, s) * 2.0 ** np.random.default_rng(s).integers(-200, 200, (n, 1)),
    "tiny": lambda n, s: inputs.circle_f64(n, s) * 2.0 ** -300,
    "one": lambda n, s: np.full((n, 2), 0.1 * s),
    "idisk": inputs.disk_i32,
    "icircle": lambda n, s: np.floor(inputs.circle_f64(n, s) * 2.0 ** 28).astype(np.int32),
    "iwide": lambda n, s: np.random.default_rng(s).integers(-2 ** 31, 2 ** 31, (n, 2)).astype(np.int32),
}


@pytest.mark.parametrize("kind", list(KINDS))
def test_single_sets(kind):
    for n in (1023, 1024, 2047, 2049, 4095, 8191, 12_287, 12_288, 30_001):
        p = np.ascontiguousarray(KINDS[kind](n, n % 89 + 1))
        assert np.array_equal(cch.hull(torch.from_numpy(p).to(DEV)).cpu().numpy(), oracle.hull(p)), n


@pytest.mark.parametrize("count", [2, 37, 39])
@pytest.mark.parametrize("kind", ["disk", "circle", "huge", "icircle"])
def test_batches_on_both_sides_of_the_limit(kind, count):
    """38 sets are split on 152 SMs, 39 are not; on another GPU the limit lies elsewhere, the hulls are the same."""
    sizes = [[1024, 5000, 16_383][i % 3] for i in range(count)] + [300, 0, 1]
    base = {n: np.ascontiguousarray(KINDS[kind](n, 5)) for n in set(sizes) if n}
    want = {n: oracle.hull(p) for n, p in base.items()}
    off = np.concatenate([[0], np.cumsum(sizes)])
    got = cch.hull_batched(torch.from_numpy(np.concatenate([base[n] for n in sizes if n])).to(DEV), off)
    for n, h in zip(sizes, got):
        assert np.array_equal(h.cpu().numpy(), want[n] if n else np.zeros(0, np.int32)), n


def test_domain_errors_of_split_sets():
    for n in (1024, 9000):
        for v, code in ((np.nan, -3), (np.inf, -3), (2.0 ** 401, -4), (2.0 ** -410, -4)):
            p = inputs.disk_f64(n, 4)
            p[n // 2, 1] = v
            _, cnt = cch.hull_async(torch.from_numpy(p).to(DEV))
            assert int(cnt.item()) == code, (n, v)
