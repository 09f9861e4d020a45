"""Batches by the number and the sizes of their sets: one set, few sets, sets
above 2^18 points in few and in many, small sets beside larger ones, and sets
of which some are refused by the sieve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GEN = {"disk": inputs.disk_f64, "square": inputs.square_f64, "circle": inputs.circle_f64,
       "degenerate": inputs.degenerate_f64, "idisk": inputs.disk_i32, "isquare": inputs.square_i32}
_cache = {}


def set_of(kind, n):
    if (kind, n) not in _cache:
        p = np.ascontiguousarray(GEN[kind](n, n % 83 + 1)) if n else np.zeros((0, 2), np.int32 if kind[0] == "i" else np.float64)
        _cache[kind, n] = (torch.from_numpy(p).to(DEV), oracle.hull(p) if n else np.zeros(0, np.int32))
    return _cache[kind, n]


def check(sets):
    pts = torch.cat([set_of(*k)[0] for k in sets])
    off = np.concatenate([[0], np.cumsum([k[1] for k in sets])])
    for _ in range(2):
        got = cch.hull_batched(pts, off)
        for k, h in zip(sets, got):
            assert np.array_equal(h.cpu().numpy(), set_of(*k)[1]), k


@pytest.mark.parametrize("n", [0, 1, 1000, 16_000, 50_003, 300_001])
def test_one_set(n):
    check([("disk", n)])
    check([("isquare", n)])


def test_few_larger_sets():
    check([("disk", 17_003), ("square", 40_001)])
    check([("idisk", 262_144), ("isquare", 262_145)])
    check([("disk", 20_011), ("circle", 30_011), ("square", 262_144), ("disk", 60_001)])        # one is refused: all are
    check([("degenerate", 38_000 + 501 * i) for i in range(6)])                                 # about half of them


def test_small_beside_larger():
    sizes = [300, 1500, 9000, 16_383, 700, 0, 4096]
    for larger in ([("disk", 70_001)], [("circle", 30_011), ("disk", 20_011)], [("square", 500_003)],
                   [("disk", 500_003), ("disk", 20_011)], [("disk", 20_011)] * 130 + [("square", 500_003)]):
        check([("disk", n) for n in sizes] + larger + [("square", n) for n in sizes])


def test_many_sets_above_2_to_18():
    """One for every SM at least: sieved, the disks among them refused by their lists' length or not."""
    check([("idisk" if i % 3 else "isquare", 270_001) for i in range(160)] + [("idisk", 900), ("isquare", 20_011)])


def test_small_sets_of_several_calls_in_flight():
    """The small sets run on a stream of the workspace: later calls on the caller's stream come after them."""
    a = [("disk", 9000)] * 20 + [("disk", 70_001)]
    b = [("circle", 16_000), ("square", 40_001), ("disk", 1200)]
    ops = []
    for sets in (a, b) * 4:
        pts = torch.cat([set_of(*k)[0] for k in sets])
        off = np.concatenate([[0], np.cumsum([k[1] for k in sets])])
        idx, cnt = cch.hull_batched_async(pts, off)
        ops.append((sets, off, idx.clone(), cnt.clone()))
    for sets, off, idx, cnt in ops:
        cnt = cnt.cpu().numpy()
        for i, k in enumerate(sets):
            assert np.array_equal(idx[int(off[i]):int(off[i]) + int(cnt[i])].cpu().numpy(), set_of(*k)[1]), k
