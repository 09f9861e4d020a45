"""Calls that are known to reach the pipeline behind the sieve, by the route
that the library reports: every run-time choice, float32 vectors at every
alignment, int32 batches, and the repairs of the sort by quantised keys."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs
from test_gpu_bigsort import SETS as BIG_SETS
from test_gpu_tune import CANDIDATES

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def circle_i32(n, seed):
    return np.floor(inputs.circle_f64(n, seed) * 2.0 ** 28).astype(np.int32)


def run(p):
    got = cch.hull(torch.from_numpy(np.ascontiguousarray(p)).to(DEV)).cpu().numpy()
    assert np.array_equal(got, oracle.hull(p))
    return cch.route()


@pytest.mark.parametrize("kind,sieved", [("square_f64", 1), ("disk_f64", 1), ("gauss_f64", 1), ("shell_f64", 1),
                                         ("disk_i32", 1), ("circle_f64", 0)])
def test_route_of_single_sets(kind, sieved):
    for n in (20_011, 300_007):
        r = run(getattr(inputs, kind)(n, 3))
        assert r["sieved"] == sieved, (kind, n, r)
        assert (r["small_regions"] + r["sort_tiles"] == 0) == bool(sieved), (kind, n, r)


def test_repairs_of_the_sort_by_quantised_keys():
    r = run(BIG_SETS["circle"](400_003))
    assert r["sort_tiles"] > 0 and r["fast_fail"] == 0
    r = run(BIG_SETS["arc_short"](400_003))
    assert r["sort_tiles"] > 0 and r["fast_runs"] > 0 and r["fast_fail"] == 0
    r = run(BIG_SETS["arc_long"](400_003))
    assert r["sort_tiles"] > 0 and r["fast_fail"] == 1


@pytest.mark.parametrize("dx", range(4))
def test_float32_vectors_in_the_pipeline(dx):
    for n in (20_011, 90_003):
        q = inputs.circle_f64(n, 7).astype(np.float32)
        want = oracle.hull(q.astype(np.float64))
        for dy in range(4):
            bx, by = torch.zeros(n + 4, device=DEV), torch.zeros(n + 4, device=DEV)
            x, y = bx[dx:dx + n], by[dy:dy + n]
            x.copy_(torch.from_numpy(q[:, 0].copy()))
            y.copy_(torch.from_numpy(q[:, 1].copy()))
            assert np.array_equal(cch.hull_f32soa(x, y).cpu().numpy(), want), (n, dx, dy)
            assert cch.route()["sieved"] == 0


@pytest.mark.parametrize("dtype", [np.int32, np.float64])
def test_every_choice_in_the_pipeline(dtype):
    """A batch of refused sets, one above 2^21 points and small ones, under every candidate of every choice."""
    circ, disk = (circle_i32, inputs.disk_i32) if dtype == np.int32 else (inputs.circle_f64, inputs.disk_f64)
    sets = [circ(n, i + 1) for i, n in enumerate((17_003, 20_011, 33_333, 70_001, 150_001))]
    sets += [disk(2_100_001, 6), disk(900, 7), circ(40_001, 8), disk(60_001, 9)]
    want = [oracle.hull(p) for p in sets]
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])]).astype(np.int64)
    d = torch.from_numpy(np.concatenate(sets)).to(DEV)
    code = cch.CCH_I32 if dtype == np.int32 else cch.CCH_F64
    bucket = cch.lib().cch_tune_bucket(int(off[-1]), len(sets))
    base, _ = cch.tune_get(code, True, bucket)
    try:
        for cand in [dict()] + CANDIDATES:
            cch.tune_set(dict(base, **cand), code, True, bucket)
            got = cch.hull_batched(d, off)
            for s, w in enumerate(want):
                assert np.array_equal(got[s].cpu().numpy(), w), (cand, s)
            r = cch.route()
            assert r["sieved"] == 0 and r["small_regions"] + r["sort_tiles"] > 0, cand
    finally:
        cch.lib().cch_tune_clear()


def test_single_set_choices():
    """The largest region of the shared-memory sort: the choice of a set that the quantised sort would take."""
    n = 40_001
    p = inputs.circle_f64(n, 4)
    bucket = cch.lib().cch_tune_bucket(n, 1)
    base, _ = cch.tune_get(cch.CCH_F64, False, bucket)
    try:
        assert run(p)["sort_tiles"] > 0                          # above 4096 points a region
        for m, big in ((8192, True), (16_383, False), (4096, True), (1, True)):
            cch.tune_set(dict(base, small_max=m), cch.CCH_F64, False, bucket)
            assert (run(p)["sort_tiles"] > 0) == big, m
    finally:
        cch.lib().cch_tune_clear()
