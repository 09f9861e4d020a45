"""The tuner on batches that its choices act on, and on batches that never
reach the pipeline: there it searches nothing and changes nothing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tune(sets):
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])]).astype(np.int64)
    d = torch.from_numpy(np.concatenate(sets)).to(DEV)
    idx = torch.zeros(int(off[-1]), dtype=torch.int32, device=DEV)
    cnt = torch.zeros(len(sets), dtype=torch.int32, device=DEV)
    bucket = cch.lib().cch_tune_bucket(int(off[-1]), len(sets))
    before, _ = cch.tune_get(cch.CCH_F64, len(sets) > 1, bucket)
    for _ in range(2):
        cch.hull_batched_async(d, off, idx, cnt)
    l0 = cch.launch_count()
    cch.hull_batched_async(d, off, idx, cnt)
    per_call = cch.launch_count() - l0
    l0 = cch.launch_count()
    best = cch.autotune_batched(d, off, idx, cnt, reps=2)
    calls = (cch.launch_count() - l0) / per_call
    now, found = cch.tune_get(cch.CCH_F64, len(sets) > 1, bucket)
    assert found and now == best
    cnt = cnt.cpu().numpy()
    for s, p in enumerate(sets):
        assert np.array_equal(idx[int(off[s]):int(off[s]) + int(cnt[s])].cpu().numpy(), oracle.hull(p)), s
    return before, best, calls


@pytest.fixture(autouse=True)
def table():
    cch.lib().cch_tune_clear()
    yield
    cch.lib().cch_tune_clear()


@pytest.mark.parametrize("sets", [
    [inputs.disk_f64(n, n) for n in (300, 5000, 16_000, 900)],                 # small ones
    [inputs.square_f64(n, n) for n in (20_011, 60_001, 800, 250_000)],         # sieved ones
    [inputs.circle_f64(9000, 1)],
    [inputs.disk_f64(300_007, 1)],
])
def test_nothing_to_choose(sets):
    before, best, calls = tune(sets)
    assert best == before and calls <= 1


def test_sets_of_the_pipeline():
    _, _, calls = tune([inputs.circle_f64(n, n) for n in (20_011, 50_003, 40_001)])
    assert calls > 20
