"""Calls of several host threads, each on its own stream, while the workspaces
are released under them: every call has a workspace of its stream and the
right result."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_threads_and_release():
    sets = [inputs.disk_f64(60_001, 1), inputs.circle_f64(30_011, 2), inputs.square_f64(200_003, 3), inputs.disk_i32(40_001, 4)]
    pts = [torch.from_numpy(np.ascontiguousarray(p)).to(DEV) for p in sets]
    want = [oracle.hull(p) for p in sets]
    off = np.array([0, 900, 25_000, 60_001], dtype=np.int64)
    want_b = [oracle.hull(sets[0][off[k]:off[k + 1]]) for k in range(3)]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for k in range(40):
                    j = (i + k) % len(sets)
                    if not np.array_equal(cch.hull(pts[j]).cpu().numpy(), want[j]):
                        errors.append((i, k, j))
                    if k % 5 == 0:
                        for h, w in zip(cch.hull_batched(pts[0], off), want_b):
                            if not np.array_equal(h.cpu().numpy(), w):
                                errors.append((i, k, "batch"))
        except Exception as e:            # noqa: BLE001 -- reported by the main thread
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for _ in range(10):
        cch.release_workspace()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
