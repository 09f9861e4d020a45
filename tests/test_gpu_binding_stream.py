"""The synchronous forms with a stream that is not the current one read its
result, not what the output buffers held before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_results_of_another_stream():
    p = inputs.disk_f64(5000, 1)
    t = torch.from_numpy(p).to(DEV)
    q = p.astype(np.float32)
    x, y = (torch.from_numpy(np.ascontiguousarray(q[:, k])).to(DEV) for k in (0, 1))
    want, want32 = oracle.hull(p), oracle.hull(q.astype(np.float64))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)                 # some 10 ms of work in front of the call
        assert np.array_equal(cch.hull(t, stream=s).cpu().numpy(), want)
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)
        assert np.array_equal(cch.hull_f32soa(x, y, stream=s).cpu().numpy(), want32)
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)
        got = cch.hull_batched(t, [0, 5000], stream=s)
        assert np.array_equal(got[0].cpu().numpy(), want)
