"""A batch that fails for want of device memory launches nothing: the small
sets of a mixed batch need no workspace, its larger ones do."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_mixed_batch_without_memory_for_its_workspace():
    small = inputs.square_i32(1000, 1)
    n = 150_000_000
    need = cch.lib().cch_workspace_bytes(n, cch.CCH_I32)
    pts = torch.zeros((1000 + n, 2), dtype=torch.int32, device=DEV)
    pts[:1000] = torch.from_numpy(small).to(DEV)
    idx = torch.full((1000 + n,), -7, dtype=torch.int32, device=DEV)
    cnt = torch.full((2,), -7, dtype=torch.int32, device=DEV)
    s = torch.cuda.Stream()                          # a stream without a workspace
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(max(free - need // 2, 0), dtype=torch.uint8, device=DEV)
    assert torch.cuda.mem_get_info()[0] < need
    off = np.array([0, 1000, 1000 + n], dtype=np.int64)
    rc = cch.lib().cch_hull_batched(pts.data_ptr(), off.ctypes.data, 2, cch.CCH_I32, idx.data_ptr(), cnt.data_ptr(),
                                    ctypes.c_void_p(s.cuda_stream))
    torch.cuda.synchronize()
    del hold
    torch.cuda.empty_cache()
    assert rc == -5
    assert cnt.tolist() == [-7, -7] and int(idx[0]) == -7
    # the small set alone needs no workspace, and the stream is as it was
    got = cch.hull_batched(pts[:1000], off[:2], stream=s)
    s.synchronize()
    assert np.array_equal(got[0].cpu().numpy(), oracle.hull(small))
