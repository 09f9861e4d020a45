"""Captured calls replayed on other points: sets that the sieve refuses go
through the multi-block sort, the SPA scan and the output compaction, whose
look-back words a run must not take from the run before it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N = 150_001


def grid_circle(n, seed):
    return np.round(inputs.circle_f64(n, seed) * 2.0 ** 17) / 2.0 ** 17


def circle_i32(n, seed):
    return np.floor(inputs.circle_f64(n, seed) * 2.0 ** 28).astype(np.int32)


SETS = [(inputs.circle_f64, 1), (inputs.circle_f64, 2), (grid_circle, 3), (inputs.disk_f64, 4), (inputs.circle_f64, 5),
        (inputs.degenerate_f64, 6), (inputs.shell_f64, 7), (inputs.circle_f64, 8)]


class Captured:
    """A call on points of a shape, captured on a stream of its own after one plain call."""

    def __init__(self, form, n):
        self.form, self.n, self.stream = form, n, torch.cuda.Stream()
        self.idx = torch.zeros(n, dtype=torch.int32, device=DEV)
        self.cnt = torch.zeros(1, dtype=torch.int32, device=DEV)
        if form == "f32":
            self.buf = [torch.zeros(n, dtype=torch.float32, device=DEV) for _ in range(2)]
        else:
            self.buf = torch.zeros((n, 2), dtype=torch.int32 if form == "i32" else torch.float64, device=DEV)
        self.fill(self.points(*SETS[0]))
        with torch.cuda.stream(self.stream):
            self.call()
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph, stream=self.stream):
            self.call()

    def points(self, gen, seed):
        if self.form == "i32":
            return circle_i32(self.n, seed) if seed % 2 else inputs.disk_i32(self.n, seed)
        p = gen(self.n, seed)
        return p.astype(np.float32) if self.form == "f32" else p

    def fill(self, p):
        p = np.ascontiguousarray(p)
        if self.form == "f32":
            for k in (0, 1):
                self.buf[k].copy_(torch.from_numpy(p[:, k].copy()))
        else:
            self.buf.copy_(torch.from_numpy(p))
        torch.cuda.synchronize()

    def call(self):
        if self.form == "f32":
            cch.hull_f32soa_async(*self.buf, self.idx, self.cnt)
        elif self.form == "noalloc":
            assert cch.lib().cch_hull_noalloc(self.buf.data_ptr(), self.n, cch.CCH_F64, self.idx.data_ptr(),
                                              self.cnt.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
        else:
            cch.hull_async(self.buf, self.idx, self.cnt)

    def check(self, p):
        torch.cuda.synchronize()
        want = oracle.hull(p.astype(np.float64) if self.form == "f32" else p)
        assert np.array_equal(self.idx[:max(int(self.cnt.item()), 0)].cpu().numpy(), want), self.form
        self.cnt.zero_()
        torch.cuda.synchronize()

    def replay(self, p):
        self.fill(p)
        self.graph.replay()
        self.check(p)


@pytest.mark.parametrize("form", ["f64", "f32", "i32", "noalloc"])
def test_replays_of_refused_and_sieved_sets(form):
    c = Captured(form, 100_003 if form == "noalloc" else N)
    for gen, seed in SETS:
        c.replay(c.points(gen, seed))


def test_replays_between_plain_calls_across_the_epoch_wrap():
    """Plain calls of the same stream meet no word of a replay, whatever their epoch."""
    c = Captured("f64", N)
    p, q = inputs.circle_f64(N, 11), grid_circle(N, 12)
    small = torch.from_numpy(inputs.circle_f64(20_000, 13)).to(DEV)     # bumps the epoch cheaply
    idx, cnt = torch.zeros(20_000, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    for _ in range(3):
        c.replay(p)
        c.fill(q)
        with torch.cuda.stream(c.stream):
            c.call()
            c.check(q)
            for _ in range(1400):
                cch.hull_async(small, idx, cnt)
    with torch.cuda.stream(c.stream):
        c.fill(p)
        c.call()
        c.check(p)


def test_replay_after_the_workspace_has_grown():
    c = Captured("f64", 60_001)
    big = inputs.circle_f64(400_003, 21)
    for seed in (22, 23):
        with torch.cuda.stream(c.stream):
            got = cch.hull(torch.from_numpy(big).to(DEV))
        assert np.array_equal(got.cpu().numpy(), oracle.hull(big))
        c.replay(inputs.circle_f64(60_001, seed))


def batch_sets(sizes, seed):
    gens = [inputs.disk_f64, inputs.circle_f64, inputs.square_f64]
    return [gens[k % 3](n, seed + k) for k, n in enumerate(sizes)]


def test_captured_batch_between_plain_batches():
    """A batch's graph keeps its own tables; a plain batch of other sizes on the stream is not in its way, nor
    is an earlier capture that the mode refused."""
    sizes, other = [500, 30_001, 1500, 9000, 20_011, 70_003, 40_000], [700, 25_000, 16_000, 3000]
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])
    s = torch.cuda.Stream()
    pts = torch.zeros((n, 2), dtype=torch.float64, device=DEV)
    idx = torch.zeros(n, dtype=torch.int32, device=DEV)
    cnt = torch.zeros(len(sizes), dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()

    def check(sets):
        torch.cuda.synchronize()
        for k, p in enumerate(sets):
            a = int(off[k])
            assert np.array_equal(idx[a:a + int(cnt[k])].cpu().numpy(), oracle.hull(p)), k

    def plain():
        sets = batch_sets(other, 50)
        with torch.cuda.stream(s):
            got = cch.hull_batched(torch.from_numpy(np.concatenate(sets)).to(DEV), np.concatenate([[0], np.cumsum(other)]))
        for h, p in zip(got, sets):
            assert np.array_equal(h.cpu().numpy(), oracle.hull(p))

    with torch.cuda.stream(s):
        cch.hull_batched_async(pts, off, idx, cnt)
    s.synchronize()
    with pytest.raises(Exception):
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s, capture_error_mode="global"):
            cch.hull_batched_async(pts, off, idx, cnt)
    plain()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        cch.hull_batched_async(pts, off, idx, cnt)
    for seed in (1, 20, 40):
        plain()
        sets = batch_sets(sizes, seed)
        pts.copy_(torch.from_numpy(np.concatenate(sets)))
        torch.cuda.synchronize()
        g.replay()
        check(sets)
