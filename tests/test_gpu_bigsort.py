"""The multi-block sort by quantised keys (k_big) against the oracle: sets whose
points mostly survive round 1, with equal keys, keys that differ below the
quantisation (put right run by run) and runs too long for that (full sort)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1508_05488_gb300 as cch
from paper_1508_05488_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def with_arc(n, m, seed):
    """A circle and m points of a tiny convex arc inside its leftmost point's neighbourhood: their x agree to
    2^-30 of the width and all of them survive."""
    rng = np.random.default_rng(seed)
    t = rng.permutation(m) * (1e-7 / max(m, 1)) + 1e-9
    arc = np.stack([-1.5 + t * t * 1e3, -t], axis=1)
    return rng.permutation(np.concatenate([inputs.circle_f64(n, seed), arc]))


SETS = {
    "circle": lambda n: inputs.circle_f64(n, 3),
    "grid_circle": lambda n: np.round(inputs.circle_f64(n, 4) * 2.0 ** 17) / 2.0 ** 17,       # equal keys, duplicates
    "degenerate": lambda n: inputs.degenerate_f64(n, 5),
    "offset": lambda n: inputs.circle_f64(n, 6) * [1.0, 1e-3] + [3.0, -100.0],
    "arc_short": lambda n: with_arc(n, 40, 7),
    "arc_long": lambda n: with_arc(n, 3000, 8),
    "log_spiral": lambda n: (lambda t: np.stack([-np.exp(-t), np.exp(-t) ** 2 - 1], axis=1))(
        np.random.default_rng(9).uniform(0, 60, n)),                                          # every exponent
}


@pytest.mark.parametrize("kind", list(SETS))
def test_multi_block_sort(kind):
    for n in (70_001, 131_072, 400_003):
        p = np.ascontiguousarray(SETS[kind](n))
        t = torch.from_numpy(p).to(DEV)
        want = oracle.hull(p)
        assert np.array_equal(cch.hull(t).cpu().numpy(), want), (kind, n)
        assert np.array_equal(cch.hull(t[torch.arange(len(p) - 1, -1, -1, device=DEV)].contiguous()).cpu().numpy(),
                              oracle.hull(p[::-1].copy())), (kind, n, "reversed")
