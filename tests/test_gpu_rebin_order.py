"""The canonical bucket order (stayers, then movers, both in storage order) for
mover segments around every line of the re-bin: one mover, segments ordered by
counting, sorted by a warp, sorted by a block; few and many keys (scans in one
block and in three launches); rows (2D) and records (3D)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("d,depth,n,m", [(2, 2, 3000, 0), (2, 2, 3000, 1), (2, 2, 3000, 63), (2, 2, 3000, 64),
                                         (2, 2, 3000, 65), (2, 2, 3000, 127), (2, 2, 3000, 128),
                                         (2, 2, 3000, 129), (2, 3, 9000, 1023), (2, 3, 9000, 1024), (2, 3, 9000, 1025),
                                         (3, 2, 5000, 129), (2, 3, 9000, 2047), (2, 3, 9000, 2048), (2, 3, 9000, 2049),
                                         (2, 5, 70_001, 40_000), (3, 1, 1000, 64), (3, 2, 5000, 65),
                                         (3, 4, 60_001, 3000), (2, 2, 31, 31), (2, 2, 64, 40), (2, 6, 900_000, 300)])
@pytest.mark.parametrize("scheme,precision", [(pic.PIT, pic.FP32_SPLIT), (pic.PIDT, pic.FP32_SPLIT), (pic.PIT, pic.FP64),
                                              (pic.PIDT, pic.FP64)])
def test_order_around_segment_lines(d, depth, n, m, scheme, precision):
    rng = np.random.default_rng(17 + m)
    x = rng.random((d, n))
    v = np.zeros((d, n))
    go = rng.choice(n, m, replace=False)
    # into the first quarter of one cell (one leaf and one quadrant), a third of the others one cell along x
    v[:, go] = (rng.random((d, m)) * 0.25 + 1.0) / 3 ** depth - x[:, go]
    rest = np.setdiff1d(rng.choice(n, n // 3, replace=False), go)
    v[0, rest] = 1.0 / 3 ** depth
    g = pic.Pic(d, W.uniform_tree_flags(d, depth), x, v, scheme=scheme, precision=precision, q=0.0, sweeps=0,
                path=pic.PATH_GENERIC)
    (_, ids0), keys0 = g.bins(), g.keys()
    by_input = np.empty(n, np.int64)
    by_input[ids0] = np.arange(n)
    fresh_keys = keys0[by_input]          # at creation every particle is a mover: stable by key in input order
    assert np.array_equal(ids0, np.argsort(fresh_keys, kind="stable"))
    g.step_particles(1.0, reflect=False)
    g.sync()
    (start, ids1), keys1 = g.bins(), g.keys()
    new = np.empty(n, np.int64)
    new[ids1] = keys1
    moved = new[ids0] != keys0
    want = ids0[np.argsort(2 * new[ids0] + moved, kind="stable")]
    assert np.array_equal(ids1, want)
    counts = np.bincount(keys1 >> (d if scheme == pic.PIDT else 0), minlength=len(start) - 1)
    assert np.array_equal(np.diff(start), counts)
    assert g.stats().movers == int(moved.sum())
    assert g.stats().max_bucket == int(np.bincount(keys1).max())
