"""Brick handles whose bricks hold more particles than the shared-memory
kernels take run the generic passes: same bits as a generic handle, and still
the brick path's contract (charges are up to date after a step, so captured
steps go on after a deposit is read)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


# 9 bricks in 2D, 27 in 3D: one particle per half brick below and above 3,200 on average
@pytest.mark.parametrize("d,n", [(2, 18 * 3200), (2, 18 * 3200 + 1), (3, 54 * 3200), (3, 54 * 3200 + 1), (2, 100_001)])
def test_steps_replays_and_deposits(d, n):
    flags = W.uniform_tree_flags(d, 3)
    x, v = W.random_particles(d, n, 3, vmax=0.3)
    kw = dict(q=-1.0 / n, ion=1.0, sweeps=5, scheme=pic.PIT, precision=pic.FP32_SPLIT)
    a = pic.Pic(d, flags, x, v, stream=torch.cuda.Stream(), **kw)
    b = pic.Pic(d, flags, x, v, path=pic.PATH_GENERIC, **kw)
    assert a.info().brick == 1 and b.info().brick == 0
    a.graph_capture_step(0.05)
    b.step(0.05)
    for _ in range(3):
        a.graph_launch(1)
        b.step(0.05)
        a.sync()
        b.sync()
        for p, q in zip(a.get_state(), b.get_state()):
            assert np.array_equal(p, q)
        assert np.array_equal(a.deposit(), b.deposit())
        assert np.array_equal(a.bins()[1], b.bins()[1])
        assert a.stats().movers == b.stats().movers and a.stats().max_bucket == b.stats().max_bucket


# one brick among 9 (27) sparse ones: parts of up to 3,200 particles, their last one full or short, and units whose
# arrivals overflow
@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("dense", [6400, 6401, 9599, 9600, 9601, 12801, 50_003])
def test_uneven_bricks(d, dense):
    rng = np.random.default_rng(dense)
    flags = W.uniform_tree_flags(d, 3)
    x, v = W.random_particles(d, dense + 1001, 4, vmax=0.3)
    x[:, :dense] = (1 + rng.random((d, dense))) / 3
    order = rng.permutation(x.shape[1])
    x, v = x[:, order], v[:, order]
    kw = dict(q=-1.0 / x.shape[1], ion=1.0, sweeps=5, scheme=pic.PIT, precision=pic.FP32_SPLIT)
    a = pic.Pic(d, flags, x, v, track_ids=True, **kw)
    assert a.info().brick == 1
    b = pic.Pic(d, flags, x, v, path=pic.PATH_GENERIC, track_ids=True, **kw)
    for _ in range(4):
        a.step(0.05)
        b.step(0.05)
        for p, q in zip(a.get_state(), b.get_state()):
            assert np.array_equal(p, q)
        assert np.array_equal(a.bins()[1], b.bins()[1])
        assert np.array_equal(a.deposit(), b.deposit())
        assert a.stats().movers == b.stats().movers and a.stats().max_bucket == b.stats().max_bucket
