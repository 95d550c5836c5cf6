"""A 2D and a 3D handle alive together: each solves with its own element matrix,
whichever was created last, in the sweeps, the two passes and the rows that a
re-tree assembles again."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


def adaptive_flags(d, second):
    """Trees whose rows the FP64 solve assembles (21 to 41 entries)."""
    if d == 2:
        return W.random_tree_flags(2, 5, *((0.25, 25) if second else (0.1, 2)), min_depth=2 if second else 3)
    return W.random_tree_flags(3, 3, 0.02, 3 if second else 2, min_depth=2)


def make(d, tree, precision, sweeps):
    flags = W.uniform_tree_flags(d, 3) if tree == "uniform" else adaptive_flags(d, False)
    n = 5003
    x, v = W.random_particles(d, n, 3, vmax=0.1)
    h = pic.Pic(d, flags, x, v, precision=precision, q=-1.0 / n, ion=0.3, sweeps=sweeps, omega=0.8)
    assert h.info().uniform == (tree == "uniform")
    return h


def advance(h, tree):
    """Two steps, with a re-tree between them on adaptive trees; what they leave behind."""
    h.step(0.05)
    if tree == "adaptive":
        h.retree(adaptive_flags(h.d, True))
    h.step(0.05)
    h.sync()
    return [*h.get_state(), h.potential(), h.field(), np.array(h.stats().residual)]


@pytest.mark.parametrize("sweeps", [7, 20])
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("tree", ["uniform", "adaptive"])
@pytest.mark.parametrize("first", [2, 3])
def test_dimensions_do_not_mix(first, tree, precision, sweeps):
    alone = make(first, tree, precision, sweeps)
    want = advance(alone, tree)
    alone.close()
    h = make(first, tree, precision, sweeps)
    other = make(5 - first, tree, precision, sweeps)
    other.step(0.05)
    got = advance(h, tree)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    other.close()
