"""pic_set_state from device arrays is done with them when it returns: a handle on
a side stream keeps the state that was handed over although the arrays are
overwritten at once on the current stream.  Ordered and unordered states, 2D and
3D, PIT and PIDT, uniform and adaptive trees."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("ordered", [False, True])
@pytest.mark.parametrize("scheme", [pic.PIT, pic.PIDT])
@pytest.mark.parametrize("precision", [pic.FP32_SPLIT, pic.FP64])
@pytest.mark.parametrize("tree", ["uniform", "adaptive"])
@pytest.mark.parametrize("d", [2, 3])
def test_arrays_are_free_on_return(d, tree, precision, scheme, ordered):
    n = 1_500_001
    flags = W.uniform_tree_flags(d, 3) if tree == "uniform" else W.random_tree_flags(d, 4, 0.3, 6, min_depth=2)
    x, v = W.random_particles(d, n, 1, vmax=0.1)
    kw = dict(scheme=scheme, precision=precision, q=-1.0 / n, sweeps=0)
    h = pic.Pic(d, flags, x, v, stream=torch.cuda.Stream(), **kw)
    ref = pic.Pic(d, flags, x, v, **kw)
    state = [a.copy() for a in ref.get_state()]
    if not ordered:
        p = np.random.default_rng(2).permutation(n)
        state = [None if a is None else np.ascontiguousarray(a[..., p]) for a in state]
    ref.set_state(*state)
    ref.sync()
    want = ref.get_state()
    for _ in range(3):
        arrays = [torch.from_numpy(a).cuda() for a in state]
        torch.cuda.synchronize()
        h.set_state(*arrays)
        for a in arrays:  # in-range values, so that whatever reads them stays inside the tree
            a.fill_(0 if a.dtype == torch.int32 else 0.25)
        torch.cuda.synchronize()
        h.sync()
        for a, b in zip(h.get_state(), want):
            assert np.array_equal(a, b)
        assert np.array_equal(h.keys(), ref.keys())
        assert np.array_equal(h.deposit(), ref.deposit())
