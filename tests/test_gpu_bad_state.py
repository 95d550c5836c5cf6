"""A split state with a leaf outside the tree or an offset outside [0, 1): the next
sync reports it, what is stored stays inside the tree (later passes index by it),
and the other particles are as they were handed over."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("what,value", [("leaf", -1), ("leaf", "n"), ("leaf", 2 ** 31 - 1), ("leaf", -2 ** 31), ("offset", 1.0),
                                        ("offset", -0.25), ("offset", -3e38), ("offset", np.inf), ("offset", np.nan)])
@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("scheme", [pic.PIT, pic.PIDT])
@pytest.mark.parametrize("d", [2, 3])
def test_stored_state_is_in_range(d, scheme, where, ordered, what, value):
    n = 1003
    flags = W.random_tree_flags(d, 4, 0.3, 6, min_depth=2)
    x, v = W.random_particles(d, n, 1, vmax=0.1)
    h = pic.Pic(d, flags, x, v, scheme=scheme, precision=pic.FP32_SPLIT, q=-1.0 / n, sweeps=0)
    leaf, o, vel = (a.copy() for a in h.get_state())
    if not ordered:
        p = np.random.default_rng(2).permutation(n)
        leaf, o, vel = leaf[p], np.ascontiguousarray(o[:, p]), np.ascontiguousarray(vel[:, p])
    bad = [0, 31, 32, n - 1]
    vel[0] = np.arange(n)  # names the particles
    n_leaves = h.info().n_leaves
    if what == "leaf":
        leaf[bad] = n_leaves if value == "n" else value
    else:
        o[d - 1, bad] = value
    args = (leaf, o, vel)
    if where == "device":
        args = tuple(torch.from_numpy(a).cuda() for a in args)
    h.set_state(*args)
    with pytest.raises(pic.PicError):
        h.sync()
    l2, o2, v2 = h.get_state()
    assert np.all((l2 >= 0) & (l2 < n_leaves)) and np.all((o2 >= 0) & (o2 < 1))
    was = v2[0].astype(np.int64)
    assert np.array_equal(np.sort(was), np.arange(n))
    good = ~np.isin(was, bad)
    assert np.array_equal(l2[good], leaf[was[good]]) and np.array_equal(o2[:, good], o[:, was[good]])
    assert np.array_equal(v2, vel[:, was])
    if where == "device":
        for a, b in zip(args, (leaf, o, vel)):  # the caller's arrays stay as they were
            assert np.array_equal(a.cpu().numpy(), b, equal_nan=b.dtype != np.int32)
