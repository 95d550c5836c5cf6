"""pic_set_state with split states: unordered and ordered, from host arrays and
from device arrays (read where they are, also off 16-byte boundaries), against
the stable order by key; the caller's arrays stay as they were."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


def shifted(a):
    """The array on the device, one element past an allocation's start."""
    t = torch.empty(a.size + 1, dtype=torch.from_numpy(a).dtype, device="cuda")[1:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("ordered", [False, True])
@pytest.mark.parametrize("scheme", [pic.PIT, pic.PIDT])
@pytest.mark.parametrize("d,tree,n", [(2, "uniform", 1), (2, "uniform", 257), (2, "adaptive", 10_001),
                                      (3, "uniform", 4099), (3, "adaptive", 30_001)])
def test_state_is_ordered_by_key(d, tree, n, scheme, ordered):
    flags = W.uniform_tree_flags(d, 2) if tree == "uniform" else W.random_tree_flags(d, 4, 0.3, 6, min_depth=1)
    x, v = W.random_particles(d, n, 1, vmax=0.1)
    g = pic.Pic(d, flags, x, v, scheme=scheme, precision=pic.FP32_SPLIT, q=-1.0 / n, sweeps=0)
    leaf, o, vel = (a.copy() for a in g.get_state())
    keys = g.keys()
    if not ordered:
        p = np.random.default_rng(2).permutation(n)
        leaf, o, vel, keys = leaf[p], np.ascontiguousarray(o[:, p]), np.ascontiguousarray(vel[:, p]), keys[p]
    order = np.argsort(keys, kind="stable")
    rho = None
    for where in ("host", "device"):
        args = (leaf, o, vel) if where == "host" else tuple(shifted(a) for a in (leaf, o, vel))
        g.set_state(*args)
        g.sync()
        l2, o2, v2 = g.get_state()
        assert np.array_equal(l2, leaf[order]) and np.array_equal(o2, o[:, order]) and np.array_equal(v2, vel[:, order])
        assert np.array_equal(g.keys(), keys[order])
        q = g.deposit()
        assert rho is None or np.array_equal(q, rho)
        rho = q
        if where == "device":
            for a, b in zip(args, (leaf, o, vel)):
                assert np.array_equal(a.cpu().numpy(), b)


def test_bad_leaf_or_offset_is_reported():
    x, v = W.random_particles(3, 1000, 1, vmax=0.1)
    for bad in ("leaf", "offset"):
        g = pic.Pic(3, W.uniform_tree_flags(3, 2), x, v, precision=pic.FP32_SPLIT, q=-1e-3, sweeps=0)
        leaf, o, vel = (torch.from_numpy(a.copy()).cuda() for a in g.get_state())
        if bad == "leaf":
            leaf[7] = 27 ** 2
        else:
            o[1, 7] = 1.5
        g.set_state(leaf, o, vel)
        with pytest.raises(pic.PicError):
            g.sync()
