"""The assembled rows of the FP64 solve on adaptive trees are as close to exact
sweeps as leaf-by-leaf sums in double precision, over the sweeps of a usual solve and
more: the spread of the potential's error against sweeps in extended precision, and
the field's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


def plain_sweeps(d, flags, b, sweeps, x):
    """Jacobi sweeps from zero in precision x, leaf by leaf."""
    b = b.astype(x)
    t = pic.tree_tables(d, flags)
    level = oracle.Tree(d, flags).leaf_info()[0]
    nc = 1 << d
    kref = [4 / 6, -1 / 6, -2 / 6] if d == 2 else [4 / 12, 0.0, -1 / 12, -1 / 12]
    k = np.array([[kref[bin(e ^ f).count("1")] for f in range(nc)] for e in range(nc)], x)
    ptr, vid, w = t["cexp_ptr"], t["cexp_vid"], t["cexp_w"].astype(x)
    width = (x(1) / x(3) ** (level if d == 3 else 0 * level))[:, None]
    corner = np.repeat(np.arange(len(ptr) - 1), np.diff(ptr))
    by_vertex = np.argsort(vid, kind="stable")
    first = np.searchsorted(vid[by_vertex], np.arange(len(b)))
    step = x(0.8) / t["diag"].astype(x)
    V = np.zeros(len(b), x)
    for _ in range(sweeps):
        at = np.add.reduceat(w * V[vid], ptr[:-1]).reshape(-1, nc)
        part = ((at @ k.T) * width).reshape(-1)
        V = V + step * (b - np.add.reduceat((w * part[corner])[by_vertex], first))
    return V


@pytest.mark.parametrize("sweeps", [100, 300])
@pytest.mark.parametrize("d,p,seed,depth,min_depth", [(2, 0.1, 2, 5, 3), (2, 0.25, 25, 5, 2), (3, 0.02, 2, 3, 2),
                                                      (3, 0.02, 3, 3, 2)])
def test_rows_are_as_accurate_as_leaf_by_leaf_sums(d, p, seed, depth, min_depth, sweeps):
    flags = W.random_tree_flags(d, depth, p, seed, min_depth=min_depth)
    n = 3001
    x, v = W.random_particles(d, n, 8, vmax=0.1)
    h = pic.Pic(d, flags, x, v, precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=sweeps)
    h.init_leapfrog(0.0)
    tree = oracle.Tree(d, flags)
    b = h.deposit() - h.stats().total_charge * pic.tree_tables(d, flags)["ion_load"]  # as the handle rounds it
    plain = plain_sweeps(d, flags, b, sweeps, np.float64)
    V = plain_sweeps(d, flags, b, sweeps, np.longdouble)
    exact = V.astype(np.float64)
    E = tree.efield64(exact)

    def off(potential, field):
        return np.std((potential - V).astype(np.float64)), np.std(field.reshape(E.shape) - E)

    here, there = off(h.potential(), h.field()), off(plain, tree.efield64(plain))
    # no further off, with room for the chance of a thousand roundings
    assert here[0] <= 1.5 * there[0] and here[1] <= 1.5 * there[1]
