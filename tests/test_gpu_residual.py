"""The reported residual is the norm of b - A V for any damping factor, zero and
subnormal ones included: every form of the built-in solve (one cluster, a thread
per vertex, strips, tiles, a batch; assembled rows and the two passes)."""
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

OMEGAS = [0.0, 1e-310, 1e-6, 0.01, 0.8, 1.0]


def row_bounds(d, flags, tree):
    """Per vertex at most: terms of (A V), and the sum of their magnitudes where |V| <= 1."""
    nc, level = 1 << d, tree.leaf_info()[0]
    kref = 8 / 6 if d == 2 else 8 / 12  # a row of the reference element's matrix
    t = pic.tree_tables(d, flags)
    if t["uniform"]:
        return nc * nc, kref * nc * 3.0 ** (-(d - 2) * int(level[0]))
    ptr, vid, w = t["cexp_ptr"], t["cexp_vid"], t["cexp_w"]
    corner = np.repeat(np.arange(len(ptr) - 1), np.diff(ptr))
    width = 3.0 ** (-(d - 2.0) * level[corner // nc])
    expansions = np.add.reduceat(np.diff(ptr), np.arange(0, len(ptr) - 1, nc))  # of a leaf's corners
    terms = np.bincount(vid, weights=expansions[corner // nc])
    return terms, kref * np.bincount(vid, weights=w * width)


def check(h, flags, omega, precision):
    """Residual of the handle's charges and potential against the oracle's residual of the same."""
    h.init_leapfrog(0.0)
    Q, V, vs = h.deposit(), h.potential(), h.instances()[1]
    eps = 2.0 ** -53 if precision == pic.FP64 else 2.0 ** -24
    want, bound = 0.0, 0.0
    for i, f in enumerate(flags):
        tree = oracle.Tree(h.d, f)
        q, v = Q[vs[i]:vs[i + 1]].copy(), V[vs[i]:vs[i + 1]].copy()
        if precision == pic.FP64:
            res = tree.solve64(q, v, 0, omega)
        else:
            res = tree.solve32(q.astype(np.float32), v.astype(np.float32), 0, np.float32(omega))
        want += res * res
        terms, size = row_bounds(h.d, f, tree)
        # both sides round every term, product and weight included; |b| <= |Q| + |sum Q| times the ion load (at most 1)
        err = 2 * eps * (4 * terms + 16) * (np.abs(q) + abs(q.sum()) + size * np.abs(v).max())
        bound += np.sum(err * err)
    got = h.stats().residual
    assert abs(got - np.sqrt(want)) <= np.sqrt(bound) + 1e-12 * got
    assert got > 0 or len(Q) == 1


@pytest.mark.parametrize("omega", OMEGAS)
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d,depth", [(2, 0), (2, 3), (2, 4), (2, 6), (3, 1), (3, 2), (3, 3), (3, 4)])
def test_uniform(d, depth, precision, omega):
    flags = W.uniform_tree_flags(d, depth)
    n = 3001
    x, v = W.random_particles(d, n, 5, vmax=0.1)
    h = pic.Pic(d, flags, x, v, precision=precision, q=-1.0 / n, ion=0.3, sweeps=9, omega=omega)
    check(h, [flags], omega, precision)


@pytest.mark.parametrize("omega", OMEGAS)
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d", [2, 3])
def test_batch(d, precision, omega):
    flags = [W.uniform_tree_flags(d, k) for k in (1, 3, 2)]
    parts = [W.random_particles(d, n, n, vmax=0.1) for n in (301, 2003, 907)]
    h = pic.Pic.batch(d, flags, [p[0] for p in parts], [p[1] for p in parts], precision=precision, q=-1e-3, ion=0.3,
                      sweeps=9, omega=omega)
    check(h, flags, omega, precision)


@pytest.mark.parametrize("omega", OMEGAS)
@pytest.mark.parametrize("sweeps", [9, 20])
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d,depth,p,seed,min_depth", [(2, 5, 0.1, 2, 3), (2, 6, 0.3, 2, 2),  # rows of 21, 139 entries
                                                      (3, 3, 0.02, 2, 2), (3, 3, 0.3, 6, 1)])  # 41, 275
def test_adaptive(d, depth, p, seed, min_depth, precision, sweeps, omega):
    flags = W.random_tree_flags(d, depth, p, seed, min_depth=min_depth)
    n = 3001
    x, v = W.random_particles(d, n, 5, vmax=0.1)
    h = pic.Pic(d, flags, x, v, precision=precision, q=-1.0 / n, ion=0.3, sweeps=sweeps, omega=omega)
    assert not h.info().uniform
    check(h, [flags], omega, precision)
