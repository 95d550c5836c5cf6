"""The FP32 sweep of 243^3 cells marches in blocks over groups of planes; its sums
are in leaf order bit for bit, on planes either side of every kind of group
boundary and in the wrapped first and last ones."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)

DEPTH, M = 5, 243
F = np.float32


def spread(c):
    """Base-27 number of the base-3 digits of c: the share of x in the depth-first leaf index (y: 3 times, z: 9 times)."""
    out, mul = np.zeros_like(c), 1
    for _ in range(DEPTH):
        out, c, mul = out + c % 3 * mul, c // 3, mul * 27
    return out


def apply_plane(V, z):
    """(A V) of plane z of V[z][y][x], FP32: per leaf the corners in ascending order, the leaves by ascending index."""
    h = F(1.0 / M)
    k = [F(4 / 12) * h, F(0.0) * h, F(-1 / 12) * h, F(-1 / 12) * h]
    s = spread(np.arange(M))
    leaf, part = [], []
    for f in range(8):  # the leaf that has the vertex as its corner f
        o = [f & 1, f >> 1 & 1, f >> 2]
        j = np.arange(M)
        leaf.append(9 * s[(z - o[2]) % M] + 3 * s[(j - o[1]) % M][:, None] + s[(j - o[0]) % M][None, :])
        acc = None
        for g in range(8):
            p = np.roll(V[(z - o[2] + (g >> 2)) % M], (o[1] - (g >> 1 & 1), o[0] - (g & 1)), (0, 1))
            term = k[bin(f ^ g).count("1")] * p
            acc = term if acc is None else acc + term
        part.append(acc)
    order = np.argsort(np.array(leaf), axis=0)
    part = np.take_along_axis(np.array(part), order, axis=0)
    y = np.zeros((M, M), F)
    for i in range(8):
        y = y + part[i]
    return y


def test_sums_in_leaf_order_across_plane_groups():
    x, v = W.random_particles(3, 200_001, 17, vmax=0.2)
    g = pic.Pic(3, W.uniform_tree_flags(3, DEPTH), x, v, precision=pic.FP32_SPLIT, q=-1.0 / x.shape[1], ion=0.3, sweeps=1,
                omega=0.8)
    g.init_leapfrog(0.0)  # V = omega b / diag
    V0 = g.potential().astype(F).reshape(M, M, M)
    g.init_leapfrog(0.0)  # one sweep from there: the positions, so b, are the same
    V1 = g.potential().astype(F).reshape(M, M, M)
    h = 1.0 / M
    ion = F(h * h * h)
    b = g.deposit().astype(F).reshape(M, M, M) - F(g.stats().total_charge) * ion
    diag = F(8 * (4 / 12) * h)
    assert np.any(V0)
    planes = sorted({p % M for q in range(0, M, 27) for p in (q - 1, q, q + 1)} | set(range(12)) | {17, 18, 19, M - 2})
    for z in planes:
        want = V0[z] + F(0.8) * (b[z] - apply_plane(V0, z)) / diag
        assert np.array_equal(V1[z], want), z
