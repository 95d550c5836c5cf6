"""Potentials that are not finite (as a run that diverged leaves them) spread over the
same vertices as in the oracle, whatever form of the solve runs: the sweeps leave
out terms whose matrix entry is zero, and those must still pass on what is not
finite.  FP32 values that stay finite keep their bits.  The potential comes in by
a checkpoint."""
from __future__ import annotations

import struct

import numpy as np
import pytest

import oracle
from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

from .test_checkpoint_file import fold

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


def with_potential(path, V, d):
    """The checkpoint's potential section (before the field's, which is last) replaced by V."""
    data = bytearray(path.read_bytes())
    size, field = V.nbytes, d * V.nbytes
    end = len(data) - (field + -field % 8)
    start = end - (size + -size % 8)
    data[start:start + size] = V.tobytes()
    data[16:24] = struct.pack("<Q", fold(0x243F6A8885A308D3, bytes(data[24:])))
    path.write_bytes(data)


@pytest.mark.parametrize("sweeps", [1, 2, 17])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d,tree", [(2, 3), (2, 4), (2, 6), (3, 1), (3, 2), (3, 3), (3, 4), (2, "adaptive"), (3, "adaptive")])
def test_spreads_as_in_the_oracle(d, tree, precision, value, sweeps, tmp_path):
    if tree != "adaptive":
        flags = W.uniform_tree_flags(d, tree)
    else:  # rows of 36 and 41 entries: assembled from 16 sweeps on
        flags = W.random_tree_flags(2, 6, 0.2, 2, min_depth=4) if d == 2 else W.random_tree_flags(3, 3, 0.02, 2, min_depth=2)
    if sweeps > 2 and tree in (4, 6) and d + tree > 6:
        pytest.skip("the oracle's sweeps of large grids take long; the launches are those of few sweeps")
    n = 301
    x, v = W.random_particles(d, n, 5, vmax=0.1)
    kw = dict(q=-1.0 / n, ion=0.3, sweeps=sweeps, omega=0.8)
    g = pic.Pic(d, flags, x, v, precision=precision, **kw)
    ft = np.float64 if precision == pic.FP64 else np.float32
    nv = g.info().n_vertices
    V = np.random.default_rng(1).standard_normal(nv).astype(ft)
    V[[0, nv // 2, nv - 1]] = value
    g.save(tmp_path / "v.pic")
    with_potential(tmp_path / "v.pic", V, d)
    g = pic.Pic.load(tmp_path / "v.pic")
    assert np.array_equal(g.potential(), V.astype(np.float64), equal_nan=True)
    Q = g.deposit().astype(ft)
    g.init_leapfrog(0.0)
    got, E = g.potential(), g.field()
    t = oracle.Tree(d, flags)
    with np.errstate(invalid="ignore"):
        if precision == pic.FP64:
            t.solve64(Q, V, sweeps, 0.8)
            Eo = t.efield64(V)
        else:
            t.solve32(Q, V, sweeps, np.float32(0.8))
            Eo = t.efield32(V)
    assert np.array_equal(np.isfinite(got), np.isfinite(V))
    assert np.array_equal(np.isfinite(E), np.isfinite(Eo.reshape(E.shape)))
    ok = np.isfinite(V)
    if precision == pic.FP32_SPLIT:
        assert np.array_equal(got[ok], V[ok].astype(np.float64))
    else:
        # sums of up to a few dozen roundings a sweep, on values of scale one
        assert np.max(np.abs(got[ok] - V[ok]), initial=0.0) <= 1e-12
    assert not np.isfinite(g.stats().residual) or ok.all()
