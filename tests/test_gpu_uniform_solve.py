"""The built-in solve and the vertex field on uniform trees against the oracle:
FP32 bit for bit (same order of every sum), FP64 within rounding, on grids of
one cell, of fewer cells than a block has columns and of several blocks, for
even and odd numbers of sweeps, single plasmas and a batch."""
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

# a few hundred roundings of 1.1e-16 per sum and sweep, on fields of scale one
TOL64 = 1e-12


def states(d, depth, n, seed, precision, sweeps, scheme):
    flags = W.uniform_tree_flags(d, depth)
    x, v = W.random_particles(d, n, seed, vmax=0.2)
    # ion 0.3: the charge total is far from zero, so its FP32 value does not hang on the order of the FP64 sum
    kw = dict(q=-1.0 / n, qm=-1.0, ion=0.3, sweeps=sweeps, omega=0.8)
    g = pic.Pic(d, flags, x, v, scheme=scheme, precision=precision, **kw)
    S = oracle.State64 if precision == pic.FP64 else oracle.State32
    return g, S(oracle.Tree(d, flags), x, v, oracle.Params(scheme=scheme, **kw))


def close(a, b):
    return np.max(np.abs(a - b)) <= TOL64 * max(1e-300, np.max(np.abs(b)))


@pytest.mark.parametrize("sweeps", [1, 8])
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d,depth", [(2, 0), (2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (3, 0), (3, 1), (3, 2), (3, 3),
                                     (3, 4)])
def test_solve_and_field_match_oracle(d, depth, precision, sweeps):
    scheme = pic.PIDT if depth % 2 else pic.PIT
    g, st = states(d, depth, 3001 + 7 * depth, 5 + depth, precision, sweeps, scheme)
    for _ in range(2):
        _, _, res, E = st.step(0.05)
        g.step(0.05)
        g.sync()
        V, Eg = g.potential(), g.field()
        if precision == pic.FP32_SPLIT:
            assert np.array_equal(V, st.V.astype(np.float64))
            assert np.array_equal(Eg, np.asarray(E, np.float64).reshape(Eg.shape))
        else:
            assert close(V, st.V)
            # a difference of potentials over h: the potential's rounding divided by h
            assert np.max(np.abs(Eg - E.reshape(Eg.shape))) <= TOL64 * max(1e-300, np.max(np.abs(st.V))) * 3 ** depth
        assert abs(g.stats().residual - res) <= 1e-6 * res + 1e-12


@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d", [2, 3])
def test_batch_solve_matches_single_plasmas(d, precision):
    depths, ns = [0, 2, 1, 3], [50, 2000, 301, 4007]
    parts = [W.random_particles(d, n, 40 + n, vmax=0.2) for n in ns]
    flags = [W.uniform_tree_flags(d, k) for k in depths]
    kw = dict(qm=-1.0, ion=0.3, sweeps=7, omega=0.8, precision=precision)
    qs = [-1.0 / n for n in ns]
    b = pic.Pic.batch(d, flags, [p[0] for p in parts], [p[1] for p in parts], qs, **kw)
    b.step(0.05)
    b.sync()
    V, E, vs = b.potential(), b.field(), b.instances()[1]
    for i, n in enumerate(ns):
        one = pic.Pic(d, flags[i], *parts[i], q=qs[i], **kw)
        one.step(0.05)
        one.sync()
        a, c = V[vs[i]:vs[i + 1]], one.potential()
        ea, ec = E[:, vs[i]:vs[i + 1]], one.field()
        if precision == pic.FP32_SPLIT:
            assert np.array_equal(a, c) and np.array_equal(ea, ec)
        else:
            assert np.max(np.abs(a - c)) <= TOL64 * max(1e-300, np.max(np.abs(c)))
            assert np.max(np.abs(ea - ec)) <= TOL64 * max(1e-300, np.max(np.abs(c))) * 3 ** depths[i]


@pytest.mark.parametrize("sweeps", [1, 4])
def test_long_march_matches_fp64(sweeps):
    """243^3: blocks that march over several groups of planes, against the FP64
    solve of the same particles.  A sweep rounds the at most 64 terms of a vertex
    by 2^-24 each, and its iteration matrix does not amplify (norm 1)."""
    x, v = W.random_particles(3, 200001, 17, vmax=0.2)
    kw = dict(q=-1.0 / len(x), qm=-1.0, ion=0.3, sweeps=sweeps, omega=0.8, scheme=pic.PIT)
    V = []
    for precision in (pic.FP32_SPLIT, pic.FP64):
        g = pic.Pic(3, W.uniform_tree_flags(3, 5), x, v, precision=precision, **kw)
        g.step(0.05)
        g.sync()
        V.append(g.potential())
        del g
    assert np.max(np.abs(V[1])) > 0
    assert np.max(np.abs(V[0] - V[1])) <= sweeps * 64 * 2.0 ** -24 * np.max(np.abs(V[1]))
