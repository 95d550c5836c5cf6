"""The built-in FP64 solve on adaptive trees by assembled rows (enough sweeps)
and by the two passes (few sweeps), and the FP32 one, against the oracle: 2D and
3D, hanging vertices over several level jumps, ragged last slices of rows, odd
and even numbers of sweeps, and a re-tree in between."""
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

TOL64 = 1e-11  # some hundred roundings of 1.1e-16 per sum and sweep, fields of scale one


@pytest.mark.parametrize("sweeps", [7, 15, 16, 33])
@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_SPLIT])
@pytest.mark.parametrize("d,depth,min_depth,p", [(2, 3, 1, 0.3), (2, 5, 2, 0.25), (2, 6, 3, 0.2), (3, 2, 1, 0.2),
                                                  (3, 4, 1, 0.15)])
def test_potential_and_field_match_oracle(d, depth, min_depth, p, precision, sweeps):
    flags = [W.random_tree_flags(d, depth, p, 20 + depth, min_depth=min_depth),
             W.random_tree_flags(d, depth, p, 40 + depth, min_depth=min_depth)]
    n = 3001
    x, v = W.random_particles(d, n, 8, vmax=0.1)
    kw = dict(q=-1.0 / n, qm=-1.0, ion=0.3, sweeps=sweeps, omega=0.8)
    g = pic.Pic(d, flags[0], x, v, precision=precision, **kw)
    for k in range(2):
        if k:
            g.retree(flags[1])
        S = oracle.State64 if precision == pic.FP64 else oracle.State32
        xs, vs = g.particles()
        st = S(oracle.Tree(d, flags[k]), xs, vs, oracle.Params(**kw))
        for _ in range(2):  # the second solve starts from the first one's potential
            Q, _, res, E = st.field()
            g.init_leapfrog(0.0)
        V, Eg = g.potential(), g.field()
        # the deposit's rounding enters V through the charges, the same relative size
        scale = max(1e-300, float(np.max(np.abs(st.V))))
        Eo = np.asarray(E, np.float64).reshape(Eg.shape)
        if precision == pic.FP64:
            assert np.max(np.abs(V - st.V)) <= TOL64 * scale
            assert np.max(np.abs(Eg - Eo)) <= TOL64 * scale * 3 ** depth
        elif k == 0:  # the re-located offsets of the second tree are not the oracle's conversion of FP64 positions
            assert np.array_equal(V, st.V.astype(np.float64)) and np.array_equal(Eg, Eo)
        assert abs(g.stats().residual - res) <= 1e-5 * res + 1e-12
