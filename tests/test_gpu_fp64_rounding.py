"""FP64 on uniform trees: the first sweep from zero is omega b / diag rounded once,
and the field is the difference of potentials over the rounded leaf width, without
a systematic error."""
from __future__ import annotations

from fractions import Fraction

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("omega", [0.8, 0.7, 1.0, 1.3])
@pytest.mark.parametrize("d,depth", [(2, 3), (2, 4), (2, 6), (3, 2), (3, 3), (3, 4)])
def test_first_sweep_is_rounded_once(d, depth, omega):
    n = 3001
    x, v = W.random_particles(d, n, 5, vmax=0.1)
    g = pic.Pic(d, W.uniform_tree_flags(d, depth), x, v, precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=1, omega=omega)
    g.init_leapfrog(0.0)
    V, Q = g.potential(), g.deposit()
    h = 1.0 / 3 ** depth
    ion = 1.0
    for _ in range(d):
        ion *= h
    b = Q - g.stats().total_charge * ion
    diag = 2 ** d * (4 / 6 if d == 2 else 4 / 12) * (1.0 if d == 2 else h)
    w = Fraction(omega) / Fraction(diag)
    for i in np.random.default_rng(3).choice(len(V), 400):
        # the two-double factor and the product's tail are off by 2^-100 or so: half an ulp and a little
        assert abs(Fraction(float(V[i])) - w * Fraction(float(b[i]))) <= Fraction(float(np.spacing(abs(V[i])))) * Fraction(501, 1000)


@pytest.mark.parametrize("depth", [3, 4, 5, 6])
def test_field_has_no_systematic_error(depth):
    n = 20_011
    x, v = W.random_particles(2, n, 5, vmax=0.1)
    g = pic.Pic(2, W.uniform_tree_flags(2, depth), x, v, precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=9)
    g.init_leapfrog(0.0)
    M = 3 ** depth
    V = g.potential().reshape(M, M)
    h = Fraction(1.0 / M)
    f = float(1 / (2 * h))
    own = abs(Fraction(f) * 2 * h - 1)  # the factor's rounding, which the product cannot avoid
    for a, E in enumerate(g.field().reshape(2, M, M)):
        diff = np.roll(V, 1, 1 - a) - np.roll(V, -1, 1 - a)
        ok = np.abs(diff) > 0
        # one rounding of at most 2^-53 relative each, of either sign: five deviations of their mean
        noise = 5 * 2.0 ** -53 / np.sqrt(ok.sum())
        err = (E[ok] - diff[ok] * (M / 2)) / (diff[ok] * (M / 2))  # against an exact factor M / 2
        assert abs(err.mean() - float(1 / (M * h) - 1)) <= float(own) + 2 * noise
