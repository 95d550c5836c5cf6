"""Captured fixed-field steps take the field as it is when they are launched, also
where a call between the capture and the launch changed it without a step: an
unchanged re-refinement clears it, the leapfrog start solves it again.  Field
copies that the push reads (leaf corners, bricks) follow."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)

DT = 1e-7  # kicks show in the velocities, and no particle leaves its leaf


def pair(d, precision, depth, ppc):
    n = 20_011
    x, _ = W.random_particles(d, n, 4, vmax=0.0)
    kw = dict(precision=precision, q=-1.0 / n, ion=1.0, sweeps=5)
    out = []
    for _ in range(2):
        h = pic.Pic(d, W.uniform_tree_flags(d, depth), x, np.zeros_like(x), stream=torch.cuda.Stream(), **kw)
        if ppc:
            h.adapt(ppc, 1, depth + 2)
            assert not h.info().uniform
        out.append(h)
    return out


def velocities(h):
    h.sync()
    return h.get_state()[2]


@pytest.mark.parametrize("d,precision,depth,ppc", [(2, pic.FP64, 3, 30), (2, pic.FP32_SPLIT, 3, 30), (3, pic.FP64, 2, 25),
                                                   (3, pic.FP32_SPLIT, 2, 25), (3, pic.FP32_SPLIT, 3, 0),
                                                   (2, pic.FP32_SPLIT, 4, 0), (2, pic.FP64, 4, 0)])
def test_unchanged_refinement_clears_the_field(d, precision, depth, ppc):
    a, b = pair(d, precision, depth, ppc)
    for h in (a, b):
        h.step(DT)
    a.graph_capture(DT)
    b.step_fixed_field(DT)
    for h in (a, b):
        before = h.info().n_leaves
        if ppc:
            h.adapt(ppc, 1, depth + 2)
        else:
            h.adapt(0, depth, depth)
        assert h.info().n_leaves == before and not np.any(h.field())
    a.graph_launch(2)
    for _ in range(2):
        b.step_fixed_field(DT)
    va, vb = velocities(a), velocities(b)
    assert np.any(vb) and np.array_equal(va, vb)


@pytest.mark.parametrize("d,depth", [(3, 3), (2, 4)])
def test_leapfrog_start_between_brick_replays(d, depth):
    a, b = pair(d, pic.FP32_SPLIT, depth, 0)
    assert a.info().brick
    for h in (a, b):
        h.step(DT)
    a.graph_capture(DT)
    b.step_fixed_field(DT)
    for h in (a, b):
        h.init_leapfrog(0.0)  # five more sweeps from the potential before
    a.graph_launch(2)
    for _ in range(2):
        b.step_fixed_field(DT)
    assert np.array_equal(velocities(a), velocities(b))
