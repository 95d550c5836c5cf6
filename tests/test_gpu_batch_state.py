"""A split state handed to a batch may hold other numbers of particles per
instance than before (an instance may be left empty): every particle belongs to
the instance of its leaf, and steps are those of single handles, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)

DEPTHS = [3, 1, 2]


def setup(d, scheme, counts, new, device, seed=7):
    """A batch with `counts` particles per instance that was handed `new` ones, and a single handle of each."""
    kw = dict(scheme=scheme, precision=pic.FP32_SPLIT, qm=-1.0, ion=0.3, sweeps=4)
    flags = [W.uniform_tree_flags(d, k) for k in DEPTHS]
    first = [W.random_particles(d, n, n, vmax=0.3) for n in counts]
    qs = [-1e-3, -2e-3, -5e-4]
    b = pic.Pic.batch(d, flags, [p[0] for p in first], [p[1] for p in first], qs, **kw)
    singles = [pic.Pic(d, f, *W.random_particles(d, n, seed + i, vmax=0.3), q=q, path=pic.PATH_GENERIC, **kw)
               if n else None for i, (f, n, q) in enumerate(zip(flags, new, qs))]
    off = np.concatenate([[0], np.cumsum([(3 ** d) ** k for k in DEPTHS])])
    parts = [(s.get_state(), off[i]) for i, s in enumerate(singles) if s]
    leaf = np.concatenate([p[0] + o for p, o in parts]).astype(np.int32)
    pos, vel = (np.ascontiguousarray(np.concatenate([p[k] for p, _ in parts], axis=1)) for k in (1, 2))
    mix = np.random.default_rng(seed).permutation(len(leaf))
    args = leaf[mix], np.ascontiguousarray(pos[:, mix]), np.ascontiguousarray(vel[:, mix])
    # the same order within every instance as the singles are given
    for i, s in enumerate(singles):
        if s:
            mine = (args[0] >= off[i]) & (args[0] < off[i + 1])
            s.set_state(args[0][mine] - np.int32(off[i]), np.ascontiguousarray(args[1][:, mine]),
                        np.ascontiguousarray(args[2][:, mine]))
    b.set_state(*(torch.from_numpy(a).cuda() for a in args) if device else args)
    return b, singles, off


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("scheme", [pic.PIT, pic.PIDT])
@pytest.mark.parametrize("new", [[2000, 300, 900], [100, 2500, 600], [0, 1, 3199], [3200, 0, 0], [1, 0, 3199]])
def test_steps_match_single_plasmas(d, scheme, new, device):
    b, singles, off = setup(d, scheme, [700, 2100, 400], new, device)
    at = np.concatenate([[0], np.cumsum(new)])
    for h in [b, *filter(None, singles)]:
        h.step(0.05)
        h.step_fixed_field(0.07)
        h.step_particles(0.3, reflect=True)
        h.sync()
    leaf, pos, vel = b.get_state()
    vs = b.instances()[1]
    Q = b.deposit()
    for i, s in enumerate(singles):
        if s is None:
            continue
        r = slice(at[i], at[i + 1])
        l1, p1, v1 = s.get_state()
        assert np.array_equal(leaf[r], l1 + off[i]) and np.array_equal(pos[:, r], p1) and np.array_equal(vel[:, r], v1)
        assert np.array_equal(Q[vs[i]:vs[i + 1]], s.deposit())


@pytest.mark.parametrize("scheme", [pic.PIT, pic.PIDT])
@pytest.mark.parametrize("new", [[2000, 300, 900], [0, 1, 3199], [3200, 0, 0]])
def test_ranges_and_checkpoint_follow(scheme, new, tmp_path):
    b, _, off = setup(2, scheme, [700, 2100, 400], new, True)
    want = np.concatenate([[0], np.cumsum(new)])
    assert np.array_equal(b.instances()[0], want)
    b.step(0.05)
    assert np.array_equal(b.instances()[0], want)
    b.save(tmp_path / "batch.pic")
    c = pic.Pic.load(tmp_path / "batch.pic")
    assert np.array_equal(c.instances()[0], want)
    for h in (b, c):
        h.step(0.05)
        h.sync()
    for u, w in zip(b.get_state(), c.get_state()):
        assert np.array_equal(u, w)
    leaf = b.get_state()[0]
    assert np.array_equal(np.searchsorted(leaf, off[:-1]), want[:-1]) or scheme == pic.PIDT
