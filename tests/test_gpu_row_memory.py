"""The assembled rows of the FP64 solve on adaptive trees are optional: where one
of their blocks is refused, at creation or at a re-tree, the handle solves by the
two passes and gives the other blocks back."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU hosts
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROWS_FROM = 16  # sweeps from which rows are assembled


class Requests:
    """Device blocks from torch, their sizes on record; request number `refuse` gets none, nor do those of `bytes`."""

    def __init__(self, refuse=None):
        self.sizes, self.refuse, self.bytes, self.refused = [], refuse, None, 0
        self.calls = (pic.ALLOC_FN(self.take), pic.FREE_FN(self.give))

    def take(self, user, nbytes, stream):
        self.sizes.append(int(nbytes))
        if len(self.sizes) - 1 == self.refuse or int(nbytes) == self.bytes:
            self.refused += 1
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))

    def give(self, user, p, nbytes, stream):
        torch.cuda.caching_allocator_delete(int(p))


def trees(d):
    """A small and a larger tree; the larger one's rows are short enough to be assembled (36 and 41 entries)."""
    if d == 2:
        return W.random_tree_flags(2, 3, 0.3, 1, min_depth=1), W.random_tree_flags(2, 6, 0.2, 2, min_depth=4)
    return W.random_tree_flags(3, 2, 0.2, 22, min_depth=1), W.random_tree_flags(3, 3, 0.02, 2, min_depth=2)


def handle(d, flags, sweeps, refuse=None):
    req = Requests(refuse)
    lib = pic.load()
    n = 3001
    x, v = W.random_particles(d, n, 8, vmax=0.1)
    assert lib.pic_set_allocator(*req.calls, None) == 0
    try:
        h = pic.Pic(d, flags, x, v, precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=sweeps)
    finally:
        assert lib.pic_set_allocator(pic.ALLOC_FN(), pic.FREE_FN(), None) == 0
    h.requests = req  # the callbacks outlive the handle's blocks
    return h


def extra_requests(few, many):
    """Positions in `many` of the requests that `few` does not make (in the same order)."""
    out, i = [], 0
    for k, s in enumerate(many):
        if i < len(few) and few[i] == s:
            i += 1
        else:
            out.append(k)
    assert i == len(few)
    return out


def close(V, want):
    # a sum of at most 64 terms per vertex and sweep, in another order; two solves
    return np.max(np.abs(V - want)) <= 2 * ROWS_FROM * 64 * 2.0 ** -53 * np.max(np.abs(want))


def stepped(h):
    h.step(0.05)
    h.sync()
    return h.potential()


@pytest.mark.parametrize("d", [2, 3])
def test_refused_rows_leave_the_two_passes(d):
    small, large = trees(d)
    few = handle(d, large, ROWS_FROM - 1)
    rows = handle(d, large, ROWS_FROM)
    extra = extra_requests(few.requests.sizes, rows.requests.sizes)
    assert len(extra) >= 4
    V = stepped(rows)
    for k in extra:
        h = handle(d, large, ROWS_FROM, refuse=k)
        assert h.requests.refused == 1
        assert close(stepped(h), V)
        assert h.info().device_bytes == few.info().device_bytes  # nothing of them is kept
        h.close()
    # the same at a re-tree, for the two largest blocks
    a = handle(d, small, ROWS_FROM)
    a.retree(large)
    Va = stepped(a)
    for size in sorted(rows.requests.sizes[k] for k in extra)[-2:]:
        h = handle(d, small, ROWS_FROM)
        h.requests.bytes = size
        h.retree(large)
        assert h.requests.refused >= 1
        assert close(stepped(h), Va)
        h.close()
    # a block that every handle needs is still an error
    with pytest.raises(pic.PicError):
        handle(d, large, ROWS_FROM, refuse=0)


@pytest.mark.parametrize("d", [2, 3])
def test_rows_wait_for_the_first_solve(d):
    """Creations and re-trees leave the rows to the first solve outside a capture; the solves of a captured
    step before it are by the two passes."""
    small, large = trees(d)
    n = 3001
    x, v = W.random_particles(d, n, 8, vmax=0.1)
    kw = dict(precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=ROWS_FROM)
    s = torch.cuda.Stream()
    a = pic.Pic(d, small, x, v, stream=s, **kw)
    b = pic.Pic(d, large, *a.particles(), **kw)
    a.retree(large)
    held = a.info().device_bytes
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        a.init_leapfrog(0.0)
    graph.replay()
    torch.cuda.synchronize()
    b.init_leapfrog(0.0)  # rows, from the same charges and a potential of zero
    b.sync()
    assert close(a.potential(), b.potential()) and np.any(b.potential())
    for h in (a, b):
        h.step(0.05)
        h.sync()
    assert close(a.potential(), b.potential())
    assert a.info().device_bytes == held  # a step takes no memory


def test_first_solve_leaves_another_threads_capture_alone():
    flags = trees(2)[1]
    n = 3001
    x, v = W.random_particles(2, n, 8, vmax=0.1)
    kw = dict(precision=pic.FP64, q=-1.0 / n, ion=0.3, sweeps=ROWS_FROM)
    want = stepped(pic.Pic(2, flags, x, v, **kw))
    h = pic.Pic(2, flags, x, v, stream=torch.cuda.Stream(), **kw)
    a = torch.zeros(1000, device="cuda")
    graph, failed = torch.cuda.CUDAGraph(), []

    def step():
        try:
            h.step(0.05)
        except pic.PicError as e:
            failed.append(e)

    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="global"):
        a += 1
        other = threading.Thread(target=step)
        other.start()
        other.join()
        a += 1
    graph.replay()
    torch.cuda.synchronize()
    assert not failed and torch.all(a == 2)
    h.sync()
    assert np.array_equal(h.potential(), want)
