"""Batches whose sizes or shapes the schedule could be slow on: a batch of a
quarter of the graphs against the whole one.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")


def takes(parts):
    """Microseconds (the fastest of nine) of a batch of (n, edges), its labels checked."""
    vtx = np.cumsum([0] + [n for n, _ in parts]).astype(np.int64)
    off = np.cumsum([0] + [len(e) for _, e in parts]).astype(np.int64)
    edges = np.ascontiguousarray(np.concatenate([e for _, e in parts]), dtype=np.uint32)
    v, o, d = torch.from_numpy(vtx).cuda(), torch.from_numpy(off).cuda(), torch.from_numpy(edges.view(np.int32)).cuda()
    L = torch.empty(int(vtx[-1]), dtype=torch.int32, device="cuda")
    best = float("inf")
    with cc.Batch(len(parts)) as b:
        for _ in range(9):
            torch.cuda.synchronize()
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            b.run(len(parts), v, o, d, L)
            end.record()
            end.synchronize()
            best = min(best, start.elapsed_time(end) * 1e3)
        assert cc.cc_batch_sync_status(b.h) == cc.CC_OK
    want = oracle.batch_min_labels(edges, vtx.astype(np.uint64), off.astype(np.uint64))
    np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), want)
    return best


def test_a_quarter_of_the_graphs():
    # at most 0.6 of the time: it cannot fill the GPU as well, but need not be slower a graph
    parts = [(1 << 16, graphgen.rmat(16, 1 << 18, 100 + k % 20)) for k in range(400)]
    assert takes(parts[:100]) <= 0.6 * takes(parts)


def lattice(side):
    """Rows of a lattice with its diagonals, by first vertex."""
    c = np.arange(side * side).reshape(side, side)
    pairs = [(c[:, :-1], c[:, 1:]), (c[:-1], c[1:]), (c[:-1, :-1], c[1:, 1:]), (c[:-1, 1:], c[1:, :-1])]
    e = np.concatenate([np.stack([a.ravel(), b.ravel()], 1) for a, b in pairs])
    return e[np.argsort(e[:, 0], kind="stable")]


def test_lattices():
    # with 40% more vertices, of no edges, the same graphs are hooked whole: the sampled route may cost a third more
    e = lattice(200)
    assert takes([(40_000, e)] * 200) <= 1.33 * takes([(56_000, e)] * 200)
