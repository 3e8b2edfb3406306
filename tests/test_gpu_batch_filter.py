"""The batched path's sampled hooking and its filter by reference tree: graphs
at the lines where the sampling starts (edge count, edges per vertex, vertices
whose bits fit), ragged chunks, odd offsets, graphs whose largest component
does not hold vertex 0, and bad ids in the chunks that only the filter reads.
Bit for bit against the CPU oracle."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

MIN_EDGES, BITS = 1 << 15, 1 << 18


def run(parts, shift=0, **cfg):
    """parts: (n, edges) per graph; shift: the labels start that many words past a 16-byte boundary."""
    vtx = np.cumsum([0] + [n for n, _ in parts]).astype(np.uint64)
    off = np.cumsum([0] + [len(e) for _, e in parts]).astype(np.uint64)
    edges = np.concatenate([np.asarray(e, dtype=np.uint32).reshape(-1, 2) for _, e in parts])
    L = torch.full((int(vtx[-1]) + 4,), -1, dtype=torch.int32, device="cuda")[shift:shift + int(vtx[-1])]
    with cc.Batch(len(parts)) as b:
        if cfg:
            cc.cc_batch_set_config(b.h, **cfg)
        b.run(len(parts), torch.from_numpy(vtx.view(np.int64)).cuda(), torch.from_numpy(off.view(np.int64)).cuda(),
              torch.from_numpy(edges.view(np.int32)).cuda(), L)
        status = cc.cc_batch_sync_status(b.h)
    return L.cpu().numpy().view(np.uint32), status, (edges, vtx, off)


def check(parts, **kw):
    got, status, (edges, vtx, off) = run(parts, **kw)
    assert status == cc.CC_OK
    np.testing.assert_array_equal(got, oracle.batch_min_labels(edges, vtx, off))


@pytest.mark.parametrize("count", [MIN_EDGES - 1, MIN_EDGES, MIN_EDGES + 1, MIN_EDGES + 127, 100_003])
@pytest.mark.parametrize("ratio", [2.99, 3.0, 3.01, 9.7, 400.0])
def test_lines_of_the_sampling(count, ratio):
    n = max(2, int(count / ratio))
    check([(n, graphgen.er(n, count, 5)), (3, [[0, 2]]), (n, graphgen.rmat(18, count, 6) % np.uint32(n))])


@pytest.mark.parametrize("n", [BITS - 1, BITS, BITS + 1])
def test_vertices_whose_bits_fit(n):
    check([(n, graphgen.er(n, 3 * n + 1, 7)), (1000, graphgen.er(1000, 40_000, 8))])


@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("cfg", [{}, dict(filter=0, edges_per_thread=4), dict(block_size=256, tile_edges=256)],
                         ids=["default", "lanes", "small tiles"])
def test_components_of_every_shape(shift, cfg):
    rng = np.random.default_rng(9)
    n = 9001
    upper = rng.integers(n // 2, n, (60_000, 2))            # the large component, away from vertex 0
    halves = np.concatenate([rng.integers(0, 4000, (40_000, 2)), rng.integers(4000, 8001, (40_000, 2))])
    rng.shuffle(halves)                                      # two components of one size
    star = np.stack([np.full(50_000, 17), rng.integers(0, 5000, 50_000)], 1)
    path = np.repeat(np.stack([np.arange(4999), np.arange(1, 5000)], 1), 8, axis=0)
    loops = np.repeat(np.arange(2000), 20)
    check([(n, upper), (0, []), (8001, halves), (5000, star), (5000, path[::-1]), (2000, np.stack([loops, loops], 1)),
           (1, np.zeros((40_000, 2)))], shift=shift, **cfg)


def test_bad_ids_in_filtered_chunks_are_reported():
    n, count = 2000, 60_000
    e = graphgen.er(n, count, 10)
    bad = [129, 300, count - 1]
    e[bad, [0, 1, 0]] = [n, 0xFFFFFFFF, n + 5]
    got, status, _ = run([(n, e)])
    assert status == cc.CC_ERR_OUT_OF_RANGE
    np.testing.assert_array_equal(got, oracle.min_labels(n, np.delete(e, bad, axis=0)))  # the bad edges are skipped
    got, status, _ = run([(0, np.zeros((40_000, 2))), (4, [[1, 2]])])  # a graph of edges without vertices
    assert status == cc.CC_ERR_OUT_OF_RANGE
    np.testing.assert_array_equal(got, [0, 1, 1, 3])
