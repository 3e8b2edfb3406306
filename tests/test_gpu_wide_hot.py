"""The edge pass with the wide hot-vertex table (2^22 vertices, 2^27 and 12 n
edges and up, default launch shape; a shorter list, repeated on the device) against the CPU oracle and the general pass, bit for bit: every
field width the table can have at sizes that fit a test, both forms (P within
and beyond the zero-tree threshold), odd and misaligned edge lists, a graph
without a hub, and an out-of-range id.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

MIN_EDGES = 1 << 27  # the shortest list that takes this pass
COUNT = (1 << 23) + 1  # edges made on the host


def on_device(n, e, misalign):
    """The list, repeated until it is long enough: an odd number of edges."""
    repeats = (max(MIN_EDGES, 12 * n) // len(e) + 1) | 1
    assert len(e) & 1 and repeats * len(e) >= max(MIN_EDGES, 12 * n)
    buf = torch.empty((repeats * len(e) + 1, 2), dtype=torch.int32, device="cuda")
    view = buf[1:] if misalign else buf[:-1]
    view.view(repeats, len(e), 2).copy_(torch.from_numpy(e.view(np.int32)).cuda().expand(repeats, -1, -1))
    return view


def run(n, d, **options):
    with cc.Graph(n, **options) as g:
        L = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        g.run(d, L)
        g.sync()
        return L.cpu().numpy().view(np.uint32), g.num_components(), g.root_vertex()


# 2^22: four fields of 8 bits; 2^22 + 3 and 2^24: three of 9 and 10; 2^25 + 1:
# two of 12, and P beyond 128 MiB (the zero-tree form)
@pytest.mark.parametrize("n", [1 << 22, (1 << 22) + 3, 1 << 24, (1 << 25) + 1])
@pytest.mark.parametrize("misalign", [False, True])
@pytest.mark.parametrize("kind", ["rmat", "uniform"])
def test_labels_match_the_oracle(n, misalign, kind):
    scale = (n - 1).bit_length()
    count = COUNT + 64 * (n % 7)
    e = graphgen.rmat(scale, count, 31) % np.uint32(n) if kind == "rmat" else graphgen.pairs(n, count, 32)
    d = on_device(n, np.ascontiguousarray(e), misalign)
    want = oracle.min_labels(n, e)
    got, comps, m = run(n, d)
    np.testing.assert_array_equal(got, want)
    assert comps == oracle.num_components(want)
    assert m == oracle.max_degree_vertex(n, e)
    other, comps2, m2 = run(n, d, block_size=512)  # the general pass
    np.testing.assert_array_equal(other, want)
    assert (comps2, m2) == (comps, m)


@pytest.mark.parametrize("at", [0, 1, MIN_EDGES // 2, -1])
def test_out_of_range_id_is_reported(at):
    n = 1 << 22
    e = graphgen.rmat(22, COUNT, 33)
    d = on_device(n, e, False)
    good = d[at, at & 1].clone()
    d[at, at & 1] = n
    with cc.Graph(n) as g:
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(d, L)
        assert cc.cc_sync_status(g.h) == cc.CC_ERR_OUT_OF_RANGE
        d[at, at & 1] = good
        g.run(d, L)  # the handle stays usable
        g.sync()
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, e))
