"""The edge pass by vertex bits (cc_bits.cu) at the sizes where it begins and
ends, on graph shapes its linking rounds could get wrong, against the CPU
oracle and the general pass; and the handle's budget, which its scratch must
not take from what a run needs."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

MOST, FEWEST = 1536 << 10, 1 << 15  # vertices, edges


def on_device(e, misalign):
    buf = torch.empty((len(e) + 1, 2), dtype=torch.int32, device="cuda")
    view = buf[1:] if misalign else buf[:-1]
    view.copy_(torch.from_numpy(np.ascontiguousarray(e, dtype=np.uint32).view(np.int32)))
    return view


def run(n, d, **options):
    with cc.Graph(n, **options) as g:
        L = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        g.run(d, L)
        g.sync()
        return L.cpu().numpy().view(np.uint32), g.num_components(), g.root_vertex()


def check(n, e, misalign=False, modes=(cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY)):
    d, want = on_device(e, misalign), oracle.min_labels(n, np.ascontiguousarray(e, dtype=np.uint32))
    for mode in modes:
        got, comps, m = run(n, d, mode=mode)
        np.testing.assert_array_equal(got, want)
        assert comps == oracle.num_components(want)
        assert (m, comps) == run(n, d, mode=mode, block_size=512)[:0:-1]  # the general pass


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 127, 128, 129, 4099, FEWEST // 3, FEWEST // 3 + 1])
@pytest.mark.parametrize("count", [FEWEST - 1, FEWEST, FEWEST + 1, FEWEST + 255])
@pytest.mark.parametrize("misalign", [False, True])
def test_where_it_begins(n, count, misalign):
    check(n, graphgen.er(n, count, n + count), misalign)


@pytest.mark.parametrize("n", [MOST - 1, MOST, MOST + 1])
def test_where_it_ends(n):
    check(n, graphgen.er(n, 3 * n + 1, 3), modes=(cc.CC_ROOT_MAXDEG,))


def shapes():
    rng = np.random.default_rng(5)
    path = np.stack([np.arange(39_999), np.arange(1, 40_000)], 1)
    yield "path", 40_000, np.repeat(path, 4, axis=0)
    yield "path backwards", 40_000, np.repeat(path[::-1, ::-1], 4, axis=0)
    yield "long path", 1_000_000, np.tile(np.stack([np.arange(999_999), np.arange(1, 1_000_000)], 1), (4, 1))
    yield "star at the top", 20_000, np.stack([np.full(80_000, 19_999), rng.integers(0, 20_000, 80_000)], 1)
    halves = np.concatenate([rng.integers(0, 9000, (60_000, 2)), rng.integers(9000, 18_001, (60_000, 2))])
    yield "two halves", 18_001, rng.permutation(halves)
    loops = np.repeat(np.arange(5000), 20)
    yield "self-loops", 5000, np.stack([loops, loops], 1)
    yield "cliques", 12_000, (rng.integers(0, 1200, 100_000)[:, None] * 10 + rng.integers(0, 10, (100_000, 2)))
    yield "skewed", 50_021, graphgen.rmat(16, 700_001, 8) % np.uint32(50_021)
    e = graphgen.rmat(15, 1 << 19, 9)
    yield "by source", 1 << 15, e[np.argsort(e[:, 0], kind="stable")]


@pytest.mark.parametrize("name, n, e", list(shapes()), ids=lambda v: v if isinstance(v, str) else "")
def test_shapes(name, n, e):
    check(n, e)


@pytest.mark.parametrize("at", [0, 1, 130, 99_999, 100_000])
def test_out_of_range_id_is_reported(at):
    n = 5000
    e = graphgen.er(n, 100_001, 11)
    e[at, at & 1] = n + at
    with cc.Graph(n) as g:
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(on_device(e, False), L)
        assert cc.cc_sync_status(g.h) == cc.CC_ERR_OUT_OF_RANGE
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, np.delete(e, at, axis=0)))


@pytest.mark.parametrize("n", [1 << 16, 1 << 22])
def test_budget_without_the_scratch_is_enough(n):
    e = graphgen.rmat(16, 1 << 18, 12)
    want = oracle.min_labels(n, e)
    with cc.Graph(n, block_size=512) as g:  # the general pass alone: no scratch of the others
        least = cc.cc_device_bytes(g.h)
    with cc.Graph(n) as g:
        assert cc.cc_device_bytes(g.h) > least
    with cc.Graph(n, hbm_budget_bytes=least) as g:
        assert cc.cc_device_bytes(g.h) == least
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(on_device(e, False), L)
        g.sync()
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), want)
    # a later buffer displaces it: the labels of a host run
    with cc.Graph(n, len(e), hbm_budget_bytes=least + 8 * len(e) + 4 * n) as g:
        host, out = torch.from_numpy(e.view(np.int32)).pin_memory(), torch.empty(n, dtype=torch.int32).pin_memory()
        cc.cc_run_host(g.h, host, L_out_host=out)
        np.testing.assert_array_equal(out.numpy().view(np.uint32), want)
        g.run(on_device(e, False))
        assert g.num_components() == oracle.num_components(want)
