"""The one-block run (cc_tiny.cu) at its limits, over the options that reach
it, against the CPU oracle and the general path."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

VERTICES, EDGES = 48 << 10, (1 << 15) - 1


def on_device(e, misalign):
    buf = torch.empty((len(e) + 1, 2), dtype=torch.int32, device="cuda")
    view = buf[1:] if misalign else buf[:-1]
    view.copy_(torch.from_numpy(np.ascontiguousarray(e, dtype=np.uint32).view(np.int32)))
    return view


def run(n, d, label=True, **options):
    with cc.Graph(n, **options) as g:
        L = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")[1:]  # labels need no 16-byte alignment
        g.run(d, L if label else None)
        first = g.num_components(), g.root_vertex()
        g.labels(L)  # from the parent array that the run left
        g.sync()
        return (L.cpu().numpy().view(np.uint32), *first)


OPTIONS = [dict(), dict(mode=cc.CC_ROOT_IDENTITY), dict(label_space=cc.CC_LABEL_ROOT_VALUE),
           dict(root_select=cc.CC_ROOT_SELECT_SAMPLED), dict(root_select=cc.CC_ROOT_SELECT_SAMPLED, sample_stride=3),
           dict(root_hint=0)]


@pytest.mark.parametrize("n, count", [(1, 0), (1, 5), (2, 1), (3, 2), (1023, 1024), (1025, 4097), (4099, 12_289),
                                      (VERTICES - 1, EDGES), (VERTICES, EDGES - 1), (VERTICES + 1, EDGES),
                                      (VERTICES, EDGES + 1), (30_000, 7), (500, EDGES)])
@pytest.mark.parametrize("misalign", [False, True])
def test_limits(n, count, misalign):
    scale = max(1, (n - 1).bit_length())
    e = graphgen.rmat(scale, count, n + count) % np.uint32(n)
    d, want = on_device(e, misalign), oracle.min_labels(n, e)
    for options in OPTIONS:
        got, comps, m = run(n, d, label=count % 2 == 0, **options)
        general = run(n, d, block_size=512, **options)
        np.testing.assert_array_equal(got, general[0])
        assert (comps, m) == general[1:] and comps == oracle.num_components(want)
        if options.get("label_space") is None:
            np.testing.assert_array_equal(got, want)


def test_shapes():
    n = 20_000
    rng = np.random.default_rng(3)
    path = np.stack([np.arange(n - 1), np.arange(1, n)], 1)
    hub = np.stack([np.full(30_000, n - 1), rng.integers(0, n, 30_000)], 1)
    for e in (path, path[::-1, ::-1], rng.permutation(path), hub, hub[:, ::-1], np.repeat(path[:16], 1000, axis=0)):
        e = np.ascontiguousarray(e, dtype=np.uint32)
        want = oracle.min_labels(n, e)
        for mode in (cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY):
            got, comps, m = run(n, on_device(e, False), mode=mode)
            np.testing.assert_array_equal(got, want)
            assert comps == oracle.num_components(want)
            if mode == cc.CC_ROOT_MAXDEG:
                assert m == oracle.max_degree_vertex(n, e)


@pytest.mark.parametrize("at", [0, 1, 2, 4998, 4999])
def test_out_of_range_id_is_reported_and_inserts_follow(at):
    n = 2000
    e = graphgen.er(n, 5000, 4)
    e[at, at & 1] = n
    good = np.delete(e, at, axis=0)
    with cc.Graph(n) as g:
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(on_device(e, True), L)
        assert cc.cc_sync_status(g.h) == cc.CC_ERR_OUT_OF_RANGE
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, good))
        more = graphgen.pairs(n, 700, 5)
        g.insert(on_device(more, False))
        g.labels(L)
        g.sync()
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, np.concatenate([good, more])))
