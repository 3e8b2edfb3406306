"""Inserts at the sizes where their route changes: one block up to 4096 pairs, and
into settled trees a full or a small grid by what the list meets. Labels and
counts against the oracle, all or nothing when an id is out of range.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

SLOWER = 1.4  # the worst that a route may be to the same insert into a fresh handle


def on_device(e, misalign):
    buf = torch.empty((len(e) + 1, 2), dtype=torch.int32, device="cuda")
    view = buf[1:] if misalign else buf[:-1]
    view.copy_(torch.from_numpy(np.ascontiguousarray(e, dtype=np.uint32).view(np.int32)))
    return view


def launches(call):
    before = cc.cc_kernel_launches()
    call()
    return cc.cc_kernel_launches() - before


@pytest.mark.parametrize("mode", [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY])
@pytest.mark.parametrize("settled", [False, True])
@pytest.mark.parametrize("count", [1, 511, 4095, 4096, 4097, 70_001])
@pytest.mark.parametrize("misalign", [False, True])
def test_routes(mode, settled, count, misalign):
    n = 1 << 16
    base = graphgen.rmat(15, 2 * n if settled else n, 91)  # the upper half stays empty
    near = graphgen.pairs(n // 2, count, 92)
    far = graphgen.rmat(15, count, 93) + np.uint32(n // 2)
    with cc.Graph(n, mode=mode) as g:
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(on_device(base, False))
        seen = [base]
        for e in (near, far, near):
            bad = e.copy()
            bad[-1, 1] = n
            g.insert(on_device(bad, misalign))
            assert cc.cc_sync_status(g.h) == cc.CC_ERR_OUT_OF_RANGE
            g.labels(L)
            np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, np.concatenate(seen)))
            d = on_device(e, misalign)
            assert (launches(lambda: g.insert(d)) == 1) == (count <= 4096)
            seen.append(e)
            g.labels(L)
            want = oracle.min_labels(n, np.concatenate(seen))
            np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), want)
            assert g.num_components() == oracle.num_components(want)


def test_a_new_part_of_the_graph_is_not_taken_to_be_settled():
    n, count = 1 << 17, 1 << 20
    first, new = graphgen.rmat(16, count, 94), graphgen.rmat(16, count, 95) + np.uint32(n // 2)
    d, m = on_device(first, False), on_device(new, False)

    def insert_takes(start, mode):
        with cc.Graph(n, mode=mode) as g:
            best = float("inf")
            for _ in range(9):
                g.run(start)
                torch.cuda.synchronize()
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                g.insert(m)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b) * 1e3)
            g.sync()
            return best

    for mode in (cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY):
        assert insert_takes(d, mode) <= SLOWER * insert_takes(d[: n // 8], mode)
