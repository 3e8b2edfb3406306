"""Host-memory runs of small graphs, which take the device-resident run's route
on the staged edges: plain and packed ids, every selection, both sides of the
sizes where that route begins and ends, against the device-resident run and the
oracle; consecutive calls of other sizes on one handle.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

CAP = 1 << 18


def on_device(n, e, **options):
    with cc.Graph(n, **options) as g:
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        g.run(torch.from_numpy(e.view(np.int32)).cuda(), L)
        g.sync()
        return L.cpu().numpy().view(np.uint32), g.num_components(), g.root_vertex()


SIZES = [(1, 5), (300, 1), (300, 900), (49152, 32767), (49153, 32767), (20000, 32768), (20000, 60000),
         (20000, 59999), (70000, 210000), (70000, 209999)]


@pytest.mark.parametrize("options", [
    dict(), dict(mode=cc.CC_ROOT_IDENTITY), dict(label_space=cc.CC_LABEL_ROOT_VALUE),
    dict(root_select=cc.CC_ROOT_SELECT_SAMPLED), dict(root_hint=0)])
def test_matches_the_device_run(options):
    for n, count in SIZES:
        e = np.ascontiguousarray(graphgen.rmat(max(1, (n - 1).bit_length()), count, 61) % np.uint32(n))
        labels, comps, root = on_device(n, e, **options)
        if options.get("label_space") is None:
            np.testing.assert_array_equal(labels, oracle.min_labels(n, e))
        small = e[: max(1, count // 7)]
        with cc.Graph(n, CAP, **options) as g:
            for host in (torch.from_numpy(e.view(np.int32)).pin_memory(), torch.from_numpy(e.view(np.int32))):
                L = torch.full((n,), -1, dtype=torch.int32).pin_memory()
                cc.cc_run_host(g.h, host, count, L)
                np.testing.assert_array_equal(L.numpy().view(np.uint32), labels)
                assert (g.num_components(), g.root_vertex()) == (comps, root)
                # another list in between, without labels
                cc.cc_run_host_packed(g.h, torch.from_numpy(graphgen.pack_ids(small, 3)), len(small), 3, None)
            L.fill_(-1)
            cc.cc_run_host_packed(g.h, torch.from_numpy(graphgen.pack_ids(e, 3)), count, 3, L)
            np.testing.assert_array_equal(L.numpy().view(np.uint32), labels)
            assert (g.num_components(), g.root_vertex()) == (comps, root)


@pytest.mark.parametrize("count", [1000, 40000])
def test_out_of_range_id_is_reported(count):
    n = 5000
    e = graphgen.pairs(n, count, 62)
    bad = e.copy()
    bad[count // 2, 1] = n
    with cc.Graph(n, CAP) as g:
        L = torch.empty(n, dtype=torch.int32)
        with pytest.raises(cc.CCError):
            cc.cc_run_host(g.h, torch.from_numpy(bad.view(np.int32)), count, L)
        cc.cc_run_host(g.h, torch.from_numpy(e.view(np.int32)), count, L)
        np.testing.assert_array_equal(L.numpy().view(np.uint32), oracle.min_labels(n, e))
