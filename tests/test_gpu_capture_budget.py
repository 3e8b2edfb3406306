"""Captured runs on a handle with a memory budget: scratch that a later buffer
of the handle may displace is not named by the captured launches, so a replay
after such a call is sound. Without a budget nothing is displaced and a
captured run takes the same passes as any other, but for the wide hot-vertex
table's.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")


def capture(g, d, L):
    """The captured run and how many kernels it holds."""
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        g.run(d, L, s)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        before = cc.cc_kernel_launches()
        graph.capture_begin()
        g.run(d, L, s)
        graph.capture_end()
        return graph, cc.cc_kernel_launches() - before


def launches(g, d, L):
    before = cc.cc_kernel_launches()
    g.run(d, L)
    return cc.cc_kernel_launches() - before


# the vertex bits of small graphs; the wide hot-vertex table (a short list, repeated on the device)
@pytest.mark.parametrize("scale, repeats", [(16, 1), (22, 65)])
@pytest.mark.parametrize("mode", [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY])
def test_replay_after_the_scratch_was_displaced(scale, repeats, mode):
    n, e = 1 << scale, graphgen.rmat(scale, (1 << 21) + 1 if repeats > 1 else 1 << 18, 71)
    want = oracle.min_labels(n, e)
    d = torch.from_numpy(e.view(np.int32)).cuda().repeat(repeats, 1)
    L = torch.empty(n, dtype=torch.int32, device="cuda")
    host, out = torch.from_numpy(e.view(np.int32)).pin_memory(), torch.empty(n, dtype=torch.int32).pin_memory()
    with cc.Graph(n, len(e), mode=mode, block_size=512) as g:
        least, general = cc.cc_device_bytes(g.h), launches(g, d, L)
    with cc.Graph(n, len(e), mode=mode) as g:
        fast = launches(g, d, L)
        graph, held = capture(g, d, L)
        # (the pass with the wide table waits for a server's executor: never captured)
        assert held == (fast if repeats == 1 else general)
    # room for the scratch, or for the labels of a host run, not for both
    with cc.Graph(n, len(e), mode=mode, hbm_budget_bytes=least + 4 * n) as g:
        assert launches(g, d, L) == fast
        graph, held = capture(g, d, L)
        assert held == general
        cc.cc_run_host(g.h, host, L_out_host=out)
        assert cc.cc_device_bytes(g.h) == least + 4 * n
        np.testing.assert_array_equal(out.numpy().view(np.uint32), want)
        for _ in range(2):
            L.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), want)
        assert g.num_components() == oracle.num_components(want)
