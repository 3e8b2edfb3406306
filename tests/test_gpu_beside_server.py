"""Graph calls while a server's executor holds its share of every SM: they run
beside it instead of waiting until it leaves. The executor is resident and idle
here, with an idle timeout far above the time that the calls may take.
"""
import time

import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

IDLE, LIMIT = 8.0, 2.0  # seconds
MOST = 1504 << 10
HUB = (1 << 21) + 1, 65  # edges of the list, repeated on the device: 2^27 and more


def edges(n, count, repeats=1):
    e = np.ascontiguousarray(graphgen.rmat((n - 1).bit_length(), count, 81) % np.uint32(n))
    return e, torch.from_numpy(e.view(np.int32)).cuda().repeat(repeats, 1)


# vertices, edges, repeats: one block; the vertex bits, smallest and largest; the general pass; the wide table's sizes
SIZES = [(4096, 12_289, 1), (48 << 10, 32_767, 1), (1 << 14, 1 << 16, 1), (MOST, 3 * MOST + 1, 1), (1 << 17, 1 << 18, 1),
         (1 << 22, *HUB)]


@pytest.mark.parametrize("blocks", [3, 4])
@pytest.mark.parametrize("mode", [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY])
def test_runs_and_inserts_do_not_wait_for_the_executor(mode, blocks):
    if blocks == 4 and mode == cc.CC_ROOT_MAXDEG:
        pytest.skip("the exact selection's counting pass needs the room that three blocks leave")
    stream = torch.cuda.current_stream()
    cases = []
    for n, count, repeats in SIZES:
        e, d = edges(n, count, repeats)
        more = graphgen.pairs(n, 4000, 82)
        g = cc.Graph(n, mode=mode)  # (its kernels run once before the executor is there)
        L = torch.empty(n, dtype=torch.int32, device="cuda")
        m = torch.from_numpy(more.view(np.int32)).cuda()
        L.fill_(-1)
        g.run(d, L)
        g.insert(m)
        g.labels(L)
        g.sync()
        L.cpu()
        cases.append((g, d, L, m, oracle.min_labels(n, np.concatenate([e, more]))))
    base, base_d = edges(1 << 12, 1 << 14)
    q = torch.from_numpy(graphgen.pairs(1 << 12, 4000, 83).view(np.int32)).cuda()
    out = torch.empty(4000, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    try:
        with cc.Server(1 << 28, mode=mode, executor_blocks_per_sm=blocks, idle_timeout_us=int(IDLE * 1e6)) as s:
            t, graph = s.new_graph(1 << 12, base_d)
            assert s.wait(t) == cc.CC_OK
            assert s.wait(s.query(graph, q, out)) == cc.CC_OK  # the executor is resident now
            for g, d, L, m, want in cases:
                t0 = time.perf_counter()
                L.fill_(-1)
                g.run(d, L)
                g.insert(m)
                g.labels(L)
                stream.synchronize()
                assert time.perf_counter() - t0 < LIMIT
                np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), want)
            assert s.wait(s.query(graph, q, out)) == cc.CC_OK
            assert s.stats()["executor_launches"] == 1  # it was there all the time
    finally:
        for g, *_ in cases:
            g.close()
