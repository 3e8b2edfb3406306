"""The exact root of graphs without a hub, whose degrees are all counted: runs
of equal sources (summed before they are added) of every length and position,
odd and misaligned lists, and vertex counts that leave a remainder of four.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")


@pytest.mark.parametrize("n", [50001, 65536, 65539, 200002])
@pytest.mark.parametrize("count", [65535, 100002, 400003])
@pytest.mark.parametrize("kind", ["random", "source", "target", "runs"])
def test_root_is_the_largest_degree(n, count, kind):
    e = graphgen.pairs(n, count, 51 + n % 5)
    if kind == "source":
        e = e[np.argsort(e[:, 0], kind="stable")]
    elif kind == "target":
        e = e[np.argsort(e[:, 1], kind="stable")]
    elif kind == "runs":  # 1 to 9 equal sources, one after the other
        lengths = np.random.RandomState(n).randint(1, 10, count)
        e[:, 0] = np.repeat(e[:, 0], lengths)[:count]
    e = np.ascontiguousarray(e)
    want = oracle.max_degree_vertex(n, e)
    buf = torch.empty((count + 1, 2), dtype=torch.int32, device="cuda")
    for view in (buf[:-1], buf[1:]):
        view.copy_(torch.from_numpy(e.view(np.int32)))
        with cc.Graph(n) as g:
            g.run(view, None)
            g.sync()
            assert g.root_vertex() == want
