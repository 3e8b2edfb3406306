"""Shapes whose order or degrees the specialised routes could be slow on: labels
against the oracle, and no route takes much longer than the general pass on the
same call (the fastest of several runs each).
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

SLOWER = 1.5  # the worst that a route may be to the general pass


def microseconds(call, before=lambda: None, runs=9):
    best = float("inf")
    for _ in range(runs):
        before()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def path(n):
    return np.stack([np.arange(n - 1), np.arange(1, n)], 1)


def by_source(e):
    return e[np.argsort(e[:, 0], kind="stable")]


def lattice(*sides):
    """Every pair of neighbours of a lattice, diagonal ones too, by first vertex."""
    c = np.arange(np.prod(sides)).reshape(sides)
    out = []
    for step in np.ndindex(*(3,) * len(sides)):
        d = np.array(step) - 1
        if tuple(d) > (0,) * len(sides):
            a = c[tuple(slice(max(0, -k), s - max(0, k)) for k, s in zip(d, sides))]
            b = c[tuple(slice(max(0, k), s - max(0, -k)) for k, s in zip(d, sides))]
            out.append(np.stack([a.ravel(), b.ravel()], 1))
    return by_source(np.concatenate(out))


def star(n, count, others=0):
    rng = np.random.default_rng(7)
    e = np.concatenate([np.stack([np.full(count, n - 1), rng.integers(0, n, count)], 1), rng.integers(0, n, (others, 2))])
    return rng.permutation(e)


def cliques(n, k, count):
    rng = np.random.default_rng(8)
    return rng.integers(0, n // k, (count, 1)) * k + rng.integers(0, k, (count, 2))


ONE_BLOCK = {
    "path": (20_000, path(20_000)), "path backwards": (20_000, path(20_000)[::-1]), "short path": (4000, path(4000)),
    "path, shuffled": (30_000, np.random.default_rng(9).permutation(path(30_000))), "lattice": (8000, lattice(80, 100)[:32_767]),
}


def check(n, e, mode):
    e = np.ascontiguousarray(e, dtype=np.uint32)
    d = torch.from_numpy(e.view(np.int32)).cuda()
    L = torch.empty(n, dtype=torch.int32, device="cuda")
    with cc.Graph(n, mode=mode) as g, cc.Graph(n, mode=mode, block_size=512) as general:
        took, usual = microseconds(lambda: g.run(d, L)), microseconds(lambda: general.run(d))
        np.testing.assert_array_equal(L.cpu().numpy().view(np.uint32), oracle.min_labels(n, e))
    assert took <= SLOWER * usual, (took, usual)


@pytest.mark.parametrize("mode", [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY])
@pytest.mark.parametrize("shape", ONE_BLOCK)
def test_one_block_run(shape, mode):
    check(*ONE_BLOCK[shape], mode)


VERTEX_BITS = {
    "lattice": lambda: (10**6, lattice(1000, 1000)), "long lattice": lambda: (960_000, lattice(60_000, 16)),
    "small lattice": lambda: (40_000, lattice(200, 200)), "cube": lambda: (10**6, lattice(100, 100, 100)),
    "path": lambda: (10**6, np.tile(path(10**6), (4, 1))), "star at the top": lambda: (10**6, star(10**6, 4 * 10**6)),
    "quarter star": lambda: (10**6, star(10**6, 10**6, 3 * 10**6)), "cliques": lambda: (10**6, cliques(10**6, 10, 10**7)),
    "cliques by source": lambda: (10**6, by_source(cliques(10**6, 10, 10**7))),
}


@pytest.mark.parametrize("mode", [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY])
@pytest.mark.parametrize("shape", VERTEX_BITS)
def test_vertex_bits(shape, mode):
    check(*VERTEX_BITS[shape](), mode)
