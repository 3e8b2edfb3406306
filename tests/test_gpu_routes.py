"""Which passes a run takes on both sides of every line of the dispatch, by the
number of kernels it launches: the routes give the same labels, so the other
tests would not notice one that is never taken.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
cc = pytest.importorskip("paper_2507_03695_gb300")

MODES = [cc.CC_ROOT_MAXDEG, cc.CC_ROOT_IDENTITY]


def edges(n, count):
    g = torch.Generator("cuda").manual_seed(count)
    return torch.randint(0, n, (count, 2), generator=g, dtype=torch.int32, device="cuda")


def launches(call):
    before = cc.cc_kernel_launches()
    call()
    return cc.cc_kernel_launches() - before


def of_run(n, d, **options):
    with cc.Graph(n, **options) as g:
        return launches(lambda: g.run(d))


@pytest.mark.parametrize("mode", MODES)
def test_one_block(mode):
    for n, count, one in ((49_152, 32_767, True), (49_153, 32_767, False), (49_152, 32_768, False), (1, 0, True)):
        assert (of_run(n, edges(n, count), mode=mode) == 1) == one


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("n, count, bits", [(10_000, 32_768, True), (60_000, 180_000, True), (60_000, 179_999, False),
                                            (1504 << 10, 4512 << 10, True), ((1504 << 10) + 1, (4512 << 10) + 3, False)])
def test_vertex_bits(n, count, bits, mode):
    d = edges(n, count)
    assert (of_run(n, d, mode=mode) != of_run(n, d, mode=mode, block_size=512)) == bits


@pytest.mark.parametrize("n, least", [(1 << 22, 1 << 27), (1 << 24, 12 << 24), ((1 << 25) + 1, 1 << 27)])
def test_wide_table(n, least):
    d = edges(n, least)
    for take, wide in ((d, True), (d[:-1], False)):
        more = of_run(n, take) - of_run(n, take, block_size=512)
        assert more == (1 if wide else 0)  # the table's packing
    if n < 1 << 25:  # (with the bitmap it stays: the other form fits no better beside an executor)
        with cc.Server(1 << 26):
            assert of_run(n, d) == of_run(n, d, block_size=512)
    assert of_run(n, d) == of_run(n, d, block_size=512) + 1


@pytest.mark.parametrize("n, count, same", [(762, 809, True), (60_000, 180_000, True), (60_000, 179_999, False)])
def test_host_lists(n, count, same):
    d = edges(n, count)
    host = d.cpu().pin_memory()
    with cc.Graph(n, count) as g:
        from_host = launches(lambda: cc.cc_run_host(g.h, host, count, None))
        assert (from_host == launches(lambda: g.run(d))) == same
