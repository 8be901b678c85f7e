"""The tuning knobs on small launches, whose lanes work in groups on one lineage:
no setting may make the groups slower than the same launch on single lanes (a
work-counting trace always takes those, and counts besides).  Best of nine
launches each; 1.25 leaves room for the clock."""
import pytest

from paper_1912_03998_gb300 import btrace, synth

pytestmark = pytest.mark.gpu

SLOWER = 1.25


@pytest.fixture(scope="module")
def city():
    with btrace.Tracer(0) as t:
        yield t, {n: t.load(synth.tiny_city(seed=1, level=4, max_order=4, n_sources=n)) for n in (1, 2, 8)}


def kernel_ms(t, sid, **kw):
    p, best = t.params(4, **kw), float("inf")
    for _ in range(9):
        btrace.bt_trace(t.ctx, sid, p)
        best = min(best, btrace.bt_read_levels(t.ctx, sid)["trace_kernel_ms"])
    return best


def check(city, sources, **kw):
    t, sid = city
    groups, single = kernel_ms(t, sid[sources], **kw), kernel_ms(t, sid[sources], count_work=1, **kw)
    assert groups <= SLOWER * single, (sources, kw, groups, single)


@pytest.mark.parametrize("tiles", [1, 4])
@pytest.mark.parametrize("sources,beams_per_warp", [(1, 32), (1, 256), (8, 64), (8, 1024)])
def test_reserved_lineages(city, tiles, sources, beams_per_warp):
    check(city, sources, tiles_x=tiles, tiles_y=tiles, beams_per_warp=beams_per_warp)


@pytest.mark.parametrize("sources,queue_depth", [(1, 32), (1, 1024), (2, 256), (8, 32), (8, 256), (8, 4096)])
def test_shallow_queues(city, sources, queue_depth):
    check(city, sources, tiles_x=4, tiles_y=4, queue_depth=queue_depth)


@pytest.mark.parametrize("tiles", [1, 4])
@pytest.mark.parametrize("sources,blocks_per_sm", [(1, 1), (2, 1), (2, 2), (8, 1), (8, 2), (8, 4)])
def test_fewer_blocks(city, tiles, sources, blocks_per_sm):
    check(city, sources, tiles_x=tiles, tiles_y=tiles, blocks_per_sm=blocks_per_sm)
