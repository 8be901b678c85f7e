"""Small launches, whose lanes work in groups on one lineage, against the same
trace with one lane per lineage (a work-counting trace always takes that path):
the same hits, so counts are exact and intensities agree to the rounding of
their float64 sums (1e-9 relative, as for the other orders of accumulation).
Sizes on both sides of the rule's lines and down to one beam per face."""
import numpy as np
import pytest

from paper_1912_03998_gb300 import btrace, synth

pytestmark = pytest.mark.gpu


def both(t, sid, n_m, nb, order, **kw):
    out = []
    for count_work in (0, 1):
        btrace.bt_trace(t.ctx, sid, t.params(order, count_work=count_work, **kw))
        I, cnt = np.empty((n_m, nb)), np.empty(n_m, np.int32)
        st = btrace.bt_read_levels(t.ctx, sid, None, I, cnt)
        out.append((I, cnt, st))
    (I0, c0, s0), (I1, c1, s1) = out
    for k in ("segments", "hits", "escapes", "emitted", "contributions"):
        assert s0[k] == s1[k], k
    assert (c0 == c1).all()
    np.testing.assert_allclose(I0, I1, rtol=1e-9, atol=0.0)


@pytest.mark.parametrize("precision", [btrace.BT_PREC_FP32, btrace.BT_PREC_MIXED])
@pytest.mark.parametrize("tiles", [(1, 1), (3, 2)])
@pytest.mark.parametrize("sources,level", [(1, 0), (3, 1), (1, 4), (2, 4), (7, 4), (10, 4), (11, 4)])
def test_groups_match_single_lanes(precision, tiles, sources, level):
    w = synth.tiny_city(seed=3, level=level, max_order=4, n_grid=24, n_sources=sources)
    with btrace.Tracer(0) as t:
        both(t, t.load(w), len(w.mics), 8, w.max_order, precision=precision, tiles_x=tiles[0], tiles_y=tiles[1])


def test_groups_few_triangles():
    """Hierarchies of one leaf, of a few, and of none."""
    with btrace.Tracer(0) as t:
        for w in (synth.boxes(1, level=3), synth.ground_only(level=3), synth.single_wall(level=3),
                  synth.free_field(level=2)):
            both(t, t.load(w), len(w.mics), 8, w.max_order)
        w = synth.ground_only(level=3)
        w.scene.tris, w.scene.mat = w.scene.tris[:1], w.scene.mat[:1]
        both(t, t.load(w), len(w.mics), 8, w.max_order)


def test_groups_coincident_triangles():
    """Stacks of coincident triangles: every box overlaps every ray, so the
    groups' stacks grow past the depth at which they take one node a step."""
    w = synth.ground_only(level=2)
    w.scene.tris = np.concatenate([w.scene.tris] * 1500).astype(np.int32)
    w.scene.mat = np.concatenate([w.scene.mat] * 1500).astype(np.uint8)
    with btrace.Tracer(0) as t:
        both(t, t.load(w), len(w.mics), 8, w.max_order)


def test_groups_in_a_batch():
    ws = [synth.tiny_city(seed=s, level=lv, max_order=k, n_grid=16, n_sources=n)
          for s, lv, k, n in ((1, 3, 2, 1), (2, 4, 5, 1), (3, 2, 3, 4))]
    with btrace.Tracer(0) as t:
        sids = [t.load(w) for w in ws]
        got = []
        for count_work in (0, 1):
            b = btrace.bt_batch_create(t.ctx, sids, [t.params(w.max_order, count_work=count_work) for w in ws])
            btrace.bt_batch_run(t.ctx, b)
            for sid, w in zip(sids, ws):
                I, cnt = np.empty((len(w.mics), 8)), np.empty(len(w.mics), np.int32)
                btrace.bt_read_levels(t.ctx, sid, None, I, cnt)
                got.append((I, cnt))
            btrace.bt_batch_destroy(b)
        for (I0, c0), (I1, c1) in zip(got[:3], got[3:]):
            assert (c0 == c1).all()
            np.testing.assert_allclose(I0, I1, rtol=1e-9, atol=0.0)


def test_groups_few_triangles_split():
    """Sub-domains with hierarchies of one leaf, of a few, and of none."""
    with btrace.Tracer(0) as t:
        for w in (synth.boxes(1, level=3), synth.boxes(4, level=3), synth.ground_only(level=3), synth.single_wall(level=3)):
            both(t, t.load(w), len(w.mics), 8, w.max_order, tiles_x=3, tiles_y=4)
        w = synth.ground_only(level=3)
        w.scene.tris, w.scene.mat = w.scene.tris[:1], w.scene.mat[:1]
        both(t, t.load(w), len(w.mics), 8, w.max_order, tiles_x=5, tiles_y=2)


@pytest.mark.parametrize("precision", [btrace.BT_PREC_FP32, btrace.BT_PREC_MIXED])
def test_chunks_on_both_sides_of_the_rule(precision):
    """A lineage rounds alike whatever the size of its launch: 163,840 lineages in
    one launch on single lanes, in chunks of 60,000 with the rest on groups of
    eight, in chunks of 45,000 on those and of 7,000 on groups of sixteen."""
    w = synth.tiny_city(seed=6, level=5, max_order=5, n_grid=40, n_sources=8)
    with btrace.Tracer(0) as t:
        sid = t.load(w)
        out = []
        for chunk in (0, 60000, 45000, 7000):
            btrace.bt_trace(t.ctx, sid, t.params(w.max_order, precision=precision, chunk_beams=chunk))
            I, cnt = np.empty((len(w.mics), 8)), np.empty(len(w.mics), np.int32)
            st = btrace.bt_read_levels(t.ctx, sid, None, I, cnt)
            out.append((I, cnt, st))
        for I, cnt, st in out[1:]:
            for k in ("segments", "hits", "escapes", "emitted", "contributions"):
                assert st[k] == out[0][2][k], k
            assert (cnt == out[0][1]).all()
            # (float32 contributions in float64 sums: only their order differs)
            np.testing.assert_allclose(I, out[0][0], rtol=1e-12, atol=0.0)
