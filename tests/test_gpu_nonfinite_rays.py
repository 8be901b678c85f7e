"""bt_cast_rays with rays that are not finite (a missing point is usually marked
by NaN): they hit nothing, and the ordinary rays of the same warps are not
disturbed.  A NaN ray meets every box, unused lanes of a wide node included,
so scenes of a few triangles, whose nodes have unused lanes, and larger ones,
with leaves of one and of several triangles."""
import numpy as np
import pytest

from paper_1912_03998_gb300 import btrace, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf_size", [1, 4])
@pytest.mark.parametrize("scene", ["two", "three", "box", "city"])
def test_nonfinite_rays_hit_nothing(scene, leaf_size):
    w = {"two": lambda: synth.ground_only(level=0), "three": lambda: synth.single_wall(level=0),
         "box": lambda: synth.boxes(1, level=0), "city": lambda: synth.tiny_city(seed=2, level=0, n_grid=8)}[scene]()
    if scene == "three":
        w.scene.tris, w.scene.mat = w.scene.tris[:3], w.scene.mat[:3]
    rng = np.random.default_rng(5)
    n = 1000
    o = rng.uniform([-20, -20, 0.5], [60, 60, 40], (n, 3)).astype(np.float32)
    d = rng.standard_normal((n, 3)).astype(np.float32)
    ns = rng.standard_normal((n, 3)).astype(np.float32)
    bad = np.zeros(n, bool)
    for k, (where, value) in enumerate(((o, np.nan), (d, np.nan), (o, np.inf), (d, -np.inf), (o, -np.inf))):
        rows = np.arange(k, n, 9)
        where[rows[::2]] = value        # all three components
        where[rows[1::2], k % 3] = value  # one
        bad[rows] = True
    zero = np.arange(5, n, 9)
    d[zero] = 0.0
    bad[zero] = True
    with btrace.Tracer(0) as t:
        sid = t.load(w)
        # (a trace sets the hierarchy's leaf size)
        btrace.bt_trace(t.ctx, sid, t.params(0, leaf_size=leaf_size))
        for normals in (None, ns):
            got_t, got_id = btrace.bt_cast_rays(t.ctx, sid, o, d, normals)
            assert np.isinf(got_t[bad]).all() and (got_id[bad] == -1).all()
            sub = None if normals is None else normals[~bad]
            ref_t, ref_id = btrace.bt_cast_rays(t.ctx, sid, o[~bad], d[~bad], sub)
            assert np.array_equal(got_t[~bad], ref_t) and np.array_equal(got_id[~bad], ref_id)
            assert (ref_id >= 0).any()
        ns[::4] = np.nan
        got_t, got_id = btrace.bt_cast_rays(t.ctx, sid, o, d, ns)
        assert np.isinf(got_t[::4]).all() and (got_id[::4] == -1).all()
