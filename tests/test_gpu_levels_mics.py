"""The level readout's logarithm over the whole float64 range, and microphone
binning at the sizes where its scan and its cells change."""
import numpy as np
import pytest

from paper_1912_03998_gb300 import btrace, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bands", [1, 3, 8])
def test_levels_of_installed_intensities(n_bands):
    rng = np.random.default_rng(n_bands)
    n = 1500
    I = 10.0 ** rng.uniform(-300.0, 300.0, (n, n_bands))
    I.flat[:400] = 10.0 ** rng.uniform(-20.0, 3.0, 400)
    # powers of two, their neighbours, denormals, zero and infinity
    p = 2.0 ** np.arange(-40, 40)
    special = np.concatenate([p, np.nextafter(p, 0), np.nextafter(p, 1e9), [5e-324, 1e-310, 0.0, np.inf, 1.0, 1e-12]])
    I.flat[400:400 + len(special)] = special
    w = synth.ground_only(level=1)
    mics = rng.uniform(-50.0, 50.0, (n, 3)).astype(np.float32)
    cnt = rng.integers(0, 9, n).astype(np.int32)
    with btrace.Tracer(0) as t:
        sid = btrace.bt_load_scene(t.ctx, w.scene.verts, w.scene.tris, w.scene.mat, synth.refl_table(n_bands=n_bands))
        btrace.bt_set_microphones(t.ctx, sid, mics)
        btrace.bt_set_result(t.ctx, sid, I, cnt)
        L, J, c = np.empty((n, n_bands)), np.empty((n, n_bands)), np.empty(n, np.int32)
        btrace.bt_read_levels(t.ctx, sid, L, J, c)
        L2 = np.empty((n, n_bands))
        btrace.bt_read_levels(t.ctx, sid, L2)
    assert (J == I).all() and (c == cnt).all() and np.array_equal(L, L2)
    with np.errstate(divide="ignore"):
        ref = 10.0 * np.log10(I) + 120.0
    f = np.isfinite(ref)
    assert np.array_equal(L[~f], ref[~f])
    # the reference and the kernel each round a few times at the size of the
    # largest intermediate: four units in the last place between them
    assert (np.abs(L[f] - ref[f]) <= 4 * np.spacing(np.maximum(np.abs(ref[f]), 128.0))).all()


@pytest.mark.parametrize("n,kind", [(1, "spread"), (2, "same"), (33, "same"), (1000, "line"), (4097, "spread"),
                                    (65530, "spread"), (65541, "spread"), (70000, "volume"), (5000, "same")])
def test_every_microphone_binned_once(n, kind):
    """Free field, one source: every microphone lies in exactly one beam and
    receives W / (4 pi d^2)."""
    rng = np.random.default_rng(n)
    m = rng.uniform(-80.0, 80.0, (n, 3))
    if kind == "same":
        m[:] = m[0]
    if kind == "line":
        m[:, 1:] = m[0, 1:]
    if kind == "spread":
        m[:, 2] = 1.5
    m = m.astype(np.float32)
    w = synth.free_field(level=3).with_mics(m)
    with btrace.Tracer(0) as t:
        g = t.run(w)
    assert (g["cnt"] == 1).all()
    d2 = ((m.astype(np.float64) - w.src[0].astype(np.float64)) ** 2).sum(1)
    ref = w.power[0].astype(np.float64)[None] / (4.0 * np.pi * d2[:, None])
    # float32 distance and quotient: a few 2^-24 relative
    np.testing.assert_allclose(g["I"], ref, rtol=1e-6)


def test_levels_are_rounded_once():
    """Against 50-digit arithmetic: half a unit in the last place of the level,
    and 1e-16 dB for all that the readout adds below it (its largest small part
    is 0.02 dB, rounded a few times, and a float32 tail of 6e-17 dB)."""
    from decimal import Decimal, localcontext
    rng = np.random.default_rng(3)
    n, nb = 500, 8
    I = 10.0 ** rng.uniform(-18.0, 2.0, (n, nb))
    I[:100] = 10.0 ** rng.uniform(-300.0, 300.0, (100, nb))
    I[100:150] = 1e-12 * (1.0 + rng.uniform(-1e-3, 1e-3, (50, nb)))
    w = synth.ground_only(level=1)
    with btrace.Tracer(0) as t:
        sid = btrace.bt_load_scene(t.ctx, w.scene.verts, w.scene.tris, w.scene.mat, synth.refl_table(n_bands=nb))
        btrace.bt_set_microphones(t.ctx, sid, rng.uniform(-50.0, 50.0, (n, 3)).astype(np.float32))
        btrace.bt_set_result(t.ctx, sid, I, np.zeros(n, np.int32))
        L = np.empty((n, nb))
        btrace.bt_read_levels(t.ctx, sid, L)
    with localcontext() as ctx:
        ctx.prec = 50
        ref = [10 * Decimal(float(x)).log10() + 120 for x in I.ravel()]
        err = np.array([abs(float(Decimal(float(y)) - r)) for y, r in zip(L.ravel(), ref)])
    tol = 0.5 * np.spacing(np.abs(np.array([float(r) for r in ref]))) + 1e-16
    assert (err <= tol).all(), (err / tol).max()


@pytest.mark.parametrize("precision", [btrace.BT_PREC_MIXED, btrace.BT_PREC_FP64])
@pytest.mark.parametrize("kind", ["planes", "clusters", "one off", "top and bottom", "column"])
def test_layers_without_microphones(kind, precision):
    """Volumes whose microphones fill few of the grid's layers or few of its
    cells, alone and in a batch beside a planar set: free field, every
    microphone once."""
    rng = np.random.default_rng(len(kind))
    n = 40000
    m = rng.uniform(-80.0, 80.0, (n, 3))
    if kind == "planes":
        m[:, 2] = rng.choice([-3.0, 35.0], n)
    if kind == "clusters":
        m = rng.uniform(-60.0, 60.0, (7, 3))[rng.integers(0, 7, n)] + rng.uniform(0.0, 1.0, (n, 3))
    if kind == "one off":
        m[:, 2] = 1.5
        m[n // 2, 2] = 70.0
    if kind == "top and bottom":
        m[:, 2] = np.where(rng.random(n) < 0.5, -40.0, 40.0) + rng.uniform(0.0, 0.1, n)
    if kind == "column":
        m[:, :2] = 20.0 + rng.uniform(0.0, 0.1, (n, 2))
    w = synth.free_field(level=3).with_mics(m.astype(np.float32))
    flat = synth.free_field(level=3)

    def check(sid, mics, w):
        I, cnt = np.empty((len(mics), 8)), np.empty(len(mics), np.int32)
        btrace.bt_read_levels(t.ctx, sid, None, I, cnt)
        assert (cnt == 1).all()
        d2 = ((mics.astype(np.float64) - w.src[0].astype(np.float64)) ** 2).sum(1)
        np.testing.assert_allclose(I, w.power[0].astype(np.float64)[None] / (4.0 * np.pi * d2[:, None]), rtol=1e-6)

    with btrace.Tracer(0) as t:
        sids = [t.load(w), t.load(flat)]
        p = t.params(1, precision=precision)
        btrace.bt_trace(t.ctx, sids[0], p)
        check(sids[0], w.mics, w)
        b = btrace.bt_batch_create(t.ctx, sids, [p, p])
        btrace.bt_batch_run(t.ctx, b)
        check(sids[0], w.mics, w)
        check(sids[1], flat.mics, flat)
        btrace.bt_batch_destroy(b)
