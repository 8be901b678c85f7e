"""What this framework is asked to do, as measurable cases.

A case is a dict of plain values; its "kind" says which public entry points a
pass goes through:

  trace    a resident city with its sources and microphones: bt_trace, then
           bt_read_levels into device arrays
  frame    bt_trace_noalloc into the caller's device arrays
  query    one traffic-noise query served whole (serve.run_plain): sources and
           microphones set, traced, read back to the host, dropped
  burst    several queries at once through the continuous-batching server
           (serve.Server.run)
  batch    several resident cities in one bt_batch_run, every result read
  ingest   a new city model loaded, traced and dropped (Tracer.run on host
           arrays)
  cast     axis rays against a resident city (bt_cast_rays)

The city's plan is drawn once per (buildings) by the framework's generators;
the seed scales the buildings' heights and draws reflection coefficients,
sources, powers, queries and rays.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1912_03998_gb300 import btrace, serve, synth

PREC = {"mixed": btrace.BT_PREC_MIXED, "fp32": btrace.BT_PREC_FP32, "fp64": btrace.BT_PREC_FP64,
        "mixed64": btrace.BT_PREC_MIXED64}
# air damping per octave band, dB/m (63 Hz .. 8 kHz)
ALPHA = (1e-4, 4e-4, 1e-3, 2e-3, 4e-3, 9e-3, 2.3e-2, 7.7e-2)


def listed():
    return [
        # the smallest whole call: one car in eight by eight blocks; latency and launches count
        _trace("tiny_city", scene="tiny", sources=1, level=4, order=4, side=32),
        # the same city traced finely with air damping and an odd microphone grid
        _trace("tiny_city_fine", scene="tiny", sources=2, level=6, order=5, side=45, damping=True),
        # a per-frame update loop in float32, no allocation
        dict(_trace("frame_fp32", buildings=300, sources=1, level=4, order=4, side=63, precision="fp32"), kind="frame"),
        # one small query against a resident city: what a lightly loaded service answers
        {"name": "query_small", "kind": "query", "buildings": 5000, "sources": 3, "level": 4, "order": 4, "side": 33},
        # eight queries waiting at once
        {"name": "query_burst", "kind": "burst", "cities": 2, "queries": 8, "max_sources": 300, "max_mics": 40000},
        # line-of-sight and distance queries by the axis ray alone
        {"name": "cast_rays", "kind": "cast", "buildings": 5000, "rays": 200000, "reflected": True},
        # a changed city model: ingest, hierarchy build and a first look at the levels
        dict(_trace("new_city", buildings=5000, sources=5, level=4, order=4, side=128), kind="ingest"),
        # uneven cities in one launch sequence
        {"name": "batch_cities", "kind": "batch", "cities": 8, "max_sources": 200, "max_mics": 60000, "precision": "mixed"},
        # the district as the paper runs it: split into sub-domains with hand-off queues
        _trace("district_split", buildings=5000, sources=1000, level=5, order=6, side=500, tiles_x=4, tiles_y=4),
        # the district unsplit, directional sources and air damping
        _trace("district_directional", buildings=5000, sources=250, level=5, order=6, side=500, damping=True,
               directional=True),
        # the precision reference: everything in float64
        _trace("district_fp64", buildings=5000, sources=24, level=5, order=6, side=500, precision="fp64"),
        # microphones through the city's whole volume on the 4 m grid, 13.75 M of them
        _trace("district_volume", buildings=5000, sources=40, level=5, order=6, side=500, heights=55, tiles_x=4,
               tiles_y=4),
    ]


def _trace(name, scene="district", buildings=64, sources=1, level=4, order=4, side=32, heights=1, tiles_x=1,
           tiles_y=1, precision="mixed", damping=False, directional=False, bands=8):
    return {"name": name, "kind": "trace", "scene": scene, "buildings": buildings, "sources": sources,
            "level": level, "order": order, "side": side, "heights": heights, "tiles_x": tiles_x,
            "tiles_y": tiles_y, "precision": precision, "damping": damping, "directional": directional,
            "bands": bands}


# -------------------------------------------------------------------- draw
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace"] * 8 + ["frame", "query", "query", "burst", "batch", "ingest", "cast"])
    buildings = _log(rng, 100, 5000)
    if kind == "query":
        return {"kind": "query", "buildings": buildings, "sources": _log(rng, 1, 2000), "level": 4,
                "order": rng.randint(3, 6), "side": _log(rng, 32, 500)}
    if kind == "burst":
        return {"kind": "burst", "cities": rng.randint(1, 4), "queries": rng.randint(2, 16),
                "max_sources": _log(rng, 10, 1000), "max_mics": _log(rng, 2000, 100000)}
    if kind == "batch":
        return {"kind": "batch", "cities": rng.randint(2, 16), "max_sources": _log(rng, 10, 300),
                "max_mics": _log(rng, 2000, 100000), "precision": rng.choice(["mixed", "mixed", "fp32"])}
    if kind == "cast":
        return {"kind": "cast", "buildings": buildings, "rays": _log(rng, 100, 2000000),
                "reflected": rng.random() < 0.5}
    c = _trace("", scene=rng.choice(["tiny", "district", "district"]), buildings=buildings, level=rng.randint(3, 6),
               order=rng.randint(2, 8), side=_log(rng, 16, 500), bands=rng.choice([8, 8, 8, 1, 3, 5]),
               damping=rng.random() < 0.4, directional=rng.random() < 0.3)
    c["kind"] = kind
    c["precision"] = rng.choice(["mixed"] * 5 + ["fp32", "fp64", "mixed64"])
    if kind == "trace" and rng.random() < 0.5:
        c["tiles_x"], c["tiles_y"] = rng.choice([(2, 2), (4, 4), (3, 5), (1, 4), (8, 8)])
    if kind == "trace" and rng.random() < 0.25:
        c["heights"] = rng.randint(2, 55)
    # segments of a pass at most those of the largest listed case of its type
    most = {"mixed": 1000 * 20480 * 7, "fp32": 1000 * 20480 * 7, "fp64": 24 * 20480 * 7,
            "mixed64": 400 * 20480 * 7}[c["precision"]]
    if c["heights"] > 1:
        most = min(most, 40 * 20480 * 7 * (55 * 500 * 500) / (c["heights"] * c["side"] ** 2))
    if kind == "ingest":
        c["scene"], c["directional"], most = "district", False, most / 10
    if kind == "frame":
        most /= 50
    per_source = 20 * 4 ** c["level"] * (c["order"] + 1)
    c["sources"] = _log(rng, 1, max(1, min(1000, int(most // per_source))))
    if c["scene"] == "tiny":
        c["buildings"] = 64
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=16)
def _plan(scene, buildings, variant):
    """The plan of a city, (verts, tris, mat): the generators' own."""
    if scene == "tiny":
        s = synth.tiny_city(seed=1 + variant).scene
    else:
        s = synth.district(seed=2 + variant, n_buildings=buildings, n_sources=1, n_mic_side=2).scene
    return s.verts, s.tris, s.mat


def _city(rng, scene="district", buildings=64, bands=8, variant=0):
    verts, tris, mat = _plan(scene, buildings, variant)
    verts = verts * np.array([1.0, 1.0, rng.uniform(0.8, 1.25)], np.float32)
    refl = np.stack([rng.uniform(0.6, 0.8, bands), rng.uniform(0.85, 0.95, bands)]).astype(np.float32)
    return synth.Scene(verts.astype(np.float32), tris, mat, refl)


def _sources(rng, scene, n, bands):
    """Cars on the streets at 0.5 m, per-band power log-uniform 0.01-1 W."""
    if scene == "tiny":
        pitch, width, blocks, off = synth.TINY_PITCH, synth.TINY_PITCH - synth.TINY_BLOCK, synth.TINY_N, 0.0
    else:
        pitch, width, blocks, off = synth.DIST_PITCH, synth.DIST_ROAD, synth.DIST_NBLK, 0.5 * synth.DIST_ROAD
    road = rng.integers(0 if scene != "tiny" else 1, blocks, n) * pitch + off
    across = road + rng.uniform(-0.4, 0.4, n) * width
    along = rng.uniform(0.0, pitch * blocks, n)
    flip = rng.random(n) < 0.5
    src = np.stack([np.where(flip, along, across), np.where(flip, across, along), np.full(n, 0.5)], 1)
    return src.astype(np.float32), (10.0 ** rng.uniform(-2.0, 0.0, (n, bands))).astype(np.float32)


def _extent(scene):
    return synth.TINY_PITCH * synth.TINY_N if scene == "tiny" else synth.DIST_MIC_SIDE


def _mics(case):
    e = _extent(case["scene"])
    plane = synth.mic_grid(0.0, 0.0, e, e, case["side"], case["side"], 1.5)
    if case["heights"] == 1:
        return plane
    p = torch.from_numpy(plane).cuda().repeat(case["heights"], 1, 1)
    p[:, :, 2] += 4.0 * torch.arange(case["heights"], device="cuda", dtype=torch.float32)[:, None]
    torch.cuda.synchronize()  # the library's stream reads it
    return p.reshape(-1, 3)


def _workload(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    scene = _city(rng, case["scene"], case["buildings"], case["bands"])
    src, power = _sources(rng, case["scene"], case["sources"], case["bands"])
    d = None
    if case["directional"]:
        d = synth.Directivity([synth.cardioid((1, 0, 0), 0.8), synth.cardioid((0, 1, 0.2), 0.5)],
                              rng.integers(-1, 2, case["sources"]).astype(np.int32))
    return synth.Workload(case["kind"], scene, src, power, _mics(case), case["level"], case["order"],
                          (case["tiles_x"], case["tiles_y"]), {}, d)


def _options(case):
    o = {"precision": PREC[case["precision"]], "tiles_x": case["tiles_x"], "tiles_y": case["tiles_y"]}
    if case["damping"]:
        o["air_atten_db_per_m"] = ALPHA[:case["bands"]]
    return o


def _uneven(n, lo, hi):
    """n sizes from lo to hi, log-spaced, in a fixed mixed order."""
    v = [int(round(lo * (hi / lo) ** (i / max(1, n - 1)))) for i in range(n)]
    return [v[(5 * i) % n] if n % 5 else v[i] for i in range(n)]


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.Generator(np.random.PCG64(seed))
    tr = btrace.Tracer(0)
    if kind in ("trace", "frame", "ingest"):
        w = _workload(case, seed)
        if kind == "ingest":
            return {"kind": kind, "tr": tr, "w": w, "options": _options(case)}
        st = {"kind": kind, "tr": tr, "sid": tr.load(w), "params": tr.params(case["order"], **_options(case))}
        st["level"] = torch.empty((len(w.mics), case["bands"]), dtype=torch.float64, device="cuda")
        st["count"] = torch.empty(len(w.mics), dtype=torch.int32, device="cuda")
        return st
    if kind == "query":
        w = synth.Workload("city", _city(rng, "district", case["buildings"]), None, None, None, 0, 0)
        src, power = _sources(rng, "district", case["sources"], 8)
        span = min(synth.DIST_MIC_SIDE, 4.0 * case["side"])
        x0, y0 = np.clip(src[0, :2] - 0.5 * span, 0.0, synth.DIST_MIC_SIDE - span)
        mics = synth.mic_grid(x0, y0, x0 + span, y0 + span, case["side"], case["side"], 1.5)
        q = synth.Query(0.0, 0, src, power, mics, case["level"], case["order"])
        return {"kind": kind, "tr": tr, "city": tr.load_geometry(w), "query": q}
    if kind == "burst":
        cities = [synth.Workload("city", _city(rng, "district", b, 8, i), None, None, None, 0, 0)
                  for i, b in enumerate(_uneven(case["cities"], 500, 5000))]
        # the stream's sizes and windows are the case's, its cars the seed's
        qs = synth.serving_queries(7, case["queries"], case["cities"], 200.0, max_sources=case["max_sources"],
                                   max_mics=case["max_mics"])
        for q in qs:
            q.src, q.power = _sources(rng, "district", len(q.src), 8)
        return {"kind": kind, "tr": tr, "server": serve.Server(tr, cities), "queries": qs}
    if kind == "batch":
        n = case["cities"]
        sids, params, out = [], [], []
        sizes = zip(_uneven(n, 100, 5000), _uneven(n, case["max_sources"], 1), _uneven(n, case["max_mics"], 1000))
        for i, (b, n_s, n_m) in enumerate(sizes):
            src, power = _sources(rng, "district", n_s, 8)
            side = int(round(math.sqrt(n_m)))
            mics = synth.mic_grid(0.0, 0.0, synth.DIST_MIC_SIDE, synth.DIST_MIC_SIDE, side, side, 1.5)
            w = synth.Workload("city", _city(rng, "district", b, 8, i), src, power, mics, 3 + i % 4, 2 + (3 * i) % 7)
            sids.append(tr.load(w))
            params.append(tr.params(w.max_order, precision=PREC[case["precision"]]))
            out.append((torch.empty((side * side, 8), dtype=torch.float64, device="cuda"),
                        torch.empty(side * side, dtype=torch.int32, device="cuda")))
        return {"kind": kind, "tr": tr, "sids": sids, "batch": btrace.bt_batch_create(tr.ctx, sids, params), "out": out}
    # cast: from points in the streets and on the buildings' walls, in all directions
    w = synth.Workload("city", _city(rng, "district", case["buildings"]), None, None, None, 0, 0)
    n = case["rays"]
    d = rng.standard_normal((n, 3)).astype(np.float32)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    if case["reflected"]:
        v, t = w.scene.verts, w.scene.tris[rng.integers(0, len(w.scene.tris) - 2, n)]
        b = rng.dirichlet((1.0, 1.0, 1.0), n).astype(np.float32)[:, :, None]
        o = (v[t] * b).sum(1).astype(np.float32)
        ns = np.cross(v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]])
        ns = (ns / np.linalg.norm(ns, axis=1, keepdims=True)).astype(np.float32)
    else:
        o, ns = np.empty((n, 3), np.float32), None
        o[:, :2] = rng.uniform(0.0, synth.DIST_MIC_SIDE, (n, 2))
        o[:, 2] = rng.uniform(0.5, 60.0, n)
    return {"kind": kind, "tr": tr, "city": tr.load_geometry(w), "o": o, "d": d, "ns": ns}


# --------------------------------------------------------------------- run
def run(state):
    kind, tr = state["kind"], state["tr"]
    if kind == "trace":
        btrace.bt_trace(tr.ctx, state["sid"], state["params"])
        btrace.bt_read_levels(tr.ctx, state["sid"], state["level"], None, state["count"])
        return {"level": state["level"], "count": state["count"]}
    if kind == "frame":
        btrace.bt_trace_noalloc(tr.ctx, state["sid"], state["params"], state["level"], state["count"])
        return {"level": state["level"], "count": state["count"]}
    if kind == "ingest":
        r = tr.run(state["w"], **state["options"])
        btrace.bt_unload_scene(tr.ctx, r["scene_id"])
        return {"level": r["level"], "intensity": r["I"], "count": r["cnt"]}
    if kind == "query":
        d = serve.run_plain(tr, [state["city"]], [state["query"]], realtime=False)[0]
        return {"level": d.level, "count": d.count}
    if kind == "burst":
        done = state["server"].run(state["queries"], realtime=False)
        return [{"level": d.level, "count": d.count} for d in done]
    if kind == "batch":
        btrace.bt_batch_run(tr.ctx, state["batch"])
        for sid, (level, count) in zip(state["sids"], state["out"]):
            btrace.bt_read_levels(tr.ctx, sid, level, None, count)
        return [{"level": level, "count": count} for level, count in state["out"]]
    t, tri = btrace.bt_cast_rays(tr.ctx, state["city"], state["o"], state["d"], state["ns"])
    return {"t": t, "tri": tri}


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: geometry, sources and microphones read once, levels and counts
    written once.  Operations: for every beam segment one axis-ray query down
    a tree of the triangles (two boxes of 15 operations a level, one triangle
    of 60) and one reflection of the image source, cone and axis (120); on
    these cities about half of the orders are reached."""
    kind = case["kind"]
    bands = case.get("bands", 8)

    def city(b):
        return 40 * b  # triangles

    def cost(tris, lineages, order, sources, mics):
        seg = lineages * (1 + 0.5 * order)
        flops = seg * (2 * 15 * math.log2(tris) + 60 + 120)
        return 36 * tris + (12 + 4 * bands) * sources + mics * (12 + 8 * bands + 4), flops

    if kind == "cast":
        t = city(case["buildings"])
        return {"bytes": 36 * t + case["rays"] * (24 + 8 + (12 if case["reflected"] else 0)),
                "flops": case["rays"] * (2 * 15 * math.log2(t) + 60)}
    if kind == "burst":
        lin = case["queries"] * 5120 * case["max_sources"] / max(1.0, math.log(case["max_sources"]))
        mics = case["queries"] * case["max_mics"] / 3
        parts = [cost(city(2000), lin, 4.5, lin / 5120, mics)]
    elif kind == "batch":
        n = case["cities"]
        parts = [cost(city(b), 20 * 4 ** (3 + i % 4) * s, 2 + (3 * i) % 7, s, m) for i, (b, s, m) in enumerate(
            zip(_uneven(n, 100, 5000), _uneven(n, case["max_sources"], 1), _uneven(n, case["max_mics"], 1000)))]
    else:
        mics = case["side"] ** 2 * case.get("heights", 1)
        tris = 770 if case.get("scene") == "tiny" else city(case["buildings"])
        parts = [cost(tris, 20 * 4 ** case["level"] * case["sources"], case["order"], case["sources"], mics)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """The levels in 64 bits by testing every axis ray against every triangle
    and every microphone against every beam segment, where that is quick."""
    if case["kind"] not in ("trace", "frame") or case["directional"]:
        return None
    rays = case["sources"] * 20 * 4 ** case["level"] * (case["order"] + 1)
    tris = 770 if case["scene"] == "tiny" else 41 * case["buildings"]
    if rays * (tris + case["side"] ** 2 * case["heights"]) > 5e9:
        return None
    w = _workload(case, seed)
    alpha = ALPHA[:case["bands"]] if case["damping"] else None
    return {"level": _levels64(w, case["order"], alpha), "count": None}


def _icosphere(level):
    phi = 0.5 * (1.0 + math.sqrt(5.0))
    v = np.array([(s * a, t * b, 0.0) for s in (-1, 1) for t in (-1, 1) for a, b in ((1.0, phi),)])
    v = np.concatenate([np.roll(v[:, [2, 0, 1]], k, axis=1) for k in range(3)])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    near = v @ v.T > 0.4
    f = [(i, j, k) for i in range(12) for j in range(i + 1, 12) for k in range(j + 1, 12)
         if near[i, j] and near[j, k] and near[i, k]]
    f = [(i, j, k) if np.linalg.det(v[[i, j, k]]) > 0 else (i, k, j) for i, j, k in f]
    c = v[np.array(f)]
    for _ in range(level):
        a, b, d = c[:, 0], c[:, 1], c[:, 2]
        m = [x / np.linalg.norm(x, axis=1, keepdims=True) for x in (a + b, b + d, d + a)]
        c = np.concatenate([np.stack(t, 1) for t in ((a, m[0], m[2]), (m[0], b, m[1]), (m[2], m[1], d), m)])
    return c


def _levels64(w, max_order, alpha):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
    dot = lambda a, b: (a * b).sum(-1)  # noqa: E731
    corner = f64(_icosphere(w.level))
    n_s, n_b = len(w.src), len(corner)
    cone = torch.stack([torch.linalg.cross(corner[:, k], corner[:, (k + 1) % 3]) for k in range(3)], 1)
    axis = torch.nn.functional.normalize(corner.sum(1), dim=-1)
    mic = w.mics.double() if isinstance(w.mics, torch.Tensor) else f64(w.mics)
    tri = f64(w.scene.verts)[torch.as_tensor(w.scene.tris, device=dev).long()]
    refl = f64(w.scene.refl)[torch.as_tensor(w.scene.mat, device=dev).long()]
    v0, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    nrm = torch.nn.functional.normalize(torch.linalg.cross(e1, e2), dim=-1)
    A = f64(w.src).repeat_interleave(n_b, 0)
    P = f64(w.power).repeat_interleave(n_b, 0)
    C, D, O = cone.repeat(n_s, 1, 1), axis.repeat(n_s, 1), A.clone()
    sn, sv, dns = torch.zeros_like(A), torch.zeros_like(A), torch.zeros(len(A), device=dev, dtype=torch.float64)
    out = torch.zeros((len(mic), P.shape[1]), device=dev, dtype=torch.float64)
    for order in range(max_order + 1):
        # the nearest triangle in front of each axis ray
        T = torch.full((len(A),), math.inf, device=dev, dtype=torch.float64)
        hit = torch.full((len(A),), -1, device=dev, dtype=torch.long)
        step = max(1, (1 << 23) // max(1, len(v0)))
        for b in range(0, len(A), step):
            o, d = O[b:b + step, None], D[b:b + step, None]
            p = torch.linalg.cross(d.expand(-1, len(v0), -1), e2.expand(d.shape[0], -1, -1))
            det = dot(e1, p)
            s = o - v0
            u = dot(s, p) / det
            q = torch.linalg.cross(s, e1.expand_as(s))
            v = dot(d, q) / det
            t = dot(e2, q) / det
            g = dns[b:b + step, None]
            ok = (det != 0) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1) & (t > 1e-3) & ((g == 0) | (t * g > 1e-3))
            t = torch.where(ok, t, math.inf)
            best = t.amin(1)
            T[b:b + step] = best
            tied = t <= (best + 1e-9 * (1 + best))[:, None]
            hit[b:b + step] = torch.where(torch.isfinite(best), tied.to(torch.uint8).argmax(1), -1)
        on = hit >= 0
        h = hit.clamp(min=0)
        en = nrm[h] * torch.where(dot(nrm[h], D) < 0, 1.0, -1.0)[:, None]
        # microphones inside each segment
        step = max(1, (1 << 22) // len(mic))
        for b in range(0, len(A), step):
            e = slice(b, b + step)
            v = mic - A[e, None]
            inside = dot(C[e, 0, None], v) >= 0
            for k in (1, 2):
                inside &= dot(C[e, k, None], v) >= 0
            if order:
                inside &= dot(sn[e, None], mic - sv[e, None]) > 0
            inside &= ~on[e, None] | (dot(en[e, None], mic - v0[h[e]][:, None]) >= 0)
            d2 = dot(v, v)
            gain = torch.where(inside, 1.0 / (4.0 * math.pi * d2), 0.0)
            if alpha is None:
                out += gain.T @ P[e]
            else:
                dist = d2.sqrt()
                for k, a in enumerate(alpha):
                    a32 = float(np.float32(a))
                    out[:, k] += (gain * 10.0 ** (-a32 * dist / 10.0)).T @ P[e, k]
        if order == max_order:
            break
        # reflect what hit
        A, C, D, O, P, T, h = A[on], C[on], D[on], O[on], P[on], T[on], h[on]
        n = nrm[h]
        O = O + T[:, None] * D
        A = A - 2 * dot(A - v0[h], n)[:, None] * n
        D = D - 2 * dot(D, n)[:, None] * n
        C = C - 2 * dot(C, n[:, None])[..., None] * n[:, None]
        P = P * refl[h]
        s = dot(n, D)
        sn, sv, dns = n * torch.sign(s)[:, None], v0[h], s.abs()
    return 10.0 * torch.log10(out) + 120.0
