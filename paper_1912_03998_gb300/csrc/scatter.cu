// scatter.cu -- the microphone half of the hot path (Section 2 of the
// paper): a microphone measures a beam when it lies inside the beam's cone,
// past its start plane and before its end plane, and receives the beam's
// per-band intensity W_b prod(r_b) 10^(-alpha_b d / 10) / (4 pi d^2); the
// level readout turns the accumulated intensity into 10 log10(I / 1e-12) dB.
//
//   k_scatter each lane of a warp builds the footprint of one segment record
//             written by the trace kernels; the warp then flattens the
//             (segment, cell row) pairs and the microphone runs of those
//             rows, tests every candidate microphone and adds the beam's
//             intensity with float64 atomics.
//   k_levels  intensity -> level, back to the caller's microphone order.
//
// Precision.  Microphone tests are float32 relative to the apex and are
// re-tested with float pairs when a microphone lies within the rounding band
// of a cone or start/end plane (BT_PREC_MIXED and FP32).  In BT_PREC_FP64
// float32 only sorts out what it finds outside by more than its rounding;
// every other test and every contribution is float64.  Intensity accumulates
// in float64.
#include "bt_internal.cuh"

namespace bt {

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// ------------------------------------------------------- footprint polygon
// Conservative xy footprint of a segment on the microphone slab: each 3D
// half-space a.m >= b becomes, over z in [zlo, zhi], the weaker half-plane
// ax x + ay y >= b - max(az zlo, az zhi), grown by a 1 cm slack; the grid
// rectangle is clipped by those half-planes (Sutherland-Hodgman).
constexpr int kPolyMax = 12;

// A polygon's vertices in one lane's column of a [vertex][32] shared-memory
// array: vertex i at x[32 i], y[32 i].
struct PolyCol {
  float *x, *y;
};

// q = p (n vertices) clipped by ax x + ay y >= b; returns q's vertex count.
// Every vertex's plane value is evaluated once; an edge that crosses the
// line contributes its crossing.
__device__ __forceinline__ int poly_clip(PolyCol p, int n, PolyCol q, float ax, float ay, float b) {
  int m = 0;
  const float f0 = ax * p.x[0] + ay * p.y[0] - b;
  float fi = f0, xi = p.x[0], yi = p.y[0];
  for (int i = 0; i < n; i++) {
    const bool last = i + 1 == n;
    const float xj = last ? p.x[0] : p.x[32 * (i + 1)], yj = last ? p.y[0] : p.y[32 * (i + 1)];
    const float fj = last ? f0 : ax * xj + ay * yj - b;
    if (fi >= 0.0f && m < kPolyMax) { q.x[32 * m] = xi; q.y[32 * m] = yi; m++; }
    if ((fi >= 0.0f) != (fj >= 0.0f) && m < kPolyMax) {
      // fi and fj have opposite signs, so |fi - fj| >= |fi| > 0
      const float t = __fdividef(fi, fi - fj);
      q.x[32 * m] = xi + t * (xj - xi);
      q.y[32 * m] = yi + t * (yj - yi);
      m++;
    }
    fi = fj; xi = xj; yi = yj;
  }
  return m;
}

// Clip polygon P (n vertices) by the relaxation of a.m >= b into Q and swap
// the two; returns false when the footprint is empty.
__device__ __forceinline__ bool poly_halfspace(PolyCol &P, PolyCol &Q, int &n, float3 a, float b, float zl, float zh) {
  if (!(b > -kInf)) return true;  // missing plane
  float bz = fmaxf(a.z * zl, a.z * zh);
  float axy = fabsf(a.x) + fabsf(a.y);
  float bb = b - bz - 0.01f * axy - 1e-6f * fabsf(b);
  if (axy == 0.0f) return bb <= 0.0f;
  n = poly_clip(P, n, Q, a.x, a.y, bb);
  PolyCol t = P;
  P = Q;
  Q = t;
  return n >= 3;
}

// Footprint of segment s over layer `layer` of the grid (the whole height
// slab when the grid has one layer), built in the columns A and B; returns
// its vertex count (0 if it is empty) with the polygon left in A.  Planes
// are relative to the apex: n . (m - A) >= w  <=>  n . m >= w + n . A.
// Reads only the apex, the cone normals and the start and end planes of s.
__device__ __forceinline__ int seg_footprint(const Seg &s, const MicGrid &g, int layer, PolyCol A, PolyCol B) {
  float zl = g.zlo, zh = g.zhi;
  if (g.nz > 1) {
    zl = fmaxf(g.zlo, g.z0 + layer * g.dz) - 1e-3f;
    zh = fminf(g.zhi, g.z0 + (layer + 1) * g.dz) + 1e-3f;
  }
  float m = 0.01f;
  float X0 = g.x0 - m, X1 = g.x0 + g.cw * g.nx + m, Y0 = g.y0 - m, Y1 = g.y0 + g.ch * g.ny + m;
  PolyCol P = A, Q = B;
  int n = 4;
  P.x[0] = X0; P.y[0] = Y0;
  P.x[32] = X1; P.y[32] = Y0;
  P.x[64] = X1; P.y[64] = Y1;
  P.x[96] = X0; P.y[96] = Y1;
  float3 ap = make_float3(s.ahi[0], s.ahi[1], s.ahi[2]);
  float3 n0 = f3(s.n0), n1 = f3(s.n1), n2 = f3(s.n2);
  float3 ns = f3(s.start), ne = f3(s.end);
  if (!poly_halfspace(P, Q, n, n0, dot3(n0, ap), zl, zh)) return 0;
  if (!poly_halfspace(P, Q, n, n1, dot3(n1, ap), zl, zh)) return 0;
  if (!poly_halfspace(P, Q, n, n2, dot3(n2, ap), zl, zh)) return 0;
  if (!poly_halfspace(P, Q, n, ns, s.start.w + dot3(ns, ap), zl, zh)) return 0;
  if (!poly_halfspace(P, Q, n, ne, s.end.w + dot3(ne, ap), zl, zh)) return 0;
  if (P.x != A.x) {
    for (int i = 0; i < n; i++) { A.x[32 * i] = P.x[32 * i]; A.y[32 * i] = P.y[32 * i]; }
  }
  return n;
}

// ------------------------------------------------------------------ scatter
// Per-warp shared state of the scatter: 32 segments, one per lane, stored as
// [field][lane] so that lanes reading different segments hit different banks.
// The rows hold what every candidate reads; what only the rare float-pair
// re-tests (and every FP64 test) need -- the cone normals' low parts, the
// apex's third word, the start and end planes' triangle slots -- is read
// from the segment record (F_SI) when needed.
constexpr int kScatterWarps = 4;
enum : int {
  F_AX = 0, F_RX = 3, F_N0 = 6, F_NS = 15, F_NE = 19, F_P = 23, F_SI = 31, F_CY0 = 32, F_PN = 33,
  F_VI = 34, F_LAYER = 35, F_PX = 36, F_PY = F_PX + kPolyMax,
  // batches only: the view's microphone array, accumulators and band count
  // (plus an air-damping flag), read for every candidate
  F_MP = F_PY + kPolyMax, F_EP = F_MP + 2, F_CP = F_EP + 2, F_FL = F_CP + 2, F_COUNT = F_FL + 1
};
// While a lane clips its footprint, its columns of the rows below F_PX
// (written only afterwards) hold the clip's second vertex buffer.
constexpr int F_QX = 0, F_QY = kPolyMax;
static_assert(F_QY + kPolyMax <= F_PX, "clip scratch overlaps the polygon rows");
// Rows a variant needs: 60 for one scene, 67 for a batch, either way six
// 128-thread blocks per SM.
template <bool kBatch>
constexpr int scatter_rows() {
  return kBatch ? F_COUNT : F_MP;
}
template <bool kBatch>
struct ScatterSmem {
  float f[kScatterWarps][scatter_rows<kBatch>()][32];
};

// A pointer kept as two float rows (bit patterns).
__device__ __forceinline__ void put_ptr(float (*F)[32], int row, unsigned lane, const void *p) {
  const unsigned long long u = (unsigned long long)p;
  F[row][lane] = __uint_as_float((unsigned)u);
  F[row + 1][lane] = __uint_as_float((unsigned)(u >> 32));
}
template <typename T>
__device__ __forceinline__ T *get_ptr(const float (*F)[32], int row, int s) {
  return (T *)((unsigned long long)__float_as_uint(F[row][s]) |
               ((unsigned long long)__float_as_uint(F[row + 1][s]) << 32));
}

__device__ __forceinline__ int warp_incl_scan(int v, unsigned lane) {
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, v, o);
    if ((int)lane >= o) v += y;
  }
  return v;
}

// Largest lane whose exclusive prefix is <= i (the owner of item i).
__device__ __forceinline__ int warp_owner(int excl, int i) {
  int owner = 0;
  for (int step = 16; step >= 1; step >>= 1) {
    int ex = __shfl_sync(0xffffffffu, excl, owner + step);
    if (ex <= i) owner += step;
  }
  return owner;
}

// m - apex as float pairs (apex hi in F[F_AX..], lo parts in F[F_RX..])
__device__ __forceinline__ df3 rel_df(const float (*F)[32], int s, float4 m) {
  return df3_sub(mkdf3(make_float3(m.x, m.y, m.z)),
                 df3{df{F[F_AX][s], F[F_RX][s]}, df{F[F_AX + 1][s], F[F_RX + 1][s]}, df{F[F_AX + 2][s], F[F_RX + 2][s]}});
}

// Signed distance of m from the plane of leaf slot `slot` as a float pair,
// oriented like the float32 normal `nf` of the segment record.
__device__ __forceinline__ float plane_side_df(const SceneView &a, int slot, float3 nf, float4 m) {
  PlaneDF pd = a.sc.planes_df[slot];
  float4 v0 = __ldg(&a.sc.tris[slot].v0);
  df3 n = df3{df{pd.hi.x, pd.lo.x}, df{pd.hi.y, pd.lo.y}, df{pd.hi.z, pd.lo.z}};
  df3 rel = df3_sub(mkdf3(make_float3(m.x, m.y, m.z)), mkdf3(f3(v0)));
  df e = df3_dot(n, rel);
  float sg = pd.hi.x * nf.x + pd.hi.y * nf.y + pd.hi.z * nf.z < 0.0f ? -1.0f : 1.0f;
  return sg * (e.hi + e.lo);
}

// Signed distance of m from the float64 plane of leaf slot `slot`, oriented
// like the float32 normal `nf` of the segment record (FP64 mode).
__device__ __forceinline__ double plane_side64(const SceneView &a, int slot, float3 nf, float4 m) {
  Plane64 pl = ldg_d4(&a.sc.planes64[slot]);
  double e = pl.x * (double)m.x + pl.y * (double)m.y + pl.z * (double)m.z - pl.w;
  return pl.x * nf.x + pl.y * nf.y + pl.z * nf.z < 0.0 ? -e : e;
}

// FP64: test microphone e.x against segment record e.y and add its
// contribution, all in float64 (apex exact from its three words, cone normals
// from their float pairs, start and end planes from the triangles' float64
// planes).  1 if it contributed.
template <bool kBatch>
__device__ __forceinline__ int contribute64(const ScatterArgs &a, int2 e) {
  const Seg *const rec = a.segs + e.y;
  const SceneView &V = kBatch ? a.views[rec->view] : a.v;
  const float4 m = __ldg(&V.mics[e.x]);
  const float4 n0 = __ldg(&rec->n0), n1 = __ldg(&rec->n1), n2 = __ldg(&rec->n2);
  const float4 st = __ldg(&rec->start), en = __ldg(&rec->end);
  double3 vd;
  vd.x = (double)m.x - (((double)__ldg(&rec->ahi[0]) + __ldg(&rec->alo[0])) + __ldg(&rec->pad[0]));
  vd.y = (double)m.y - (((double)__ldg(&rec->ahi[1]) + __ldg(&rec->alo[1])) + __ldg(&rec->pad[1]));
  vd.z = (double)m.z - (((double)__ldg(&rec->ahi[2]) + __ldg(&rec->alo[2])) + __ldg(&rec->pad[2]));
  const float3 nh[3] = {f3(n0), f3(n1), f3(n2)};
  bool in = true;
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const double3 nd = make_double3((double)nh[j].x + __ldg(&rec->nlo[3 * j]), (double)nh[j].y + __ldg(&rec->nlo[3 * j + 1]),
                                    (double)nh[j].z + __ldg(&rec->nlo[3 * j + 2]));
    in = in && dot3(nd, vd) >= 0.0;
  }
  if (in) {
    const int s_slot = __float_as_int(n0.w), e_slot = __float_as_int(n1.w);
    const double fs = s_slot >= 0 ? plane_side64(V, s_slot, f3(st), m) : 1.0;
    const double fe = e_slot >= 0 ? plane_side64(V, e_slot, f3(en), m) : 1.0;
    in = fs > 0.0 && fe >= 0.0;
  }
  const double d2 = dot3(vd, vd);
  if (!(in && d2 > 1e-18)) return 0;
  const double gf = 1.0 / (4.0 * 3.141592653589793 * d2);
  const bool has_alpha = V.has_alpha != 0;
  const double dist = has_alpha ? sqrt(d2) : 0.0;
  const float4 p0 = __ldg(&rec->p03), p1 = __ldg(&rec->p47);
  const float p[kMaxBands] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
  double *const out = V.energy + (size_t)e.x * kMaxBands;
  const int nb = V.sc.n_bands;
#pragma unroll
  for (int b = 0; b < kMaxBands; b++) {
    if (b < nb) {
      double c = (double)p[b] * gf;
      if (has_alpha) c *= exp2((double)V.alpha_log2[b] * dist);
      atomicAdd(out + b, c);
    }
  }
  atomicAdd(V.count + e.x, 1);
  return 1;
}

// One warp takes 32 segments at a time.  Each lane loads one segment and
// builds its footprint; the warp then walks the (segment, cell row) pairs of
// all 32 footprints 32 at a time, turns each into its run of microphones, and
// walks the runs 32 candidates at a time, so every lane has work whatever
// the footprint sizes.
template <bool kF64, bool kBatch>
__global__ void __launch_bounds__(32 * kScatterWarps) k_scatter(ScatterArgs a) {
  __shared__ ScatterSmem<kBatch> sm;
  const unsigned lane = lane_id();
  const int w = threadIdx.x >> 5;
  float(*F)[32] = sm.f[w];
  const long long n_seg = (long long)min(*a.seg_count, a.seg_capacity);
  // work items: (segment, microphone layer) pairs; one per segment when the
  // microphones lie in one layer.  By groups of 32 segments, layer by layer: a
  // warp then takes one layer of 32 neighbours and not the 32 layers of one
  // segment, which for a long beam over the roofs hold tens of thousands of
  // candidates (13.75 M microphones, 8 sources: 40 % of the chip's time went
  // by waiting for such warps; 10.1 -> 5.9 ms, 40 sources 29.9 -> 24.6 ms).
  // Only layers that hold microphones count, and fewer items are taken where the
  // microphones crowd (mic_layers).
  int n_layers = 1, most_log2 = 5;
  if (a.max_nz > 1) {
    if (kBatch) {
      n_layers = a.max_nz;
      for (int v = lane; v < a.n_views; v += 32) most_log2 = min(most_log2, a.views[v].grid->take_log2);
      most_log2 = (int)__reduce_min_sync(0xffffffffu, (unsigned)most_log2);
    } else {
      n_layers = a.v.grid->n_lay;
      most_log2 = a.v.grid->take_log2;
    }
  }
  const long long n_items = n_layers > 1 ? (n_seg + 31) / 32 * 32 * n_layers : n_seg;
  unsigned long long n_cand = 0, n_contrib = 0;
  // FP64: candidates that wait for their float64 test, (microphone, segment),
  // tested 32 at a time: whole-warp float64 instructions cost the same for one
  // lane as for 32, and one candidate in ten comes this far (24 district
  // sources: 1.07 -> 0.32 ms)
  __shared__ int2 wait_q[kF64 ? kScatterWarps : 1][kF64 ? 64 : 1];
  int2 *const wait = wait_q[kF64 ? w : 0];
  int n_wait = 0;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  // Items a warp takes at a time: 32, one per lane, and fewer once less than
  // that is left for every warp.  The first take is the warp's own, the
  // others come from the launch's counter.  Segments differ by orders of
  // magnitude -- a wide beam over open ground holds thousands of candidates,
  // which a warp tests 32 at a time -- so with fixed shares a launch lasted as
  // long as its fullest warp (eight uneven cities, 4.4 M segments: batch call
  // 5.0 -> 4.3 ms; 17,700 segments of 28 candidates each on average: 617 -> 121
  // us).  The next take is under way while a warp works.
  auto share = [&](long long left) {
    int lg = most_log2;
    while (lg > 0 && left < n_warps << lg) lg--;
    return lg;
  };
  const long long warp0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  int lg = share(n_items);
  const long long own = n_warps << lg;  // items of the first takes
  unsigned long long taken = 0;
  for (long long base = warp0 << lg; base < n_items;) {
    const unsigned per = 1u << lg;
    const int lg_next = share(n_items - max(base, own));
    if (lane == 0 && own < n_items) taken = own + atomicAdd(a.next, 1ull << lg_next);
    // ---- 1. one item per lane: segment parameters and the layer's footprint
    const long long it = base + lane;
    long long ii = it;
    int layer = 0;
    if (n_layers > 1) {
      const long long group = it / (32 * n_layers);
      const int rest = (int)(it - group * (32 * n_layers));
      layer = rest >> 5;
      ii = group * 32 + (rest & 31);
    }
    // the segment record: in order of place when the scene orders its scatter
    const long long si = a.order && ii < n_seg ? (long long)__ldg(&a.order[ii]) : ii;
    int nrows = 0;
    if (lane < per && ii < n_seg) {
      // the footprint needs the apex, the cone normals and the start and end
      // planes (the record's first 112 bytes); the rest is read only for a
      // non-empty footprint
      Seg sl;
      const float4 *src4 = reinterpret_cast<const float4 *>(a.segs + si);
      float4 *dst4 = reinterpret_cast<float4 *>(&sl);
#pragma unroll
      for (int q = 0; q < 7; q++) dst4[q] = __ldg(src4 + q);
      const int vi = kBatch ? sl.view : 0;
      const MicGrid &g = *(kBatch ? a.views[vi] : a.v).grid;
      // the footprint is clipped in the lane's own columns: the polygon rows
      // and, as scratch, the rows of the segment fields written below
      if (a.max_nz > 1) layer = layer < g.n_lay ? (int)g.lay[layer] : g.nz;
      const int pn = layer < g.nz ? seg_footprint(sl, g, layer, PolyCol{&F[F_PX][lane], &F[F_PY][lane]},
                                                  PolyCol{&F[F_QX][lane], &F[F_QY][lane]})
                                  : 0;
      int cy0 = 0, cy1 = -1;
      if (pn > 0) {
        float ymin = kInf, ymax = -kInf;
        for (int i = 0; i < pn; i++) { ymin = fminf(ymin, F[F_PY + i][lane]); ymax = fmaxf(ymax, F[F_PY + i][lane]); }
        if (ymin <= ymax) {
          cy0 = clampi((int)floorf((ymin - g.y0) * g.inv_ch), 0, g.ny - 1);
          cy1 = clampi((int)floorf((ymax - g.y0) * g.inv_ch), 0, g.ny - 1);
        }
      }
      nrows = cy1 >= cy0 ? cy1 - cy0 + 1 : 0;
      if (nrows > 0) {
        // band powers (p03, p47); the normals' low parts stay in the record
        dst4[7] = __ldg(src4 + 7);
        dst4[8] = __ldg(src4 + 8);
        F[F_VI][lane] = __int_as_float(vi);
        F[F_SI][lane] = __int_as_float((int)si);
        if (kBatch) {
          const SceneView &V = a.views[vi];
          put_ptr(F, F_MP, lane, V.mics);
          put_ptr(F, F_EP, lane, V.energy);
          put_ptr(F, F_CP, lane, V.count);
          F[F_FL][lane] = __int_as_float(V.sc.n_bands | (V.has_alpha ? 0x100 : 0));
        }
        F[F_LAYER][lane] = __int_as_float(layer);
        for (int q = 0; q < 3; q++) {
          F[F_AX + q][lane] = sl.ahi[q];
          F[F_RX + q][lane] = sl.alo[q];
        }
        F[F_N0][lane] = sl.n0.x; F[F_N0 + 1][lane] = sl.n0.y; F[F_N0 + 2][lane] = sl.n0.z;
        F[F_N0 + 3][lane] = sl.n1.x; F[F_N0 + 4][lane] = sl.n1.y; F[F_N0 + 5][lane] = sl.n1.z;
        F[F_N0 + 6][lane] = sl.n2.x; F[F_N0 + 7][lane] = sl.n2.y; F[F_N0 + 8][lane] = sl.n2.z;
        F[F_NS][lane] = sl.start.x; F[F_NS + 1][lane] = sl.start.y; F[F_NS + 2][lane] = sl.start.z;
        F[F_NS + 3][lane] = sl.start.w;
        F[F_NE][lane] = sl.end.x; F[F_NE + 1][lane] = sl.end.y; F[F_NE + 2][lane] = sl.end.z;
        F[F_NE + 3][lane] = sl.end.w;
        F[F_P][lane] = sl.p03.x; F[F_P + 1][lane] = sl.p03.y; F[F_P + 2][lane] = sl.p03.z;
        F[F_P + 3][lane] = sl.p03.w; F[F_P + 4][lane] = sl.p47.x; F[F_P + 5][lane] = sl.p47.y;
        F[F_P + 6][lane] = sl.p47.z; F[F_P + 7][lane] = sl.p47.w;
        F[F_CY0][lane] = __int_as_float(cy0);
        F[F_PN][lane] = __int_as_float(pn);
      }
    }
    __syncwarp();
    // ---- 2. (segment, row) pairs of the 32 footprints, 32 at a time
    const int rincl = warp_incl_scan(nrows, lane);
    const int total_rows = __shfl_sync(0xffffffffu, rincl, 31);
    const int rexcl = rincl - nrows;
    for (int rb = 0; rb < total_rows; rb += 32) {
      int r = rb + (int)lane;
      int so = warp_owner(rexcl, r);  // segment lane owning pair r
      int so_excl = __shfl_sync(0xffffffffu, rexcl, so);
      int first = 0, cnt = 0;
      if (r < total_rows) {
        const SceneView &V = kBatch ? a.views[__float_as_int(F[F_VI][so])] : a.v;
        const MicGrid &g = *V.grid;
        int row = __float_as_int(F[F_CY0][so]) + (r - so_excl);
        float ya = g.y0 + row * g.ch, yb = ya + g.ch;
        float my = 1e-3f * g.ch;
        // x extent of the owner's footprint within the row's strip
        int pn = __float_as_int(F[F_PN][so]);
        float xmin = kInf, xmax = -kInf;
        float y0s = ya - my, y1s = yb + my;
        for (int i = 0; i < pn; i++) {
          int j = i + 1 == pn ? 0 : i + 1;
          float xi = F[F_PX + i][so], yi = F[F_PY + i][so], xj = F[F_PX + j][so], yj = F[F_PY + j][so];
          if (yi >= y0s && yi <= y1s) { xmin = fminf(xmin, xi); xmax = fmaxf(xmax, xi); }
          // crossings of the strip's edges; yi != yj whenever an edge
          // crosses, and the quotient lies in [0, 1]
          if ((yi < y0s) != (yj < y0s)) {
            float x = xi + __fdividef(y0s - yi, yj - yi) * (xj - xi);
            xmin = fminf(xmin, x); xmax = fmaxf(xmax, x);
          }
          if ((yi < y1s) != (yj < y1s)) {
            float x = xi + __fdividef(y1s - yi, yj - yi) * (xj - xi);
            xmin = fminf(xmin, x); xmax = fmaxf(xmax, x);
          }
        }
        if (xmin <= xmax) {
          int cx0 = clampi((int)floorf((xmin - g.x0) * g.inv_cw), 0, g.nx - 1);
          int cx1 = clampi((int)floorf((xmax - g.x0) * g.inv_cw), 0, g.nx - 1);
          const int cell0 = (__float_as_int(F[F_LAYER][so]) * g.ny + row) * g.nx;
          first = __ldg(&V.cell_start[cell0 + cx0]);
          cnt = __ldg(&V.cell_start[cell0 + cx1 + 1]) - first;
        }
      }
      // ---- 3. candidates of those runs, 32 at a time
      const int cincl = warp_incl_scan(cnt, lane);
      const int total_c = __shfl_sync(0xffffffffu, cincl, 31);
      const int cexcl = cincl - cnt;
      for (int cb = 0; cb < total_c; cb += 32) {
        int c = cb + (int)lane;
        int ro = warp_owner(cexcl, c);
        int ofirst = __shfl_sync(0xffffffffu, first, ro);
        int oexcl = __shfl_sync(0xffffffffu, cexcl, ro);
        int s = __shfl_sync(0xffffffffu, so, ro);
        [[maybe_unused]] bool near = false;
        [[maybe_unused]] int2 entry = make_int2(0, 0);
        if (c < total_c) {
          int mi = ofirst + (c - oexcl);
          // where the contribution goes: the scene's accumulators, band
          // count and air damping (kernel parameters for one scene, the
          // segment's rows in a batch)
          const float4 *mics;
          double *energy;
          int *count;
          int nb;
          bool has_alpha;
          if (kBatch) {
            mics = get_ptr<const float4>(F, F_MP, s);
            energy = get_ptr<double>(F, F_EP, s);
            count = get_ptr<int>(F, F_CP, s);
            const int fl = __float_as_int(F[F_FL][s]);
            nb = fl & 0xff;
            has_alpha = (fl & 0x100) != 0;
          } else {
            mics = a.v.mics;
            energy = a.v.energy;
            count = a.v.count;
            nb = a.v.sc.n_bands;
            has_alpha = a.v.has_alpha != 0;
          }
          const Seg *rec = a.segs + __float_as_int(F[F_SI][s]);
          float4 m = __ldg(&mics[mi]);
          // m - apex with the apex as hi + lo: one extra rounding at most
          float3 v = make_float3((m.x - F[F_AX][s]) - F[F_RX][s], (m.y - F[F_AX + 1][s]) - F[F_RX + 1][s],
                                 (m.z - F[F_AX + 2][s]) - F[F_RX + 2][s]);
          n_cand++;
          if (kF64) {
            // FP64: a candidate that float32 finds outside by more than its
            // rounding is outside; the rest wait for float64.  With v the
            // microphone from the apex, u = 2^-24 and |.| the sum of magnitudes:
            // v and the normals n are rounded to u, a dot product of three
            // terms to 3 u |n||v|, so a cone plane's value errs by at most
            // 5 u |n||v| = 3e-7 |n||v| against 2e-6.  Start and end planes: the
            // same with |n| < 1.8, and the offset, formed in float64 with the
            // float64 normal, rounded to u of itself (within the slack, of at
            // most 1.8 |v|): 7e-7 |v| against 4e-6 |v| + 1 mm, whatever the
            // size of the triangle and its distance.
            const float v1 = fabsf(v.x) + fabsf(v.y) + fabsf(v.z), side = 1e-3f + 4e-6f * v1;
            near = true;
#pragma unroll
            for (int j = 0; j < 3; j++) {
              const float3 nj = make_float3(F[F_N0 + 3 * j][s], F[F_N0 + 3 * j + 1][s], F[F_N0 + 3 * j + 2][s]);
              near = near && dot3(nj, v) >= -2e-6f * v1 * (fabsf(nj.x) + fabsf(nj.y) + fabsf(nj.z));
            }
            const float3 ns = make_float3(F[F_NS][s], F[F_NS + 1][s], F[F_NS + 2][s]);
            const float3 ne = make_float3(F[F_NE][s], F[F_NE + 1][s], F[F_NE + 2][s]);
            near = near && dot3(ns, v) - F[F_NS + 3][s] >= -side && dot3(ne, v) - F[F_NE + 3][s] >= -side;
            if (near) entry = make_int2(mi, __float_as_int(F[F_SI][s]));
          } else {
            // cone planes: float32; within the rounding band of a plane the
            // test is redone with float pairs
            const float band_v = 2e-6f * (fabsf(v.x) + fabsf(v.y) + fabsf(v.z));
            bool in = true;
#pragma unroll
            for (int j = 0; j < 3; j++) {
              float3 nj = make_float3(F[F_N0 + 3 * j][s], F[F_N0 + 3 * j + 1][s], F[F_N0 + 3 * j + 2][s]);
              float e = dot3(nj, v);
              if (fabsf(e) <= band_v * (fabsf(nj.x) + fabsf(nj.y) + fabsf(nj.z))) {
                df3 nd = df3{df{nj.x, __ldg(&rec->nlo[3 * j])}, df{nj.y, __ldg(&rec->nlo[3 * j + 1])},
                             df{nj.z, __ldg(&rec->nlo[3 * j + 2])}};
                df ed = df3_dot(nd, rel_df(F, s, m));
                e = ed.hi + ed.lo;
              }
              in = in && e >= 0.0f;
            }
            if (in) {
              // start/end planes: float32 relative to the apex; within the
              // rounding band the test is redone with float pairs against the
              // triangle's own plane, the form the definition uses
              float3 ns = make_float3(F[F_NS][s], F[F_NS + 1][s], F[F_NS + 2][s]);
              float3 ne = make_float3(F[F_NE][s], F[F_NE + 1][s], F[F_NE + 2][s]);
              float band = 1e-4f + 1e-6f * (fabsf(v.x) + fabsf(v.y) + fabsf(v.z));
              float fs = dot3(ns, v) - F[F_NS + 3][s], fe = dot3(ne, v) - F[F_NE + 3][s];
              if (fabsf(fs) <= band || fabsf(fe) <= band) {
                const SceneView &V = kBatch ? a.views[__float_as_int(F[F_VI][s])] : a.v;
                int s_slot = __float_as_int(__ldg(&rec->n0.w)), e_slot = __float_as_int(__ldg(&rec->n1.w));
                if (fabsf(fs) <= band && s_slot >= 0) fs = plane_side_df(V, s_slot, ns, m);
                if (fabsf(fe) <= band && e_slot >= 0) fe = plane_side_df(V, e_slot, ne, m);
              }
              in = fs > 0.0f && fe >= 0.0f;
            }
            float d2 = dot3(v, v);
            if (in && d2 > 1e-18f) {
              float gf = 1.0f / (4.0f * 3.14159265358979f * d2);
              float dist = has_alpha ? sqrtf(d2) : 0.0f;
              double *e = energy + (size_t)mi * kMaxBands;
              if (has_alpha) {
                const float *alpha = (kBatch ? a.views[__float_as_int(F[F_VI][s])] : a.v).alpha_log2;
#pragma unroll
                for (int b = 0; b < kMaxBands; b++)
                  if (b < nb) atomicAdd(e + b, (double)(F[F_P + b][s] * gf * exp2f(alpha[b] * dist)));
              } else {
#pragma unroll
                for (int b = 0; b < kMaxBands; b++)
                  if (b < nb) atomicAdd(e + b, (double)(F[F_P + b][s] * gf));
              }
              atomicAdd(&count[mi], 1);
              n_contrib++;
            }
          }
        }
        if (kF64) {
          const unsigned b = __ballot_sync(0xffffffffu, near);
          if (near) wait[n_wait + __popc(b & ((1u << lane) - 1u))] = entry;
          n_wait += __popc(b);
          if (n_wait >= 32) {
            __syncwarp();
            n_contrib += contribute64<kBatch>(a, wait[lane]);
            n_wait -= 32;
            const int2 rest = wait[32 + lane];
            __syncwarp();
            wait[lane] = rest;
            __syncwarp();
          }
        }
      }
    }
    __syncwarp();
    if (own >= n_items) break;
    base = (long long)__shfl_sync(0xffffffffu, taken, 0);
    lg = lg_next;
  }
  __syncwarp();
  if (kF64 && (int)lane < n_wait) n_contrib += contribute64<kBatch>(a, wait[lane]);
  for (int o = 16; o > 0; o >>= 1) {
    n_cand += __shfl_xor_sync(0xffffffffu, n_cand, o);
    n_contrib += __shfl_xor_sync(0xffffffffu, n_contrib, o);
  }
  if (lane == 0) {
    atomicAdd(&a.ctr->candidates, n_cand);
    atomicAdd(&a.ctr->contributions, n_contrib);
  }
}

// ------------------------------------------------------ order of place
// With microphones through a whole volume, the accumulators and positions
// are many times the L2; segments taken in the order they were traced reach
// microphones all over the city, so nearly every atomic update and position
// load goes to HBM.  Taken in order of the cell under each segment (bins of
// 2^kOrderBits x 2^kOrderBits cells along a Morton curve), the warps
// resident at any time work in one neighbourhood and its accumulators stay
// in L2.  A counting sort: bin histogram, exclusive scan, placement; the
// order within a bin is immaterial (every contribution is added, whatever
// the order).
__device__ __forceinline__ int order_bin(const MicGrid &g, int key) {
  const unsigned x = ((unsigned)(key & 0xffff) << kOrderBits) / (unsigned)max(g.nx, 1);
  const unsigned y = ((unsigned)key >> 16 << kOrderBits) / (unsigned)max(g.ny, 1);
  unsigned m = 0;
#pragma unroll
  for (int b = 0; b < kOrderBits; b++) m |= ((x >> b) & 1u) << (2 * b) | ((y >> b) & 1u) << (2 * b + 1);
  return (int)(m & (kOrderBins - 1));
}

__global__ void __launch_bounds__(256) k_order_hist(const Seg *segs, const unsigned long long *seg_count,
                                                    unsigned long long cap, const MicGrid *grid, uint32_t *hist) {
  __shared__ uint32_t h[kOrderBins];
  for (int i = threadIdx.x; i < kOrderBins; i += blockDim.x) h[i] = 0u;
  __syncthreads();
  const MicGrid g = *grid;
  const long long n = (long long)min(*seg_count, cap);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    atomicAdd(&h[order_bin(g, __ldg(&segs[i].key))], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < kOrderBins; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Exclusive scan of the kOrderBins counts in place, one block.
__global__ void __launch_bounds__(1024) k_order_scan(uint32_t *hist) {
  constexpr int kPer = kOrderBins / 1024;
  __shared__ uint32_t part[1024];
  uint32_t v[kPer], sum = 0;
#pragma unroll
  for (int q = 0; q < kPer; q++) {
    v[q] = hist[threadIdx.x * kPer + q];
    sum += v[q];
  }
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const uint32_t y = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0u;
    __syncthreads();
    part[threadIdx.x] += y;
    __syncthreads();
  }
  uint32_t run = part[threadIdx.x] - sum;
#pragma unroll
  for (int q = 0; q < kPer; q++) {
    hist[threadIdx.x * kPer + q] = run;
    run += v[q];
  }
}

// Each record index to its bin's next place; lanes of a warp with the same
// bin take their places with one atomic.
__global__ void __launch_bounds__(256) k_order_place(const Seg *segs, const unsigned long long *seg_count,
                                                     unsigned long long cap, const MicGrid *grid, uint32_t *offs,
                                                     uint32_t *order) {
  const MicGrid g = *grid;
  const long long n = (long long)min(*seg_count, cap);
  const unsigned lane = lane_id();
  for (long long b0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) & ~31ll; b0 < n;
       b0 += (long long)gridDim.x * blockDim.x) {
    const long long i = b0 + lane;
    const bool ok = i < n;
    const int bin = ok ? order_bin(g, __ldg(&segs[i].key)) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, bin);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (ok && (int)lane == leader) base = atomicAdd(&offs[bin], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (ok) order[base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
  }
}

cudaError_t launch_seg_order(cudaStream_t st, const Seg *segs, const unsigned long long *seg_count,
                             unsigned long long cap, const MicGrid *grid, uint32_t *hist, uint32_t *order, int n_sm) {
  static_assert(kOrderBins % 1024 == 0, "scan layout");
  cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(uint32_t) * kOrderBins, st);
  if (e != cudaSuccess) return e;
  const int blocks = n_sm * 4;
  k_order_hist<<<blocks, 256, 0, st>>>(segs, seg_count, cap, grid, hist);
  k_order_scan<<<1, 1024, 0, st>>>(hist);
  k_order_place<<<blocks, 256, 0, st>>>(segs, seg_count, cap, grid, hist, order);
  note_launches(3);
  return cudaGetLastError();
}

template <bool kF64, bool kBatch>
static cudaError_t launch_scatter_t(cudaStream_t st, const ScatterArgs &a, int n_sm) {
  static OccCache occ;
  int per_sm = 0;
  cudaError_t e = occ.get(&per_sm, k_scatter<kF64, kBatch>, 32 * kScatterWarps);
  if (e != cudaSuccess) return e;
  k_scatter<kF64, kBatch><<<n_sm * per_sm, 32 * kScatterWarps, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_scatter(cudaStream_t st, const ScatterArgs &a, int n_sm) {
  cudaError_t e;
  if (a.views) e = a.fp64 ? launch_scatter_t<true, true>(st, a, n_sm) : launch_scatter_t<false, true>(st, a, n_sm);
  else e = a.fp64 ? launch_scatter_t<true, false>(st, a, n_sm) : launch_scatter_t<false, false>(st, a, n_sm);
  note_launches(1);
  return e;
}

// ------------------------------------------------------------------ levels
// L = 10 log10(I / 1e-12) dB; -inf where no beam reached the microphone.
//
// One thread per microphone and band.  The logarithm is table-driven (after
// Tang, "Table-driven implementation of the logarithm function", 1990):
// I = 2^e m with c ~ 1/m from the mantissa's seven leading bits, r = m c - 1
// (|r| < 2^-8, one fused multiply-add), L = 10 log10(2) e + (120 - 10 log10 c)
// + 10 log10(1 + r), the series' terms from r^4 on in float32.  The two large
// terms are split so that their leading parts add without rounding, and all
// else is below 0.02: one rounding at the size of the result.  That is 10
// float64 operations against some 35 of the library logarithm, and float64
// issue is what bounds this kernel on GB300 (13.75 M microphones x 8 bands:
// 6.7 ms, 0.4 ms of it memory).  Against 50-digit arithmetic over 1e-18..1e2
// W/m^2 its largest error is 1.42e-14 dB, half a unit in the last place, and its
// root mean square 3.5e-15 (the rounded 10 log10(I) + 120: 1.47e-14 and 6.1e-15).
struct LevelEntry {
  double c, hi, lo;  // hi + lo = 120 - 10 log10(c), hi a multiple of 2^-17
};
__device__ const LevelEntry c_level_tab[128] = {
    {0x1.fe01fep-1, 0x1.e01156p+6, 0x1.065c61b4a559ap-19}, {0x1.fa11cap-1, 0x1.e033dp+6, -0x1.41d50cee7acccp-24},
    {0x1.f6310ap-1, 0x1.e05606p+6, -0x1.d2bf4682256fcp-20}, {0x1.f25f64p-1, 0x1.e077f8p+6, 0x1.da73e3c8d5202p-21},
    {0x1.ee9c8p-1, 0x1.e099aap+6, -0x1.db104f983811fp-19}, {0x1.eae808p-1, 0x1.e0bb1ap+6, -0x1.cf888eac8a48bp-19},
    {0x1.e741aap-1, 0x1.e0dc4ap+6, -0x1.7d9a79dd9c438p-19}, {0x1.e3a918p-1, 0x1.e0fd3ap+6, 0x1.b7b999b5145d1p-20},
    {0x1.e01e02p-1, 0x1.e11deep+6, -0x1.7a96848d41e9ap-20}, {0x1.dca01ep-1, 0x1.e13e64p+6, -0x1.244a53ef3e708p-20},
    {0x1.d92f22p-1, 0x1.e15e9ep+6, -0x1.9b55a0e639356p-20}, {0x1.d5cac8p-1, 0x1.e17e9cp+6, 0x1.be8e9f4b58e98p-22},
    {0x1.d272cap-1, 0x1.e19e6p+6, 0x1.09f54d7654a34p-21}, {0x1.cf26e6p-1, 0x1.e1bdeap+6, 0x1.ccede9987c72dp-20},
    {0x1.cbe6dap-1, 0x1.e1dd3cp+6, -0x1.6a3dc703daca1p-22}, {0x1.c8b266p-1, 0x1.e1fc56p+6, -0x1.559dfd69877f7p-19},
    {0x1.c5894ep-1, 0x1.e21b38p+6, -0x1.239a3d6aea982p-19}, {0x1.c26b54p-1, 0x1.e239e4p+6, -0x1.e879d03304b59p-19},
    {0x1.bf583ep-1, 0x1.e25858p+6, 0x1.d4a0b519628b5p-19}, {0x1.bc4fd6p-1, 0x1.e2769ap+6, -0x1.57a2f7cfc0eb1p-20},
    {0x1.b951e2p-1, 0x1.e294a6p+6, 0x1.e7f87e8ed1c89p-22}, {0x1.b65e2ep-1, 0x1.e2b27ep+6, 0x1.d43d7d5ba5d91p-19},
    {0x1.b37484p-1, 0x1.e2d024p+6, 0x1.9cf8074397a42p-19}, {0x1.b094b4p-1, 0x1.e2ed98p+6, 0x1.6a5e061fb7f08p-20},
    {0x1.adbe88p-1, 0x1.e30adap+6, 0x1.949ceba3fdf9cp-20}, {0x1.aaf1d2p-1, 0x1.e327ecp+6, -0x1.0639e36e5fe89p-19},
    {0x1.a82e66p-1, 0x1.e344ccp+6, 0x1.265c70ae2b138p-21}, {0x1.a5741p-1, 0x1.e3617ep+6, -0x1.85d27808810d4p-19},
    {0x1.a2c2a8p-1, 0x1.e37ep+6, -0x1.9cd3db43aeeddp-19}, {0x1.a01a02p-1, 0x1.e39a52p+6, 0x1.41719a6de3314p-19},
    {0x1.9d79f2p-1, 0x1.e3b678p+6, 0x1.8faabaf5162e1p-21}, {0x1.9ae24ep-1, 0x1.e3d27p+6, 0x1.006ca0ef1c38ep-19},
    {0x1.9852fp-1, 0x1.e3ee3cp+6, 0x1.bb5b477aab93dp-25}, {0x1.95cbbp-1, 0x1.e409dcp+6, -0x1.5d8d508d107a8p-19},
    {0x1.934c68p-1, 0x1.e4254ep+6, 0x1.e257ed31d20b4p-19}, {0x1.90d4f2p-1, 0x1.e44098p+6, -0x1.1a8a98a09a905p-19},
    {0x1.8e6528p-1, 0x1.e45bb6p+6, -0x1.25bfca82973dep-19}, {0x1.8bfce8p-1, 0x1.e476aap+6, -0x1.5aeed4b8f38e3p-19},
    {0x1.899c1p-1, 0x1.e49174p+6, -0x1.90213df5004a7p-20}, {0x1.87427cp-1, 0x1.e4ac14p+6, 0x1.c0249582c54dcp-19},
    {0x1.84f00cp-1, 0x1.e4c68ep+6, -0x1.c301680e76de8p-20}, {0x1.82a4ap-1, 0x1.e4e0dep+6, 0x1.02ee8b5dfa635p-21},
    {0x1.806018p-1, 0x1.e4fb08p+6, -0x1.de61e7e665f21p-19}, {0x1.7e2256p-1, 0x1.e51508p+6, 0x1.9a807acfc9931p-19},
    {0x1.7beb3ap-1, 0x1.e52ee4p+6, -0x1.012cef0926b4p-21}, {0x1.79baa6p-1, 0x1.e54898p+6, 0x1.83c8ffcf9a001p-19},
    {0x1.779082p-1, 0x1.e56228p+6, -0x1.50eeb3aa18876p-20}, {0x1.756cacp-1, 0x1.e57b92p+6, -0x1.5ce6aa3b9e3a9p-19},
    {0x1.734f0cp-1, 0x1.e594d6p+6, -0x1.23a4ce871f33dp-23}, {0x1.713786p-1, 0x1.e5adf6p+6, 0x1.445e618da2e6p-22},
    {0x1.6f2602p-1, 0x1.e5c6f2p+6, -0x1.0e49f57ce00acp-23}, {0x1.6d1a62p-1, 0x1.e5dfcap+6, 0x1.e34144b22c427p-21},
    {0x1.6b149p-1, 0x1.e5f88p+6, -0x1.ba1bff2ec8fb9p-19}, {0x1.691474p-1, 0x1.e61112p+6, -0x1.ef995be98c7c5p-19},
    {0x1.6719f4p-1, 0x1.e6298p+6, 0x1.9b5b4b005a7b6p-20}, {0x1.6524f8p-1, 0x1.e641cep+6, -0x1.67b880a5bdab4p-20},
    {0x1.63356cp-1, 0x1.e659f8p+6, 0x1.ffeb1e8e9745bp-19}, {0x1.614b36p-1, 0x1.e67202p+6, 0x1.fbf9415459c13p-19},
    {0x1.5f6644p-1, 0x1.e689ecp+6, -0x1.b084a62361978p-21}, {0x1.5d867cp-1, 0x1.e6a1b4p+6, -0x1.26ecdcf736fcep-23},
    {0x1.5babccp-1, 0x1.e6b95cp+6, -0x1.24d4ddb955355p-20}, {0x1.59d62p-1, 0x1.e6d0e4p+6, -0x1.4d2df0977e1e3p-19},
    {0x1.58056p-1, 0x1.e6e84cp+6, -0x1.34525bac141b2p-19}, {0x1.56397cp-1, 0x1.e6ff94p+6, 0x1.ea5305a613146p-28},
    {0x1.54725ep-1, 0x1.e716bep+6, -0x1.8384107b4e8cbp-20}, {0x1.52aff6p-1, 0x1.e72dc8p+6, 0x1.b5c78450e3c43p-20},
    {0x1.50f22ep-1, 0x1.e744b4p+6, 0x1.d2c77918cff35p-19}, {0x1.4f38f6p-1, 0x1.e75b84p+6, -0x1.73f56a3c7adbfp-19},
    {0x1.4d843cp-1, 0x1.e77234p+6, -0x1.5e752f2c8ec57p-21}, {0x1.4bd3eep-1, 0x1.e788c6p+6, 0x1.d0e6028559568p-19},
    {0x1.4a27fap-1, 0x1.e79f3cp+6, 0x1.b617a2f8c6157p-19}, {0x1.488052p-1, 0x1.e7b596p+6, -0x1.7166770a338fdp-21},
    {0x1.46dce4p-1, 0x1.e7cbd2p+6, 0x1.5dc92392d2ce6p-21}, {0x1.453d9ep-1, 0x1.e7e1f2p+6, 0x1.2dd74abd67f6bp-20},
    {0x1.43a274p-1, 0x1.e7f7f6p+6, 0x1.1471a2dedbb3p-20}, {0x1.420b52p-1, 0x1.e80ddep+6, 0x1.3ad734236971p-19},
    {0x1.40782ep-1, 0x1.e823acp+6, -0x1.5a7f63374ed0ep-19}, {0x1.3ee8f4p-1, 0x1.e8395cp+6, 0x1.e1387f5c1991bp-19},
    {0x1.3d5d9ap-1, 0x1.e84ef4p+6, -0x1.0a639f9846eb1p-19}, {0x1.3bd60ep-1, 0x1.e8647p+6, -0x1.30f443735abep-19},
    {0x1.3a5244p-1, 0x1.e879dp+6, 0x1.b7f6fc4e53bbfp-19}, {0x1.38d22ep-1, 0x1.e88f18p+6, 0x1.c266311f596ap-22},
    {0x1.3755bep-1, 0x1.e8a446p+6, -0x1.2244687a7a8f2p-19}, {0x1.35dce6p-1, 0x1.e8b95ap+6, -0x1.c4453fa984053p-19},
    {0x1.34679ap-1, 0x1.e8ce54p+6, -0x1.4e1adaf23c834p-19}, {0x1.32f5cep-1, 0x1.e8e334p+6, 0x1.4933be6474213p-20},
    {0x1.318776p-1, 0x1.e8f7fcp+6, 0x1.f4126b97fb48dp-21}, {0x1.301c82p-1, 0x1.e90cacp+6, -0x1.c3ba9642d0397p-20},
    {0x1.2eb4eap-1, 0x1.e92142p+6, 0x1.0dd4a0c4597d2p-20}, {0x1.2d50ap-1, 0x1.e935cp+6, 0x1.6a268837f7ae2p-19},
    {0x1.2bef98p-1, 0x1.e94a28p+6, -0x1.baaa6251f6cf9p-19}, {0x1.2a91cap-1, 0x1.e95e76p+6, -0x1.b87ee2d2959abp-20},
    {0x1.293726p-1, 0x1.e972acp+6, 0x1.02e6f18a7a988p-19}, {0x1.27dfa4p-1, 0x1.e986ccp+6, -0x1.20eb7a5b1099ap-24},
    {0x1.268b38p-1, 0x1.e99ad4p+6, 0x1.1f989ab0f5da4p-20}, {0x1.2539d8p-1, 0x1.e9aec6p+6, -0x1.b4c42a13b79f2p-20},
    {0x1.23eb7ap-1, 0x1.e9c2ap+6, 0x1.4a9e27d91f3bap-23}, {0x1.22a012p-1, 0x1.e9d664p+6, -0x1.65ca05b7aa4dep-25},
    {0x1.215798p-1, 0x1.e9ea12p+6, -0x1.017f07b3e44dp-19}, {0x1.201202p-1, 0x1.e9fda8p+6, 0x1.895645e783d7dp-19},
    {0x1.1ecf44p-1, 0x1.ea112ap+6, 0x1.15b06b18f886bp-21}, {0x1.1d8f56p-1, 0x1.ea2496p+6, -0x1.3436aec5e4785p-20},
    {0x1.1c523p-1, 0x1.ea37ecp+6, -0x1.be1d0db15b264p-20}, {0x1.1b17c6p-1, 0x1.ea4b2cp+6, 0x1.6c2d3b989528ep-22},
    {0x1.19e012p-1, 0x1.ea5e58p+6, -0x1.757876b3d22aap-19}, {0x1.18ab08p-1, 0x1.ea716ep+6, -0x1.08f4b9a8d70c7p-19},
    {0x1.1778a2p-1, 0x1.ea846ep+6, 0x1.78821b1d97036p-19}, {0x1.1648d6p-1, 0x1.ea975cp+6, -0x1.69b5a9a819ffep-19},
    {0x1.151b9ap-1, 0x1.eaaa34p+6, -0x1.23f8154b11c7ep-19}, {0x1.13f0e8p-1, 0x1.eabcf8p+6, -0x1.a744f2cb316acp-19},
    {0x1.12c8b8p-1, 0x1.eacfa6p+6, 0x1.5e44424cab5bdp-19}, {0x1.11a302p-1, 0x1.eae242p+6, 0x1.0709b84b5bafep-21},
    {0x1.107fbcp-1, 0x1.eaf4cap+6, -0x1.8c8351c1e5262p-21}, {0x1.0f5eep-1, 0x1.eb073ep+6, -0x1.d5e259c8089ap-21},
    {0x1.0e4066p-1, 0x1.eb199ep+6, 0x1.a6c3af2faa0c6p-21}, {0x1.0d2446p-1, 0x1.eb2becp+6, -0x1.635dfaa2dda05p-19},
    {0x1.0c0a78p-1, 0x1.eb3e26p+6, -0x1.770a16843b19ep-19}, {0x1.0af2f8p-1, 0x1.eb504cp+6, 0x1.25ab9096cf361p-23},
    {0x1.09ddbap-1, 0x1.eb626p+6, 0x1.4a91cdd27e1d3p-22}, {0x1.08cabcp-1, 0x1.eb7462p+6, -0x1.8bfaea606335cp-19},
    {0x1.07b9f2p-1, 0x1.eb865p+6, -0x1.5fedcb1b43bf4p-23}, {0x1.06ab5ap-1, 0x1.eb982cp+6, 0x1.ae60edb965f84p-22},
    {0x1.059eeap-1, 0x1.eba9f6p+6, 0x1.210fc73336283p-23}, {0x1.04949cp-1, 0x1.ebbbaep+6, -0x1.2a1a7e28925c3p-21},
    {0x1.038c6cp-1, 0x1.ebcd54p+6, -0x1.d6f841d63da3ep-20}, {0x1.02865p-1, 0x1.ebdee8p+6, -0x1.0c97e507f5645p-19},
    {0x1.018244p-1, 0x1.ebf06ap+6, -0x1.689c7675517b5p-20}, {0x1.00804p-1, 0x1.ec01dap+6, 0x1.45e717b058f0bp-20}};

__device__ __forceinline__ double level_of(double I) {
  if (!(I > 0.0)) return -__builtin_huge_val();
  const unsigned long long u = (unsigned long long)__double_as_longlong(I);
  const int ex = (int)(u >> 52);
  if (ex == 0 || ex == 0x7ff) return 10.0 * log10(I) + 120.0;  // denormal or infinite
  const LevelEntry *const ct = &c_level_tab[(int)(u >> 45) & 127];
  const double m = __longlong_as_double((long long)((u & 0xfffffffffffffull) | 0x3ff0000000000000ull));
  const double r = fma(m, __ldg(&ct->c), -1.0);
  // 10 / ln 10, and 10 log10(2) in two parts, the first of 24 bits
  const double k = 0x1.15f2ced384f29p+2, hi = 0x1.815182p+1, lo = 0x1.31d61fabf59b6p-25;
  const float f = (float)r, kf = (float)k;
  const float t = f * fmaf(f, fmaf(f, -kf / 6.0f, kf / 5.0f), -kf / 4.0f);
  const double e = (double)(ex - 1023);
  const double p = fma(r, fma(r, k / 3.0 + (double)t, -k / 2.0), k);
  // e hi + ct->hi is exact: multiples of 2^-22 below 2^12
  return fma(e, hi, __ldg(&ct->hi)) + fma(r, p, fma(e, lo, __ldg(&ct->lo)));
}

// The outputs that are wanted, in the caller's microphone order.
__global__ void __launch_bounds__(256) k_levels(const double *energy, const int *count, const float4 *mics, int64_t n_m,
                                                int n_bands, double *level_db, double *intensity, int *path_count) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t p = i / kMaxBands;
  const int b = (int)(i % kMaxBands);
  if (p >= n_m) return;
  const int64_t orig = __float_as_int(__ldg(&mics[p].w));
  if (b == 0 && path_count) path_count[orig] = count[p];
  if (b >= n_bands) return;
  const double I = energy[i];
  if (level_db) level_db[orig * n_bands + b] = level_of(I);
  if (intensity) intensity[orig * n_bands + b] = I;
}

cudaError_t launch_levels(cudaStream_t st, const double *energy, const int *count, const float4 *mics,
                          int64_t n_m, int n_bands, double *level_db, double *intensity, int *path_count) {
  if (n_m == 0 || (!level_db && !intensity && !path_count)) return cudaSuccess;
  const int threads = 256;
  k_levels<<<(int)((n_m * kMaxBands + threads - 1) / threads), threads, 0, st>>>(energy, count, mics, n_m, n_bands,
                                                                                level_db, intensity, path_count);
  note_launches(1);
  return cudaGetLastError();
}

// Clear a scene's accumulators and a trace's counters and cursors, in one
// launch instead of five (which took longer than a small trace's scatter).
__global__ void __launch_bounds__(256) k_clear(double2 *energy, int *count, int64_t n_m, Counters *ctr,
                                               unsigned long long *cursors) {
  static_assert(sizeof(Counters) % 8 == 0, "cleared by words");
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = i0; i < n_m * (kMaxBands / 2); i += step) energy[i] = make_double2(0.0, 0.0);
  for (int64_t i = i0; i < n_m; i += step) count[i] = 0;
  if (i0 < (int64_t)(sizeof(Counters) / 8)) ((unsigned long long *)ctr)[i0] = 0ull;
  if (i0 < kCursors) cursors[i0] = 0ull;
}

cudaError_t launch_clear(cudaStream_t st, double *energy, int *count, int64_t n_m, Counters *ctr,
                         unsigned long long *cursors, int n_sm) {
  const int64_t need = (n_m * (kMaxBands / 2) + 255) / 256, most = (int64_t)n_sm * 8;
  k_clear<<<(int)(need < 1 ? 1 : need < most ? need : most), 256, 0, st>>>((double2 *)energy, count, n_m, ctr, cursors);
  note_launches(1);
  return cudaGetLastError();
}

// Install a result given in input microphone order (partial results of
// source shards, summed by the caller) into a scene's accumulators, which are
// kept in binned order.
__global__ void k_set_result(const double *intensity, const int *count_in, const float4 *mics, int64_t n_m,
                             int n_bands, double *energy, int *count) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n_m) return;
  int64_t orig = __float_as_int(mics[p].w);
  for (int b = 0; b < kMaxBands; b++) energy[p * kMaxBands + b] = b < n_bands ? intensity[orig * n_bands + b] : 0.0;
  count[p] = count_in ? count_in[orig] : 0;
}

cudaError_t launch_set_result(cudaStream_t st, const double *intensity, const int *count_in, const float4 *mics,
                              int64_t n_m, int n_bands, double *energy, int *count) {
  if (n_m == 0) return cudaSuccess;
  int threads = 256;
  k_set_result<<<(int)((n_m + threads - 1) / threads), threads, 0, st>>>(intensity, count_in, mics, n_m,
                                                                         n_bands, energy, count);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace bt
