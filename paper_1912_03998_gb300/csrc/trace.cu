// trace.cu -- the tracing half of the hot path of the hybrid beam/ray
// tracer (Section 2 of the paper): beam generation, axis-ray traversal and
// image-source reflection, with and without the sub-domain split (Section 3).
// The microphone-in-beam test, the energy scatter and the level readout are
// in scatter.cu.
//
//   k_trace   persistent warps, one lineage (source, icosahedron face) per
//             lane: for orders 0..K it casts the beam's axis ray through the
//             BVH, writes the segment (apex, cone planes, start/end planes,
//             band power) unless it cannot reach the microphones' height, and
//             reflects the beam about the hit triangle's plane (image source);
//             a lane whose lineage ends takes the next one at once.
//   k_trace_tiled  the same over sub-domains (Section 3): one hierarchy per
//             tile, hand-off queues between tiles and work stealing, all in
//             one persistent launch.
//   k_cast    the axis-ray query on its own (closest hit of given rays).
//
// Precision.  BT_PREC_FP32 carries the lineage in float32.  BT_PREC_MIXED
// carries the image-source chain -- apex, cone normals, ray origin and
// direction -- as float pairs (about 48 bits, on the float32 pipe) from a
// float64 beam table through every reflection, on the triangles' float64
// planes.  Traversal is float32; a triangle whose float32 test is ambiguous
// (the ray within a relative 1e-4 of an edge) is re-tested in float64, near-
// equal hit distances are compared in float64 -- both after the search, from
// a short per-lane list, so that no float64 code sits in the traversal loop.
// The reflection's float-pair arithmetic runs in stages, each reading its
// rows from shared memory and writing them back.  The microphone tests are
// in scatter.cu.
#include <stdio.h>

#include <type_traits>

#include "bt_internal.cuh"

namespace bt {

// precision variants of the trace kernels (BT_PREC_*)
constexpr int kPF32 = 0, kPMixed = 1, kPF64 = 2, kPMixed64 = 3;
// What each variant does: the image-source chain (apex, cone normals, ray
// origin and direction) as float pairs (`pairs`, MIXED) or in float64
// (`chain64`, FP64 and MIXED64), else float32; float32 triangle tests whose
// ambiguous cases and near ties are settled in float64 after the search
// (`defer`, MIXED and MIXED64), or every triangle test in float64 (`all64`,
// FP64).
template <int kP>
struct Prec {
  static constexpr bool pairs = kP == kPMixed;
  static constexpr bool chain64 = kP == kPF64 || kP == kPMixed64;
  static constexpr bool defer = kP == kPMixed || kP == kPMixed64;
  static constexpr bool all64 = kP == kPF64;
};

// Regular icosahedron: unit vertices (the cyclic permutations of
// (0, +-1, +-phi), normalised) and its 20 faces, counter-clockwise seen
// from outside.  Vertex coordinates are 0, +-A or +-B with
// A = 1/sqrt(1+phi^2), B = phi/sqrt(1+phi^2); the table holds 0, +-1 (A),
// +-2 (B).
__constant__ signed char c_ico_s[12][3] = {
    {0, -1, 2}, {0, 1, 2},   {2, 0, 1},   {-2, 0, 1},  {-1, -2, 0}, {1, -2, 0},
    {1, 2, 0},  {-1, 2, 0},  {2, 0, -1},  {-2, 0, -1}, {0, -1, -2}, {0, 1, -2},
};
__constant__ int c_ico_f[20][3] = {
    {0, 2, 1},  {0, 1, 3},  {0, 5, 2},  {0, 3, 4},  {1, 2, 6},   {1, 7, 3},  {0, 4, 5},
    {1, 6, 7},  {2, 5, 8},  {2, 8, 6},  {3, 9, 4},  {3, 7, 9},   {4, 10, 5}, {6, 11, 7},
    {4, 9, 10}, {5, 10, 8}, {6, 8, 11}, {7, 11, 9}, {8, 10, 11}, {9, 11, 10},
};

template <typename T>
struct Vec3;
template <>
struct Vec3<float> { using type = float3; };
template <>
struct Vec3<double> { using type = double3; };

template <typename T>
__device__ __forceinline__ typename Vec3<T>::type ico_vertex(int v) {
  const T phi = (T)0.5 * ((T)1 + sqrt((T)5));
  const T inv = (T)1 / sqrt((T)1 + phi * phi);
  const T A = inv, B = phi * inv;
  T c[3];
  for (int k = 0; k < 3; k++) {
    int s = c_ico_s[v][k];
    c[k] = s == 0 ? (T)0 : (s == 1 ? A : (s == -1 ? -A : (s == 2 ? B : -B)));
  }
  typename Vec3<T>::type r;
  r.x = c[0];
  r.y = c[1];
  r.z = c[2];
  return r;
}

// Edge directions of face `i` of the level-L geodesic icosahedron.  The base
// face is i >> 2L; each further pair of bits picks one of the four children
// (a,ab,ca), (ab,b,bc), (ca,bc,c), (ab,bc,ca), ab = midpoint pushed to the
// sphere.  A vertex shared by two faces is computed from the same operands in
// both, so both faces get the bit-identical direction.
template <typename T>
__device__ __forceinline__ void beam_dirs(int level, int64_t i, typename Vec3<T>::type &a,
                                          typename Vec3<T>::type &b, typename Vec3<T>::type &c) {
  int f = (int)(i >> (2 * level));
  a = ico_vertex<T>(c_ico_f[f][0]);
  b = ico_vertex<T>(c_ico_f[f][1]);
  c = ico_vertex<T>(c_ico_f[f][2]);
  for (int l = level - 1; l >= 0; --l) {
    int ch = (int)((i >> (2 * l)) & 3);
    auto ab = normalize3(a + b), bc = normalize3(b + c), ca = normalize3(c + a);
    if (ch == 0) { b = ab; c = ca; }
    else if (ch == 1) { a = ab; c = bc; }
    else if (ch == 2) { a = ca; b = bc; }
    else { a = ab; b = bc; c = ca; }
  }
}

// Beam table of one icosahedron level, formed in float64 and stored as float
// pairs: per beam the three cone-face normals d_j x d_{j+1} (no FMA, so
// neighbours share exactly opposite normals; the split keeps that) and the
// unit axis -- 12 hi floats, then 12 lo floats.
__global__ void k_beam_table(int level, int64_t n_beams, float *table) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_beams) return;
  double3 d0, d1, d2;
  beam_dirs<double>(level, i, d0, d1, d2);
  double3 v[4] = {cross_exact(d0, d1), cross_exact(d1, d2), cross_exact(d2, d0), normalize3((d0 + d1) + d2)};
  float *o = table + 24 * i;
  for (int k = 0; k < 4; k++) {
    double c[3] = {v[k].x, v[k].y, v[k].z};
    for (int q = 0; q < 3; q++) {
      df h = d_to_df(c[q]);
      o[3 * k + q] = h.hi;
      o[12 + 3 * k + q] = h.lo;
    }
  }
}

// The same in float64 for the float64-chain variants, 12 doubles a beam.  Those
// formed each lineage's beam in the trace kernel: some thousand float64
// operations for the few lanes of a service phase that start a lineage, which
// cost as much of the float64 pipe as everything else together (FP64, 24
// district sources: trace kernel 3.23 -> 2.31 ms).  From kBeamFaces on a thread
// forms the four beams of one face of the level above, whose descent they
// share: a call without allocation makes the table anew each time, and a beam a
// thread took longer at level 6 than the trace saves by it (MIXED64, one source
// in the 8 x 8-block city: 652 -> 602 us a call, 628 without a table).  Below,
// the table is a chain of latencies, which four beams a thread lengthen (level
// 4: 209 -> 217 us).
constexpr int kBeamFaces = 5;
__device__ __forceinline__ void put_beam64(double *o, double3 d0, double3 d1, double3 d2) {
  const double3 v[4] = {cross_exact(d0, d1), cross_exact(d1, d2), cross_exact(d2, d0), normalize3((d0 + d1) + d2)};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    o[3 * k] = v[k].x;
    o[3 * k + 1] = v[k].y;
    o[3 * k + 2] = v[k].z;
  }
}
__global__ void k_beam_table64(int level, int64_t n_threads, double *table) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_threads) return;
  double3 a, b, c;
  beam_dirs<double>(level < kBeamFaces ? level : level - 1, i, a, b, c);
  if (level < kBeamFaces) {
    put_beam64(table + 12 * i, a, b, c);
    return;
  }
  const double3 ab = normalize3(a + b), bc = normalize3(b + c), ca = normalize3(c + a);
  double *const o = table + 48 * i;
  put_beam64(o, a, ab, ca);
  put_beam64(o + 12, ab, b, bc);
  put_beam64(o + 24, ca, bc, c);
  put_beam64(o + 36, ab, bc, ca);
}

cudaError_t launch_beam_table(cudaStream_t st, int prec, int level, float *table) {
  int64_t n = (int64_t)20 << (2 * level);
  if (prec == kPMixed) k_beam_table<<<(int)((n + 127) / 128), 128, 0, st>>>(level, n, table);
  else {
    const int64_t threads = level < kBeamFaces ? n : n / 4;
    k_beam_table64<<<(int)((threads + 127) / 128), 128, 0, st>>>(level, threads, (double *)table);
  }
  note_launches(1);
  return cudaGetLastError();
}

// Unit axis of every beam of a level, float32 [n_beams][3] (the order of the
// lineages' beam index: a directional source's gains are given in it).
__global__ void k_beam_axes(int level, int64_t n_beams, float *axes) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_beams) return;
  double3 d0, d1, d2;
  beam_dirs<double>(level, i, d0, d1, d2);
  const double3 ax = normalize3((d0 + d1) + d2);
  axes[3 * i] = (float)ax.x;
  axes[3 * i + 1] = (float)ax.y;
  axes[3 * i + 2] = (float)ax.z;
}

cudaError_t launch_beam_axes(cudaStream_t st, int level, float *axes) {
  const int64_t n = (int64_t)20 << (2 * level);
  k_beam_axes<<<(int)((n + 127) / 128), 128, 0, st>>>(level, n, axes);
  note_launches(1);
  return cudaGetLastError();
}

// float64 distance along the ray to the plane of leaf slot `slot`.
__device__ __forceinline__ double plane_t64(const DevScene &sc, int slot, double3 od, double3 dd) {
  Plane64 pl = ldg_d4(&sc.planes64[slot]);
  double3 n = make_double3(pl.x, pl.y, pl.z);
  return (pl.w - dot3(n, od)) / dot3(n, dd);
}

// Best hit so far.  In MIXED mode t64 holds the float64 distance when known.
struct Best {
  float t;
  int slot, id;
  double t64;
  bool has64;
};

// Candidates a MIXED search leaves to float64 (kPend at most per search):
// triangles whose float32 test was ambiguous (slot | kPendAmb) and near ties
// of the best hit (slot).  Past kPend a candidate is decided in float32 like
// any other (a search meets that many only on a ray running along a line of
// triangle edges).
constexpr int kPend = 8;
constexpr int kPendAmb = 0x40000000;

// Ray as float pairs in shared memory: rows 0..5 of `hi` and `lo` hold origin
// xyz and direction xyz, `stride` floats apart.
// In FP64 mode `dv` points at the same rows held as float64.  MIXED: `pend`
// is the lane's column of the pending list (entry 0 the count, entries 1..
// kPend the candidates, `stride` ints apart).
struct RaySrc {
  const float *hi, *lo;
  int stride;
  const double *dv;
  int *pend;
  __device__ __forceinline__ void get(double3 &o, double3 &d) const {
    if (dv) {
      o = make_double3(dv[0], dv[stride], dv[2 * stride]);
      d = make_double3(dv[3 * stride], dv[4 * stride], dv[5 * stride]);
      return;
    }
    o = make_double3((double)hi[0] + lo[0], (double)hi[stride] + lo[stride], (double)hi[2 * stride] + lo[2 * stride]);
    d = make_double3((double)hi[3 * stride] + lo[3 * stride], (double)hi[4 * stride] + lo[4 * stride],
                     (double)hi[5 * stride] + lo[5 * stride]);
  }
};

// Record a candidate for float64 after the search; false if the list is full.
__device__ __forceinline__ bool pend_add(const RaySrc &rs, int entry) {
  const int n = rs.pend[0];
  if (n >= kPend) return false;
  rs.pend[(n + 1) * rs.stride] = entry;
  rs.pend[0] = n + 1;
  return true;
}

// An event count of a warp, in shared memory: every lane that passes an
// increment adds one, the lanes that execute it together with one atomic.
struct WarpCount {
  unsigned *p;
  __device__ __forceinline__ void operator++(int) const {
    const unsigned m = __activemask();
    if ((int)(threadIdx.x & 31u) == __ffs(m) - 1) atomicAdd(p, (unsigned)__popc(m));
  }
};

// What a triangle test found: an accepted hit at distance t (t64 in FP64), or
// (deferring variants) an ambiguous one, or nothing.
struct TriHit {
  float t;
  double t64;
  int id;
  bool ok, amb;
};

// Test leaf slot `slot` against ray r; hits beyond `tmax` are dropped.
template <int kP, bool kCount>
__device__ __forceinline__ TriHit test_tri(const Tri *tris, const Ray &r, const RaySrc &rs, double dns64, int slot,
                                           const WarpCount &n_tris, float tmax) {
  constexpr bool kDefer = Prec<kP>::defer, kAll64 = Prec<kP>::all64;
  if (kCount) n_tris++;
  const Tri *tp = tris + slot;
  const float4 v0 = __ldg(&tp->v0), v1 = __ldg(&tp->v1), v2 = __ldg(&tp->v2);
  TriHit h = {0.0f, 0.0, __float_as_int(v1.w), false, false};
  if (kAll64) {
    // FP64: every candidate in float64 Moller-Trumbore on the float64 ray
    double3 o, d;
    rs.get(o, d);
    double tt;
    if (!hit_mt64(o, d, v0, v1, v2, tt)) return h;
    if (!(tt > (double)r.t_eps && (dns64 == 0.0 || tt * dns64 > (double)r.t_eps))) return h;
    h.t64 = tt;
    h.t = (float)tt;
    h.ok = !(h.t > tmax);
    return h;
  }
  bool amb;
  h.t = hit_watertight(r, v0, v1, v2, amb);
  h.ok = h.t < kInf && accept_hit(r, h.t) && !(h.t > tmax);
  h.amb = kDefer && amb;
  return h;
}

// The window of distances around the best hit that is settled in float64.
__device__ __forceinline__ float tie_window(float t) { return 1e-5f * fabsf(t) + 1e-4f; }

// A hit (or an ambiguous test) of leaf slot `slot` against the best hit so
// far.
template <int kP>
__device__ __forceinline__ void weigh_hit(const RaySrc &rs, Best &best, int slot, const TriHit &h) {
  constexpr bool kDefer = Prec<kP>::defer;
  // MIXED: an ambiguous candidate is decided in float64 after the search
  if (kDefer && h.amb && pend_add(rs, slot | kPendAmb)) return;
  if (!h.ok) return;
  if (kP == kPF32) {
    if (h.t < best.t || (h.t == best.t && h.id < best.id)) { best.t = h.t; best.slot = slot; best.id = h.id; }
    return;
  }
  // MIXED and FP64: a clearly nearer or farther float32 distance decides; a
  // near tie is settled in float64, where distances within 1e-9 relative tie
  // and go to the lowest triangle index (MIXED: after the search)
  const float win = tie_window(best.t);
  if (best.slot < 0 || h.t < best.t - win) {
    best.t = h.t; best.slot = slot; best.id = h.id; best.t64 = h.t64; best.has64 = !kDefer;
    return;
  }
  if (h.t > best.t + win) return;
  if (kDefer) {
    if (!pend_add(rs, slot) && (h.t < best.t || (h.t == best.t && h.id < best.id))) {
      best.t = h.t; best.slot = slot; best.id = h.id; best.t64 = 0.0; best.has64 = false;
    }
    return;
  }
  const double tol = 1e-9 * (1.0 + fabs(h.t64));
  if (h.t64 < best.t64 - tol || (fabs(h.t64 - best.t64) <= tol && h.id < best.id)) {
    best.t = (float)h.t64; best.slot = slot; best.id = h.id; best.t64 = h.t64; best.has64 = true;
  }
}

// MIXED, after a search: the candidates it left to float64.  An ambiguous
// triangle is tested with float64 Moller-Trumbore; a near tie compares the
// float64 plane distances of both triangles.  Each is then weighed against
// the best hit as during the search.
__device__ __forceinline__ void settle_pending(const DevScene &sc, const Ray &r, const RaySrc &rs, double dns64,
                                               Best &best, float tlim);
__device__ __noinline__ void settle_pending_call(const DevScene &sc, const Ray &r, const RaySrc &rs, double dns64,
                                                 Best &best, float tlim) {
  settle_pending(sc, r, rs, dns64, best, tlim);
}
// kOutOfLine: the rarely needed float64 code as a call, out of the caller's
// instruction stream (the sub-domain trace, whose service code measured
// faster the smaller it was: 46.1 -> 45.2 ms on the district)
template <bool kOutOfLine = false>
__device__ __forceinline__ void settle_search(const DevScene &sc, const Ray &r, const RaySrc &rs, double dns64,
                                              Best &best, float tlim) {
  if (rs.pend[0] == 0) return;
  if (kOutOfLine) settle_pending_call(sc, r, rs, dns64, best, tlim);
  else settle_pending(sc, r, rs, dns64, best, tlim);
}
__device__ __forceinline__ void settle_pending(const DevScene &sc, const Ray &r, const RaySrc &rs, double dns64,
                                               Best &best, float tlim) {
  const int n = rs.pend[0];
  const Tri *const tris = sc.tris;
  double3 o, d;
  rs.get(o, d);
#pragma unroll 1
  for (int q = 1; q <= n; q++) {
    const int e = rs.pend[q * rs.stride];
    const int slot = e & ~kPendAmb;
    const Tri *tp = tris + slot;
    const float4 v1 = __ldg(&tp->v1);
    double tt;
    if (e & kPendAmb) {
      if (!hit_mt64(o, d, __ldg(&tp->v0), v1, __ldg(&tp->v2), tt)) continue;
      if (!(tt > (double)r.t_eps && (dns64 == 0.0 || tt * dns64 > (double)r.t_eps))) continue;
    } else {
      tt = plane_t64(sc, slot, o, d);
    }
    const float t = (float)tt;
    if (t > tlim) continue;
    const int id = __float_as_int(v1.w);
    const float win = 1e-5f * fabsf(best.t) + 1e-4f;
    if (best.slot < 0 || t < best.t - win) {
      best.t = t; best.slot = slot; best.id = id; best.t64 = tt; best.has64 = true;
      continue;
    }
    if (t > best.t + win) continue;
    if (!best.has64) {
      best.t64 = plane_t64(sc, best.slot, o, d);
      best.has64 = true;
    }
    const double tol = 1e-9 * (1.0 + fabs(tt));
    if (tt < best.t64 - tol || (fabs(tt - best.t64) <= tol && id < best.id)) {
      best.t = t; best.slot = slot; best.id = id; best.t64 = tt; best.has64 = true;
    }
  }
}

// Order two (distance, child) pairs by distance.
__device__ __forceinline__ void sort_pair(float &ka, int &ca, float &kb, int &cb) {
  const bool sw = kb < ka;
  const float k = sw ? kb : ka;
  const int c = sw ? cb : ca;
  kb = sw ? ka : kb;
  cb = sw ? ca : cb;
  ka = k;
  ca = c;
}

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

constexpr int kTraceThreads = 128;

// Triangle tests a warp owes: (lane, leaf code) pairs that its lanes' node
// steps exposed.  Once there are kPairTest of them (or the phase ends) the warp
// tests 32 at a time, each lane one pair, whichever lane's ray it belongs to.
// A node step exposes a triangle on about one lane in six, so testing them
// where they arise ran the triangle code for 4.4 of 32 lanes nearly as often as
// the node code; by pairs it runs for 18 (both counted on the CPU over the
// axis rays of 4 district sources).  The best hits the node steps cull by are
// then up to kPairTest tests old, which costs 2 % more node visits at 12 (8
// and 16 measured 2-5 % slower).
constexpr int kPairTest = 12;
constexpr int kPairCap = 4 * 32 + kPairTest;  // a step adds at most four per lane
template <int kWarps>
struct PairQueue {
  int code[kWarps][kPairCap];
  int n[kWarps];
  unsigned char lane[kWarps][kPairCap];
};
struct WarpPairs {
  int *code, *n;
  unsigned char *lane;
};
template <int kWarps>
__device__ __forceinline__ WarpPairs warp_pairs(PairQueue<kWarps> &q) {
  const int w = threadIdx.x >> 5;
  if (lane_id() == 0) q.n[w] = 0;
  __syncwarp();
  return WarpPairs{q.code[w], &q.n[w], q.lane[w]};
}

// A closest-hit search that can stop after any node and resume later: its
// state is the current node, the stack (an array the caller keeps: the inner
// children not yet visited) and the best hit so far.
struct HitSearch {
  int node, sp, budget;
  Best best;
  __device__ __forceinline__ void start(int root, int64_t n_tris) {
    node = root;
    sp = 0;
    budget = (int)n_tris + 64;
    best.t = kInf;
    best.slot = -1;
    best.id = 0x7fffffff;
    best.t64 = 0.0;
    best.has64 = false;
  }
  // Distances beyond which nothing is of interest: in MIXED and FP64 mode
  // near ties must still be visited.
  template <int kP>
  __device__ __forceinline__ float limit(float tlim) const {
    return fminf(kP != kPF32 ? best.t + tie_window(best.t) : best.t, tlim);
  }
};

// Test the warp's `n` pairs, 32 at a time.  Each lane takes one pair and makes
// its owner's ray again from the rows in shared memory (which costs less than
// holding the test's part of every ray in registers); the hits then go back to
// their owners, one per owner and round, through a mailbox in the pairs' own
// (read) entries.  Warp-collective; t_eps, dns, dns64 and tlim are the calling
// lane's own.
template <int kP, bool kCount, bool kLeaves>
__device__ __forceinline__ void test_pairs(const WarpPairs &wp, int n, const Tri *tris, bool lane_tris, float t_eps,
                                           float dns, const RaySrc &rs, double dns64, HitSearch &hs,
                                           const WarpCount &n_tris, float tlim, int lg = 0) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = (int)lane_id();
  volatile int *const mail = wp.code;
  for (int base = 0; base < n; base += 32) {
    bool have = base + lane < n;
    int code = 0, owner = lane;
    if (have) {
      code = wp.code[base + lane];
      owner = wp.lane[base + lane];
      have = code != ~kNoChild;  // (an unused lane, met by a NaN ray)
    }
    __syncwarp();
    RaySrc qs = rs;
    const int col = (owner >> lg) - (lane >> lg);  // the owner's column, from one's own
    const float *h6 = rs.hi + col;
    const float3 qo = make_float3(h6[0], h6[rs.stride], h6[2 * rs.stride]);
    const float3 qd = make_float3(h6[3 * rs.stride], h6[4 * rs.stride], h6[5 * rs.stride]);
    const Ray q = make_ray(qo, qd, lane_tris ? __shfl_sync(kAll, t_eps, owner) : t_eps,
                           kP == kPF64 ? 0.0f : __shfl_sync(kAll, dns, owner));
    const Tri *qt = tris;
    if (lane_tris) qt = (const Tri *)__shfl_sync(kAll, (unsigned long long)tris, owner);
    double qdns64 = 0.0;
    if (kP == kPF64) {
      qdns64 = __shfl_sync(kAll, dns64, owner);
      qs.dv += col;
    }
    int left = 1;
    if (kLeaves) {
      left = have ? leaf_count(code) : 0;
      code = leaf_slot(code);
    }
    // (kLeaves: a pair may stand for several consecutive triangles)
    for (int j = 0; kLeaves ? __any_sync(kAll, j < left) != 0 : j < 1; j++) {
      const float tmax = __shfl_sync(kAll, hs.limit<kP>(tlim), owner);
      TriHit h = {0.0f, 0.0, 0, false, false};
      if (kLeaves ? j < left : have) h = test_tri<kP, kCount>(qt, q, qs, qdns64, code + j, n_tris, tmax);
      bool todo = h.ok || h.amb;
      while (__any_sync(kAll, todo)) {
        mail[lane] = -1;
        __syncwarp();
        if (todo) mail[owner] = lane;
        __syncwarp();
        const int from = mail[lane];
        if (todo && mail[owner] == lane) todo = false;
        const int src = from < 0 ? lane : from;
        TriHit g;
        g.t = __shfl_sync(kAll, h.t, src);
        g.id = __shfl_sync(kAll, h.id, src);
        g.t64 = kP == kPF64 ? __shfl_sync(kAll, h.t64, src) : 0.0;
        const int flags = __shfl_sync(kAll, (int)h.ok | (int)h.amb << 1, src);
        const int slot = __shfl_sync(kAll, code + j, src);
        g.ok = flags & 1;
        g.amb = flags >> 1;
        if (from >= 0) weigh_hit<kP>(rs, hs.best, slot, g);
        __syncwarp();
      }
    }
  }
  if (lane == 0) *wp.n = 0;
  __syncwarp();
}

// The search phase of a warp: every lane with `more` nodes to visit takes node
// steps until at most `few` lanes have nodes left.  kPairs: the exposed
// triangles are tested by pairs, else each lane tests its own at once.
// lane_tris: the lanes' scenes differ.  Warp-collective.
//
// A node step is one wide node: the boxes of its up to four children in one
// 128-byte fetch, each axis' near and far planes told apart by the sign of the
// ray's direction; the nearest inner child hit next, the others pushed
// farthest first.
template <int kP, bool kCount, bool kLeaves, bool kPairs>
__device__ __forceinline__ void search_phase(const DevScene &sc, bool lane_tris, const Ray &r, const RaySrc &rs,
                                             double dns64, int *stack, int *err, HitSearch &hs, bool &more,
                                             const WarpPairs &wp, const WarpCount &n_nodes, const WarpCount &n_tris,
                                             float tlim, int few) {
  // the hot fields in registers: in a batch `sc` lives in device memory and
  // would otherwise be re-read on every node
  const char *const nodes = (const char *)sc.nodes;
  const Tri *const tris = sc.tris;
  const float3 inv = r.inv, oi = origin_scaled(r);
  const float t_eps = r.t_eps, dns = r.dns;
  auto expose = [&](int c, int pos) {
    wp.code[pos] = ~c;
    wp.lane[pos] = (unsigned char)lane_id();
  };
  // the leaves ~lc of the lanes in lm, tested at once (a leaf of several
  // triangles is one run of slots)
  auto test_now = [&](int4 lc, unsigned lm) {
#pragma unroll 1
    while (lm) {
      const int c = __ffs(lm) - 1;
      lm &= lm - 1;
      const int v = ~(c == 0 ? lc.x : c == 1 ? lc.y : c == 2 ? lc.z : lc.w);
      for (int j = 0; j < (kLeaves ? leaf_count(v) : 1); j++) {
        const int slot = (kLeaves ? leaf_slot(v) : v) + j;
        const TriHit h = test_tri<kP, kCount>(tris, r, rs, dns64, slot, n_tris, hs.limit<kP>(tlim));
        if (h.ok || h.amb) weigh_hit<kP>(rs, hs.best, slot, h);
      }
    }
  };
  if (more && (hs.node < 0 || sc.n_tris == 0)) {
    // nothing to search, or the root of a one-leaf hierarchy
    if (sc.n_tris > 0 && hs.node != kNoChild) {
      if (kPairs) expose(hs.node, atomicAdd(wp.n, 1));
      else test_now(make_int4(hs.node, 0, 0, 0), 1u);
    }
    more = false;
  }
  unsigned run;
  do {
    int4 lc = make_int4(0, 0, 0, 0);
    unsigned lm = 0;
    if (more) {
      if (kCount) n_nodes++;
      const char *nd = nodes + (size_t)(unsigned)hs.node * sizeof(Node4);
      // (by address where throughput counts; by value in the split trace, whose
      // smaller launches wait for the longest chain of fetches, which address
      // arithmetic lengthens: 81,920 lineages split 4 x 4 1,002 -> 855 us, the
      // district 38.4 -> 38.0 ms, but the unsplit district 28.9 -> 30.0 ms)
      const int sx = inv.x < 0.0f ? 16 : 0, sy = inv.y < 0.0f ? 16 : 0, sz = inv.z < 0.0f ? 16 : 0;
      float4 nx, fx, ny, fy, nz, fz;
      if (kPairs) {
        nx = __ldg((const float4 *)(nd + sx)); fx = __ldg((const float4 *)(nd + (sx ^ 16)));
        ny = __ldg((const float4 *)(nd + 32 + sy)); fy = __ldg((const float4 *)(nd + 32 + (sy ^ 16)));
        nz = __ldg((const float4 *)(nd + 64 + sz)); fz = __ldg((const float4 *)(nd + 64 + (sz ^ 16)));
      } else {
        auto pair = [](const char *p, bool flip, float4 &n, float4 &f) {
          const float4 lo = __ldg((const float4 *)p), hi = __ldg((const float4 *)(p + 16));
          n = make_float4(flip ? hi.x : lo.x, flip ? hi.y : lo.y, flip ? hi.z : lo.z, flip ? hi.w : lo.w);
          f = make_float4(flip ? lo.x : hi.x, flip ? lo.y : hi.y, flip ? lo.z : hi.z, flip ? lo.w : hi.w);
        };
        pair(nd, sx != 0, nx, fx);
        pair(nd + 32, sy != 0, ny, fy);
        pair(nd + 64, sz != 0, nz, fz);
      }
      const int4 ch = __ldg((const int4 *)(nd + 96));
      const float tmax = hs.limit<kP>(tlim);
      float k0, k1, k2, k3;
      const bool h0 = slab_nf(inv, oi, nx.x, fx.x, ny.x, fy.x, nz.x, fz.x, tmax, k0);
      const bool h1 = slab_nf(inv, oi, nx.y, fx.y, ny.y, fy.y, nz.y, fz.y, tmax, k1);
      const bool h2 = slab_nf(inv, oi, nx.z, fx.z, ny.z, fy.z, nz.z, fz.z, tmax, k2);
      const bool h3 = slab_nf(inv, oi, nx.w, fx.w, ny.w, fy.w, nz.w, fz.w, tmax, k3);
      int c0 = ch.x, c1 = ch.y, c2 = ch.z, c3 = ch.w;
      // (to a NaN ray an unused lane looks like a leaf: test_pairs tells them
      // apart, and without pairs no NaN ray is searched)
      const bool l0 = h0 && c0 < 0, l1 = h1 && c1 < 0, l2 = h2 && c2 < 0, l3 = h3 && c3 < 0;
      if (kPairs) {
        const int cnt = (int)l0 + (int)l1 + (int)l2 + (int)l3;
        if (cnt) {
          int pos = atomicAdd(wp.n, cnt);
          if (l0) expose(c0, pos++);
          if (l1) expose(c1, pos++);
          if (l2) expose(c2, pos++);
          if (l3) expose(c3, pos);
        }
      } else {
        lc = ch;
        lm = (unsigned)l0 | (unsigned)l1 << 1 | (unsigned)l2 << 2 | (unsigned)l3 << 3;
      }
      // inner children hit, nearest first (a sorting network on the entry
      // distances; misses sort last)
      k0 = h0 && !l0 ? k0 : kInf;
      k1 = h1 && !l1 ? k1 : kInf;
      k2 = h2 && !l2 ? k2 : kInf;
      k3 = h3 && !l3 ? k3 : kInf;
      sort_pair(k0, c0, k1, c1);
      sort_pair(k2, c2, k3, c3);
      sort_pair(k0, c0, k2, c2);
      sort_pair(k1, c1, k3, c3);
      sort_pair(k1, c1, k2, c2);
      // a well-formed BVH is visited at most once per node; the bound only
      // guarantees termination should the structure ever be malformed
      if (--hs.budget < 0 || hs.sp + 3 > kStackDepth) {
        atomicExch(err, hs.budget < 0 ? BT_E_TIMEOUT : BT_E_QUEUE_FULL);
        more = false;
      } else if (k0 < kInf) {
        if (k1 < kInf) {
          if (k2 < kInf) {
            if (k3 < kInf) stack[hs.sp++] = c3;
            stack[hs.sp++] = c2;
          }
          stack[hs.sp++] = c1;
        }
        hs.node = c0;
      } else if (hs.sp > 0) {
        hs.node = stack[--hs.sp];
      } else {
        more = false;
      }
    }
    if (!kPairs) test_now(lc, lm);
    run = __ballot_sync(0xffffffffu, more);
    if (kPairs) {
      __syncwarp();
      // (one lane's reading for all: no lane may go on to the next step's
      // additions before every lane has it, and all must decide alike)
      const int n = __shfl_sync(0xffffffffu, *(volatile int *)wp.n, 0);
      // (the phase's end flushes, so that every lane without nodes is done)
      if (n >= kPairTest || (n > 0 && __popc(run) <= few))
        test_pairs<kP, kCount, kLeaves>(wp, n, tris, lane_tris, t_eps, dns, rs, dns64, hs, n_tris, tlim);
    }
  } while (__popc(run) > few);
}

// ------------------------------------------------------- groups of lanes
// Small launches: fewer lineages than the chip has lanes.  Their time is the
// latency of the longest lineage, one dependent node fetch after the other, so
// a group of G = 8 or 16 lanes works on one lineage: a step takes the top
// G / 4 nodes of the group's stack at once, four lanes to a node and one child
// box to a lane.
constexpr int kGroupMin = 8, kGroupMax = 16;               // lanes
constexpr int kGroupCols = kTraceThreads / kGroupMin;      // groups in a block
// A group takes several nodes a step only while its stack is shallow, so that
// taking one at a time from there on (at most three more entries per level of
// the binary hierarchy, kStackDepth in all) still fits.
constexpr int kGroupShallow = 40;
constexpr int kGroupDepth = kGroupShallow + 3 * (kGroupMax / 4) + kStackDepth;
constexpr int kGroupPairTest = 8;
struct GroupStack {
  int node[kGroupCols][kGroupDepth];
  unsigned short near[kGroupCols][kGroupDepth];  // upper half of the entry distance's bits (not above it)
};

// The search phase of a warp whose lanes work in groups of 1 << lg: every
// group whose leader (lowest lane) has `more` nodes searches to the end.  rs
// points at the group's column and r holds its ray in all of its lanes (r.dns,
// dns64, hs, more and tlim count in the leader).  Warp-collective.
template <int kP>
__device__ __forceinline__ void search_groups(const DevScene &sc, bool lane_tris, const Ray &r, const RaySrc &rs,
                                              double dns64, int *near_node, unsigned short *near_dist, int *err,
                                              HitSearch &hs, bool &more, const WarpPairs &wp, const WarpCount &n_tris,
                                              float tlim, int lg) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = (int)lane_id(), G = 1 << lg;
  const int leader = lane & ~(G - 1), sub = lane & 3, q = (lane & (G - 1)) >> 2;
  const unsigned group = (1u << G) - 1u;
  const Tri *const tris = sc.tris;
  const float3 inv = r.inv, oi = origin_scaled(r);
  const char *const nodes = (const char *)sc.nodes + 4 * sub;
  int root = hs.node, n = 0;
  if (!more || sc.n_tris == 0) root = kNoChild;
  {
    // the root of a one-leaf hierarchy
    const bool leaf = root < 0 && root != kNoChild;
    const unsigned lb = __ballot_sync(kAll, leaf);
    if (leaf) {
      const int pos = __popc(lb & ((1u << lane) - 1u));
      wp.code[pos] = ~root;
      wp.lane[pos] = (unsigned char)lane;
    }
    n = __popc(lb);
  }
  root = __shfl_sync(kAll, root, leader);
  int sp = root >= 0 ? 1 : 0;  // (the same in all lanes of the group)
  if (sp && lane == leader) {
    near_node[0] = root;
    near_dist[0] = 0;
  }
  unsigned run = __ballot_sync(kAll, sp > 0);
  __syncwarp();
  while (run != 0u || n > 0) {
    if (run != 0u) {
      const float tmax = __shfl_sync(kAll, hs.limit<kP>(tlim), leader);
      // this step's nodes: the top `take` of the stack, the nearest first
      const int take = min(sp, sp <= kGroupShallow ? G >> 2 : 1);
      const int at = sp - 1 - q;
      bool hit = false;
      int code = kNoChild;
      float tn = kInf;
      if (q < take && __uint_as_float((unsigned)near_dist[at] << 16) <= tmax) {
        const char *nd = nodes + (size_t)(unsigned)near_node[at] * sizeof(Node4);
        const float lx = __ldg((const float *)nd), hx = __ldg((const float *)(nd + 16));
        const float ly = __ldg((const float *)(nd + 32)), hy = __ldg((const float *)(nd + 48));
        const float lz = __ldg((const float *)(nd + 64)), hz = __ldg((const float *)(nd + 80));
        code = __ldg((const int *)(nd + 96));
        const bool sx = inv.x < 0.0f, sy = inv.y < 0.0f, sz = inv.z < 0.0f;
        hit = slab_nf(inv, oi, sx ? hx : lx, sx ? lx : hx, sy ? hy : ly, sy ? ly : hy, sz ? hz : lz, sz ? lz : hz,
                      tmax, tn);
      }
      const bool leaf = hit && code < 0, inner = hit && code >= 0;
      const unsigned lb = __ballot_sync(kAll, leaf), ib = (__ballot_sync(kAll, inner) >> leader) & group;
      if (leaf) {
        const int pos = n + __popc(lb & ((1u << lane) - 1u));
        wp.code[pos] = ~code;
        wp.lane[pos] = (unsigned char)leader;
      }
      n += __popc(lb);
      // the inner children hit: the nearest node's on top, nearest first
      const unsigned key = inner ? (__float_as_uint(tn) & ~3u) | (unsigned)sub : ~0u;
      const int rank = (int)(__shfl_xor_sync(kAll, key, 1) < key) + (int)(__shfl_xor_sync(kAll, key, 2) < key) +
                       (int)(__shfl_xor_sync(kAll, key, 3) < key);
      const int total = __popc(ib);
      sp += total - take;
      // a well-formed BVH is visited at most once per node; the bound only
      // guarantees termination should the structure ever be malformed.  (The
      // shuffle before the branch: sp differs between a warp's groups.)
      hs.budget -= take;
      const int budget = __shfl_sync(kAll, hs.budget, leader);
      if (sp > kGroupDepth || budget < 0) {
        if (lane == leader) atomicExch(err, sp > kGroupDepth ? BT_E_QUEUE_FULL : BT_E_TIMEOUT);
        sp = 0;
      } else if (inner) {
        const int to = sp - 1 - (__popc(ib & ((1u << (4 * q)) - 1u)) + rank);
        near_node[to] = code;
        near_dist[to] = (unsigned short)(__float_as_uint(tn) >> 16);
      }
      run = __ballot_sync(kAll, sp > 0);
      __syncwarp();
    }
    if (n >= kGroupPairTest || (run == 0u && n > 0)) {
      test_pairs<kP, false, false>(wp, n, tris, lane_tris, r.t_eps, r.dns, rs, dns64, hs, n_tris, tlim, lg);
      n = 0;
    }
  }
  more = false;
}

// Cheap rejection of a segment that cannot reach the microphones' height
// slab: the cone lies on one side of its apex height when all three edge
// directions point the same way in z.  Edge j is along n_{j-1} x n_j times
// the sign of det(n0, n1, n2), which a mirror image flips.  Everything else
// goes to the scatter, which clips the footprint exactly.
__device__ __forceinline__ bool may_reach_slab(float3 n0, float3 n1, float3 n2, float az, const MicGrid &g) {
  float det = n0.x * (n1.y * n2.z - n1.z * n2.y) + n0.y * (n1.z * n2.x - n1.x * n2.z) +
              n0.z * (n1.x * n2.y - n1.y * n2.x);
  float sg = det >= 0.0f ? 1.0f : -1.0f;
  float dz0 = sg * (n2.x * n0.y - n2.y * n0.x);
  float dz1 = sg * (n0.x * n1.y - n0.y * n1.x);
  float dz2 = sg * (n1.x * n2.y - n1.y * n2.x);
  float m = 1e-3f;
  if (dz0 < 0.0f && dz1 < 0.0f && dz2 < 0.0f && az < g.zlo - m) return false;
  if (dz0 > 0.0f && dz1 > 0.0f && dz2 > 0.0f && az > g.zhi + m) return false;
  return true;
}

// The microphone-grid cell under the middle of a segment (of its first 200 m
// when it is longer or escapes), x | y << 16: the place the scatter orders
// segments by, so that segments processed together reach the same
// microphones and accumulators.
__device__ __forceinline__ int seg_cell_key(const MicGrid &g, const Ray &r, float t) {
  const float h = 0.5f * fminf(t, 200.0f);
  const int cx = clampi((int)((r.o.x + r.d.x * h - g.x0) * g.inv_cw), 0, g.nx - 1);
  const int cy = clampi((int)((r.o.y + r.d.y * h - g.y0) * g.inv_ch), 0, g.ny - 1);
  return (cx & 0xffff) | cy << 16;
}

// Warp-aggregated append of a segment record.
__device__ __forceinline__ void emit_segment(const TraceArgs &a, const Seg &s, bool emit,
                                             const WarpCount &n_emit) {
  unsigned mask = __activemask();
  unsigned bal = __ballot_sync(mask, emit);
  if (!bal) return;
  int leader = __ffs(bal) - 1;
  unsigned long long base = 0;
  if ((int)lane_id() == leader) {
    base = atomicAdd(a.seg_count, (unsigned long long)__popc(bal));
    atomicAdd(n_emit.p, (unsigned)__popc(bal));
  }
  base = __shfl_sync(mask, base, leader);
  if (emit) {
    unsigned long long idx = base + __popc(bal & ((1u << lane_id()) - 1u));
    if (idx < a.seg_capacity) a.segs[idx] = s;
    else atomicExch(&a.ctr->error, BT_E_QUEUE_FULL);
  }
}

// Lineage state of one thread, in shared memory (one column per thread) so
// that it holds no registers across the traversal.  Rows: apex 0..2, cone
// normals 3..11, ray origin 12..14, ray direction 15..17; `lo` holds the low
// parts of the float pairs (MIXED only).

constexpr int kRowA = 0, kRowN = 3, kRowO = 12, kRowD = 15, kRows = 18;
// a sub-domain accepts hits up to this far (m along the ray) past its exit
constexpr float kTileEps = 1e-2f;
// per-lane event counters (rows of LineageSmem::cnt)
enum { kCSeg, kCHit, kCEsc, kCEmit, kCHand, kCSteal, kCNodes, kCTris, kNumCounts };
// kC columns, one per lineage a block holds.
template <int kP, int kC>
struct LineageSmem {
  double dv[Prec<kP>::chain64 ? kRows : 1][Prec<kP>::chain64 ? kC : 1];  // float64 chain; `hi` holds its float32 rounding
  float hi[kRows][kC];
  float lo[Prec<kP>::pairs ? kRows : 1][Prec<kP>::pairs ? kC : 1];
  float p[kMaxBands][kC];  // band power W_b prod(r_b)
  float st[4][kC];         // start plane (relative to the apex)
  int pend[Prec<kP>::defer ? kPend + 1 : 1][Prec<kP>::defer ? kC : 1];  // candidates left to float64
};

template <int kP, int kC>
__device__ __forceinline__ df3 ld_df3(const LineageSmem<kP, kC> &sm, int row, int t) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  df3 v;
  v.x = df{sm.hi[row][t], kPairs ? sm.lo[row][t] : 0.0f};
  v.y = df{sm.hi[row + 1][t], kPairs ? sm.lo[row + 1][t] : 0.0f};
  v.z = df{sm.hi[row + 2][t], kPairs ? sm.lo[row + 2][t] : 0.0f};
  return v;
}
template <int kP, int kC>
__device__ __forceinline__ void st_df3(LineageSmem<kP, kC> &sm, int row, int t, df3 v) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  sm.hi[row][t] = v.x.hi;
  sm.hi[row + 1][t] = v.y.hi;
  sm.hi[row + 2][t] = v.z.hi;
  if (kPairs) {
    sm.lo[row][t] = v.x.lo;
    sm.lo[row + 1][t] = v.y.lo;
    sm.lo[row + 2][t] = v.z.lo;
  }
}
template <int kP, int kC>
__device__ __forceinline__ float3 ld_hi3(const LineageSmem<kP, kC> &sm, int row, int t) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  return make_float3(sm.hi[row][t], sm.hi[row + 1][t], sm.hi[row + 2][t]);
}
template <int kP, int kC>
__device__ __forceinline__ void st_f3(LineageSmem<kP, kC> &sm, int row, int t, float3 v) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  sm.hi[row][t] = v.x;
  sm.hi[row + 1][t] = v.y;
  sm.hi[row + 2][t] = v.z;
}

// FP64 rows: the float64 value and its float32 rounding in `hi` (read by the
// float32 traversal and the segment records).
template <int kP, int kC>
__device__ __forceinline__ double3 ld_d3(const LineageSmem<kP, kC> &sm, int row, int t) {
  return make_double3(sm.dv[row][t], sm.dv[row + 1][t], sm.dv[row + 2][t]);
}
template <int kP, int kC>
__device__ __forceinline__ void st_d3(LineageSmem<kP, kC> &sm, int row, int t, double3 v) {
  sm.dv[row][t] = v.x;
  sm.dv[row + 1][t] = v.y;
  sm.dv[row + 2][t] = v.z;
  sm.hi[row][t] = (float)v.x;
  sm.hi[row + 1][t] = (float)v.y;
  sm.hi[row + 2][t] = (float)v.z;
}

// Start lineage `lin` (source si, beam bi) in this thread's column.
template <int kP, int kC>
__device__ __forceinline__ void init_lineage(const SceneView &a, LineageSmem<kP, kC> &sm, int t, int64_t lin) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  const int nb = a.sc.n_bands;
  int64_t si = lin / a.n_beams, bi = lin - si * a.n_beams;
  float4 s4 = __ldg(&a.src[si]);
  float3 A = make_float3(s4.x, s4.y, s4.z);
  if (kChain64) {
    const double2 *bt = reinterpret_cast<const double2 *>(a.beam_table) + 6 * bi;
    double d[12];
#pragma unroll
    for (int q = 0; q < 6; q++) {
      const double2 x = __ldg(bt + q);
      d[2 * q] = x.x;
      d[2 * q + 1] = x.y;
    }
#pragma unroll
    for (int j = 0; j < 3; j++) st_d3(sm, kRowN + 3 * j, t, make_double3(d[3 * j], d[3 * j + 1], d[3 * j + 2]));
    st_d3(sm, kRowD, t, make_double3(d[9], d[10], d[11]));
    const double3 A64 = make_double3(s4.x, s4.y, s4.z);
    st_d3(sm, kRowA, t, A64);
    st_d3(sm, kRowO, t, A64);
  } else if (kPairs) {
    // table: 9 normal components then the 3 axis components, hi parts
    // first, lo parts 12 floats later
    const float *bt = a.beam_table + 24 * bi;
    for (int q = 0; q < 9; q++) {
      sm.hi[kRowN + q][t] = __ldg(bt + q);
      sm.lo[kRowN + q][t] = __ldg(bt + 12 + q);
    }
    for (int q = 0; q < 3; q++) {
      sm.hi[kRowD + q][t] = __ldg(bt + 9 + q);
      sm.lo[kRowD + q][t] = __ldg(bt + 21 + q);
      sm.lo[kRowA + q][t] = 0.0f;
      sm.lo[kRowO + q][t] = 0.0f;
    }
  } else {
    float3 d0, d1, d2;
    beam_dirs<float>(a.level, bi, d0, d1, d2);
    st_f3(sm, kRowN, t, cross_exact(d0, d1));
    st_f3(sm, kRowN + 3, t, cross_exact(d1, d2));
    st_f3(sm, kRowN + 6, t, cross_exact(d2, d0));
    st_f3(sm, kRowD, t, normalize3((d0 + d1) + d2));
  }
  st_f3(sm, kRowA, t, A);
  st_f3(sm, kRowO, t, A);
  // a directional source: its power in this beam's direction (Section 2),
  // the pattern's gain times the omnidirectional power
  float gain = 1.0f;
  if (a.dir_of) {
    const int pat = __ldg(&a.dir_of[si]);
    if (pat >= 0) gain = __ldg(&a.dir_gain[pat * a.n_beams + bi]);
  }
#pragma unroll
  for (int b = 0; b < kMaxBands; b++) sm.p[b][t] = b < nb ? gain * __ldg(&a.power[si * nb + b]) : 0.0f;
  sm.st[0][t] = 0.0f;
  sm.st[1][t] = 0.0f;
  sm.st[2][t] = 0.0f;
  sm.st[3][t] = -kInf;
}

// Per-lane scalars of a lineage besides its shared-memory column.
struct LaneState {
  int64_t lin;
  int k, start_slot;
  float dns;
  double dns64;
};

// Event counts of one launch per warp, in shared memory rather than in
// registers or per lane (4 KB less shared memory a block).  A warp handles at
// most some ten thousand segments per launch, so even its node count stays
// far below 2^32; the launch totals are formed in 64-bit.
struct TraceCounts {
  unsigned *p;  // the warp's counts
  __device__ WarpCount operator[](int i) const { return WarpCount{p + i}; }
};
__device__ __forceinline__ TraceCounts init_counts(unsigned (*wc)[kNumCounts], int t) {
  if ((t & 31) < kNumCounts) wc[t >> 5][t & 31] = 0u;
  __syncwarp();
  return TraceCounts{wc[t >> 5]};
}

// A segment is resolved: its axis ray hit triangle `slot` (or escaped, slot
// < 0).  Write the segment record and, if the beam goes on, reflect it: the
// image source (Section 2), mirrored cone and axis, energy lost at the
// reflection.  Returns true if the lineage continues.
template <int kP, int kC>
__device__ __forceinline__ bool finish_segment(const TraceArgs &a, const SceneView &v, int vi, LineageSmem<kP, kC> &sm,
                                               int t, const Ray &r, const Best &best, int slot, LaneState &ls,
                                               const TraceCounts &cn) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  const int nb = v.sc.n_bands;
  cn[kCSeg]++;
  float4 end = make_float4(0.0f, 0.0f, 0.0f, -kInf);
  float4 v0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float4 plf = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (a.hit_log) {
    // (measurement aid: which triangle each segment's axis ray hit)
    a.hit_log[ls.lin * a.hit_log_stride + ls.k] = slot >= 0 ? __float_as_int(__ldg(&v.sc.tris[slot].v1.w)) : -1;
  }
  if (slot >= 0) {
    cn[kCHit]++;
    v0 = __ldg(&v.sc.tris[slot].v0);
    plf = __ldg(&v.sc.planes[slot]);
    // end plane on the incident side, offset relative to the apex
    float3 pn = f3(plf);
    const bool facing = dot3(pn, r.d) < 0.0f;
    float3 en = facing ? pn : pn * -1.0f;
    float ew;
    if (kChain64) {
      // (with the float64 normal: the float32 one errs by its rounding times
      // the distance to v0, which a triangle of many km makes centimetres, and
      // FP64's scatter sorts microphones out by this offset)
      const Plane64 pl = ldg_d4(&v.sc.planes64[slot]);
      const double w = dot3(make_double3(pl.x, pl.y, pl.z), make_double3(v0.x, v0.y, v0.z) - ld_d3(sm, kRowA, t));
      ew = (float)(facing ? w : -w);
    } else if (kPairs) {
      ew = df3_dot2(mkdf3(en), df3_sub(mkdf3(f3(v0)), ld_df3(sm, kRowA, t))).hi;
    } else {
      ew = dot3(en, f3(v0) - ld_hi3(sm, kRowA, t));
    }
    end = make_float4(en.x, en.y, en.z, ew);
  } else {
    cn[kCEsc]++;
  }
  {
    Seg s;
    for (int q = 0; q < 3; q++) {
      s.ahi[q] = sm.hi[kRowA + q][t];
      s.alo[q] = kPairs ? sm.lo[kRowA + q][t] : 0.0f;
    }
    float3 n0 = ld_hi3(sm, kRowN, t), n1 = ld_hi3(sm, kRowN + 3, t), n2 = ld_hi3(sm, kRowN + 6, t);
    s.n0 = make_float4(n0.x, n0.y, n0.z, __int_as_float(ls.start_slot));
    s.n1 = make_float4(n1.x, n1.y, n1.z, __int_as_float(slot));
    s.n2 = make_float4(n2.x, n2.y, n2.z, __int_as_float(ls.k));
    for (int q = 0; q < 9; q++) s.nlo[q] = kPairs ? sm.lo[kRowN + q][t] : 0.0f;
    s.pad[0] = s.pad[1] = s.pad[2] = 0.0f;
    if (kChain64) {
      // float64 values as float pairs, the apex with a third word so that
      // hi + lo + pad gives it back exactly
      for (int q = 0; q < 3; q++) {
        double x = sm.dv[kRowA + q][t];
        s.alo[q] = (float)(x - (double)s.ahi[q]);
        s.pad[q] = (float)((x - (double)s.ahi[q]) - (double)s.alo[q]);
      }
      for (int q = 0; q < 9; q++) s.nlo[q] = (float)(sm.dv[kRowN + q][t] - (double)sm.hi[kRowN + q][t]);
    }
    s.start = make_float4(sm.st[0][t], sm.st[1][t], sm.st[2][t], sm.st[3][t]);
    s.end = end;
    s.p03 = make_float4(sm.p[0][t], sm.p[1][t], sm.p[2][t], sm.p[3][t]);
    s.p47 = make_float4(sm.p[4][t], sm.p[5][t], sm.p[6][t], sm.p[7][t]);
    s.view = vi;
    const MicGrid &g = *v.grid;
    s.key = v.seg_key ? seg_cell_key(g, r, best.t) : 0;
    emit_segment(a, s, g.n_mics > 0 && may_reach_slab(n0, n1, n2, s.ahi[2], g), cn[kCEmit]);
  }
  if (slot < 0 || ls.k == v.max_order) return false;
  // energy lost at the reflection
  int mat = __float_as_int(v0.w);
  float wmax = 0.0f;
#pragma unroll
  for (int b = 0; b < kMaxBands; b++) {
    float p = sm.p[b][t];
    if (b < nb) p *= __ldg(&v.sc.refl[mat * nb + b]);
    sm.p[b][t] = p;
    wmax = fmaxf(wmax, p);
  }
  if (v.energy_threshold > 0.0f && wmax < v.energy_threshold) return false;
  // Image source: mirror the apex, the cone and the axis in the hit plane;
  // the reflected beam starts at the hit point on that plane.
  float3 pn = f3(plf), pv0 = f3(v0);
  float3 Dn;
  if (kChain64) {
    Plane64 pl = ldg_d4(&v.sc.planes64[slot]);
    const double3 n = make_double3(pl.x, pl.y, pl.z), v0d = make_double3(v0.x, v0.y, v0.z);
    double3 A = ld_d3(sm, kRowA, t), O = ld_d3(sm, kRowO, t), D = ld_d3(sm, kRowD, t);
    const double th = best.has64 ? best.t64 : (pl.w - dot3(n, O)) / dot3(n, D);
    const double3 H = O + D * th;
    A = A - n * (2.0 * dot3(A - v0d, n));
    st_d3(sm, kRowA, t, A);
#pragma unroll
    for (int j = 0; j < 3; j++) {
      double3 nj = ld_d3(sm, kRowN + 3 * j, t);
      st_d3(sm, kRowN + 3 * j, t, nj - n * (2.0 * dot3(nj, n)));
    }
    D = D - n * (2.0 * dot3(D, n));
    st_d3(sm, kRowO, t, H);
    st_d3(sm, kRowD, t, D);
    const double dn = dot3(n, D);
    ls.dns64 = fabs(dn);
    ls.dns = (float)ls.dns64;
    Dn = make_float3((float)D.x, (float)D.y, (float)D.z);
    const double3 sn = dn > 0.0 ? n : n * -1.0;
    const double sw = dot3(sn, v0d - A);
    sm.st[0][t] = (float)sn.x; sm.st[1][t] = (float)sn.y; sm.st[2][t] = (float)sn.z; sm.st[3][t] = (float)sw;
  } else if (kPairs) {
    // in stages, each reading its rows from shared memory and writing them
    // back before the next starts, so that few float pairs are live at once
    // (the compiler fences keep the stages apart)
    PlaneDF pd = v.sc.planes_df[slot];
    const df3 n = df3{df{pd.hi.x, pd.lo.x}, df{pd.hi.y, pd.lo.y}, df{pd.hi.z, pd.lo.z}};
    df kd = df{0.0f, 0.0f}, ka = df{0.0f, 0.0f};
    {
      // the hit point on the plane (the reflected beam's origin); n . D is
      // also the axis' own coefficient in the mirror loop below
      const df3 O = ld_df3(sm, kRowO, t), D = ld_df3(sm, kRowD, t);
      kd = df3_dot2(D, n);
      const df th = best.has64 ? d_to_df(best.t64) : df_div2(df_sub(df{pd.hi.w, pd.lo.w}, df3_dot2(n, O)), kd);
      st_df3(sm, kRowO, t, df3{df_axpy(O.x, th, D.x), df_axpy(O.y, th, D.y), df_axpy(O.z, th, D.z)});
    }
    // the cone normals, the axis and the apex (the image source) mirrored
    // by one copy of the code: v - 2 ((v - p) . n) n with p = 0 for the
    // directions and p = v0, a point of the plane, for the apex
    const df3 p0 = mkdf3(pv0);
#pragma unroll 1
    for (int j = 0; j < 5; j++) {
      asm volatile("" ::: "memory");
      const int row = j < 3 ? kRowN + 3 * j : (j == 3 ? kRowD : kRowA);
      const df3 v = ld_df3(sm, row, t);
      df k = kd;
      if (j != 3) k = df3_dot2(j == 4 ? df3_sub(v, p0) : v, n);
      if (j == 4) ka = k;
      st_df3(sm, row, t, df3_sub2kn(v, k, n));
    }
    asm volatile("" ::: "memory");
    // |n . D| is the same for the axis and its mirror image, and the image
    // source lies as far behind the plane as the apex in front of it
    ls.dns64 = fabs((double)kd.hi + (double)kd.lo);
    ls.dns = (float)ls.dns64;
    Dn = ld_hi3(sm, kRowD, t);
    const bool fwd = dot3(pn, Dn) > 0.0f;
    float3 sn = fwd ? pn : pn * -1.0f;
    float sw = fwd ? ka.hi : -ka.hi;
    sm.st[0][t] = sn.x; sm.st[1][t] = sn.y; sm.st[2][t] = sn.z; sm.st[3][t] = sw;
  } else {
    float3 A = ld_hi3(sm, kRowA, t), O = ld_hi3(sm, kRowO, t), D = ld_hi3(sm, kRowD, t);
    A = A - pn * (2.0f * dot3(A - pv0, pn));
    st_f3(sm, kRowA, t, A);
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float3 nj = ld_hi3(sm, kRowN + 3 * j, t);
      st_f3(sm, kRowN + 3 * j, t, nj - pn * (2.0f * dot3(nj, pn)));
    }
    float3 H = O + D * best.t;
    Dn = D - pn * (2.0f * dot3(D, pn));
    st_f3(sm, kRowO, t, H);
    st_f3(sm, kRowD, t, Dn);
    ls.dns = fabsf(dot3(pn, Dn));
    ls.dns64 = 0.0;
    float3 sn = dot3(pn, Dn) > 0.0f ? pn : pn * -1.0f;
    float sw = dot3(sn, pv0 - A);
    sm.st[0][t] = sn.x; sm.st[1][t] = sn.y; sm.st[2][t] = sn.z; sm.st[3][t] = sw;
  }
  ls.start_slot = slot;
  ls.k++;
  return true;
}

__device__ __forceinline__ void flush_counts(const TraceArgs &a, const TraceCounts &cn, bool count_work) {
  // warp sums in 64-bit
  __syncwarp();
  unsigned long long v[kNumCounts];
  for (int q = 0; q < kNumCounts; q++) v[q] = cn.p[q];
  if (lane_id() == 0) {
    if (count_work) {
      atomicAdd(&a.ctr->nodes_visited, v[kCNodes]);
      atomicAdd(&a.ctr->tris_tested, v[kCTris]);
    }
    atomicAdd(&a.ctr->segments, v[kCSeg]);
    atomicAdd(&a.ctr->hits, v[kCHit]);
    atomicAdd(&a.ctr->escapes, v[kCEsc]);
    atomicAdd(&a.ctr->emitted, v[kCEmit]);
    if (v[kCHand]) atomicAdd(&a.ctr->handoffs, v[kCHand]);
    if (v[kCSteal]) atomicAdd(&a.ctr->steals, v[kCSteal]);
  }
}

// A warp's reservation of lineages, [next, end) relative to the launch's
// first lineage, in shared memory; `last` once the launch's counter has run
// past the end (nothing more to reserve).
struct WarpLineages {
  unsigned long long next, end;
  int last;
};

// Lineages a warp reserves at a time: what its lanes need now, or at least
// beams_per_warp, so that it draws from the launch's counter less often (at
// the price of a coarser end of the launch).
__device__ __forceinline__ unsigned long long reserve_size(const TraceArgs &a, unsigned long long need) {
  const unsigned long long b = (unsigned long long)a.beams_per_warp;
  return need > b ? need : b;
}

// Take the next lineage of the batch for every lane in `need` (warp-vote
// refill): first from the warp's reservation, then from a new one.  Returns
// the lineage index or -1 when the batch is used up.
__device__ __forceinline__ int64_t take_lineage(const TraceArgs &a, bool need, WarpLineages &wl) {
  unsigned nm = __ballot_sync(0xffffffffu, need);
  if (!nm) return -1;
  const unsigned lane = lane_id();
  if (a.beams_per_warp == 0) {
    // as many as the lanes need, straight from the launch's counter
    const int leader = __ffs(nm) - 1;
    unsigned long long base = 0;
    if ((int)lane == leader) base = atomicAdd(a.lineage_next, (unsigned long long)__popc(nm));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (!need) return -1;
    const int64_t mine = a.lineage_begin + (int64_t)(base + __popc(nm & ((1u << lane) - 1u)));
    return mine < a.lineage_end ? mine : -1;
  }
  const unsigned long long total = (unsigned long long)(a.lineage_end - a.lineage_begin);
  const unsigned long long n = (unsigned long long)__popc(nm);
  const unsigned long long next = wl.next, end = wl.end, have = end - next;
  const int last = wl.last;
  unsigned long long b = total, got = 0;
  if (have < n && !last && (int)lane == __ffs(nm) - 1) {
    const unsigned long long R = reserve_size(a, n - have);
    b = atomicAdd(a.lineage_next, R);
    got = b < total ? (b + R < total ? R : total - b) : 0;
    if (b + R >= total) wl.last = 1;
  }
  b = __shfl_sync(0xffffffffu, b, __ffs(nm) - 1);
  got = __shfl_sync(0xffffffffu, got, __ffs(nm) - 1);
  __syncwarp();
  if (lane == 0) {
    if (have < n && !last) {
      const unsigned long long used = n - have < got ? n - have : got;
      wl.next = b + used;
      wl.end = b + got;
    } else {
      wl.next = next + (n < have ? n : have);
    }
  }
  __syncwarp();
  if (!need) return -1;
  const unsigned long long r = (unsigned long long)__popc(nm & ((1u << lane) - 1u));
  if (r < have) return a.lineage_begin + (int64_t)(next + r);
  return r - have < got ? a.lineage_begin + (int64_t)(b + (r - have)) : -1;
}

// Persistent warps: every lane works on one lineage at a time and takes the
// next one from a global counter as soon as its lineage ends, so a warp stays
// full until the batch runs out (warp-vote refill of finished lanes).
// Index of the view whose lineage range holds global lineage `g`; `base`
// holds the views' first lineages in order (a shared-memory copy).
__device__ __forceinline__ int find_view(const int64_t *base, int n_views, int64_t g) {
  int lo = 0, hi = n_views - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (base[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Lanes whose search ended (or whose lineage needs replacing) before a warp
// leaves its search phase to serve them; lanes still searching keep their
// search state and resume afterwards.  Measured on the district: 28 beat 32
// (wait for every lane) by 2.5 %; 24 and below lost, the service phase then
// running too often for too few lanes.
constexpr int kRefillLanes = 28;

// Resident blocks per SM: the traversal is latency-bound, so more warps
// help as long as the spills they force stay light.  Seven (at most 72
// registers a thread) for the single-scene MIXED kernel, whose reflection
// code is small enough (district unsplit 34.2 -> 32.8 ms against six);
// six (80 registers) for the other variants and for batches, whose lanes
// hold their scene's arrays in registers.  kBatch: the lineages of many
// scenes (views) in one launch, each lane on its own lineage's scene.
//
// Each warp alternates two phases.  In the search phase every lane with a ray
// steps through the BVH one node at a time and the warp tests the triangles
// they expose (by pairs: district unsplit 32.8 -> 28.6 ms together with the
// near/far slab test and the wider-first nodes, FP64 on 24 of its sources
// 8.4 -> 4.8 ms a call); the phase ends once kRefillLanes lanes have nothing to
// search (their search finished, or they need a new lineage) or no lane is
// searching.  In the service phase, reconverged, the
// lanes whose search finished write their segment and reflect (or end their
// lineage), lanes without a lineage take new ones, and new searches start --
// while the lanes still searching keep their state, so a long search no longer
// holds the whole warp (dynamic ray fetch, after Aila & Laine 2009).
template <int kP, bool kCount, bool kBatch, bool kLeaves, bool kGroup>
__global__ void __launch_bounds__(kTraceThreads, kP == kPMixed && !kBatch ? 7 : 6) k_trace(TraceArgs a) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  __shared__ LineageSmem<kP, kGroup ? kGroupCols : kTraceThreads> sm;
  __shared__ typename std::conditional<kGroup, GroupStack, char>::type gstack;
  __shared__ int64_t view_base[kBatch ? BT_MAX_SCENES : 1];
  __shared__ WarpLineages wlin[kTraceThreads / 32];
  // kGroup: lanes work in groups of 1 << lg, each on one lineage (column t)
  const int lg = kGroup ? a.group_log2 : 0;
  const int t = (int)threadIdx.x >> lg;
  const int warp = (int)threadIdx.x >> 5;
  if (lane_id() == 0) wlin[warp] = WarpLineages{0ull, 0ull, 0};
  __syncwarp();
  if (kBatch) {
    for (int i = threadIdx.x; i < a.n_views; i += kTraceThreads) view_base[i] = a.views[i].lineage_base;
    __syncthreads();
  }
  __shared__ unsigned wcount[kTraceThreads / 32][kNumCounts];
  const TraceCounts cn = init_counts(wcount, threadIdx.x);
  LaneState ls = {-1, 0, -1, 0.0f, 0.0};
  int vi = 0;  // this lane's scene view
  __shared__ PairQueue<kTraceThreads / 32> pairs;
  const WarpPairs wp = warp_pairs(pairs);
  bool done = (lane_id() & ((1u << lg) - 1u)) != 0;  // (only a group's leader takes lineages)
  bool more = false;        // its search has nodes left to visit
  bool pending = false;     // its search is over and awaits service
  HitSearch hs;
  hs.start(-1, 0);
  int stack[kGroup ? 1 : kStackDepth];
  const RaySrc rs{&sm.hi[kRowO][t], kPairs ? &sm.lo[kRowO][t] : &sm.hi[kRowO][t], kGroup ? kGroupCols : kTraceThreads,
                  kChain64 ? &sm.dv[kRowO][t] : nullptr, kDefer ? &sm.pend[0][t] : nullptr};
  while (true) {
    // ---- service: finished searches write their segment and reflect
    bool fresh = false;
    if (__ballot_sync(0xffffffffu, pending) && pending) {
      const SceneView &v = kBatch ? a.views[vi] : a.v;
      const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
      if constexpr (kDefer) settle_search(v.sc, r, rs, ls.dns64, hs.best, kInf);
      if (finish_segment(a, v, vi, sm, t, r, hs.best, hs.best.slot, ls, cn)) fresh = true;
      else ls.lin = -1;
      pending = false;
    }
    // ---- service: lanes without a lineage take the next ones
    bool need = !done && ls.lin < 0;
    int64_t mine = take_lineage(a, need, wlin[warp]);
    if (need) {
      if (mine >= 0) {
        if (kBatch) {
          vi = find_view(view_base, a.n_views, mine);
          mine += a.views[vi].lineage_first - view_base[vi];
        }
        ls = LaneState{mine, 0, -1, 0.0f, 0.0};
        init_lineage(kBatch ? a.views[vi] : a.v, sm, t, mine);
        fresh = true;
      } else {
        done = true;
      }
    }
    if (fresh) {
      const DevScene &fs = (kBatch ? a.views[vi] : a.v).sc;
      hs.start(fs.root, fs.n_tris);
      if constexpr (kDefer) rs.pend[0] = 0;
      more = true;
    }
    if (__all_sync(0xffffffffu, done)) break;
    // ---- search
    {
      if constexpr (kGroup) {
        // (the group's other lanes read the ray its leader has just written)
        vi = __shfl_sync(0xffffffffu, vi, (int)lane_id() & ~((1 << lg) - 1));
        __syncwarp();
      }
      const SceneView &v = kBatch ? a.views[vi] : a.v;
      const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
      const bool searching = more;
      const int few = max(0, 32 - kRefillLanes - __popc(__ballot_sync(0xffffffffu, done)));
      if constexpr (kGroup) {
        search_groups<kP>(v.sc, kBatch, r, rs, ls.dns64, gstack.node[t], gstack.near[t], &a.ctr->error, hs, more, wp,
                          cn[kCTris], kInf, lg);
        pending = searching;
        continue;
      }
      search_phase<kP, kCount, kLeaves, true>(v.sc, kBatch, r, rs, ls.dns64, stack, &a.ctr->error, hs, more, wp, cn[kCNodes],
                                        cn[kCTris], kInf, few);
      pending = searching && !more;
    }
  }
  flush_counts(a, cn, kCount);
}

// --------------------------------------------------------------- sub-domains
// Device-scope ordered accesses for the hand-off queues.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long v;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
  return v;
}

// Record a watchdog expiry unless an error is already recorded.
__device__ __forceinline__ void watchdog_fired(const TraceArgs &a) { atomicCAS(&a.ctr->error, 0, BT_E_TIMEOUT); }

// Bounded wait until a queue slot's sequence word reaches `want`.  False if
// the watchdog ran out first (an error is then recorded).
__device__ __forceinline__ bool wait_slot(const TraceArgs &a, const TiledArgs &ta, const unsigned *seq, unsigned want) {
  if (ld_acquire_u32(seq) == want) return true;
  const unsigned long long t0 = global_ns();
  while (true) {
    __nanosleep(32);
    if (ld_acquire_u32(seq) == want) return true;
    if (global_ns() - t0 > ta.watchdog_ns) {
      watchdog_fired(a);
      return false;
    }
  }
}

// A lineage's state in a queue slot: S points at row 0, rows c words apart.
// Queue slots are written once and read once by another SM, so both sides
// go through L2 only.
template <int kP, int kC>
__device__ __forceinline__ void save_state(uint32_t *S, size_t c, const LineageSmem<kP, kC> &sm, int t,
                                           const LaneState &ls) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  if (kChain64) {
    // rows 0..35: the float64 chain, low word then high word
    for (int q = 0; q < kRows; q++) {
      unsigned long long b = __double_as_longlong(sm.dv[q][t]);
      __stcg(S + (2 * q) * c, (uint32_t)(b & 0xffffffffu));
      __stcg(S + (2 * q + 1) * c, (uint32_t)(b >> 32));
    }
  } else {
    for (int q = 0; q < kRows; q++) __stcg(S + q * c, __float_as_uint(sm.hi[q][t]));
    if (kPairs)
      for (int q = 0; q < kRows; q++) __stcg(S + (kRows + q) * c, __float_as_uint(sm.lo[q][t]));
  }
  for (int b = 0; b < kMaxBands; b++) __stcg(S + (36 + b) * c, __float_as_uint(sm.p[b][t]));
  for (int q = 0; q < 4; q++) __stcg(S + (44 + q) * c, __float_as_uint(sm.st[q][t]));
  __stcg(S + 48 * c, (uint32_t)(ls.lin & 0xffffffffu));
  __stcg(S + 49 * c, (uint32_t)(ls.lin >> 32));
  __stcg(S + 50 * c, (uint32_t)ls.k);
  __stcg(S + 51 * c, (uint32_t)ls.start_slot);
  __stcg(S + 52 * c, __float_as_uint(ls.dns));
  unsigned long long d = __double_as_longlong(ls.dns64);
  __stcg(S + 53 * c, (uint32_t)(d & 0xffffffffu));
  __stcg(S + 54 * c, (uint32_t)(d >> 32));
}

template <int kP, int kC>
__device__ __forceinline__ void load_state(const uint32_t *S, size_t c, LineageSmem<kP, kC> &sm, int t,
                                           LaneState &ls) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  if (kChain64) {
    for (int q = 0; q < kRows; q++) {
      unsigned long long b = (unsigned long long)__ldcg(S + (2 * q) * c) |
                             ((unsigned long long)__ldcg(S + (2 * q + 1) * c) << 32);
      double x = __longlong_as_double((long long)b);
      sm.dv[q][t] = x;
      sm.hi[q][t] = (float)x;
    }
  } else {
    for (int q = 0; q < kRows; q++) sm.hi[q][t] = __uint_as_float(__ldcg(S + q * c));
    if (kPairs)
      for (int q = 0; q < kRows; q++) sm.lo[q][t] = __uint_as_float(__ldcg(S + (kRows + q) * c));
  }
  for (int b = 0; b < kMaxBands; b++) sm.p[b][t] = __uint_as_float(__ldcg(S + (36 + b) * c));
  for (int q = 0; q < 4; q++) sm.st[q][t] = __uint_as_float(__ldcg(S + (44 + q) * c));
  ls.lin = (int64_t)__ldcg(S + 48 * c) | ((int64_t)__ldcg(S + 49 * c) << 32);
  ls.k = (int)__ldcg(S + 50 * c);
  ls.start_slot = (int)__ldcg(S + 51 * c);
  ls.dns = __uint_as_float(__ldcg(S + 52 * c));
  ls.dns64 = __longlong_as_double(
      (long long)((unsigned long long)__ldcg(S + 53 * c) | ((unsigned long long)__ldcg(S + 54 * c) << 32)));
}

// False if the ray cannot reach any triangle under a subtree root: an empty
// tile, or both child boxes of the root missed (the test a binary traversal
// would make first; the root's binary node, half the bytes of its wide one).
// A single-triangle root is always reachable.
__device__ __forceinline__ bool root_reachable(const Node *bin, int root, const Ray &r) {
  if (root == kNoChild) return false;
  if (root < 0) return true;
  const Node *nd = bin + root;
  float4 lxy = __ldg(&nd->lxy), rxy = __ldg(&nd->rxy), lrz = __ldg(&nd->lrz);
  float tl, tr;
  return slab(r, lxy.x, lxy.y, lxy.z, lxy.w, lrz.x, lrz.y, kInf, tl) ||
         slab(r, rxy.x, rxy.y, rxy.z, rxy.w, lrz.z, lrz.w, kInf, tr);
}

// Take up to `want` queued hand-offs, from the home tile if it has any, else
// from the first tile after it that has (work stealing).  Warp-collective;
// the result is warp-uniform: the tile (-1 if none was taken), the first
// position and the count.  avail[k] counts written items not yet taken; a
// take subtracts and gives back what it could not have, so it never takes
// more than were there.
__device__ __forceinline__ int take_handoffs(const TiledArgs &ta, int home, int want, unsigned &base, int &got) {
  const unsigned lane = lane_id();
  const int T = ta.n_tiles;
  int *head = ta.ctl, *avail = ta.ctl + 2 * T;
  got = 0;
  base = 0;
  int tile = -1;
  for (int off = 0; off < T && tile < 0; off += 32) {
    int q = off + (int)lane;
    int k = home + q;
    if (k >= T) k -= T;
    bool ne = q < T && *(volatile int *)&avail[k] > 0;
    unsigned b = __ballot_sync(0xffffffffu, ne);
    if (b) {
      tile = home + off + __ffs(b) - 1;
      if (tile >= T) tile -= T;
    }
  }
  if (tile < 0) return -1;
  if (lane == 0) {
    int old = atomicSub(&avail[tile], want);
    int g = old < 0 ? 0 : (old < want ? old : want);
    if (g < want) atomicAdd(&avail[tile], want - g);
    if (g > 0) base = (unsigned)atomicAdd(&head[tile], g);
    got = g;
  }
  got = __shfl_sync(0xffffffffu, got, 0);
  base = __shfl_sync(0xffffffffu, base, 0);
  return got > 0 ? tile : -1;
}

// Take up to `want` fresh lineages of the batch without exceeding qcap
// lineages in flight.  A lineage in flight holds one of qcap credits; a warp
// draws credits from the global count in chunks, keeps those of lineages
// that end on it for its next fresh lineages, and gives back any above one
// for each of the `slots` lineages it can hold (drawn for 32 by a warp of lane
// groups, they starved the other warps of a launch with shallow queues: 8 x 8-
// block city split 4 x 4, 40,960 lineages, depth 4,096: 2.51 ms, now 0.72, single
// lanes 1.86).  Warp-collective, warp-uniform result: the first lineage offset
// and the count; *exhausted is set once the batch is used up.
__device__ __forceinline__ int take_fresh(const TraceArgs &a, const TiledArgs &ta, int want, int slots, int &credits,
                                          int64_t &base, bool &exhausted, WarpLineages &wl) {
  int *used = ta.ctl + 3 * ta.n_tiles;
  int got = 0;
  unsigned long long b = 0;
  int ex = 0, c = credits;
  if (lane_id() == 0) {
    const unsigned long long n = (unsigned long long)(a.lineage_end - a.lineage_begin);
    // with beams_per_warp the warp reserves lineages ahead, and a reserved
    // lineage holds its credit from the moment it is reserved, so that
    // reservations never exceed the cap on lineages in flight
    const int bpw = a.beams_per_warp;
    const bool refill = bpw > 0 && wl.next == wl.end && !wl.last;
    const int target = bpw > slots ? bpw : slots;
    if (c < want || (refill && c < target)) {
      int req = target - c;
      int old = atomicAdd(used, req);
      int g = (int)ta.qcap - old;
      g = g < 0 ? 0 : (g < req ? g : req);
      if (g < req) atomicSub(used, req - g);
      c += g;
    }
    if (bpw == 0) {
      int k = c < want ? c : want;
      if (k > 0) {
        b = atomicAdd(a.lineage_next, (unsigned long long)k);
        unsigned long long left = b < n ? n - b : 0;
        if (left <= (unsigned long long)k) ex = 1;
        got = left < (unsigned long long)k ? (int)left : k;
        c -= got;
      }
    } else {
      if (refill && c > 0) {
        const unsigned long long R = (unsigned long long)(c < bpw ? c : bpw);
        const unsigned long long r0 = atomicAdd(a.lineage_next, R);
        wl.next = r0 < n ? r0 : n;
        wl.end = r0 + R < n ? r0 + R : n;
        if (r0 + R >= n) wl.last = 1;
        c -= (int)(wl.end - wl.next);
      }
      const unsigned long long have = wl.end - wl.next;
      got = have < (unsigned long long)want ? (int)have : want;
      b = wl.next;
      wl.next += got;
      if (wl.last && wl.next == wl.end) ex = 1;
    }
    if (ex && c > 0) {  // no fresh lineages left for this warp: its spare credits go back
      atomicSub(used, c);
      c = 0;
    }
  }
  got = __shfl_sync(0xffffffffu, got, 0);
  b = __shfl_sync(0xffffffffu, b, 0);
  credits = __shfl_sync(0xffffffffu, c, 0);
  if (__shfl_sync(0xffffffffu, ex, 0)) exhausted = true;
  base = (int64_t)b;
  return got;
}

// Lanes that must need service before a warp of the split trace leaves its
// search phase: all of them.  A service phase of the split trace polls the
// hand-off queues, so fewer, fuller ones measured faster (60.6 ms against
// 65.0 ms at 28 on the district with 4x4 sub-domains).
constexpr int kRefillTiled = 32;

// Whether the split trace tests triangles by pairs: in FP64, whose triangle
// test is long (a whole-warp float64 instruction costs the same for 4 lanes as
// for 32).  In the other variants the pairs' code, added to the queue code, no
// longer fits the instruction cache beside it (no-instruction stalls 0.9 -> 2.8
// cycles per issue): 44.1 ms against 37.4 ms on the district split 4x4.
template <int kP>
constexpr bool kTilePairs = kP == kPF64;

// Distance along r to its exit from tile (ix, iy) of the grid, in the xy plane.
__device__ __forceinline__ float tile_exit(const TileGrid &tg, int ix, int iy, const Ray &r) {
  float tex = kInf, tey = kInf;
  if (r.d.x > 0.0f) tex = (tg.gx0 + (ix + 1) * tg.wx - r.o.x) / r.d.x;
  else if (r.d.x < 0.0f) tex = (tg.gx0 + ix * tg.wx - r.o.x) / r.d.x;
  if (r.d.y > 0.0f) tey = (tg.gy0 + (iy + 1) * tg.wy - r.o.y) / r.d.y;
  else if (r.d.y < 0.0f) tey = (tg.gy0 + iy * tg.wy - r.o.y) / r.d.y;
  return fminf(tex, tey);
}

// The sub-domain trace (Section 3: the geometry is split into tiles; a beam
// whose ray leaves a tile is sent to the tile it enters; exchanged beams are
// served before new ones; idle workers take work from busy tiles), as one
// persistent launch per batch.  Every warp has a home tile.  Lanes without
// work take, in this order, hand-offs from the home tile's queue, hand-offs
// from the other tiles' queues (a steal), and fresh lineages of the batch.  A
// lineage keeps going while it stays in its tile -- a reflection starts in
// the tile of its hit point -- and is pushed to the queue of the next tile
// when its ray leaves the tile without a hit there.  The launch ends when the
// batch has no fresh lineages left and no lineage is in flight (traced or
// queued).  A warp with nothing to do waits at most watchdog_ns for work;
// waits on a queue slot are bounded the same way.
//
// As in k_trace, each warp alternates a search phase (every lane with a ray
// steps through its tile's hierarchy one node at a time, until kRefillTiled
// lanes need service or none is searching) and a service phase (finished
// searches write their segment and reflect, escape, or are handed to the
// next tile; lanes without a lineage take hand-offs or fresh lineages; new
// searches start), so a long search does not hold the whole warp.
// Resident blocks per SM as for k_trace: seven for the float32 variant,
// whose smaller state fits them (40.7 -> 38.3 ms on the district split 4x4),
// and for MIXED (39.8 against 40.7 ms at six); six for the float64-chain
// variants.
template <int kP, bool kCount, bool kLeaves, bool kGroup>
__global__ void __launch_bounds__(kTraceThreads, kP == kPF32 || kP == kPMixed ? 7 : 6) k_trace_tiled(TraceArgs a, const __grid_constant__ TiledArgs ta) {
  [[maybe_unused]] constexpr bool kPairs = Prec<kP>::pairs, kChain64 = Prec<kP>::chain64, kDefer = Prec<kP>::defer;
  __shared__ LineageSmem<kP, kGroup ? kGroupCols : kTraceThreads> sm;
  __shared__ typename std::conditional<kGroup, GroupStack, char>::type gstack;
  // kGroup: lanes work in groups of 1 << lg, each on one lineage (column t)
  const int lg = kGroup ? a.group_log2 : 0;
  const int t = (int)threadIdx.x >> lg;
  const unsigned lane = lane_id();
  const bool lead = (lane & ((1u << lg) - 1u)) == 0u;  // (only a group's leader takes lineages)
  const int slots = 32 >> lg;                          // lineages the warp can hold
  const unsigned below = (1u << lane) - 1u;
  const SceneView &v = a.v;
  const TileGrid &tg = ta.tg;  // read from parameter space, not held in registers
  __shared__ unsigned wcount[kTraceThreads / 32][kNumCounts];
  const TraceCounts cn = init_counts(wcount, threadIdx.x);
  const size_t qc = ta.qcap;
  const unsigned qmask = ta.qcap - 1u;
  int *const used = ta.ctl + 3 * ta.n_tiles;
  int *const finished = used + 1;
  const int n_batch = (int)(a.lineage_end - a.lineage_begin);
  int credits = 0;  // warp-uniform
  __shared__ WarpLineages wlin[kTraceThreads / 32];
  if (lane == 0) wlin[threadIdx.x >> 5] = WarpLineages{0ull, 0ull, 0};
  __syncwarp();
  LaneState ls = {-1, 0, -1, 0.0f, 0.0};
  bool active = false;      // the lane holds a lineage
  __shared__ PairQueue<kTraceThreads / 32> pairs;
  const WarpPairs wp = warp_pairs(pairs);
  bool more = false;        // its search has nodes left to visit
  bool pending = false;     // its search is over and awaits service
  int tile = -1;
  float tlim = kInf;        // hits are accepted up to this distance
  bool exhausted = false;   // warp-uniform: the batch has no fresh lineages left
  const int home = (int)((blockIdx.x * (kTraceThreads / 32) + (threadIdx.x >> 5)) % (unsigned)ta.n_tiles);
  unsigned long long idle_since = 0, last_prog = 0;
  HitSearch hs;
  hs.start(-1, 0);
  int stack[kGroup ? 1 : kStackDepth];
  const RaySrc rs{&sm.hi[kRowO][t], kPairs ? &sm.lo[kRowO][t] : &sm.hi[kRowO][t], kGroup ? kGroupCols : kTraceThreads,
                  kChain64 ? &sm.dv[kRowO][t] : nullptr, kDefer ? &sm.pend[0][t] : nullptr};
  while (true) {
    // ---- service: finished searches write their segment and reflect, end,
    // or go on to the next tile
    bool start = false, ended = false;
    int next = -1;
    if (__ballot_sync(0xffffffffu, pending) && pending) {
      pending = false;
      const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
      if constexpr (kDefer) settle_search<true>(v.sc, r, rs, ls.dns64, hs.best, tlim);
      // the hit lies in this tile (a reflected beam starts here as well); a
      // ray without one either leaves the grid, and with it every triangle
      // (it escapes), or goes on to the next tile
      int fslot = hs.best.slot;
      bool fin = fslot >= 0;
      if (!fin) {
        // step to the next tile along the ray whose geometry the ray can
        // reach -- tiles whose root boxes it misses could give no hit, so the
        // lane walks past them itself
        int ix = tile % tg.tx, iy = tile / tg.tx;
        bool leaves = false;
        while (true) {
          float tex = kInf, tey = kInf;
          // (by the ray's inverse direction: which tile comes next needs no
          // correctly rounded quotient, the tiles' triangle lists overlap by
          // 5 cm)
          if (r.d.x > 0.0f) tex = (tg.gx0 + (ix + 1) * tg.wx - r.o.x) * r.inv.x;
          else if (r.d.x < 0.0f) tex = (tg.gx0 + ix * tg.wx - r.o.x) * r.inv.x;
          if (r.d.y > 0.0f) tey = (tg.gy0 + (iy + 1) * tg.wy - r.o.y) * r.inv.y;
          else if (r.d.y < 0.0f) tey = (tg.gy0 + iy * tg.wy - r.o.y) * r.inv.y;
          // (a ray that has become NaN leaves too: it has no next tile, and
          // would be handed to its own without end)
          const bool sx = tex <= tey, sy = tey <= tex;
          leaves = (tex == kInf && tey == kInf) || !(sx || sy);
          if (!leaves) {
            if (sx) ix += r.d.x > 0.0f ? 1 : -1;
            if (sy) iy += r.d.y > 0.0f ? 1 : -1;
            leaves = ix < 0 || ix >= tg.tx || iy < 0 || iy >= tg.ty;
          }
          if (leaves || root_reachable(ta.bin, __ldg(&ta.roots[iy * tg.tx + ix]), r)) break;
        }
        if (leaves) fin = true;
        else next = iy * tg.tx + ix;
      }
      // one call site, so that lanes with a hit and lanes that escape run the
      // segment and reflection code together
      if (fin) {
        if (finish_segment(a, v, 0, sm, t, r, hs.best, fslot, ls, cn)) start = true;
        else ended = true;
      }
      if (ended) active = false;
    }
    unsigned em = __ballot_sync(0xffffffffu, ended);
    if (em) {
      credits += __popc(em);
      int give = credits > slots ? credits - slots : 0;
      credits -= give;
      if ((int)lane == __ffs(em) - 1) {
        if (give) atomicSub(used, give);
        atomicAdd(finished, __popc(em));
      }
    }
    // ---- hand-offs: one reservation per target tile, consecutive slots
    bool push = next >= 0;
    unsigned pm = __ballot_sync(0xffffffffu, push);
    if (pm && push) {
      unsigned grp = __match_any_sync(pm, next);
      int gl = __ffs(grp) - 1;
      int n = __popc(grp);
      unsigned base = 0;
      if ((int)lane == gl) base = (unsigned)atomicAdd(&ta.ctl[ta.n_tiles + next], n);
      base = __shfl_sync(grp, base, gl);
      unsigned pos = base + (unsigned)__popc(grp & below), gen = pos & ~qmask, slot = pos & qmask;
      unsigned *sq = ta.seq + (size_t)next * qc + slot;
      // with at most qcap lineages in flight the slot's previous item has
      // been taken; its consumer may still be reading it
      if (wait_slot(a, ta, sq, gen)) {
        save_state(ta.ring + (size_t)next * kStateRows * qc + slot, qc, sm, t, ls);
        // (test hook: the launch's first hand-off is never published, so its
        // consumer's bounded wait runs out)
        if (!ta.withhold || atomicAdd(ta.ctl + 3 * ta.n_tiles + 2, 1) != 0) st_release_u32(sq, gen + 1u);
      }
      __syncwarp(grp);
      if ((int)lane == gl) atomicAdd(&ta.ctl[2 * ta.n_tiles + next], n);
      cn[kCHand]++;
      active = false;
    }
    // ---- refill: hand-offs first (home tile, then steals), then fresh lineages
    unsigned nm = __ballot_sync(0xffffffffu, lead && !active);
    if (nm) {
      unsigned base;
      int got;
      int qt = take_handoffs(ta, home, __popc(nm), base, got);
      if (qt >= 0 && lead && !active) {
        int rank = __popc(nm & below);
        if (rank < got) {
          unsigned pos = base + (unsigned)rank, gen = pos & ~qmask, slot = pos & qmask;
          unsigned *sq = ta.seq + (size_t)qt * qc + slot;
          // the item is counted in avail only after it is written, but the
          // position handed out may belong to a producer still writing
          if (wait_slot(a, ta, sq, gen + 1u)) {
            load_state(ta.ring + (size_t)qt * kStateRows * qc + slot, qc, sm, t, ls);
            st_release_u32(sq, gen + ta.qcap);
            tile = qt;
            active = true;
            start = true;
            if (qt != home) cn[kCSteal]++;
          }
        }
      }
      nm = __ballot_sync(0xffffffffu, lead && !active);
      if (nm && !exhausted) {
        int64_t fb;
        int got_f = take_fresh(a, ta, __popc(nm), slots, credits, fb, exhausted, wlin[threadIdx.x >> 5]);
        int rank = __popc(nm & below);
        if (lead && !active && rank < got_f) {
          int64_t mine = a.lineage_begin + fb + rank;
          ls = LaneState{mine, 0, -1, 0.0f, 0.0};
          init_lineage(v, sm, t, mine);
          active = true;
          start = true;
          float3 o = ld_hi3(sm, kRowO, t);
          tile = clampi((int)floorf((o.y - tg.gy0) / tg.wy), 0, tg.ty - 1) * tg.tx +
                 clampi((int)floorf((o.x - tg.gx0) / tg.wx), 0, tg.tx - 1);
        }
      }
    }
    if (start) {
      // Hits are searched up to 1 cm past the ray's exit from the tile (the
      // tile lists hold every triangle within 5 cm of the tile): a hit there
      // is the ray's first, and a ray with none goes on to the next tile.
      const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
      tlim = tile_exit(tg, tile % tg.tx, tile / tg.tx, r) + kTileEps;
      // (a ray that has become NaN hits nothing; search_phase by single lanes
      // would take an unused lane of a node for a leaf of its)
      hs.start(isnan(r.o.x + r.o.y + r.o.z) ? kNoChild : __ldg(&ta.roots[tile]), v.sc.n_tris);
      if constexpr (kDefer) rs.pend[0] = 0;
      more = true;
    }
    if (!__any_sync(0xffffffffu, active)) {
      // nothing to trace: done once every lineage of the batch has finished
      const int fin = *(volatile int *)finished;
      if (fin == n_batch) break;
      if (*(volatile int *)&a.ctr->error) break;
      // the watchdog runs while the launch as a whole makes no progress: no
      // fresh lineage taken and none finished (both counts only grow)
      const unsigned long long now = global_ns();
      const unsigned long long prog = *(volatile unsigned long long *)a.lineage_next + (unsigned)fin;
      if (idle_since == 0 || prog != last_prog) {
        idle_since = now;
        last_prog = prog;
      } else if (now - idle_since > ta.watchdog_ns) {
        if (lane == 0) watchdog_fired(a);
        break;
      }
      __nanosleep(128);
      continue;
    }
    idle_since = 0;
    // ---- search: until kRefillTiled lanes need service (a finished search,
    // or no lineage while fresh ones remain) or no lane is searching
    {
      const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
      const bool searching = more;
      if constexpr (kGroup) {
        __syncwarp();
        const Ray r = make_ray(ld_hi3(sm, kRowO, t), ld_hi3(sm, kRowD, t), v.t_eps, ls.dns);
        search_groups<kP>(v.sc, false, r, rs, ls.dns64, gstack.node[t], gstack.near[t], &a.ctr->error, hs, more, wp,
                          cn[kCTris], tlim, lg);
        pending = searching;
        continue;
      }
      const int few = max(0, 32 - kRefillTiled - __popc(__ballot_sync(0xffffffffu, !active && exhausted)));
      search_phase<kP, kCount, kLeaves, kTilePairs<kP>>(v.sc, false, r, rs, ls.dns64, stack, &a.ctr->error, hs, more, wp, cn[kCNodes],
                                        cn[kCTris], tlim, few);
      pending = searching && !more;
    }
  }
  flush_counts(a, cn, kCount);
}

// Lanes that work on one lineage, as a power of two, for a launch of n
// lineages: 16 or 8 while the chip's lanes (seven blocks per SM) are enough to
// give every lineage some, which its chain of dependent fetches needs more than
// the launch needs throughput.  Measured (trace kernel, us, 1 / 8 / 16 lanes per
// lineage; district and an 8 x 8-block city, order 4, MIXED):
//   lineages   5,120  170/77/65 and 134/63/59
//             10,240  168/79/75 and 139/69/77
//             40,960  280/180/231 and 155/141/201
//             61,440  301/216/292 and 191/188/280
//   split 4 x 4  5,120  350/165/223 and 393/149/210
//               40,960  688/571/671 and 491/542/673
// (32 lanes were slower than 16 everywhere.)  There are no group kernels for the float64
// chain and for FP32 split: on the city 8 lanes would pay below some 10,000 and
// 30,000 lineages (5,120, 10,240, 40,960: FP64 200/128/163, 202/182/258,
// 244/489/778; MIXED64 151/92/124, 157/114/174, 176/303/535; FP32 split
// 323/129/180, 387/215/325, 426/444/525), which is left to be taken up.
// A warp of groups holds 32 >> log2 lineages, so it reserves that share of
// beams_per_warp: with all of it a warp went through its reservation two at a
// time while others had none (8 x 8-block city, 5,120 lineages, 256 a warp: 4.79
// ms, by shares 0.35, single lanes 0.86).
// With fewer blocks per SM than fit (the blocks_per_sm knob) the lines move down:
// unsplit with up to five, which do what seven do, split with all.  8 x 8-block
// city, 1 / 8 / 16 lanes:
//   1 block:  5,120 133/86/118, 10,240 135/143/217, 40,960 196/459/708
//   2 blocks: 10,240 137/96/133, 20,480 143/155/231, 40,960 157/276/411
//   split, 1 block:  5,120 167/147/192, 10,240 174/294/446, 40,960 262/849/1,288
//   split, 2 blocks: 10,240 210/229/317, 20,480 217/360/520
template <int kP>
static int group_log2(int64_t n, int n_sm, int blocks_per_sm, bool split) {
  if (Prec<kP>::chain64) return 0;
  const int blocks = blocks_per_sm > 0 && blocks_per_sm < 7 ? blocks_per_sm : 7;
  const int64_t sm_lanes = (int64_t)n_sm * kTraceThreads;
  if (split) {
    const int64_t lanes = sm_lanes * blocks;
    return n <= lanes / 16 ? 4 : (n <= lanes * 3 / 8 ? 3 : 0);
  }
  if (blocks < 5) return n <= sm_lanes * blocks * 3 / 32 ? 4 : (n <= sm_lanes * blocks * 17 / 32 ? 3 : 0);
  return n <= sm_lanes * 7 / 16 ? 4 : (n <= sm_lanes * 7 * 3 / 8 ? 3 : 0);
}

template <int kP, bool kCount, bool kLeaves, bool kGroup>
static cudaError_t launch_tiled_t(cudaStream_t st, const TraceArgs &a, const TiledArgs &ta, int n_sm) {
  static OccCache occ;
  int per_sm = 0;
  cudaError_t e = occ.get(&per_sm, k_trace_tiled<kP, kCount, kLeaves, kGroup>, kTraceThreads);
  if (e != cudaSuccess) return e;
  if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
  if (per_sm < 1) per_sm = 1;
  int64_t blocks = (int64_t)n_sm * per_sm;
  if (kGroup) {
    // no more blocks than lineages need, all or (with shallow queues) those in
    // flight: warps without work poll the queues, which slows a small launch
    // down (5,120 lineages split 4 x 4: 262 -> 190 us)
    const int cols = kTraceThreads >> a.group_log2;
    const int64_t all = a.lineage_end - a.lineage_begin, most = all < (int64_t)ta.qcap ? all : (int64_t)ta.qcap;
    const int64_t need = (most + cols - 1) / cols;
    if (blocks > need) blocks = need;
  }
  k_trace_tiled<kP, kCount, kLeaves, kGroup><<<(int)blocks, kTraceThreads, 0, st>>>(a, ta);
  return cudaGetLastError();
}

template <int kP>
static cudaError_t launch_tiled_p(cudaStream_t st, const TraceArgs &a0, const TiledArgs &ta, int n_sm) {
  TraceArgs a = a0;
  a.group_log2 = group_log2<kP>(a.lineage_end - a.lineage_begin, n_sm, a.blocks_per_sm, true);
  if (a.leaf_size > 1)
    return a.count_work ? launch_tiled_t<kP, true, true, false>(st, a, ta, n_sm)
                        : launch_tiled_t<kP, false, true, false>(st, a, ta, n_sm);
  if (a.count_work) return launch_tiled_t<kP, true, false, false>(st, a, ta, n_sm);
  if constexpr (kP == kPMixed)
    if (a.group_log2 > 0) {
      a.beams_per_warp >>= a.group_log2;
      return launch_tiled_t<kP, false, false, true>(st, a, ta, n_sm);
    }
  return launch_tiled_t<kP, false, false, false>(st, a, ta, n_sm);
}

cudaError_t launch_trace_tiled(cudaStream_t st, const TraceArgs &a, const TiledArgs &ta, int n_sm) {
  cudaError_t e;
  if (a.prec == kPMixed) e = launch_tiled_p<kPMixed>(st, a, ta, n_sm);
  else if (a.prec == kPF64) e = launch_tiled_p<kPF64>(st, a, ta, n_sm);
  else if (a.prec == kPMixed64) e = launch_tiled_p<kPMixed64>(st, a, ta, n_sm);
  else e = launch_tiled_p<kPF32>(st, a, ta, n_sm);
  note_launches(1);
  return e;
}

int tiled_resident_lanes(int n_sm) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trace_tiled<kPMixed, false, false, false>, kTraceThreads, 0) !=
      cudaSuccess)
    per_sm = 8;
  if (per_sm < 1) per_sm = 1;
  return n_sm * per_sm * kTraceThreads;
}

// Closest hit of arbitrary float32 rays (the axis-ray query of the trace
// kernel on its own), decided as in MIXED mode with the float32 origin and
// the float64-normalised direction as float pairs.  ns: optional start-plane
// normals.
__global__ void __launch_bounds__(128) k_cast(DevScene sc, const float *o, const float *d, const float *ns,
                                              int64_t n, float t_eps, float *t_out, int *tri_out, int *err) {
  __shared__ float rh[6][128], rl[6][128];
  __shared__ int pend[kPend + 1][128];
  __shared__ PairQueue<4> pairs;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool mine = i < n;  // (a warp's lanes search together, so none returns early)
  const int t = threadIdx.x;
  float3 O = make_float3(0.0f, 0.0f, 0.0f);
  double3 Dd = make_double3(0.0, 0.0, 1.0);
  double dns = 0.0;
  if (mine) {
    O = make_float3(o[3 * i], o[3 * i + 1], o[3 * i + 2]);
    Dd = normalize3(make_double3(d[3 * i], d[3 * i + 1], d[3 * i + 2]));
    if (ns) dns = fabs(dot3(Dd, make_double3(ns[3 * i], ns[3 * i + 1], ns[3 * i + 2])));
  }
  df3 D = df3{d_to_df(Dd.x), d_to_df(Dd.y), d_to_df(Dd.z)};
  rh[0][t] = O.x; rh[1][t] = O.y; rh[2][t] = O.z;
  rl[0][t] = 0.0f; rl[1][t] = 0.0f; rl[2][t] = 0.0f;
  rh[3][t] = D.x.hi; rh[4][t] = D.y.hi; rh[5][t] = D.z.hi;
  rl[3][t] = D.x.lo; rl[4][t] = D.y.lo; rl[5][t] = D.z.lo;
  pend[0][t] = 0;
  Ray r = make_ray(O, df3_hi(D), t_eps, (float)dns);
  const WarpCount none{nullptr};
  const RaySrc rs{&rh[0][t], &rl[0][t], 128, nullptr, &pend[0][t]};
  const WarpPairs wp = warp_pairs(pairs);
  int stack[kStackDepth];
  HitSearch hs;
  hs.start(sc.root, sc.n_tris);
  // a ray with a NaN or infinite origin or direction hits nothing
  bool more = mine && isfinite(O.x) && isfinite(O.y) && isfinite(O.z) && isfinite(Dd.x) && isfinite(Dd.y) && isfinite(Dd.z);
  search_phase<kPMixed, false, true, true>(sc, false, r, rs, dns, stack, err, hs, more, wp, none, none, kInf, 0);
  if (!mine) return;
  Best &best = hs.best;
  settle_search(sc, r, rs, dns, best, kInf);
  const int slot = best.slot;
  // the reported distance is the float64 one to the hit triangle's plane
  // along the float-pair ray (the search itself decides in float32)
  double t64 = best.t64;
  if (slot >= 0 && !best.has64) {
    double3 o64, d64;
    rs.get(o64, d64);
    t64 = plane_t64(sc, slot, o64, d64);
  }
  t_out[i] = slot >= 0 ? (float)t64 : kInf;
  tri_out[i] = slot >= 0 ? best.id : -1;
}

cudaError_t launch_cast(cudaStream_t st, const DevScene &sc, const float *o, const float *d, const float *ns,
                        int64_t n, float t_eps, float *t_out, int *tri_out, int *err) {
  if (n <= 0) return cudaSuccess;
  k_cast<<<(int)((n + 127) / 128), 128, 0, st>>>(sc, o, d, ns, n, t_eps, t_out, tri_out, err);
  note_launches(1);
  return cudaGetLastError();
}

// One persistent grid: enough blocks to fill every SM at the kernel's
// occupancy, each block looping until the batch's lineages are taken.
template <int kP, bool kCount, bool kBatch, bool kLeaves, bool kGroup>
static cudaError_t launch_trace_t(cudaStream_t st, const TraceArgs &a, int n_sm) {
  static OccCache occ;
  int per_sm = 0;
  cudaError_t e = occ.get(&per_sm, k_trace<kP, kCount, kBatch, kLeaves, kGroup>, kTraceThreads);
  if (e != cudaSuccess) return e;
  if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
  if (per_sm < 1) per_sm = 1;
  int64_t n = a.lineage_end - a.lineage_begin;
  int64_t blocks = (int64_t)n_sm * per_sm;
  const int cols = kTraceThreads >> (kGroup ? a.group_log2 : 0);
  int64_t need = (n + cols - 1) / cols;
  if (blocks > need) blocks = need;
  k_trace<kP, kCount, kBatch, kLeaves, kGroup><<<(int)blocks, kTraceThreads, 0, st>>>(a);
  return cudaGetLastError();
}

template <int kP, bool kBatch>
static cudaError_t launch_trace_p(cudaStream_t st, const TraceArgs &a0, int n_sm) {
  TraceArgs a = a0;
  a.group_log2 = group_log2<kP>(a.lineage_end - a.lineage_begin, n_sm, a.blocks_per_sm, false);
  if (a.leaf_size > 1)
    return a.count_work ? launch_trace_t<kP, true, kBatch, true, false>(st, a, n_sm)
                        : launch_trace_t<kP, false, kBatch, true, false>(st, a, n_sm);
  if (a.count_work) return launch_trace_t<kP, true, kBatch, false, false>(st, a, n_sm);
  if constexpr (!Prec<kP>::chain64)
    if (a.group_log2 > 0) {
      a.beams_per_warp >>= a.group_log2;  // as many for each lineage that a warp holds
      return launch_trace_t<kP, false, kBatch, false, true>(st, a, n_sm);
    }
  return launch_trace_t<kP, false, kBatch, false, false>(st, a, n_sm);
}

template <bool kBatch>
static cudaError_t launch_trace_b(cudaStream_t st, const TraceArgs &a, int n_sm) {
  if (a.prec == kPMixed) return launch_trace_p<kPMixed, kBatch>(st, a, n_sm);
  if (a.prec == kPF64) return launch_trace_p<kPF64, kBatch>(st, a, n_sm);
  if (a.prec == kPMixed64) return launch_trace_p<kPMixed64, kBatch>(st, a, n_sm);
  return launch_trace_p<kPF32, kBatch>(st, a, n_sm);
}

cudaError_t launch_trace(cudaStream_t st, const TraceArgs &a, int n_sm) {
  cudaError_t e = a.views ? launch_trace_b<true>(st, a, n_sm) : launch_trace_b<false>(st, a, n_sm);
  note_launches(1);
  return e;
}

}  // namespace bt
