// Certified FP32 geometry shared by both arithmetic policies: outward-rounded vector helpers,
// points as float pairs, the closest-point classification, box bounds, and the upper bounds
// u1..u3 of a sub-triangle.  MIXED computes its results with them; FP64 uses them as filters
// that decide where the FP64 arithmetic is needed at all (FP64 runs at 1/64 of the FP32 rate
// on GB300).
#pragma once

#include "hd_internal.cuh"

namespace hd {

constexpr float kU = 5.9604644775390625e-08f;  // 2^-24

struct F3 {
  float x, y, z;
};
__device__ inline F3 f3(float x, float y, float z) { return {x, y, z}; }
__device__ inline F3 operator+(F3 a, F3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ inline F3 operator-(F3 a, F3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ inline float dotf(F3 a, F3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ inline float sum1(F3 a) { return __fadd_ru(__fadd_ru(fabsf(a.x), fabsf(a.y)), fabsf(a.z)); }
__device__ inline float amax3(F3 a) { return fmaxf(fabsf(a.x), fmaxf(fabsf(a.y), fabsf(a.z))); }
// Square root and quotient with outward rounding: the correctly rounded (round-to-nearest)
// result is within half an ulp, so one multiplication by 1 +- 2^-23, rounded outward, bounds
// the exact value.
// Square roots rounded up / down, from x * rsqrtf(x): rsqrtf is within 2 ulp (4u relative,
// the CUDA math library's documented bound) and the product adds u, so the result is within
// 5u of sqrt(x); one multiplication by 1 +- 8u in the matching direction covers that.  Tiny
// and infinite arguments take the safe branch (the product would be 0 * inf there).
__device__ inline float sqrt_up(float x) {
  if (!(x >= 1e-30f && x < INFINITY)) return x < 1e-30f ? 1e-15f : x;
  return __fmul_ru(x * rsqrtf(x), 1.f + 8.f * kU);
}
__device__ inline float sqrt_dn(float x) {
  if (!(x >= 1e-30f && x < INFINITY)) return x < 1e-30f ? 0.f : x;
  return __fmul_rd(x * rsqrtf(x), 1.f - 8.f * kU);
}
__device__ inline float div_up(float a, float b) { return __fmul_ru(__fdiv_rn(a, b), 1.f + 2.f * kU); }
__device__ inline float div_dn(float a, float b) { return __fmul_rz(__fdiv_rn(a, b), 1.f - 2.f * kU); }
__device__ inline float norm_ru(F3 a) { return sqrt_up(__fmaf_ru(a.x, a.x, __fmaf_ru(a.y, a.y, __fmul_ru(a.z, a.z)))); }
__device__ inline float norm_rd(F3 a) { return sqrt_dn(__fmaf_rd(a.x, a.x, __fmaf_rd(a.y, a.y, __fmul_rd(a.z, a.z)))); }

// A point as the unevaluated sum h + l of two float triples.
struct FFP {
  F3 h, l;
};

// x - p for a float point x, taken locally: (x - h) - l.
__device__ inline F3 local_off(float4 x, const FFP& p) {
  return {(x.x - p.h.x) - p.l.x, (x.y - p.h.y) - p.l.y, (x.z - p.h.z) - p.l.z};
}

// Barycentric weights (v, w) of the point of triangle (A, B, C) closest to the origin,
// Voronoi-region classification, clamped so that v, w >= 0 and v + w <= 1 exactly.
// Returns the region: 0 face, 1 edge AB, 2 edge AC, 3 edge BC, 4 vertex (A, B or C).
// Degenerate triangles and extreme slivers (|AB x AC|^2 below 1e-5 |AB|^2 |AC|^2, where the
// region tests are ill-conditioned or, with a zero-length edge, wrong) take the nearest of
// the three edges.
__device__ inline int closest_edge_bary(F3 A, F3 B, F3 C, float& v, float& w) {
  F3 e[3] = {B - A, C - B, A - C};
  F3 o[3] = {A, B, C};
  float best = INFINITY;
  int region = 1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float ee = dotf(e[k], e[k]);
    float t = ee > 0.f ? fminf(fmaxf(-dotf(o[k], e[k]) / ee, 0.f), 1.f) : 0.f;
    F3 q = {fmaf(t, e[k].x, o[k].x), fmaf(t, e[k].y, o[k].y), fmaf(t, e[k].z, o[k].z)};
    float dq = dotf(q, q);
    if (dq < best) {
      best = dq;
      int r = (t == 0.f || t == 1.f) ? 4 : (k == 0 ? 1 : (k == 1 ? 3 : 2));
      region = r;
      if (k == 0) { v = t; w = 0.f; }
      else if (k == 1) { v = __fsub_rd(1.f, t); w = t; }
      else { v = 0.f; w = __fsub_rd(1.f, t); }
    }
  }
  return region;
}

__device__ inline int closest_bary(F3 A, F3 B, F3 C, float& v, float& w) {
  F3 ab = B - A, ac = C - A;
  v = 0.f;
  w = 0.f;
  float aa = dotf(ab, ab), cc = dotf(ac, ac), bc = dotf(ab, ac);
  if (!(aa * cc - bc * bc > 1e-5f * aa * cc)) return closest_edge_bary(A, B, C, v, w);
  float d1 = -dotf(ab, A), d2 = -dotf(ac, A);
  if (d1 <= 0.f && d2 <= 0.f) return 4;
  float d3 = -dotf(ab, B), d4 = -dotf(ac, B);
  if (d3 >= 0.f && d4 <= d3) {
    v = 1.f;
    return 4;
  }
  float vc = d1 * d4 - d3 * d2;
  if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) {
    float den = d1 - d3;
    v = den > 0.f ? fminf(fmaxf(d1 / den, 0.f), 1.f) : 0.f;
    return 1;
  }
  float d5 = -dotf(ab, C), d6 = -dotf(ac, C);
  if (d6 >= 0.f && d5 <= d6) {
    w = 1.f;
    return 4;
  }
  float vb = d5 * d2 - d1 * d6;
  if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) {
    float den = d2 - d6;
    w = den > 0.f ? fminf(fmaxf(d2 / den, 0.f), 1.f) : 0.f;
    return 2;
  }
  float va = d3 * d6 - d5 * d4;
  if (va <= 0.f && (d4 - d3) >= 0.f && (d5 - d6) >= 0.f) {
    float den = (d4 - d3) + (d5 - d6);
    float t = den > 0.f ? fminf(fmaxf((d4 - d3) / den, 0.f), 1.f) : 0.f;
    v = __fsub_rd(1.f, t);
    w = t;
    return 3;
  }
  float den = va + vb + vc;
  if (!(den > 0.f)) return closest_edge_bary(A, B, C, v, w);
  float inv = 1.f / den;
  v = fminf(fmaxf(vb * inv, 0.f), 1.f);
  w = fminf(fmaxf(vc * inv, 0.f), __fsub_rd(1.f, v));
  return 0;
}

// min over the vertices of n . X, rounded down, for |n| <= 1 (support-function lower bound)
__device__ inline float support_rd(F3 n, F3 A, F3 B, F3 C) {
  float da = __fmaf_rd(n.x, A.x, __fmaf_rd(n.y, A.y, __fmul_rd(n.z, A.z)));
  float db = __fmaf_rd(n.x, B.x, __fmaf_rd(n.y, B.y, __fmul_rd(n.z, B.z)));
  float dc = __fmaf_rd(n.x, C.x, __fmaf_rd(n.y, C.y, __fmul_rd(n.z, C.z)));
  return fminf(da, fminf(db, dc));
}

// n scaled so that |n| <= 1 (rounded toward zero); false if n is zero
__device__ inline bool unit_rz(F3& n) {
  float l = norm_ru(n);
  if (!(l > 0.f)) return false;
  float s = div_dn(1.f, l);
  n = {__fmul_rz(n.x, s), __fmul_rz(n.y, s), __fmul_rz(n.z, s)};
  return true;
}

// Lower bound of |p - box|^2 (downward rounding), with p given by an enclosure
// [plo, phi] of the float pair h + l on each axis (h + l rounded down and up).
__device__ inline float box_lo2(F3 plo, F3 phi, float lx, float ly, float lz, float hx, float hy, float hz) {
  float gx = fmaxf(fmaxf(__fsub_rd(lx, phi.x), __fsub_rd(plo.x, hx)), 0.f);
  float gy = fmaxf(fmaxf(__fsub_rd(ly, phi.y), __fsub_rd(plo.y, hy)), 0.f);
  float gz = fmaxf(fmaxf(__fsub_rd(lz, phi.z), __fsub_rd(plo.z, hz)), 0.f);
  return __fmaf_rd(gx, gx, __fmaf_rd(gy, gy, __fmul_rd(gz, gz)));
}

// Shared edge of triangles f, g of B (equal vertex indices of their F_B rows): returns
// true with the slots of the two shared vertices in f and the opposite slots in f and g.
__device__ inline bool shared_edge(const BvhDev& B, int f, int g, int& fs0, int& fs1, int& fo, int& go) {
  int4 a = __ldg(B.tri_vid + f), b = __ldg(B.tri_vid + g);
  int av[3] = {a.x, a.y, a.z}, bv[3] = {b.x, b.y, b.z};
  bool ash[3];
  int nsh = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) ash[i] = (av[i] == bv[0] || av[i] == bv[1] || av[i] == bv[2]);
  // distinct shared vertex indices of f
  int sl[3], ns = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (!ash[i]) continue;
    bool dup = false;
    for (int k = 0; k < ns; ++k) dup |= av[sl[k]] == av[i];
    if (!dup) sl[ns++] = i;
  }
  nsh = ns;
  if (nsh != 2) return false;
  fs0 = sl[0];
  fs1 = sl[1];
  fo = go = -1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (av[i] != av[fs0] && av[i] != av[fs1]) fo = i;
    if (bv[i] != av[fs0] && bv[i] != av[fs1]) go = i;
  }
  return fo >= 0 && go >= 0;
}

// Upper bound of the same squared distance (upward rounding): |p - box|^2 lies in
// [box_lo2, box_hi2] for every p in the enclosure.
__device__ inline float box_hi2(F3 plo, F3 phi, float lx, float ly, float lz, float hx, float hy, float hz) {
  float gx = fmaxf(fmaxf(__fsub_ru(lx, plo.x), __fsub_ru(phi.x, hx)), 0.f);
  float gy = fmaxf(fmaxf(__fsub_ru(ly, plo.y), __fsub_ru(phi.y, hy)), 0.f);
  float gz = fmaxf(fmaxf(__fsub_ru(lz, plo.z), __fsub_ru(phi.z, hz)), 0.f);
  return __fmaf_ru(gx, gx, __fmaf_ru(gy, gy, __fmul_ru(gz, gz)));
}

// Certified lower bound of d(p, S) for the float triangle S = (a4, b4, c4): the support
// function along the direction the closest-point classification gives (any direction of at
// most unit length is valid; the classification only decides how tight it is).  M receives
// the largest local coordinate.  Non-finite arithmetic ends in 0.
// With `hi`, also an upper bound (the length of the point found plus the 48 u M margin of
// pt_cert), or +inf for an ill-conditioned triangle (the classification's own threshold):
// there a closest point computed in FP64 can be farther than the true one.  The triangle B was
// given may be ill-conditioned where its float form is not, so +inf too unless eta is far
// below the edges (the threshold leaves a height of 4e-3 of the shorter edge).
__device__ inline float pt_lo(const FFP& P, float4 a4, float4 b4, float4 c4, float& M, float* hi = nullptr,
                              float eta = 0.f) {
  const F3 A = local_off(a4, P), B = local_off(b4, P), C = local_off(c4, P);
  M = fmaxf(fmaxf(amax3(A), amax3(B)), fmaxf(amax3(C), amax3(P.l)));
  float v, w;
  const int region = closest_bary(A, B, C, v, w);
  const F3 E1 = B - A, E2 = C - A;
  const F3 Q = {fmaf(w, E2.x, fmaf(v, E1.x, A.x)), fmaf(w, E2.y, fmaf(v, E1.y, A.y)), fmaf(w, E2.z, fmaf(v, E1.z, A.z))};
  if (hi) {
    const float aa = dotf(E1, E1), cc = dotf(E2, E2), bc = dotf(E1, E2);
    const bool sound = aa * cc - bc * bc > 2e-5f * aa * cc && eta * eta <= 1e-6f * fminf(aa, cc);
    *hi = sound ? __fadd_ru(norm_ru(Q), __fmul_ru(48.f * kU, M)) : INFINITY;
  }
  F3 n = Q;  // vertex region
  if (region == 0) {  // face: the plane normal
    const F3 np = {E1.y * E2.z - E1.z * E2.y, E1.z * E2.x - E1.x * E2.z, E1.x * E2.y - E1.y * E2.x};
    n = dotf(np, Q) >= 0.f ? np : F3{-np.x, -np.y, -np.z};
  } else if (region != 4) {  // edge: Q less its component along the edge
    const F3 e = region == 1 ? E1 : (region == 2 ? E2 : C - B);
    const float ee = dotf(e, e), qe = dotf(Q, e);
    if (ee > 0.f) n = {Q.x * ee - e.x * qe, Q.y * ee - e.y * qe, Q.z * ee - e.z * qe};
  }
  if (!unit_rz(n)) return 0.f;
  return fmaxf(__fsub_rd(support_rd(n, A, B, C), __fmul_ru(6.f * kU, M)), 0.f);
}

// ----------------------------------------------------------------------------- bounds u1..u3

struct VM {  // one vertex of T in the cascade
  FFP p;
  float dhi;
  int I;
  F3 q;  // closest point relative to p
  float qerr;
};

// Certified edge vector p_j - p_i (components carry a relative error of about 2u).
__device__ inline F3 edge(const VM& a, const VM& b) { return (b.p.h - a.p.h) + (b.p.l - a.p.l); }
__device__ inline float len_hi(F3 e) { return __fmul_ru(norm_ru(e), 1.f + 4.f * kU); }
__device__ inline float len_lo(F3 e) { return __fmul_rd(norm_rd(e), 1.f - 4.f * kU); }

// The edges of T, e[i] opposite vertex i (v2 - v1, v0 - v2, v1 - v0), and their lengths
// rounded up: computed once per item for u1 and u2.
struct EdgesM {
  F3 e[3];
  float hi[3];
  __device__ explicit EdgesM(const VM t[3]) {
    e[0] = edge(t[1], t[2]);
    e[1] = edge(t[2], t[0]);
    e[2] = edge(t[0], t[1]);
#pragma unroll
    for (int i = 0; i < 3; ++i) hi[i] = len_hi(e[i]);
  }
};

// u1, Eq. (u1), with edge lengths rounded up: vertex i's two edges are the two not opposite it
__device__ inline float ubm_u1(const VM t[3], const EdgesM& E) {
  const float u0 = __fadd_ru(fmaxf(E.hi[1], E.hi[2]), t[0].dhi);
  const float u1 = __fadd_ru(fmaxf(E.hi[2], E.hi[0]), t[1].dhi);
  const float u2 = __fadd_ru(fmaxf(E.hi[0], E.hi[1]), t[2].dhi);
  return fminf(u0, fminf(u1, u2));
}

// u2, Eq. (u2): g is half the longest edge when T is certainly obtuse (longest edge squared,
// rounded down, above the sum of the other two squared, rounded up), else the circumradius
// with the area rounded down.  Acute <=> s - r > 2R, so this is the paper's g wherever the
// sign of the test is certain, and the circumradius (always a valid g) elsewhere.
__device__ inline float ubm_u2(const VM t[3], const EdgesM& E) {
  // the longest edge k and the other two, selected by branches (no runtime array index, so
  // the edges stay in registers)
  F3 ek = E.e[0];
  float hk = E.hi[0], h1 = E.hi[1], h2 = E.hi[2];
  if (E.hi[1] > hk && E.hi[1] >= E.hi[2]) {
    ek = E.e[1];
    hk = E.hi[1];
    h1 = E.hi[2];
    h2 = E.hi[0];
  } else if (E.hi[2] > hk && E.hi[2] > E.hi[1]) {
    ek = E.e[2];
    hk = E.hi[2];
    h1 = E.hi[0];
    h2 = E.hi[1];
  }
  const float lok = len_lo(ek);
  float g;
  if (__fmul_rd(lok, lok) > __fmaf_ru(h1, h1, __fmul_ru(h2, h2))) {
    g = __fmul_ru(0.5f, hk);
  } else {
    F3 a = E.e[2], b = {-E.e[1].x, -E.e[1].y, -E.e[1].z};  // v1 - v0 and v2 - v0
    F3 cr = {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
    float err = __fmul_ru(__fmul_ru(32.f * kU, amax3(a)), amax3(b));
    float c2 = __fsub_rd(norm_rd(cr), err);  // lower bound of 2|T|
    g = c2 > 0.f ? div_up(__fmul_ru(__fmul_ru(E.hi[0], E.hi[1]), E.hi[2]), __fmul_rd(2.f, c2)) : INFINITY;
  }
  return __fadd_ru(g, fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi)));
}

// Lower bound of u2 for every g its acute test may choose: g is at least half the longest edge,
// and the circumradius (rounded down) where T is certainly acute, which is asked only where
// the former stays below `enough`.  0 where an edge leaves the float range.
__device__ inline float ubm_u2_lo(const VM t[3], const EdgesM& E, float enough) {
  float lo[3];  // norm_ru is within 2^-18 above the length, or 1e-15 of it (sqrt_up)
#pragma unroll
  for (int i = 0; i < 3; ++i) lo[i] = fmaxf(__fsub_rd(__fmul_rd(E.hi[i], 1.f - 0x1p-18f), 2e-15f), 0.f);
  const float hk = fmaxf(E.hi[0], fmaxf(E.hi[1], E.hi[2]));
  if (!(hk < INFINITY)) return 0.f;
  const float d = __fmul_rd(fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi)), 1.f - 0x1p-20f);
  float g = 0.5f * fmaxf(lo[0], fmaxf(lo[1], lo[2]));
  if (__fadd_rd(g, d) < enough &&
      __fmaf_rd(lo[0], lo[0], __fmaf_rd(lo[1], lo[1], __fmul_rd(lo[2], lo[2]))) > __fmul_ru(__fmul_ru(2.f, hk), hk)) {
    const F3 a = E.e[2], b = {-E.e[1].x, -E.e[1].y, -E.e[1].z};
    const F3 cr = {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
    const float c2 = __fadd_ru(norm_ru(cr), __fmul_ru(__fmul_ru(32.f * kU, amax3(a)), amax3(b)));  // 2|T|, rounded up
    g = fmaxf(g, div_dn(__fmul_rd(__fmul_rd(lo[0], lo[1]), lo[2]), __fmul_ru(2.f, c2)));
  }
  return __fadd_rd(g, d);
}

// Lower bound of u4 whichever edge of T is taken for the shortest: H(q_i, q_j) is at least the
// distance from the third vertex to the nearer of q_i and q_j.  The distances are plain float,
// within 16 u M of the exact ones (M: the largest coordinate relative to T's first vertex).
__device__ inline float ubm_u4_lo(const VM t[3]) {
  const F3 x[3] = {f3(0.f, 0.f, 0.f), edge(t[0], t[1]), edge(t[0], t[2])};
  const F3 q[3] = {t[0].q, x[1] + t[1].q, x[2] + t[2].q};
  float d2 = INFINITY;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const F3 a = x[i] - q[(i + 1) % 3], b = x[i] - q[(i + 2) % 3];
    d2 = fminf(d2, fminf(dotf(a, a), dotf(b, b)));
  }
  const float M = fmaxf(fmaxf(amax3(x[1]), amax3(x[2])), fmaxf(amax3(t[0].q), fmaxf(amax3(t[1].q), amax3(t[2].q))));
  return __fsub_rd(sqrt_dn(d2), __fmul_ru(0x1p-18f, M));
}

// Upper bound of d(x, S) for the float triangle S = (a4, b4, c4), x = h + l, computed without
// branches: the distance to the projection of x onto the plane of S when it falls inside S
// (well-conditioned triangles only), else to the nearest of the three edge projections.  Any
// point of S gives an upper bound, so the parameters need not be exact; they only have to lie
// in [0, 1] (the face point: v, w >= 0, v + w <= 1), and the point built from a vertex, the
// parameters and the edge vectors carries the same rounding as in pt_cert, covered by the
// same 48 u M margin.
__device__ inline float pt_hi(const FFP& P, float4 a4, float4 b4, float4 c4) {
  F3 A = local_off(a4, P), B = local_off(b4, P), C = local_off(c4, P);
  float M = fmaxf(fmaxf(amax3(A), amax3(B)), fmaxf(amax3(C), amax3(P.l)));
  F3 E1 = B - A, E2 = C - A, E3 = C - B;
  float d00 = dotf(E1, E1), d01 = dotf(E1, E2), d11 = dotf(E2, E2);
  float a1 = -dotf(A, E1), a2 = -dotf(A, E2);
  // edge parameters; a zero-length edge gives 0/0 = NaN, which saturates to 0
  float t1 = __saturatef(__fdividef(a1, d00)), t2 = __saturatef(__fdividef(a2, d11));
  float t3 = __saturatef(__fdividef(-dotf(B, E3), dotf(E3, E3)));
  F3 Q = {fmaf(t1, E1.x, A.x), fmaf(t1, E1.y, A.y), fmaf(t1, E1.z, A.z)};
  F3 Q2 = {fmaf(t2, E2.x, A.x), fmaf(t2, E2.y, A.y), fmaf(t2, E2.z, A.z)};
  F3 Q3 = {fmaf(t3, E3.x, B.x), fmaf(t3, E3.y, B.y), fmaf(t3, E3.z, B.z)};
  float n = dotf(Q, Q), n2 = dotf(Q2, Q2), n3 = dotf(Q3, Q3);
  if (n2 < n) { Q = Q2; n = n2; }
  if (n3 < n) Q = Q3;
  float den = d00 * d11 - d01 * d01;
  if (den > 1e-5f * d00 * d11) {
    float r = __fdividef(1.f, den);
    float v = (d11 * a1 - d01 * a2) * r, w = (d00 * a2 - d01 * a1) * r;
    if (v >= 0.f && w >= 0.f && v + w <= 1.f) {
      w = fminf(w, __fsub_rd(1.f, v));  // v + w <= 1 exactly
      Q = {fmaf(w, E2.x, fmaf(v, E1.x, A.x)), fmaf(w, E2.y, fmaf(v, E1.y, A.y)), fmaf(w, E2.z, fmaf(v, E1.z, A.z))};
    }
  }
  return __fadd_ru(norm_ru(Q), __fmul_ru(48.f * kU, M));
}

__device__ inline float dist_hi(const BvhDev& B, int j, const FFP& x, float beta) {
  const float4* t = B.tri32 + 3 * (size_t)j;
  return __fadd_ru(pt_hi(x, __ldg(t), __ldg(t + 1), __ldg(t + 2)), beta);
}

// Point base + s * e (s in [0, 1]) as a float pair, with its representation error.
__device__ inline FFP along(const VM& base, F3 e, float s, float& beta) {
  FFP x;
  x.h = base.p.h;
  x.l = {fmaf(s, e.x, base.p.l.x), fmaf(s, e.y, base.p.l.y), fmaf(s, e.z, base.p.l.z)};
  beta = __fmul_ru(8.f * kU, fmaxf(amax3(e), amax3(base.p.l)));
  return x;
}

// u3 (Kang et al. 2018), Eqs. (Kang2018_case1) and (Kang2018_case2).  Both cases start with
// point-triangle distances that are laid out as six evaluation slots, so that the lanes of a
// warp run the same code whichever case each item is in: case 1 fills four slots, (b1, S1),
// (b2, S1), (b1, S2), (b2, S2); case 2 fills all six with (v_j, S_i), j != i.
//
// With kAgree the value also bounds u3 with case 1's split points chosen in FP64 on B's own
// coordinates: the points differ by at most the error of the split parameters times the edge,
// which is added, and +inf is returned where rounding leaves open whether the split points or
// the edge midpoints are used (a vertex of T close to the bisecting plane, as where A's edges
// follow B's).
template <bool kAgree = false>
__device__ inline float ubm_u3(const BvhDev& B, const VM t[3], float l, unsigned& evals) {
  int lone = -1;
  if (!(t[0].I == t[1].I && t[1].I == t[2].I)) {
    if (t[1].I == t[2].I) lone = 0;
    else if (t[0].I == t[2].I) lone = 1;
    else if (t[0].I == t[1].I) lone = 2;
  }
  int fs0, fs1, fo, go;
  // v1 is the vertex alone on its triangle; selected by branches (no runtime array index, so
  // the three vertices stay in registers)
  VM v1 = t[0], v2 = t[1], v3 = t[2];
  if (lone == 1) { v1 = t[1]; v2 = t[2]; v3 = t[0]; }
  else if (lone == 2) { v1 = t[2]; v2 = t[0]; v3 = t[1]; }
  const bool c1 = lone >= 0 && shared_edge(B, v1.I, v2.I, fs0, fs1, fo, go);
  const int S1 = v1.I, S2 = v2.I;
  FFP b1 = v1.p, b2 = v1.p;
  float be1 = 0.f, be2 = 0.f;
  float apart = kAgree ? INFINITY : 0.f;  // kAgree: how far the FP64 split points may be from these
  if (c1) {
    F3 e12 = edge(v1, v2), e13 = edge(v1, v3);
    // split parameters: the bisecting plane of the two supporting half-planes (any value
    // in [0, 1] gives a valid split; this choice only affects tightness)
    float s2 = 0.5f, s3 = 0.5f;
    const float4* T1 = B.tri32 + 3 * (size_t)S1;
    const float4* T2 = B.tri32 + 3 * (size_t)S2;
    float4 P0 = __ldg(T1 + fs0), P1 = __ldg(T1 + fs1), O1 = __ldg(T1 + fo), O2 = __ldg(T2 + go);
    F3 p0 = {P0.x, P0.y, P0.z}, ed = F3{P1.x, P1.y, P1.z} - p0;
    // (plain fast arithmetic: any split parameter in [0, 1] gives a valid bound)
    const float ee = dotf(ed, ed);
    if (ee > 0.f) {
      const float ie = rsqrtf(ee);
      F3 eh = {ed.x * ie, ed.y * ie, ed.z * ie};
      F3 a1 = F3{O1.x, O1.y, O1.z} - p0, a2 = F3{O2.x, O2.y, O2.z} - p0;
      float k1 = dotf(a1, eh), k2 = dotf(a2, eh);
      F3 w1 = {a1.x - k1 * eh.x, a1.y - k1 * eh.y, a1.z - k1 * eh.z};
      F3 w2 = {a2.x - k2 * eh.x, a2.y - k2 * eh.y, a2.z - k2 * eh.z};
      const float q1 = dotf(w1, w1), q2 = dotf(w2, w2);
      if (q1 > 0.f && q2 > 0.f) {
        const float i1 = rsqrtf(q1), i2 = rsqrtf(q2);
        F3 nb = {w1.x * i1 - w2.x * i2, w1.y * i1 - w2.y * i2, w1.z * i1 - w2.z * i2};
        F3 r1 = (v1.p.h - p0) + v1.p.l;
        float sv1 = dotf(nb, r1), sv2 = sv1 + dotf(nb, e12), sv3 = sv1 + dotf(nb, e13);
        if constexpr (kAgree) {
          // the errors: of w1 and w2 relative to their lengths (the rounding of the projections,
          // and eta in each vertex of B), hence of nb (|nb| <= 2), and of the side values
          const float eta = __ldg(B.meta), n1 = sum1(a1), n2 = sum1(a2);
          const float d = 2.f * ((32.f * kU * n1 + 4.f * eta * (1.f + n1 * ie)) * i1 +
                                 (32.f * kU * n2 + 4.f * eta * (1.f + n2 * ie)) * i2) + 32.f * kU;
          const float s1 = sum1(r1), s12 = sum1(e12), s13 = sum1(e13);
          const float E1 = s1 * (d + 16.f * kU) + 4.f * eta, E2 = E1 + s12 * (d + 16.f * kU), E3 = E1 + s13 * (d + 16.f * kU);
          const bool yes = sv1 > E1 && sv2 < -E2 && sv3 < -E3, no = sv1 < -E1 || sv2 > E2 || sv3 > E3;
          if (yes) apart = 2.f * fmaxf(E2 * s12 / (sv1 - sv2), E3 * s13 / (sv1 - sv3));
          if (no) apart = 0.f;
        }
        if (sv1 >= 0.f && sv2 <= 0.f && sv3 <= 0.f && sv1 - sv2 > 0.f && sv1 - sv3 > 0.f) {
          s2 = __saturatef(__fdividef(sv1, sv1 - sv2));
          s3 = __saturatef(__fdividef(sv1, sv1 - sv3));
        }
      }
    }
    b1 = along(v1, e12, s2, be1);
    b2 = along(v1, e13, s3, be2);
  }
  const float dmax = fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi));
  // The slots, two at a time.  The loops below are not unrolled: with every evaluation inlined
  // (15 copies of the point-triangle code) the kernels outgrew the instruction cache, and
  // waiting for instructions was their largest stall (4 to 6 cycles per instruction issued,
  // now 1 to 1.7).  On the batch of 128 pairs the bounds went from 21.7 to 18.6 ms, on the
  // large soup from 0.093 to 0.083 ms; the torus pair's stayed at 0.10 ms.  The loops keep
  // their points in local memory, so they want 128 registers (96: 18.6, 0.089, 0.109 ms).
  float u = dmax, best = INFINITY;
#pragma unroll 1
  for (int i = 0; i < (c1 ? 2 : 3); ++i) {
    // case 1: both split points against S1, then S2; case 2: the two other vertices against S_i
    const VM &x = i == 0 ? t[1] : i == 1 ? t[2] : t[0], &y = i == 0 ? t[2] : i == 1 ? t[0] : t[1];
    const int S = c1 ? (i == 0 ? S1 : S2) : i == 0 ? t[0].I : i == 1 ? t[1].I : t[2].I;
    const float own = i == 0 ? t[0].dhi : i == 1 ? t[1].dhi : t[2].dhi;
    const FFP p0 = c1 ? b1 : x.p, p1 = c1 ? b2 : y.p;
    const float d = fmaxf(dist_hi(B, S, p0, c1 ? be1 : 0.f), dist_hi(B, S, p1, c1 ? be2 : 0.f));
    u = fmaxf(u, d);
    best = fminf(best, fmaxf(own, d));
  }
  if (c1) {
    evals += 4;
    return kAgree ? __fadd_ru(u, apart) : u;
  }
  // case 2: u3 = min(u3~, min_i h(T, S_i)).  The second term comes from the slots: once it is
  // below l the item is discarded whatever u3~ is (U of a discarded item is not used
  // further), and the quadrilateral maximum u3~ is abandoned as soon as it reaches the
  // current minimum, since it can then no longer lower it.
  evals += 6;
  if (best < l) return best;
  // quadrilaterals (v_i, m_i, b, m_{i-1}) against S_i
  F3 e01 = edge(t[0], t[1]), e02 = edge(t[0], t[2]), e12 = edge(t[1], t[2]);
  float bm[3];
  FFP m[3];
  m[0] = along(t[0], e01, 0.5f, bm[0]);
  m[1] = along(t[1], e12, 0.5f, bm[1]);
  m[2] = along(t[0], e02, 0.5f, bm[2]);  // m3 on v3v1
  F3 sum = e01 + e02;
  float bb;
  FFP bc = along(t[0], sum, 1.f / 3.f, bb);
  bb = __fmul_ru(16.f * kU, fmaxf(amax3(e01), fmaxf(amax3(e02), amax3(t[0].p.l))));
  float ut = dmax;
#pragma unroll 1
  for (int k = 0; k < 9; ++k) {
    const int i = k / 3, j = k - 3 * i;  // j: m_i, b, m_{i-1}
    if (j == 0) {
      if (ut >= best) break;
      evals += 3;
    }
    const int S = i == 0 ? t[0].I : i == 1 ? t[1].I : t[2].I;
    const int q = j == 0 ? i : i == 0 ? 2 : i - 1;
    const FFP x = j == 1 ? bc : q == 0 ? m[0] : q == 1 ? m[1] : m[2];
    ut = fmaxf(ut, dist_hi(B, S, x, j == 1 ? bb : q == 0 ? bm[0] : q == 1 ? bm[1] : bm[2]));
  }
  return fminf(ut, best);
}

}  // namespace hd
