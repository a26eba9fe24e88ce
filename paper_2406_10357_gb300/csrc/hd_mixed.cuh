// Certified FP32 policy (HD_MIXED).
//
// Distances and bounds run in float with directed rounding where a bound needs it, so that
// every lower bound stays below and every upper bound above the exact value:
//
//  * Positions of sub-triangle vertices are pairs of floats h + l (l holds the rounding
//    residual of the exact midpoint), and every geometric difference is taken locally,
//    (x - h) - l, so rounding errors scale with local sizes (distances, triangle sizes),
//    not with the coordinates.
//  * Point-triangle distance: the closest point is found on the local triangle by
//    Voronoi-region classification (Ericson 2005) with barycentric weights clamped into
//    the simplex, so it is a point of the triangle up to a few units of rounding; its
//    length plus an a-priori error term (48 u M, M the local magnitude, u = 2^-24) is an
//    upper bound.  The lower bound is a support-function certificate: for any n with
//    |n| <= 1, d(p, S) >= min over the vertices X of S of n.(X - p), evaluated with
//    downward rounding; n is chosen by the closest point's region (the plane normal for
//    the face, the closest-point direction less its along-edge component for an edge, the
//    direction itself for a vertex), which makes it tight whenever the classification was
//    right.  If the certificate is loose (near-degenerate sliver, where the barycentric
//    test is ill-conditioned), the test is redone in FP64.
//  * Terms of u3 need only upper bounds, and any point of the triangle gives one: there
//    the closest point is found without branches (plane projection if inside, else the
//    nearest edge projection) with the same margin.
//  * Box distances for pruning are lower bounds (downward rounding); pruning compares
//    them with the best certified upper bound, so the minimum of the tested lower bounds
//    is a lower bound of d(p, B).
//  * Bounds of Section 3.2 take certified vertex distances (upper bounds), edge lengths
//    rounded up, the circumradius only with the area rounded down, and the split points of
//    u3 with their representation error added.  u4 is certified in FP32 too: the vertex and
//    footpoint differences are float pairs formed with error-free sums, and each remaining
//    rounded dot product or norm is raised by a bound on its error (ubm_u4).
#pragma once

#include "hd_fp64.cuh"
#include "hd_internal.cuh"

namespace hd {

struct PtOut {
  float hi;    // >= d(p, S)
  float lo;    // <= d(p, S)
  F3 q;        // closest point relative to p
  float qerr;  // a point of S lies within qerr of p + q
  bool esc;    // redone in FP64
};

// The FP64 redo of pt_cert for ill-conditioned cases (rare): not inlined, so that its
// double-precision temporaries do not add to the register budget of the traversal.
static __device__ __noinline__ void pt_escalate(FFP P, float4 a4, float4 b4, float4 c4, float M, PtOut& o) {
  D3 p = {(double)P.h.x + (double)P.l.x, (double)P.h.y + (double)P.l.y, (double)P.h.z + (double)P.l.z};
  D3 a = {a4.x, a4.y, a4.z}, b = {b4.x, b4.y, b4.z}, c = {c4.x, c4.y, c4.z};
  D3 q = closest_on_triangle(p, a, b, c) - p;  // a point of the triangle, relative to p
  double d = len(q);
  // covers the double rounding of these few operations, done in absolute coordinates
  double m = 1e-12 * ((double)M + d + fmax(fabs(p.x), fmax(fabs(p.y), fabs(p.z)))) + 1e-30;
  // support-function lower bounds along the closest-point direction and both plane normals:
  // the first is tight when the nearest point is on an edge or vertex, the others when it
  // is inside the face
  D3 Ad = a - p, Bv = b - p, Cv = c - p;
  auto support = [&](D3 nn) {
    double s = len(nn);
    if (!(s > 0.0)) return 0.0;
    nn = (1.0 / (s * (1.0 + 1e-15))) * nn;
    return fmin(dot(nn, Ad), fmin(dot(nn, Bv), dot(nn, Cv)));
  };
  D3 N = cross(Bv - Ad, Cv - Ad);
  double lo64 = fmax(support(q), fmax(support(N), support((-1.0) * N))) - m;
  o.esc = true;
  o.lo = fmaxf(o.lo, __double2float_rd(fmax(lo64, 0.0)));
  float hi64 = __double2float_ru(d + m);
  if (hi64 < o.hi) {
    o.hi = hi64;
    o.q = {(float)q.x, (float)q.y, (float)q.z};
    // float rounding of q plus the double margin
    o.qerr = __double2float_ru(3e-7 * (fabs(q.x) + fabs(q.y) + fabs(q.z)) + m);
  }
}

// Certified distance from p = h + l to the float triangle (a, b, c).
__device__ inline void pt_cert(const FFP& P, float4 a4, float4 b4, float4 c4, bool want_lo, PtOut& o) {
  F3 A = local_off(a4, P), B = local_off(b4, P), C = local_off(c4, P);
  float M = fmaxf(fmaxf(amax3(A), amax3(B)), fmaxf(amax3(C), amax3(P.l)));
  float v, w;
  int region = closest_bary(A, B, C, v, w);
  F3 E1 = B - A, E2 = C - A;
  F3 Q = {fmaf(w, E2.x, fmaf(v, E1.x, A.x)), fmaf(w, E2.y, fmaf(v, E1.y, A.y)), fmaf(w, E2.z, fmaf(v, E1.z, A.z))};
  float nq = norm_ru(Q);
  o.hi = __fadd_ru(nq, __fmul_ru(48.f * kU, M));
  o.q = Q;
  o.qerr = __fmul_ru(40.f * kU, M);
  o.esc = false;
  o.lo = 0.f;
  if (!want_lo) return;
  // Support direction by region, so that the certificate stays tight when the triangle is
  // much larger than the distance (the direction of Q alone carries an error of about u M / d):
  // face -> the plane normal; edge -> Q with its component along the edge removed;
  // vertex -> Q, which is then the vertex itself.
  F3 n = Q;
  if (region == 0) {
    F3 np = {E1.y * E2.z - E1.z * E2.y, E1.z * E2.x - E1.x * E2.z, E1.x * E2.y - E1.y * E2.x};
    n = dotf(np, Q) >= 0.f ? np : F3{-np.x, -np.y, -np.z};
  } else if (region != 4) {
    F3 e = region == 1 ? E1 : (region == 2 ? E2 : C - B);
    float ee = dotf(e, e), qe = dotf(Q, e);
    if (ee > 0.f) n = {Q.x * ee - e.x * qe, Q.y * ee - e.y * qe, Q.z * ee - e.z * qe};
  }
  float lo = 0.f;
  if (unit_rz(n)) lo = fmaxf(__fsub_rd(support_rd(n, A, B, C), __fmul_ru(6.f * kU, M)), 0.f);
  o.lo = lo;
  // a loose certificate means the classification was ill-conditioned: redo in FP64
  if (__fsub_rd(nq, lo) > __fmul_ru(256.f * kU, M)) pt_escalate(P, a4, b4, c4, M, o);
}

struct NearestM {
  FFP P;
  const float4* tri32;
  float best_hi = INFINITY;
  float dlo = INFINITY;
  float cut = -1.f;   // the traversal may stop once best_hi < cut (cut_radius)
  float cut2 = -1.f;  // cut squared, for the farthest-point box test
  int best = -1;
  F3 q = {0.f, 0.f, 0.f};
  float qerr = 0.f;
  unsigned evals = 0, esc = 0;
  __device__ float radius2() const { return __fmul_ru(best_hi, best_hi); }
  __device__ float coop_r2() const { return radius2(); }
  __device__ void test1(int j) {
    const float4* t = tri32 + 3 * (size_t)j;
    PtOut o;
    pt_cert(P, __ldg(t), __ldg(t + 1), __ldg(t + 2), true, o);
    ++evals;
    esc += o.esc;
    dlo = fminf(dlo, o.lo);
    if (o.hi < best_hi) {
      best_hi = o.hi;
      best = j;
      q = o.q;
      qerr = o.qerr;
    }
  }
  __device__ void coop_range(int first, int count, float) {
    for (int j = first; j < first + count; ++j) test1(j);
  }
};

// Ordered depth-first traversal with certified float box bounds, in the "while-while" form
// of Aila and Laine (HPG 2009): each lane expands inner nodes until it holds a pending leaf
// range, then the lanes that hold one test one triangle each, together.  The expensive
// certified point-triangle test thus runs with most lanes of the warp active, and the cheap
// node steps absorb the divergence.  Stack entries pack a node index (count 0) or a leaf
// range (first, count) into 32 bits: count in bits 27..31, index below (n_B < 2^27).
// Compare-exchange of (distance, code) pairs, smaller distance first.
__device__ inline void sort2(float& ea, unsigned& ca, float& eb, unsigned& cb) {
  if (eb < ea) {
    float e = ea;
    ea = eb;
    eb = e;
    unsigned c = ca;
    ca = cb;
    cb = c;
  }
}

// Push a child found within the radius (distance < +inf) onto the traversal stack.
__device__ inline void push_code(unsigned* stack_code, float* stack_d, int& sp, unsigned code, float d,
                                 Counters& c) {
  if (!(d < INFINITY)) return;
  if (sp < kStack) {
    stack_code[sp] = code;
    stack_d[sp] = d;
    ++sp;
  } else {
    c.err = 1;  // stack overflow: the subtree is skipped and the error reported
  }
}

// Must be called by all 32 lanes of the warp; inactive lanes start finished.  A lane that
// has tested more than `budget` triangles stops unfinished before its next stack pop and sets
// `over` (t then holds its best so far); one whose best distance bound fell below t.cut stops
// there too and sets `cut` (kCut only: the traversal without the check is a separate
// instantiation, as in traverse_coop).
template <bool kCut>
__device__ inline void traverse_m(const BvhDev& B, NearestM& t, Counters& c, bool active, int budget,
                                  bool& over, bool& cut) {
  unsigned stack_code[kStack];
  float stack_d[kStack];
  int sp = 0;
  int node = active ? 0 : -1;  // inner node to expand next, -1 = none
  int lfirst = 0, lcount = 0;
  bool done = !active;
  // an enclosure of the query point h + l, for the box bounds
  const F3 plo = {__fadd_rd(t.P.h.x, t.P.l.x), __fadd_rd(t.P.h.y, t.P.l.y), __fadd_rd(t.P.h.z, t.P.l.z)};
  const F3 phi = {__fadd_ru(t.P.h.x, t.P.l.x), __fadd_ru(t.P.h.y, t.P.l.y), __fadd_ru(t.P.h.z, t.P.l.z)};
  for (;;) {
    while (!done && lcount == 0) {
      if (node < 0) {
        if constexpr (kCut) {
          if (t.best_hi < t.cut) {
            cut = done = true;
            continue;
          }
        }
        bool found = false;
        while (sp > 0) {
          --sp;
          if (stack_d[sp] <= t.radius2()) {
            unsigned code = stack_code[sp];
            int cnt = (int)(code >> 27), ref = (int)(code & 0x07ffffffu);
            if (cnt > 0) { lfirst = ref; lcount = cnt; }
            else node = ref;
            found = true;
            break;
          }
        }
        if (!found) done = true;
        if (!done && (int)t.evals > budget) over = done = true;  // hand the query off
        continue;
      }
      const float4* np = reinterpret_cast<const float4*>(B.nodes + node);
      const float4 lx = __ldg(np), ly = __ldg(np + 1), lz = __ldg(np + 2);
      const float4 hx = __ldg(np + 3), hy = __ldg(np + 4), hz = __ldg(np + 5);
      const uint4 cd = __ldg(reinterpret_cast<const uint4*>(np + 6));
      ++c.nodes;
      const float r2 = t.radius2();
      // children within the current radius (the others at +inf), nearest first
      float e0 = box_lo2(plo, phi, lx.x, ly.x, lz.x, hx.x, hy.x, hz.x);
      float e1 = box_lo2(plo, phi, lx.y, ly.y, lz.y, hx.y, hy.y, hz.y);
      float e2 = box_lo2(plo, phi, lx.z, ly.z, lz.z, hx.z, hy.z, hz.z);
      float e3 = box_lo2(plo, phi, lx.w, ly.w, lz.w, hx.w, hy.w, hz.w);
      unsigned c0 = cd.x, c1 = cd.y, c2 = cd.z, c3 = cd.w;
      c.boxes += (c0 != kNoChild) + (c1 != kNoChild) + (c2 != kNoChild) + (c3 != kNoChild);
      int pick = -1;  // kCut: a triangle of a child whose whole box lies within the cut radius
      if constexpr (kCut) {
        const float px = t.P.h.x, py = t.P.h.y, pz = t.P.h.z;
        const uint4 rp = __ldg(reinterpret_cast<const uint4*>(np + 7));
        if (c3 != kNoChild && box_far2(px, py, pz, lx.w, ly.w, lz.w, hx.w, hy.w, hz.w) < t.cut2) pick = (int)rp.w;
        if (c2 != kNoChild && box_far2(px, py, pz, lx.z, ly.z, lz.z, hx.z, hy.z, hz.z) < t.cut2) pick = (int)rp.z;
        if (c1 != kNoChild && box_far2(px, py, pz, lx.y, ly.y, lz.y, hx.y, hy.y, hz.y) < t.cut2) pick = (int)rp.y;
        if (c0 != kNoChild && box_far2(px, py, pz, lx.x, ly.x, lz.x, hx.x, hy.x, hz.x) < t.cut2) pick = (int)rp.x;
      }
      if (!(e0 <= r2) || c0 == kNoChild) e0 = INFINITY;
      if (!(e1 <= r2) || c1 == kNoChild) e1 = INFINITY;
      if (!(e2 <= r2) || c2 == kNoChild) e2 = INFINITY;
      if (!(e3 <= r2) || c3 == kNoChild) e3 = INFINITY;
      sort2(e0, c0, e1, c1);
      sort2(e2, c2, e3, c3);
      sort2(e0, c0, e2, c2);
      sort2(e1, c1, e3, c3);
      sort2(e1, c1, e2, c2);
      // the farther hits go on the stack (farthest first, so the nearest of them is popped
      // first); the nearest is taken now
      push_code(stack_code, stack_d, sp, c3, e3, c);
      push_code(stack_code, stack_d, sp, c2, e2, c);
      push_code(stack_code, stack_d, sp, c1, e1, c);
      if constexpr (kCut) {
        if (pick >= 0) {
          // test that one triangle; the check before the next pop then stops the query (should
          // its certified distance miss the cut by a rounding, the children are all pushed)
          push_code(stack_code, stack_d, sp, c0, e0, c);
          lfirst = pick;
          lcount = 1;
          node = -1;
          continue;
        }
      }
      if (e0 < INFINITY) {
        const int cnt = code_count(c0), ref = code_ref(c0);
        if (cnt > 0) {
          lfirst = ref;
          lcount = cnt;
          node = -1;
        } else {
          node = ref;
        }
      } else {
        node = -1;
      }
    }
    if (__all_sync(0xffffffffu, lcount == 0)) break;
    if (lcount > 0) {
      t.test1(lfirst);
      ++lfirst;
      --lcount;
    }
  }
}

// ----------------------------------------------------------------------------- bounds

// ---- u4 in certified FP32.  Differences of vertices and footpoints are formed as float pairs
// (h + l) with error-free sums: each such difference is within T = 64u (L + uM) of the exact
// one per component, where L bounds the vertices' low parts and M every coordinate involved
// (u = 2^-24; each pair operation adds at most 2u times the low parts it combines, which grow
// to a few L + uM along the chain).  Only the final dot products and norms round, and each is
// raised by a bound on its error.

// a + b as s + e exactly (Knuth's two-sum; intrinsics, so that nothing is contracted or
// reassociated).
__device__ inline void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ inline FFP pair_sub(const FFP& a, const FFP& b) {
  FFP r;
  two_sum(a.h.x, -b.h.x, r.h.x, r.l.x);
  two_sum(a.h.y, -b.h.y, r.h.y, r.l.y);
  two_sum(a.h.z, -b.h.z, r.h.z, r.l.z);
  r.l = {__fadd_rn(r.l.x, __fsub_rn(a.l.x, b.l.x)), __fadd_rn(r.l.y, __fsub_rn(a.l.y, b.l.y)),
         __fadd_rn(r.l.z, __fsub_rn(a.l.z, b.l.z))};
  return r;
}
__device__ inline FFP pair_add(const FFP& a, const FFP& b) {
  FFP r;
  two_sum(a.h.x, b.h.x, r.h.x, r.l.x);
  two_sum(a.h.y, b.h.y, r.h.y, r.l.y);
  two_sum(a.h.z, b.h.z, r.h.z, r.l.z);
  r.l = {__fadd_rn(r.l.x, __fadd_rn(a.l.x, b.l.x)), __fadd_rn(r.l.y, __fadd_rn(a.l.y, b.l.y)),
         __fadd_rn(r.l.z, __fadd_rn(a.l.z, b.l.z))};
  return r;
}
__device__ inline F3 pair_f(const FFP& a) {  // h + l rounded: within u |h + l| per component
  return {__fadd_rn(a.h.x, a.l.x), __fadd_rn(a.h.y, a.l.y), __fadd_rn(a.h.z, a.l.z)};
}

// Upper bound of the length of the exact vector whose float-pair form rounds to d: each
// component of d is within u |d_c| + 3T of it (two differences of pairs and one more pair
// operation), so the exact length is at most |d| (1 + u) + 6T; tiny >= 12T covers it.
__device__ inline float len_cert(F3 d, float tiny) { return __fadd_ru(__fmul_ru(norm_ru(d), 1.f + 4.f * kU), tiny); }

// H(a, b) of Eq. (bound_u4), the largest distance from a point of T to the nearer of a and b,
// certified.  It is attained at a vertex of T or where an edge crosses the bisector plane of a
// and b.  X are T's vertices and a, b the footpoints, as float pairs relative to T's first
// vertex.  For an edge x0 x1 with c_j = n . (x_j - mid) (n = b - a, mid = (a + b) / 2),
// computed as dot products of rounded vectors with |error| <= E_j = 8u |n|_1 |w_j|_1 +
// 4T (|n|_1 + |w_j|_1), the edge is skipped only when both c_j lie beyond E_j on the same
// side (it certainly does not cross).  Otherwise its term is the distance from a to the
// farther endpoint (|x - a| is convex along the edge, so this bounds the crossing's distance
// wherever it is) or, when |c0 - c1| > 4 (E0 + E1), the smaller of that and the distance at
// the computed crossing x0 + tau (x1 - x0) plus tau's error, (2 E0 + E1) / |c0 - c1| + 3u,
// times the edge length.  Every term bounds its exact counterpart from above, and extra terms
// only raise the maximum, so the result bounds H(a, b).
__device__ inline float u4_h_cert(const FFP X[3], const FFP& a, const FFP& b, float T) {
  const float tiny = __fmul_ru(16.f, T);
  F3 dA[3];
  float h = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    dA[i] = pair_f(pair_sub(X[i], a));
    const F3 db = pair_f(pair_sub(X[i], b));
    h = fmaxf(h, fminf(len_cert(dA[i], tiny), len_cert(db, tiny)));
  }
  const F3 n = pair_f(pair_sub(b, a));
  FFP mid = pair_add(a, b);
  mid.h = {0.5f * mid.h.x, 0.5f * mid.h.y, 0.5f * mid.h.z};
  mid.l = {0.5f * mid.l.x, 0.5f * mid.l.y, 0.5f * mid.l.z};
  const float n1 = sum1(n), m2 = __fmul_ru(4.f, T);
  float c[3], E[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const F3 w = pair_f(pair_sub(X[i], mid));
    const float w1 = sum1(w);
    c[i] = dotf(n, w);
    E[i] = __fadd_ru(__fmul_ru(__fmul_ru(8.f * kU, n1), w1), __fmul_ru(m2, __fadd_ru(n1, w1)));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int k = (i + 1) % 3;
    const float c0 = c[i], c1 = c[k], E0 = E[i], E1 = E[k];
    if ((c0 > E0 && c1 > E1) || (c0 < -E0 && c1 < -E1)) continue;
    float term = fmaxf(len_cert(dA[i], tiny), len_cert(dA[k], tiny));
    const float D = fabsf(__fsub_rn(c0, c1));
    if (D > __fmul_ru(4.f, __fadd_ru(E0, E1))) {
      const float tau = __saturatef(__fdiv_rn(c0, __fsub_rn(c0, c1)));
      const F3 e = pair_f(pair_sub(X[k], X[i]));
      // x - a = (x0 - a) + tau e, each component within u (|x0 - a| + |e| + |x - a|) + 6T
      const F3 r = {fmaf(tau, e.x, dA[i].x), fmaf(tau, e.y, dA[i].y), fmaf(tau, e.z, dA[i].z)};
      const float slop = __fadd_ru(__fmul_ru(2.f * kU, __fadd_ru(__fadd_ru(amax3(dA[i]), amax3(e)), amax3(r))), tiny);
      const float errt = __fadd_ru(__fdiv_ru(__fadd_ru(__fmul_ru(2.f, E0), E1), D), 3.f * kU);
      const float at = __fadd_ru(__fadd_ru(norm_ru(r), slop), __fmul_ru(errt, len_cert(e, tiny)));
      term = fminf(term, at);
    }
    h = fmaxf(h, term);
  }
  return h;
}

// u4, Eq. (bound_u4), certified in FP32: the footpoints q1 of the vertex opposite T's shortest
// edge and q2, q3 of its ends, u4 = min(H(q1, q2), H(q1, q3)), plus the footpoints' error
// radii (the points of B they stand for are within qerr) and twice the vertices'
// representation error.
__device__ inline float ubm_u4(const VM t[3], float slack_f) {
  const FFP zero = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  const FFP X[3] = {zero, pair_sub(t[1].p, t[0].p), pair_sub(t[2].p, t[0].p)};
  FFP Q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Q[i] = pair_add(X[i], FFP{t[i].q, {0.f, 0.f, 0.f}});
  float M = 0.f, L = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    M = fmaxf(M, fmaxf(amax3(X[i].h), amax3(Q[i].h)));
    L = fmaxf(L, amax3(t[i].p.l));
  }
  M = __fmul_ru(M, 2.f);  // also bounds midpoints and differences of two of these
  const float T = __fmul_ru(64.f * kU, __fadd_ru(L, __fmul_ru(kU, M)));
  const F3 x1 = pair_f(X[1]), x2 = pair_f(X[2]), e12 = x2 - x1;
  const float l0 = dotf(x1, x1), l1 = dotf(e12, e12), l2 = dotf(x2, x2);
  // shortest edge v1v2 with footpoints q1 (the opposite vertex's), q2, q3 (any choice is
  // valid; this one is the paper's)
  FFP q2 = Q[0], q3 = Q[1], q1 = Q[2];
  if (l1 < l0 && l1 <= l2) { q2 = Q[1]; q3 = Q[2]; q1 = Q[0]; }
  else if (l2 < l0 && l2 < l1) { q2 = Q[2]; q3 = Q[0]; q1 = Q[1]; }
  const float h = fminf(u4_h_cert(X, q1, q2, T), u4_h_cert(X, q1, q3, T));
  const float qe = fmaxf(t[0].qerr, fmaxf(t[1].qerr, t[2].qerr));
  return __fadd_ru(__fadd_ru(h, qe), __fmul_ru(2.f, slack_f));
}

// Whether ubm_u4 of T is certainly at least U, so that it can neither lower U nor discard T
// (most items: the vertex at one end of T's shortest edge is farther than U from both
// footpoints of the others).  H(a, b) is at least the distance from any vertex of T to the
// nearer of a and b; the vertex taken for each pair is the one whose own footpoint is not in
// it.  The edge is chosen with ubm_u4's own operations, so it is the same one; the distances
// are plain float, within 16 u M of the exact ones, far less than the margin asked for.
// On the batch of 128 pairs u4 lowered or discarded hardly any item, and its pass with the
// list it reads took a tenth of the call: 49.5 -> 46.3 ms with this check in the UpperBound
// kernels (bounds 18.6 -> 16.2 ms; the queries 20.6 -> 19.8, as the items that skip the pass
// keep their order); the torus pair's time does not change.
__device__ inline bool u4_idle(const VM t[3], float U) {
  const FFP zero = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  const F3 x[3] = {pair_f(zero), pair_f(pair_sub(t[1].p, t[0].p)), pair_f(pair_sub(t[2].p, t[0].p))};
  const F3 e12 = x[2] - x[1];
  const float l0 = dotf(x[1], x[1]), l1 = dotf(e12, e12), l2 = dotf(x[2], x[2]);
  F3 va = x[0], vb = x[1], qa = t[0].q, qb = t[1].q, vc = x[2], qc = t[2].q;  // shortest edge (a, b)
  if (l1 < l0 && l1 <= l2) {
    va = x[1]; qa = t[1].q;
    vb = x[2]; qb = t[2].q;
    vc = x[0]; qc = t[0].q;
  } else if (l2 < l0 && l2 < l1) {
    va = x[2]; qa = t[2].q;
    vb = x[0]; qb = t[0].q;
    vc = x[1]; qc = t[1].q;
  }
  const float M = fmaxf(fmaxf(amax3(x[1]), amax3(x[2])), fmaxf(amax3(qa), fmaxf(amax3(qb), amax3(qc))));
  const float lim = fmaf(0x1p-18f, M, U * (1.f + 0x1p-10f)), lim2 = lim * lim;
  const F3 Qa = va + qa, Qb = vb + qb, Qc = vc + qc;
  const F3 bc = vb - Qc, ba = vb - Qa, ac = va - Qc, ab = va - Qb;
  return fminf(fminf(dotf(bc, bc), dotf(ba, ba)), fminf(dotf(ac, ac), dotf(ab, ab))) >= lim2 && lim2 < INFINITY;
}

// lf is l rounded down to float: comparisons against it in float are safe, u < lf => u < l
__device__ inline float upper_bound_m(const BvhDev& B, const VM t[3], float lf, const RunParams& rp, int& code,
                                      Counters& c) {
  float U;
  if (t[0].I == t[1].I && t[1].I == t[2].I) {
    code = 0;
    U = fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi));
  } else {
    U = INFINITY;
    code = 5;
    const EdgesM E(t);  // shared by u1 and u2
    for (int k = 0; k < rp.n_bounds; ++k) {
      if (rp.order[k] == 4 && k == rp.n_bounds - 1 && rp.defer_u4) {
        // u4 (FP64) is evaluated for all such items together in the u4 pass, with full
        // warps, instead of by scattered lanes here; U so far is a valid upper bound
        code = kDeferU4;
        break;
      }
      float u;
      switch (rp.order[k]) {
        case 1: u = ubm_u1(t, E); break;
        case 2: u = ubm_u2(t, E); break;
        case 3: u = ubm_u3(B, t, lf, c.evals); break;
        default: u = ubm_u4(t, rp.slack_f); break;
      }
      U = fminf(U, u);
      if (u < lf) {
        code = rp.order[k];
        U = u;
        break;
      }
    }
  }
  return __fadd_ru(U, rp.slack_f);
}

// The cascade in the paper's order (u1, u2, u3, then u4, which the u4 pass evaluates) as
// straight-line code: the same values and result codes as upper_bound_m's loop over
// rp.order, but the edges are dead once u2 is known and the footpoints are not needed at all,
// so that fewer values are live across u3, the heaviest bound.
__device__ inline float upper_bound_m_paper(const BvhDev& B, const VM t[3], float lf, const RunParams& rp, int& code,
                                            Counters& c) {
  float U;
  if (t[0].I == t[1].I && t[1].I == t[2].I) {
    code = 0;
    U = fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi));
  } else {
    const EdgesM E(t);
    const float u1 = ubm_u1(t, E);
    if (u1 < lf) {
      code = 1;
      U = u1;
    } else {
      const float u2 = ubm_u2(t, E);
      if (u2 < lf) {
        code = 2;
        U = u2;
      } else {
        const float u3 = ubm_u3(B, t, lf, c.evals);
        if (u3 < lf) {
          code = 3;
          U = u3;
        } else {
          code = kDeferU4;
          U = fminf(fminf(u1, u2), u3);
        }
      }
    }
  }
  return __fadd_ru(U, rp.slack_f);
}

// ----------------------------------------------------------------------------- the policy

#ifndef HD_MIXED_SPREAD
#define HD_MIXED_SPREAD 8
#endif
#ifndef HD_MIXED_BOUND_REGS
#define HD_MIXED_BOUND_REGS 96
#endif
#ifndef HD_MIXED_PAPER_REGS
#define HD_MIXED_PAPER_REGS 128
#endif

struct PolicyM {
  using Vtx = VtxM;
  using Item = ItemM;
  using UT = float;
  static constexpr bool kFp64 = false;
  // resident blocks per SM of the cooperative traversal, with cuts / without
  static constexpr int kCoopBlocksCut = kCoopMinBlocksCut, kCoopBlocks = kCoopMinBlocks;
  static constexpr int kLongBudget = ::hd::kLongBudget;  // triangle tests of a lane before the hand-off
  static constexpr int kTailFront = 512;  // largest frontier of the small-round kernel
  // warps per SM that a short list of queries / of bounds is spread over (spread_lanes)
  static constexpr int kSpread = HD_MIXED_SPREAD, kSpreadBounds = HD_MIXED_SPREAD;
  static constexpr int kBoundRegs = HD_MIXED_BOUND_REGS;  // register cap of the UpperBound kernels
  static constexpr int kPaperRegs = HD_MIXED_PAPER_REGS;  // ... of their paper-order instantiation

  // 2^-40 of the largest coordinate: covers the float-pair representation of subdivided
  // vertices (2^-48 relative per level, at most 60 levels) and the double rounding of u4
  static double slack(double amax) { return ldexp(amax, -40); }
  __device__ static float ut_down(double x) { return __double2float_rd(x); }
  // the pass over the items left: u4, Eq. (bound_u4), for one item (certified FP32), plus the
  // slack; U holds the item's bound so far.
  static constexpr bool kPassVotes = false;
  __device__ static void bound_deferred(const BvhDev&, const Vtx& a, const Vtx& b, const Vtx& c, bool, double, float lo,
                                        const RunParams& rp, float& U, int& code, Counters&) {
    const VM t[3] = {{pos(a), a.dhi, a.tri, {a.qx, a.qy, a.qz}, a.qerr},
                     {pos(b), b.dhi, b.tri, {b.qx, b.qy, b.qz}, b.qerr},
                     {pos(c), c.dhi, c.tri, {c.qx, c.qy, c.qz}, c.qerr}};
    const float u = __fadd_ru(ubm_u4(t, rp.slack_f), rp.slack_f);
    code = u < lo ? 4 : 5;
    if (u < lo || u < U) U = u;
  }

  __device__ static FFP pos(const Vtx& v) { return {{v.hx, v.hy, v.hz}, {v.lx, v.ly, v.lz}}; }
  __device__ static D3 exact_pos(const Vtx& v) {
    return {(double)v.hx + (double)v.lx, (double)v.hy + (double)v.ly, (double)v.hz + (double)v.lz};
  }
  // Split further in FP32 only while the gap U - l is well above the FP32 error width of the
  // vertex distances; below that, refinement cannot make progress and the item is finished
  // in the FP64 phase.
  __device__ static bool promote(const Vtx& a, const Vtx& b, const Vtx& c, double U, double l) {
    float err = fmaxf(fmaxf(a.dhi - a.dlo, b.dhi - b.dlo), c.dhi - c.dlo);
    return U - l <= 4.0 * (double)err + ldexp(U, -18);
  }

  // a float input vertex is its own float pair (residual 0), with no FP64 arithmetic
  __device__ static void set_pos_f(Vtx& v, float x, float y, float z) {
    v.hx = x;
    v.hy = y;
    v.hz = z;
    v.lx = v.ly = v.lz = 0.f;
  }
  // the longest edge at the vertex (cut_radius) lives in pad0
  static constexpr bool kEdgePerVertex = true;
  __device__ static void set_edge(Vtx& v, float e) { v.pad0 = e; }
  __device__ static double cut_r(double l, const DynParams*, const Vtx& v) {
    return cut_radius(l, (double)v.pad0 * (1.0 + 0x1p-20));
  }
  __device__ static void set_pos(Vtx& v, double x, double y, double z) {
    v.hx = (float)x;
    v.hy = (float)y;
    v.hz = (float)z;
    v.lx = (float)(x - (double)v.hx);
    v.ly = (float)(y - (double)v.hy);
    v.lz = (float)(z - (double)v.hz);
  }

  // Called by every lane of the warp (the traversal votes with __all_sync over the full
  // warp); lanes with active == false only vote and leave v untouched.
  // Nearest triangle of v, certified.  With `over` given, a traversal that tests more than
  // `budget` triangles stops, sets *over and leaves its best triangle so far in v (hint, dhi =
  // its distance bound without eta, q, qerr) for query_coop to finish.
  // With cut_r >= 0 (cut_radius), the query may stop at a triangle within cut_r of v: it
  // then sets *was_cut and keeps that triangle with a lower bound of 0.
  __device__ static void query(const BvhDev& B, Vtx& v, Counters& c, bool active, int budget = INT_MAX,
                               bool* over = nullptr, double cut_r = -1.0, bool* was_cut = nullptr) {
    NearestM t;
    t.tri32 = B.tri32;
    if (active) {
      t.P = pos(v);
      // start from the hint, or from a triangle of the point's grid cell: a first radius
      // (often already within the cut radius)
      const int h0 = v.hint >= 0 ? v.hint : grid_hint(B, t.P.h.x, t.P.h.y, t.P.h.z);
      if (h0 >= 0) t.test1(h0);
      if (v.hint < 0 && h0 >= 0 && budget < INT_MAX) ++budget;  // the grid's triangle is not the traversal's
      t.cut = cut_bound(B, cut_r);
      if (t.cut > 0.f) t.cut2 = __fmul_rd(t.cut, t.cut);
    } else {
      t.P = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
    }
    bool unfinished = false, cut = active && t.best_hi < t.cut;  // the hint may be close enough
    if (__any_sync(0xffffffffu, t.cut > 0.f))  // one instantiation for the whole warp
      traverse_m<true>(B, t, c, active && !cut, budget, unfinished, cut);
    else
      traverse_m<false>(B, t, c, active, budget, unfinished, cut);
    if (!active) return;
    c.leaf += t.evals;
    c.escalations += t.esc;
    if (cut) {
      finish(B, v, t.best, t.best_hi, 0.f, t.q, t.qerr);
      if (was_cut) *was_cut = true;
      return;
    }
    if (unfinished) {
      *over = true;
      v.hint = t.best;
      v.dhi = t.best_hi;
      v.qx = t.q.x;
      v.qy = t.q.y;
      v.qz = t.q.z;
      v.qerr = t.qerr;
      return;
    }
    finish(B, v, t.best, t.best_hi, t.dlo, t.q, t.qerr);
  }
  // The distance bound of a handed-off query's best triangle so far.
  __device__ static double hint_dist(const Vtx& v) { return v.dhi; }
  // Whether a handed-off query's best triangle so far (hint, dhi without eta) is already
  // within the cut radius cut_r.
  __device__ static bool hint_within(const BvhDev& B, const Vtx& v, double cut_r) {
    return v.hint >= 0 && v.dhi < cut_bound(B, cut_r);
  }
  // The bound on best_hi (the certified distance to B's float triangles, before eta) below
  // which a query stops: best_hi + eta < cut_r, rounded so that it holds in exact arithmetic.
  __device__ static float cut_bound(const BvhDev& B, double cut_r) {
    if (!(cut_r > 0.0)) return -1.f;
    return __fsub_rd(__double2float_rd(cut_r), __ldg(B.meta));
  }
  // The query's result in v: eta (the distance between B's float triangles and its input)
  // widens both bounds.
  __device__ static void finish(const BvhDev& B, Vtx& v, int best, float best_hi, float dlo, F3 q, float qerr) {
    const float eta = __ldg(B.meta);
    v.tri = best;
    v.dhi = __fadd_ru(best_hi, eta);
    v.dlo = fmaxf(__fsub_rd(fminf(dlo, best_hi), eta), 0.f);
    v.qx = q.x;
    v.qy = q.y;
    v.qz = q.z;
    v.qerr = __fadd_ru(qerr, eta);
  }
  // query() of a vertex that a lane's traversal handed off, by the whole warp (every lane
  // passes the same v; lane 0 returns the result in it).  The certified lower bound is the
  // smallest lower bound over the triangles tested and the final best upper bound (every
  // pruned box lies beyond the radius of the moment, which is at least that).
  // With cut_r >= 0 the traversal may stop as query() does (the same for the whole warp);
  // returns true if it did.
  __device__ static bool query_coop(const BvhDev& B, Vtx& v, Counters& c, unsigned* s_code, float* s_e,
                                    double cut_r = -1.0) {
    const int lane = threadIdx.x & 31;
    NearestM t;
    t.tri32 = B.tri32;
    t.P = pos(v);
    if (lane == 0 && v.hint >= 0) {  // the lane traversal's best so far
      t.best = v.hint;
      t.best_hi = v.dhi;
      t.q = {v.qx, v.qy, v.qz};
      t.qerr = v.qerr;
    }
    const F3 plo = {__fadd_rd(t.P.h.x, t.P.l.x), __fadd_rd(t.P.h.y, t.P.l.y), __fadd_rd(t.P.h.z, t.P.l.z)};
    const F3 phi = {__fadd_ru(t.P.h.x, t.P.l.x), __fadd_ru(t.P.h.y, t.P.l.y), __fadd_ru(t.P.h.z, t.P.l.z)};
    auto box = [plo, phi](float lx, float ly, float lz, float hx, float hy, float hz, float) {
      return box_lo2(plo, phi, lx, ly, lz, hx, hy, hz);
    };
    const float cb = cut_bound(B, cut_r);
    const bool cut = cb > 0.f ? traverse_coop<true>(B, t, box, s_code, s_e, c, __fmul_rd(cb, cb))
                              : traverse_coop<false>(B, t, box, s_code, s_e, c, 0.f);
    c.leaf += t.evals;
    c.escalations += t.esc;
    const float m = warp_min_f(t.best_hi), dlo = cut ? 0.f : warp_min_f(t.dlo);
    const int src = __ffs(__ballot_sync(0xffffffffu, t.best_hi == m)) - 1;
    const int best = __shfl_sync(0xffffffffu, t.best, src);
    const F3 q = {__shfl_sync(0xffffffffu, t.q.x, src), __shfl_sync(0xffffffffu, t.q.y, src),
                  __shfl_sync(0xffffffffu, t.q.z, src)};
    const float qerr = __shfl_sync(0xffffffffu, t.qerr, src);
    finish(B, v, best, m, dlo, q, qerr);
    return cut;
  }
  __device__ static double lower(const Vtx& v) { return v.dlo; }
  __device__ static double out_dist(const Vtx& v) { return v.dhi; }
  __device__ static double out_dlo(const Vtx& v) { return v.dlo; }
  __device__ static D3 out_foot(const Vtx& v) {
    return {(double)v.hx + (double)v.lx + (double)v.qx, (double)v.hy + (double)v.ly + (double)v.qy,
            (double)v.hz + (double)v.lz + (double)v.qz};
  }
  __device__ static void midpoint(const Vtx& a, const Vtx& b, Vtx& m) {
    double x = 0.5 * (((double)a.hx + (double)a.lx) + ((double)b.hx + (double)b.lx));
    double y = 0.5 * (((double)a.hy + (double)a.ly) + ((double)b.hy + (double)b.ly));
    double z = 0.5 * (((double)a.hz + (double)a.lz) + ((double)b.hz + (double)b.lz));
    set_pos(m, x, y, z);
    m.qx = m.qy = m.qz = 0.f;
    m.qerr = m.dhi = m.dlo = 0.f;
    m.tri = -2;
    m.hint = a.tri;
    // every edge of a sub-triangle at m is at most the longest edge at a or at b (each edge
    // of the parent touches a or b)
    m.pad0 = fmaxf(a.pad0, b.pad0);
    m.pad1 = 0.f;
  }
  // upper_bound for the paper's cascade order with u4 deferred (only valid for those
  // options; the kernels pick it on the host): u4 comes later, if it can matter at all
  __device__ static UT upper_bound_paper(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, double,
                                         float lf, const RunParams& rp, int& code, Counters& cnt) {
    const VM t[3] = {{pos(a), a.dhi, a.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(b), b.dhi, b.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(c), c.dhi, c.tri, {0.f, 0.f, 0.f}, 0.f}};
    const float U = upper_bound_m_paper(B, t, lf, rp, code, cnt);
    if (code == kDeferU4 && skip_u4(a, b, c, U)) code = 5;
    return U;
  }
  // u4 cannot change U (u4_idle); reads the vertices again, so that the footpoints are not
  // live across u3.
  __device__ static bool skip_u4(const Vtx& a, const Vtx& b, const Vtx& c, float U) {
    const VM t[3] = {{pos(a), a.dhi, a.tri, {a.qx, a.qy, a.qz}, a.qerr},
                     {pos(b), b.dhi, b.tri, {b.qx, b.qy, b.qz}, b.qerr},
                     {pos(c), c.dhi, c.tri, {c.qx, c.qy, c.qz}, c.qerr}};
    return u4_idle(t, U);
  }
  // The paper-order cascade in two parts, for kernels that gather the items reaching u3 into
  // full warps: paper_cheap runs the exact case, u1 and u2; it returns true when u3 is still
  // needed (U so far in *u12), else the result in *U and *code as upper_bound_paper.
  // paper_u3 then finishes such an item; together they give upper_bound_paper's values.
  __device__ static bool paper_cheap(const BvhDev&, const Vtx& a, const Vtx& b, const Vtx& c, float lf,
                                     const RunParams& rp, float* U, int* code, float* u12) {
    const VM t[3] = {{pos(a), a.dhi, a.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(b), b.dhi, b.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(c), c.dhi, c.tri, {0.f, 0.f, 0.f}, 0.f}};
    if (t[0].I == t[1].I && t[1].I == t[2].I) {
      *code = 0;
      *U = __fadd_ru(fmaxf(t[0].dhi, fmaxf(t[1].dhi, t[2].dhi)), rp.slack_f);
      return false;
    }
    const EdgesM E(t);
    const float u1 = ubm_u1(t, E);
    if (u1 < lf) {
      *code = 1;
      *U = __fadd_ru(u1, rp.slack_f);
      return false;
    }
    const float u2 = ubm_u2(t, E);
    if (u2 < lf) {
      *code = 2;
      *U = __fadd_ru(u2, rp.slack_f);
      return false;
    }
    *u12 = fminf(u1, u2);
    return true;
  }
  __device__ static UT paper_u3(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, float lf, const RunParams& rp,
                                float u12, float up, int& code, Counters& cnt) {
    const VM t[3] = {{pos(a), a.dhi, a.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(b), b.dhi, b.tri, {0.f, 0.f, 0.f}, 0.f},
                     {pos(c), c.dhi, c.tri, {0.f, 0.f, 0.f}, 0.f}};
    const float u3 = ubm_u3(B, t, lf, cnt.evals);
    if (u3 < lf) {
      code = 3;
      return __fadd_ru(u3, rp.slack_f);
    }
    const float U = __fadd_ru(fminf(u12, u3), rp.slack_f);
    code = skip_u4(a, b, c, fminf(U, up)) ? 5 : kDeferU4;
    return U;
  }
  __device__ static UT upper_bound(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, double,
                                   float lf, const RunParams& rp, int& code, Counters& cnt) {
    VM t[3] = {{pos(a), a.dhi, a.tri, {a.qx, a.qy, a.qz}, a.qerr},
               {pos(b), b.dhi, b.tri, {b.qx, b.qy, b.qz}, b.qerr},
               {pos(c), c.dhi, c.tri, {c.qx, c.qy, c.qz}, c.qerr}};
    return upper_bound_m(B, t, lf, rp, code, cnt);
  }
};

}  // namespace hd
