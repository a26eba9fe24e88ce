// FP64 policy: results in IEEE double with round-to-nearest, the arithmetic of the paper's
// implementation (Section 4).  Comparisons that certified FP32 intervals settle (box distances,
// leaf triangles, bounds that discard) are settled by them, so that FP64, at 1/64 of the FP32
// rate, runs where they leave a decision open and for every value that is returned.
#pragma once

#include "hd_cert.cuh"
#include "hd_coop.cuh"
#include "hd_internal.cuh"

namespace hd {

constexpr int kStack = 96;  // up to 4 pushes per 4-wide node, one of them popped next

// Squared distance from p to triangle j of B, with the closest point, in FP64.
static __device__ __forceinline__ double tri_dist2(const double* tri64, const float4* tri32, int j, D3 p, D3& x) {
  D3 a, b, c;
  load_tri_d(tri64, tri32, j, a, b, c);
  x = closest_on_triangle(p, a, b, c);
  const D3 e = p - x;
  return dot(e, e);
}


// The nearest-triangle state of one query in FP64, with FP32 filters.  FP64 arithmetic runs
// at 1/64 of the FP32 rate on GB300, so the traversal decides everything it can from
// certified FP32 intervals (box distances, and a lower bound of each leaf triangle's
// distance) and takes an FP64 step only where the interval leaves the decision open: the
// point-triangle test of a triangle that may be nearer than the best so far, and the box
// distance where it is within FP32 rounding of the radius or of another child's.  Every
// decision is thus the one the same traversal in FP64 alone takes, so the triangles tested,
// the order among equal distances, the budget and the result are bit for bit its own.
struct NearestD {
  D3 p;
  const double* tri64;
  const float4* tri32;
  double best2 = INFINITY;
  double cut2 = -1.0;  // the traversal may stop once best2 < cut2 (cut_radius)
  int best = -1;
  D3 q = {0, 0, 0};
  unsigned evals = 0;  // triangles tested (by the filter, and in FP64 where it leaves them open)
  FFP P;               // p as a float pair
  float guard = 0.f;   // what the float forms of p and B and the FP64 test's own rounding can hide
  float pmax = 0.f;
  // The smallest squared distance so far lies in [r2lo, r2hi], its root in [rlo, rhi]: best2
  // rounded outward, or while candidates wait for their FP64 tests (traverse) what their FP32
  // bounds give.
  float r2lo = INFINITY, r2hi = INFINITY, rlo = INFINITY, rhi = INFINITY;

  __device__ void start(const BvhDev& B, double x, double y, double z) {
    p = {x, y, z};
    tri64 = B.tri64;
    tri32 = B.tri32;
    P.h = {__double2float_rn(x), __double2float_rn(y), __double2float_rn(z)};
    P.l = {__double2float_rn(x - (double)P.h.x), __double2float_rn(y - (double)P.h.y),
           __double2float_rn(z - (double)P.h.z)};
    // |p - (h + l)| <= 2^-48 |p| (1e-37 where l underflows), the FP64 test rounds within
    // 2^-48 of the coordinates it works on, and B's float vertices lie within eta of its own
    guard = __fadd_ru(__ldg(B.meta), 1e-37f);
    pmax = amax3(P.h);
  }
  // Enclosure of p on each axis, for the box intervals.
  __device__ F3 below() const {
    return {__double2float_rd(p.x), __double2float_rd(p.y), __double2float_rd(p.z)};
  }
  __device__ F3 above() const {
    return {__double2float_ru(p.x), __double2float_ru(p.y), __double2float_ru(p.z)};
  }
  __device__ void set_radius() {
    r2lo = __double2float_rd(best2);
    r2hi = __double2float_ru(best2);
    rlo = sqrt_dn(r2lo);
    rhi = sqrt_up(r2hi);
  }
  __device__ float coop_r2() const { return r2hi; }
  // Whether triangle j may be nearer than r (false: its FP64 squared distance is certainly
  // not below r^2).
  __device__ bool may(int j, float r) const {
    const float4* t = tri32 + 3 * (size_t)j;
    float M;
    const float lo = pt_lo(P, __ldg(t), __ldg(t + 1), __ldg(t + 2), M);
    return !(__fsub_rd(lo, __fmaf_ru(0x1p-40f, __fadd_ru(pmax, M), guard)) > r);
  }
  // Triangle j's FP32 bounds on the distance its FP64 test would compute.
  __device__ void bounds(int j, float& lo, float& hi) const {
    const float4* t = tri32 + 3 * (size_t)j;
    float M;
    lo = pt_lo(P, __ldg(t), __ldg(t + 1), __ldg(t + 2), M, &hi, guard);  // (guard: eta and 1e-37)
    const float g = __fmaf_ru(0x1p-40f, __fadd_ru(pmax, M), guard);
    lo = __fsub_rd(lo, g);
    hi = __fadd_ru(hi, g);
  }
  __device__ void test1(int j) {
    D3 x;
    const double d2 = tri_dist2(tri64, tri32, j, p, x);
    if (d2 < best2) {
      best2 = d2;
      best = j;
      q = x;
    }
  }
  // A leaf range in the cooperative traversal; r2 is the warp's squared radius.
  __device__ void coop_range(int first, int count, float r2) {
    const float r = sqrt_up(r2);
    for (int j = first; j < first + count; ++j) {
      ++evals;
      if (may(j, fminf(r, rhi))) {
        test1(j);
        set_radius();
      }
    }
  }
};

// Nearest triangle of B to t.p by ordered depth-first traversal of the BVH: a node's leaf
// children are tested first, nearest first, then its inner children are entered nearest
// first, each while its box lies within the radius of the moment.  Must be called by all 32
// lanes of the warp; inactive lanes start finished.  `first` (or -1) is a triangle to test
// before the traversal.
//
// The FP64 tests are put off: a triangle certainly nearer than all before it takes their
// place, one certainly farther than the nearest is dropped, and one the FP32 bounds leave
// between waits with the others (up to kWait of them).  They are tested, in their order, when a
// decision depends on it (a box distance within the bounds on the radius, a full list) and at
// the end.  Most queries then run one or two FP64 tests instead of one for every improvement,
// and all lanes of a warp run theirs together: a lane expands nodes until it has a leaf
// triangle, the lanes that have one bound it in FP32, and a lane that needs a test waits until
// every lane does or is finished.
//
// Bound by the FP64 pipe (2 lanes per clock and SM) before the filters: every node cost four
// FP64 box distances, every leaf triangle an FP64 test.  Round 0 and one round of the torus
// pair (200,000 vs 50,176 triangles, 203,860 queries): 2.20 ms in FP64 alone, 0.67 ms with an
// FP64 test for each triangle that may be nearer than the best so far, 0.47 ms so.
//
// Returns kTravOver once more than `budget` triangles have been tested, and kTravCut once the
// squared radius is below t.cut2 (cut_radius), with the traversal unfinished (t then holds
// the best triangle found so far); kTravDone when it finished.
constexpr int kWait = 4;
constexpr int kTravDone = 0, kTravOver = 1, kTravCut = 2;
template <bool kCut>
__device__ inline int traverse(const BvhDev& B, NearestD& t, Counters& c, bool active, int first, int budget) {
  unsigned stack_node[kStack];
  float2 stack_e[kStack];  // the interval of each entry's squared box distance
  int sp = 0;
  int node = active ? 0 : -1;  // inner node to expand next
  int leaf_node = 0, slots = 0, n_slots = 0;  // leaf children waiting: their slots in leaf_node, 2 bits each
  int lfirst = 0, lcount = 0;                 // leaf triangles waiting
  bool picked = false;                        // kCut: the waiting triangle is a cut query's pick
  int wait[kWait], n_wait = 0;                // triangles waiting for their FP64 test, in order
  bool test = false;                          // they are tested before anything else
#pragma unroll
  for (int q = 0; q < kWait; ++q) wait[q] = -1;
  bool done = !active;
  if (active && first >= 0) {
    lfirst = first;
    lcount = 1;
  }
  int how = kTravDone;
  const F3 plo = t.below(), phi = t.above();
  // whether the smallest squared distance so far is below cut2 (asks for the tests where that
  // is open)
  const float c2lo = kCut ? __double2float_rd(t.cut2) : 0.f, c2hi = kCut ? __double2float_ru(t.cut2) : 0.f;
  auto is_cut = [&]() {
    if (c2hi <= t.r2lo) return false;
    if (t.r2hi < c2lo) return true;
    if (n_wait > 0) {
      test = true;
      return false;
    }
    return t.best2 < t.cut2;
  };
  for (;;) {
    while (!done && !test && n_slots == 0 && lcount == 0 && !picked) {
      bool open = false;  // node's own box distance is within the bounds on the radius
      if (node < 0) {
        while (sp > 0) {
          --sp;
          const float2 e = stack_e[sp];
          if (e.x > t.r2hi) continue;
          open = !(e.y < t.r2lo);
          if (open && n_wait > 0) {  // decided after the tests
            ++sp;
            test = true;
            break;
          }
          node = (int)stack_node[sp];
          break;
        }
        if (node < 0) {
          done = !test;
          continue;
        }
      }
      const float4* np = reinterpret_cast<const float4*>(B.nodes + node);
      const float4 lx = __ldg(np), ly = __ldg(np + 1), lz = __ldg(np + 2);
      const float4 hx = __ldg(np + 3), hy = __ldg(np + 4), hz = __ldg(np + 5);
      const uint4 cd = __ldg(reinterpret_cast<const uint4*>(np + 6));
      if (open) {  // its box is the union of its children's
        const double e = box_dist2(t.p, fminf(fminf(lx.x, lx.y), fminf(lx.z, lx.w)),
                                   fminf(fminf(ly.x, ly.y), fminf(ly.z, ly.w)),
                                   fminf(fminf(lz.x, lz.y), fminf(lz.z, lz.w)),
                                   fmaxf(fmaxf(hx.x, hx.y), fmaxf(hx.z, hx.w)),
                                   fmaxf(fmaxf(hy.x, hy.y), fmaxf(hy.z, hy.w)),
                                   fmaxf(fmaxf(hz.x, hz.y), fmaxf(hz.z, hz.w)));
        if (!(e < t.best2)) {
          node = -1;
          continue;
        }
      }
      if ((int)t.evals > budget) {
        how = kTravOver;
        done = true;
        continue;
      }
      if constexpr (kCut) {
        if (is_cut()) {
          how = kTravCut;
          done = true;
          continue;
        }
        if (test) continue;  // node is kept for after the tests
      }
      ++c.nodes;
      // the children's intervals; those certainly beyond the radius, and missing ones, at +inf
      float el[4], eh[4];
      int sl[4] = {0, 1, 2, 3};
      auto child = [&](int j, unsigned k, float ax, float ay, float az, float bx, float by, float bz) {
        el[j] = box_lo2(plo, phi, ax, ay, az, bx, by, bz);
        eh[j] = box_hi2(plo, phi, ax, ay, az, bx, by, bz);
        c.boxes += k != kNoChild;
        if (k == kNoChild || el[j] > t.r2hi) el[j] = eh[j] = INFINITY;
      };
      child(0, cd.x, lx.x, ly.x, lz.x, hx.x, hy.x, hz.x);
      child(1, cd.y, lx.y, ly.y, lz.y, hx.y, hy.y, hz.y);
      child(2, cd.z, lx.z, ly.z, lz.z, hx.z, hy.z, hz.z);
      child(3, cd.w, lx.w, ly.w, lz.w, hx.w, hy.w, hz.w);
      // nearest first (sorting network on four: a pair is swapped when the later child is nearer)
      bool tie = false;  // an order the intervals leave open
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        const int a = s == 0 ? 0 : s == 1 ? 2 : s == 2 ? 0 : s == 3 ? 1 : 1;
        const int b = s == 0 ? 1 : s == 1 ? 3 : s == 2 ? 2 : s == 3 ? 3 : 2;
        if (eh[b] < el[a]) {
          const float x = el[a], y = eh[a];
          el[a] = el[b];
          eh[a] = eh[b];
          el[b] = x;
          eh[b] = y;
          const int k = sl[a];
          sl[a] = sl[b];
          sl[b] = k;
        } else {
          tie |= el[b] <= eh[a] && eh[a] > 0.f && el[a] < INFINITY && el[b] < INFINITY;
        }
      }
      if (tie) {  // rare: the same network on the FP64 distances
        double e[4];
        auto exact = [&](int j, unsigned k, float ax, float ay, float az, float bx, float by, float bz) {
          e[j] = k == kNoChild ? INFINITY : box_dist2(t.p, ax, ay, az, bx, by, bz);
          sl[j] = j;
        };
        exact(0, cd.x, lx.x, ly.x, lz.x, hx.x, hy.x, hz.x);
        exact(1, cd.y, lx.y, ly.y, lz.y, hx.y, hy.y, hz.y);
        exact(2, cd.z, lx.z, ly.z, lz.z, hx.z, hy.z, hz.z);
        exact(3, cd.w, lx.w, ly.w, lz.w, hx.w, hy.w, hz.w);
#pragma unroll
        for (int s = 0; s < 5; ++s) {
          const int a = s == 0 ? 0 : s == 1 ? 2 : s == 2 ? 0 : s == 3 ? 1 : 1;
          const int b = s == 0 ? 1 : s == 1 ? 3 : s == 2 ? 2 : s == 3 ? 3 : 2;
          if (e[b] < e[a]) {
            const double x = e[a];
            e[a] = e[b];
            e[b] = x;
            const int k = sl[a];
            sl[a] = sl[b];
            sl[b] = k;
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          el[j] = __double2float_rd(e[j]);
          eh[j] = __double2float_ru(e[j]);
          if (el[j] > t.r2hi) el[j] = eh[j] = INFINITY;
        }
      }
      if constexpr (kCut) {
        // a child box wholly within the cut radius: one of its triangles is close enough
        const uint4 rp = __ldg(reinterpret_cast<const uint4*>(np + 7));
        const float px = t.P.h.x, py = t.P.h.y, pz = t.P.h.z;
        const float c2 = (float)t.cut2;
        int pick = -1;
        if (cd.w != kNoChild && box_far2(px, py, pz, lx.w, ly.w, lz.w, hx.w, hy.w, hz.w) < c2) pick = (int)rp.w;
        if (cd.z != kNoChild && box_far2(px, py, pz, lx.z, ly.z, lz.z, hx.z, hy.z, hz.z) < c2) pick = (int)rp.z;
        if (cd.y != kNoChild && box_far2(px, py, pz, lx.y, ly.y, lz.y, hx.y, hy.y, hz.y) < c2) pick = (int)rp.y;
        if (cd.x != kNoChild && box_far2(px, py, pz, lx.x, ly.x, lz.x, hx.x, hy.x, hz.x) < c2) pick = (int)rp.x;
        if (pick >= 0) {
          lfirst = pick;
          lcount = 1;
          picked = true;
        }
      }
      // the inner children go on the stack, farthest first; the leaves wait, nearest first
      // (their tests come first and shrink the radius the stack is popped with)
      leaf_node = node;
      slots = 0;
#pragma unroll
      for (int j = 3; j >= 0; --j) {
        if (!(el[j] < INFINITY)) continue;
        const unsigned k = sl[j] == 0 ? cd.x : sl[j] == 1 ? cd.y : sl[j] == 2 ? cd.z : cd.w;
        if (code_count(k) > 0) {
          slots = (slots << 2) | sl[j];
          ++n_slots;
        } else if (sp < kStack) {
          stack_node[sp] = (unsigned)code_ref(k);
          stack_e[sp] = make_float2(el[j], eh[j]);
          ++sp;
        } else {
          c.err = 1;  // stack overflow: the subtree is skipped and the error reported
        }
      }
      node = -1;
    }
    if (!done && !test) {
      if (lcount == 0) {
        if (kCut && picked) {
          if (is_cut()) {
            how = kTravCut;
            done = true;
          }
          picked = test;  // asked again after the tests
        }
        if (!done && !test && n_slots > 0) {
          const int s = slots & 3;
          const float* nf = reinterpret_cast<const float*>(B.nodes + leaf_node) + s;
          const float ax = __ldg(nf), ay = __ldg(nf + 4), az = __ldg(nf + 8);
          const float bx = __ldg(nf + 12), by = __ldg(nf + 16), bz = __ldg(nf + 20);
          const unsigned k = __ldg(reinterpret_cast<const unsigned*>(nf) + 24);
          bool in = box_hi2(plo, phi, ax, ay, az, bx, by, bz) < t.r2lo;
          if (!in && !(box_lo2(plo, phi, ax, ay, az, bx, by, bz) > t.r2hi)) {
            if (n_wait > 0) test = true;
            else in = box_dist2(t.p, ax, ay, az, bx, by, bz) < t.best2;
          }
          if (!test) {
            slots >>= 2;
            --n_slots;
          }
          if (in) {
            lfirst = code_ref(k);
            lcount = code_count(k);
          }
        }
      }
      if (!done && !test && lcount > 0) {
        ++t.evals;
        float lo, hi;
        t.bounds(lfirst, lo, hi);
        if (hi < t.rlo) {  // certainly the nearest so far
          t.best2 = INFINITY;
          n_wait = 1;
          wait[0] = lfirst;
          t.rlo = fmaxf(lo, 0.f);
          t.rhi = hi;
          t.r2lo = __fmul_rd(t.rlo, t.rlo);
          t.r2hi = __fmul_ru(hi, hi);
        } else if (!(lo > t.rhi)) {
#pragma unroll
          for (int q = 0; q < kWait; ++q)
            if (q == n_wait) wait[q] = lfirst;
          ++n_wait;
          t.rlo = fminf(t.rlo, fmaxf(lo, 0.f));
          t.r2lo = fminf(t.r2lo, __fmul_rd(t.rlo, t.rlo));
          if (hi < t.rhi) {
            t.rhi = hi;
            t.r2hi = __fmul_ru(hi, hi);
          }
          test = n_wait == kWait || !(hi < INFINITY);  // (no upper bound: its own test is needed)
        }
        ++lfirst;
        --lcount;
      }
    }
    if (__any_sync(0xffffffffu, !done && !test)) continue;
    if (!__any_sync(0xffffffffu, n_wait > 0)) break;
    do {
      if (n_wait > 0) {
        t.test1(wait[0]);
#pragma unroll
        for (int q = 0; q + 1 < kWait; ++q) wait[q] = wait[q + 1];
        if (--n_wait == 0) {
          t.set_radius();
          test = false;
        }
      }
    } while (__any_sync(0xffffffffu, n_wait > 0));
  }
  return how;
}

// ----------------------------------------------------------------------------- bounds (Section 3.2)

struct VI {
  D3 v;
  double d;
  int I;
  D3 q;
};

__device__ inline D3 tri_vertex(const BvhDev& B, int j, int slot) {
  if (B.tri64) {
    const double* t = B.tri64 + 9 * (size_t)j + 3 * slot;
    return {t[0], t[1], t[2]};
  }
  const float4 v = __ldg(B.tri32 + 3 * (size_t)j + slot);
  return {v.x, v.y, v.z};
}

// v as a vertex of the certified FP32 bounds: its position as a float pair, its distance
// rounded up.
__device__ inline VM vertex_m(D3 v, double d, int I) {
  VM m;
  m.p.h = {__double2float_rn(v.x), __double2float_rn(v.y), __double2float_rn(v.z)};
  m.p.l = {__double2float_rn(v.x - (double)m.p.h.x), __double2float_rn(v.y - (double)m.p.h.y),
           __double2float_rn(v.z - (double)m.p.h.z)};
  m.dhi = __double2float_ru(d);
  m.I = I;
  m.q = {0.f, 0.f, 0.f};
  m.qerr = 0.f;
  return m;
}

// Eq. (uexact): the three vertices are nearest to one triangle S; h(T,S) = max_i |v_i - q_i|.
__device__ inline double ub_exact(const VI t[3]) { return fmax(t[0].d, fmax(t[1].d, t[2].d)); }

// The lengths of T's edges, e[i] opposite vertex i, for u1 and u2.
struct EdgesD {
  double e[3];
  __device__ explicit EdgesD(const VI t[3])
      : e{len(t[1].v - t[2].v), len(t[2].v - t[0].v), len(t[0].v - t[1].v)} {}
};

// Eq. (u1)
__device__ inline double ub_u1(const VI t[3], const EdgesD& E) {
  return fmin(fmax(E.e[1], E.e[2]) + t[0].d, fmin(fmax(E.e[2], E.e[0]) + t[1].d, fmax(E.e[0], E.e[1]) + t[2].d));
}

// The bounds below take `cap`, the smallest bound of T so far: where a bound is certain to be
// at least cap, it may return any value from cap up (it then neither lowers U nor, U being
// at least l, discards T).

// Eq. (u2): g + max_i d_i with g = R if s - r > 2R, else half the longest edge (g is at least
// that in either case).
__device__ inline double ub_u2(const VI t[3], const EdgesD& E, double cap) {
  double g = 0.5 * fmax(E.e[0], fmax(E.e[1], E.e[2]));
  const double dmax = fmax(t[0].d, fmax(t[1].d, t[2].d));
  if (g + dmax > cap * (1.0 + 1e-12)) return INFINITY;
  double area = 0.5 * len(cross(t[1].v - t[0].v, t[2].v - t[0].v));
  if (area > 0.0) {
    double R = E.e[0] * E.e[1] * E.e[2] / (4.0 * area);
    double s = 0.5 * (E.e[0] + E.e[1] + E.e[2]);
    double r = area / s;
    if (s - r > 2.0 * R) g = R;
  }
  return g + dmax;
}

// Kang et al. 2018 bound, Eqs. (Kang2018_case1) and (Kang2018_case2).  own[i] = d(v_i, S_i).
// Must be called by all 32 lanes of the warp; lanes with on == false only vote.
//
// Every term is a maximum of point-triangle distances, so a distance is computed in FP64 only
// where its FP32 upper bound exceeds the maximum so far, and a maximum that can no longer
// lower the minimum it enters is abandoned.  Few of the 4 (case 1) or 15 (case 2) distances
// are left then, at different places for each lane; so a lane goes through them until one
// needs FP64, waits, and the waiting lanes run the FP64 test together.  (Tested where they
// occur, some lane needs FP64 at almost every place, and the warp pays for each: the pass had
// 9 to 15 lanes active.  Bounds of the batch of 32 small pairs in FP64 4.34 -> 3.55 ms, of the
// torus pair 0.418 -> 0.376 ms.)
__device__ inline double ub_u3(const BvhDev& B, const VI t[3], const double own[3], double cap, bool on, unsigned& evals) {
  const double dmax = fmax(own[0], fmax(own[1], own[2]));
  // the distances to take, in order: case 1 (c1): the split points b1, b2 against S1, then S2
  // (v1 against S1 and v2, v3 against S2 are the vertices' own); case 2: steps 0..5 the two
  // other vertices against S_i, then 6..14 the quadrilaterals (v_i, m_i, b, m_{i-1}) against S_i
  int k = 0, kend = 0, S1 = 0, S2 = 0;
  bool c1 = false;
  D3 b1 = t[0].v, b2 = t[0].v;
  double h = own[0], best = cap;
  VM f[3];
  FFP fb1, fb2, fm[3], fbc;
  float bm[3] = {0.f, 0.f, 0.f}, bb = 0.f, guard = 0.f;
  if (on) {
    int lone = -1;
    if (!(t[0].I == t[1].I && t[1].I == t[2].I)) {
      if (t[1].I == t[2].I) lone = 0;
      else if (t[0].I == t[2].I) lone = 1;
      else if (t[0].I == t[1].I) lone = 2;
    }
    int fs0, fs1, fo, go;
    // v1 is the vertex alone on its triangle (selected by branches: no runtime array index)
    VI v1 = t[0], v2 = t[1], v3 = t[2];
    if (lone == 1) { v1 = t[1]; v2 = t[2]; v3 = t[0]; }
    else if (lone == 2) { v1 = t[2]; v2 = t[0]; v3 = t[1]; }
    c1 = lone >= 0 && shared_edge(B, v1.I, v2.I, fs0, fs1, fo, go);
#pragma unroll
    for (int i = 0; i < 3; ++i) f[i] = vertex_m(t[i].v, 0.0, t[i].I);
    // the float forms of B and the points, and the FP64 rounding (NearestD::guard)
    const float pmax = fmaxf(amax3(f[0].p.h), fmaxf(amax3(f[1].p.h), amax3(f[2].p.h)));
    guard = __fmaf_ru(0x1p-38f, pmax, __fadd_ru(__ldg(B.meta), 1e-37f));
    if (c1) {
      S1 = v1.I;
      S2 = v2.I;
      D3 p0 = tri_vertex(B, S1, fs0), e = tri_vertex(B, S1, fs1) - p0;
      b1 = 0.5 * (v1.v + v2.v);
      b2 = 0.5 * (v1.v + v3.v);
      double el = len(e);
      if (el > 0.0) {
        D3 eh = (1.0 / el) * e;
        D3 a1 = tri_vertex(B, S1, fo) - p0, a2 = tri_vertex(B, S2, go) - p0;
        D3 w1 = a1 - dot(a1, eh) * eh, w2 = a2 - dot(a2, eh) * eh;
        double n1 = len(w1), n2 = len(w2);
        if (n1 > 0.0 && n2 > 0.0) {
          D3 nb = (1.0 / n1) * w1 - (1.0 / n2) * w2;
          double s1 = dot(nb, v1.v - p0), s2 = dot(nb, v2.v - p0), s3 = dot(nb, v3.v - p0);
          if (s1 >= 0.0 && s2 <= 0.0 && s3 <= 0.0 && s1 - s2 > 0.0 && s1 - s3 > 0.0) {
            b1 = v1.v + (s1 / (s1 - s2)) * (v2.v - v1.v);
            b2 = v1.v + (s1 / (s1 - s3)) * (v3.v - v1.v);
          }
        }
      }
      fb1 = vertex_m(b1, 0.0, 0).p;
      fb2 = vertex_m(b2, 0.0, 0).p;
      h = dmax;
      kend = 4;
    } else {
      const F3 e01 = edge(f[0], f[1]), e02 = edge(f[0], f[2]), e12 = edge(f[1], f[2]);
      fm[0] = along(f[0], e01, 0.5f, bm[0]);
      fm[1] = along(f[1], e12, 0.5f, bm[1]);
      fm[2] = along(f[0], e02, 0.5f, bm[2]);
      fbc = along(f[0], e01 + e02, 1.f / 3.f, bb);
      bb = __fmul_ru(16.f * kU, fmaxf(amax3(e01), fmaxf(amax3(e02), amax3(f[0].p.l))));
      kend = 15;
    }
  }
  // step k is settled: on to the next one (and the next maximum of case 2)
  auto next = [&]() {
    ++k;
    if (!c1 && k <= 6 && (k & 1) == 0) {
      best = fmin(best, h);
      h = k == 2 ? own[1] : k == 4 ? own[2] : dmax;
    }
  };
  bool pend = false;
  int S = 0, i = 0, j = 0;
  for (;;) {
    while (k < kend && !pend) {
      if (c1) {
        if (!(h < cap)) {
          k = kend;
          break;
        }
        S = k < 2 ? S1 : S2;
      } else {
        if (!(h < best)) {  // this maximum cannot lower the minimum
          if (k < 6) {
            k |= 1;
            next();
            continue;
          }
          k = kend;
          break;
        }
        const int r = k < 6 ? k : k - 6;
        i = k < 6 ? r >> 1 : r / 3;
        j = k < 6 ? r & 1 : r - 3 * i;
        S = i == 0 ? t[0].I : i == 1 ? t[1].I : t[2].I;
      }
      FFP x;
      float beta = 0.f;
      if (c1) {
        x = (k & 1) ? fb2 : fb1;
      } else if (k < 6) {
        const int v = i + 1 + j > 2 ? i + j - 2 : i + 1 + j;  // (i + 1 + j) mod 3
        x = v == 0 ? f[0].p : v == 1 ? f[1].p : f[2].p;
      } else if (j == 2) {
        x = fbc;
        beta = bb;
      } else {
        const int q = j == 0 ? i : i == 0 ? 2 : i - 1;
        x = q == 0 ? fm[0] : q == 1 ? fm[1] : fm[2];
        beta = q == 0 ? bm[0] : q == 1 ? bm[1] : bm[2];
      }
      ++evals;
      if (__fadd_ru(dist_hi(B, S, x, beta), guard) <= __double2float_rd(h)) next();
      else pend = true;
    }
    if (!__any_sync(0xffffffffu, pend)) break;
    if (pend) {
      D3 x, q;
      if (c1) {
        x = (k & 1) ? b2 : b1;
      } else if (k < 6) {
        const int v = i + 1 + j > 2 ? i + j - 2 : i + 1 + j;
        x = v == 0 ? t[0].v : v == 1 ? t[1].v : t[2].v;
      } else if (j == 2) {
        x = (1.0 / 3.0) * (t[0].v + t[1].v + t[2].v);
      } else {
        const int e = j == 0 ? i : i == 0 ? 2 : i - 1;  // m_e is the middle of v_e and the next
        x = 0.5 * ((e == 0 ? t[0].v : e == 1 ? t[1].v : t[2].v) + (e == 0 ? t[1].v : e == 1 ? t[2].v : t[0].v));
      }
      h = fmax(h, sqrt(tri_dist2(B.tri64, B.tri32, S, x, q)));
      pend = false;
      next();
    }
  }
  return c1 ? h : fmin(h, best);
}

// Squared max over T of d(., {a, b}), attained at a vertex of T or where an edge of T crosses
// the bisector plane of a and b (Section 3.2.4), or +inf once it exceeds cap2.  Squared
// distances throughout: the one square root is taken by ub_u4 (FP64 square roots are costly
// on GB300, whose FP64 rate is low).
__device__ inline double h2_two_points(const VI t[3], D3 a, D3 b, double cap2) {
  double h2 = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    D3 ea = t[i].v - a, eb = t[i].v - b;
    h2 = fmax(h2, fmin(dot(ea, ea), dot(eb, eb)));
  }
  if (h2 > cap2) return INFINITY;
  D3 n = b - a;
  if (dot(n, n) == 0.0) return h2;
  D3 mid = 0.5 * (a + b);
  const double c[3] = {dot(n, t[0].v - mid), dot(n, t[1].v - mid), dot(n, t[2].v - mid)};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double c0 = c[i], c1 = c[(i + 1) % 3];
    if (((c0 <= 0.0 && c1 >= 0.0) || (c0 >= 0.0 && c1 <= 0.0)) && c0 != c1) {
      D3 x = t[i].v + (c0 / (c0 - c1)) * (t[(i + 1) % 3].v - t[i].v);
      D3 ea = x - a, eb = x - b;
      h2 = fmax(h2, fmin(dot(ea, ea), dot(eb, eb)));
    }
  }
  return h2;
}

// Eq. (bound_u4)
__device__ inline double ub_u4(const VI t[3], double cap) {
  D3 e0 = t[0].v - t[1].v, e1 = t[1].v - t[2].v, e2 = t[2].v - t[0].v;
  double l0 = dot(e0, e0), l1 = dot(e1, e1), l2 = dot(e2, e2);
  int k = 0;
  double m = l0;
  if (l1 < m) { k = 1; m = l1; }
  if (l2 < m) k = 2;
  D3 q2 = t[0].q, q3 = t[1].q, q1 = t[2].q;  // shortest edge v1v2 (k = 0)
  if (k == 1) { q2 = t[1].q; q3 = t[2].q; q1 = t[0].q; }
  else if (k == 2) { q2 = t[2].q; q3 = t[0].q; q1 = t[1].q; }
  double h2 = INFINITY;
  const double cap2 = cap * cap * (1.0 + 1e-12);
#pragma unroll 1
  for (int j = 0; j < 2; ++j) h2 = fmin(h2, h2_two_points(t, q1, j ? q3 : q2, fmin(cap2, h2)));
  return sqrt(h2);
}

// UpperBound(T, l) of Section 4; own(i) = d(v_i, S_i), asked for only where u3 is reached.  Must
// be called by all 32 lanes of the warp (ub_u3 votes); lanes with on == false return +inf.
// With `full`, every bound is evaluated in full (a discarded T then returns the deciding bound's
// own value).  kU3: the order may hold u3.
template <bool kU3 = true, class Own>
__device__ inline double upper_bound_d(const BvhDev& B, const VI t[3], const Own& own, double l, const uint8_t* order,
                                       int nb, bool full, bool on, int& code, unsigned& evals) {
  double U = INFINITY;
  code = 5;
  if (on && t[0].I == t[1].I && t[1].I == t[2].I) {
    code = 0;
    U = ub_exact(t);
    on = false;
  }
  const EdgesD E(t);
  for (int k = 0; k < nb; ++k) {
    double u = INFINITY;
    const double cap = full ? INFINITY : U;
    if (order[k] == 3) {
      if constexpr (kU3) {
        double d[3] = {0.0, 0.0, 0.0};
        if (on) {
#pragma unroll
          for (int i = 0; i < 3; ++i) d[i] = own(i);
        }
        const double u3 = ub_u3(B, t, d, cap, on, evals);
        if (on) u = u3;
      }
    } else if (on) {
      u = order[k] == 1 ? ub_u1(t, E) : order[k] == 2 ? ub_u2(t, E, cap) : ub_u4(t, cap);
    }
    if (on) {
      if (u < l) {
        code = order[k];
        U = u;
        on = false;
      } else {
        U = fmin(U, u);
      }
    }
  }
  return U;
}

// ----------------------------------------------------------------------------- the policy

#ifndef HD_FP64_SPREAD
#define HD_FP64_SPREAD 8
#endif
#ifndef HD_FP64_SPREAD_BOUNDS
#define HD_FP64_SPREAD_BOUNDS 3
#endif
#ifndef HD_FP64_BOUND_REGS
#define HD_FP64_BOUND_REGS 128
#endif
#ifndef HD_FP64_PAPER_REGS
#define HD_FP64_PAPER_REGS 128
#endif

struct PolicyD {
  using Vtx = VtxD;
  using Item = ItemD;
  using UT = double;
  static constexpr bool kFp64 = true;
  // resident blocks per SM of the cooperative traversal, with cuts / without
  static constexpr int kCoopBlocksCut = HD_COOP_MIN_BLOCKS_D, kCoopBlocks = HD_COOP_MIN_BLOCKS_D;
  static constexpr int kLongBudget = HD_LONG_BUDGET_D;      // triangle tests of a lane before the hand-off
  static constexpr int kTailFront = 64;  // largest frontier of the small-round kernel
  // warps per SM that a short list of queries / of bounds is spread over (spread_lanes)
  static constexpr int kSpread = HD_FP64_SPREAD, kSpreadBounds = HD_FP64_SPREAD_BOUNDS;
  static constexpr int kBoundRegs = HD_FP64_BOUND_REGS;  // register cap of the UpperBound kernels
  static constexpr int kPaperRegs = HD_FP64_PAPER_REGS;  // ... of their paper-order instantiation

  // Nearest triangle of v.  Called by every lane of the warp (the traversal votes over the
  // full warp); lanes with active == false only vote and leave v untouched.  With `over`
  // given, a traversal that tests more than `budget` triangles stops, sets *over and leaves
  // its best triangle so far in v (hint, d = its squared distance, q) for query_coop to finish.
  // With cut_r >= 0 (cut_radius), the query may stop at a triangle within cut_r of v: it
  // then sets *was_cut and keeps that triangle and its distance (not a lower bound then).
  __device__ static void query(const BvhDev& B, Vtx& v, Counters& c, bool active, int budget = INT_MAX,
                               bool* over = nullptr, double cut_r = -1.0, bool* was_cut = nullptr) {
    NearestD t;
    int h0 = -1;
    if (active) {
      t.start(B, v.x, v.y, v.z);
      if (cut_r > 0.0) t.cut2 = cut_r * cut_r;
      // start from the hint, or from a triangle of the point's grid cell (a first radius)
      h0 = v.hint >= 0 ? v.hint : grid_hint(B, t.P.h.x, t.P.h.y, t.P.h.z);
      if (v.hint < 0 && h0 >= 0 && budget < INT_MAX) ++budget;  // the grid's triangle is not the traversal's
    } else {
      t.p = {0.0, 0.0, 0.0};
    }
    // one instantiation for the whole warp
    const int how = __any_sync(0xffffffffu, t.cut2 > 0.0) ? traverse<true>(B, t, c, active, h0, budget)
                                                          : traverse<false>(B, t, c, active, h0, budget);
    if (!active) return;
    c.leaf += t.evals;
    if (how == kTravCut && was_cut) *was_cut = true;
    if (how == kTravOver) {
      *over = true;
      v.hint = t.best;
      v.d = t.best2;
      v.qx = t.q.x;
      v.qy = t.q.y;
      v.qz = t.q.z;
      return;
    }
    v.tri = t.best;
    v.d = sqrt(t.best2);
    v.qx = t.q.x;
    v.qy = t.q.y;
    v.qz = t.q.z;
  }
  // query() of a vertex that a lane's traversal handed off, by the whole warp (every lane
  // passes the same v; lane 0 returns the result in it).
  // With cut_r >= 0 the traversal may stop as query() does (the same for the whole warp);
  // returns true if it did.
  __device__ static bool query_coop(const BvhDev& B, Vtx& v, Counters& c, unsigned* s_code, float* s_e,
                                    double cut_r = -1.0) {
    const int lane = threadIdx.x & 31;
    NearestD t;
    t.start(B, v.x, v.y, v.z);
    if (lane == 0 && v.hint >= 0) {  // the lane traversal's best so far
      t.best = v.hint;
      t.best2 = v.d;
      t.q = {v.qx, v.qy, v.qz};
      t.set_radius();
    }
    // the FP64 squared box distance rounded down to float decides (e <= r2); where its FP32
    // interval lies on one side of r2, the interval's lower end decides the same
    const D3 p = t.p;
    const F3 plo = t.below(), phi = t.above();
    auto box = [p, plo, phi](float lx, float ly, float lz, float hx, float hy, float hz, float r2) {
      const float e = box_lo2(plo, phi, lx, ly, lz, hx, hy, hz);
      if (e > __fmul_ru(r2, 1.f + 4.f * kU) || box_hi2(plo, phi, lx, ly, lz, hx, hy, hz) <= r2) return e;
      return __double2float_rd(box_dist2(p, lx, ly, lz, hx, hy, hz));
    };
    const float cut2 = cut_r > 0.0 ? __double2float_rd(cut_r * cut_r) : 0.f;
    const bool cut = cut2 > 0.f ? traverse_coop<true>(B, t, box, s_code, s_e, c, cut2)
                                : traverse_coop<false>(B, t, box, s_code, s_e, c, 0.f);
    c.leaf += t.evals;
    double m = t.best2;
    for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int src = __ffs(__ballot_sync(0xffffffffu, t.best2 == m)) - 1;
    const int best = __shfl_sync(0xffffffffu, t.best, src);
    const double qx = __shfl_sync(0xffffffffu, t.q.x, src), qy = __shfl_sync(0xffffffffu, t.q.y, src),
                 qz = __shfl_sync(0xffffffffu, t.q.z, src);
    v.tri = best;
    v.d = sqrt(m);
    v.qx = qx;
    v.qy = qy;
    v.qz = qz;
    return cut;
  }
  __device__ static double lower(const Vtx& v) { return v.d; }
  __device__ static double out_dist(const Vtx& v) { return v.d; }
  __device__ static double out_dlo(const Vtx& v) { return v.d; }
  __device__ static D3 out_foot(const Vtx& v) { return {v.qx, v.qy, v.qz}; }
  static double slack(double) { return 0.0; }
  __device__ static double ut_down(double x) { return x; }
  __device__ static D3 exact_pos(const Vtx& v) { return {v.x, v.y, v.z}; }
  __device__ static bool promote(const Vtx&, const Vtx&, const Vtx&, double, double) { return false; }
  __device__ static void set_pos_f(Vtx& v, float x, float y, float z) { set_pos(v, x, y, z); }
  // the distance of a handed-off query's best triangle so far (d holds its square then)
  __device__ static double hint_dist(const Vtx& v) { return sqrt(v.d); }
  // whether a handed-off query's best triangle so far (hint, d = its squared distance) is
  // already within the cut radius cut_r
  __device__ static bool hint_within(const BvhDev&, const Vtx& v, double cut_r) {
    return v.hint >= 0 && cut_r > 0.0 && v.d < cut_r * cut_r;
  }
  // no room in the vertex for its own edge bound: the longest edge of A for every vertex
  static constexpr bool kEdgePerVertex = false;
  __device__ static void set_edge(Vtx&, float) {}
  __device__ static double cut_r(double l, const DynParams* dyn, const Vtx&) { return cut_radius(l, dyn->emax); }
  __device__ static void set_pos(Vtx& v, double x, double y, double z) {
    v.x = x;
    v.y = y;
    v.z = z;
  }
  __device__ static void midpoint(const Vtx& a, const Vtx& b, Vtx& m) {
    m.x = 0.5 * (a.x + b.x);
    m.y = 0.5 * (a.y + b.y);
    m.z = 0.5 * (a.z + b.z);
    m.d = 0.0;
    m.qx = m.qy = m.qz = 0.0;
    m.tri = -2;
    m.hint = a.tri;
  }
  // The FP32 filter of the UpperBound kernels.  An item's vertices for its bounds (q only for
  // ubm_u4_lo):
  __device__ static void vertices_m(const Vtx& a, const Vtx& b, const Vtx& c, VM t[3]) {
    t[0] = vertex_m({a.x, a.y, a.z}, a.d, a.tri);
    t[1] = vertex_m({b.x, b.y, b.z}, b.d, b.tri);
    t[2] = vertex_m({c.x, c.y, c.z}, c.d, c.tri);
  }
  __device__ static F3 foot_m(const Vtx& v) {
    return {__double2float_rn(v.qx - v.x), __double2float_rn(v.qy - v.y), __double2float_rn(v.qz - v.z)};
  }
  // What the filter compares with: an FP32 upper bound below u12 (u1, u2) or u3 discards the
  // item, as the FP64 bound then also does (it lies below the FP32 bound up to its own rounding):
  // l less 2^-14 of it, the slack, the float pairs' rounding (u1 and u2 move by no more than the
  // vertices do: g is the radius of T's smallest enclosing circle) and, for u3, the distance
  // of B's float vertices from its own.  An FP32 lower bound of at least `keep` shows that the FP64
  // bound does not discard it (2e-15: what sqrt_up adds to tiny lengths).  Between the two the
  // item is left to the FP64 cascade, so that the bound a discard is counted for is the one
  // FP64 alone finds.
  struct Limits {
    float u12, u3, keep;
  };
  __device__ static Limits limits(const BvhDev& B, const VM t[3], float lf, const RunParams& rp) {
    const float pmax = fmaxf(amax3(t[0].p.h), fmaxf(amax3(t[1].p.h), amax3(t[2].p.h)));
    const float rep = __fadd_ru(__fmaf_ru(0x1p-38f, pmax, 1e-37f), rp.slack_f);
    Limits m;
    m.u12 = __fsub_rd(__fmul_rd(lf, 1.f - 0x1p-14f), rep);
    m.u3 = __fsub_rd(m.u12, __ldg(B.meta));
    m.keep = __fadd_ru(__fmaf_ru(lf, 1.f + 0x1p-13f, rep), 2e-15f);
    return m;
  }
  // u1 or u2 (u: upper bound, lo: lower bound) decides: 1 discards, 0 does not, -1 is left open
  __device__ static int verdict(const Limits& m, float u, float lo) {
    return u < m.u12 ? 1 : lo >= m.keep && lo < INFINITY ? 0 : -1;
  }
  // The cascade's part in the UpperBound kernels: the exact case, and the items that certified
  // FP32 bounds u1..u3 discard.  Every other item is left (kDeferU4, U = +inf) to the pass
  // that bounds them in FP64 with every lane of a warp on an item of its own: about one
  // item in ten is left, and each would hold its whole warp for the FP64 cascade.  (Inlined
  // 21 times and run by every item, that cascade also outgrew the instruction cache: 45
  // cycles of instruction fetch per instruction issued.)  Torus pair in FP64: the bounds of
  // 200,000 faces and 138,480 children 4.59 -> 0.47 ms.
  __device__ static UT upper_bound_paper(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, double,
                                         float lf, const RunParams& rp, int& code, Counters& cnt) {
    UT U;
    float u12;
    if (!paper_cheap(B, a, b, c, lf, rp, &U, &code, &u12)) return U;
    return paper_u3(B, a, b, c, lf, rp, u12, INFINITY, code, cnt);
  }
  __device__ static bool paper_cheap(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, float lf,
                                     const RunParams& rp, UT* U, int* code, float* u12) {
    if (a.tri == b.tri && b.tri == c.tri) {
      *code = 0;
      *U = fmax(a.d, fmax(b.d, c.d)) + rp.slack;
      return false;
    }
    VM t[3];
    vertices_m(a, b, c, t);
    const Limits m = limits(B, t, lf, rp);
    const EdgesM E(t);
    const float u1 = ubm_u1(t, E);
    int v = verdict(m, u1, u1);
    *code = 1;
    *U = (UT)u1;
    if (v == 0) {
      const float u2 = ubm_u2(t, E);
      v = verdict(m, u2, u2 < m.u12 ? 0.f : ubm_u2_lo(t, E, m.keep));
      *code = 2;
      *U = (UT)u2;
      *u12 = fminf(u1, u2);
    }
    if (v < 0) {
      *code = kDeferU4;
      *U = INFINITY;
    }
    return v == 0;
  }
  __device__ static UT paper_u3(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, float lf, const RunParams& rp,
                                float, float, int& code, Counters& cnt) {
    VM t[3];
    vertices_m(a, b, c, t);
    const float lim = limits(B, t, lf, rp).u3;
    if (lim > 0.f) {
      const float u3 = ubm_u3<true>(B, t, lim, cnt.evals);
      if (u3 < lim) {
        code = 3;
        return (UT)u3;
      }
    }
    code = kDeferU4;
    return INFINITY;
  }
  // The same for a cascade in any order.
  __device__ static UT upper_bound(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, double, float lf,
                                   const RunParams& rp, int& code, Counters& cnt) {
    if (a.tri == b.tri && b.tri == c.tri) {
      code = 0;
      return fmax(a.d, fmax(b.d, c.d)) + rp.slack;
    }
    VM t[3];
    vertices_m(a, b, c, t);
    const Limits m = limits(B, t, lf, rp);
    code = kDeferU4;
    if (!(m.u12 > 0.f)) return INFINITY;
    const EdgesM E(t);
    for (int k = 0; k < rp.n_bounds; ++k) {
      const int o = rp.order[k];
      float u = INFINITY;
      int v;
      if (o == 1) {
        u = ubm_u1(t, E);
        v = verdict(m, u, u);
      } else if (o == 2) {
        u = ubm_u2(t, E);
        v = verdict(m, u, ubm_u2_lo(t, E, m.keep));
      } else if (o == 3) {
        if (m.u3 > 0.f) u = ubm_u3<true>(B, t, m.u3, cnt.evals);
        v = u < m.u3 ? 1 : -1;
      } else {
        t[0].q = foot_m(a);
        t[1].q = foot_m(b);
        t[2].q = foot_m(c);
        v = verdict(m, INFINITY, ubm_u4_lo(t));
      }
      if (v < 0) break;
      if (v == 1) {
        code = o;
        return (UT)u;
      }
    }
    return INFINITY;
  }
  // The pass over the items left: the whole cascade in FP64, clamped to what U holds.  Must be
  // called by all 32 lanes of the warp; only those with on == true have an item.
  static constexpr bool kPassVotes = true;
  __device__ static void bound_deferred(const BvhDev& B, const Vtx& a, const Vtx& b, const Vtx& c, bool on, double l, UT,
                                        const RunParams& rp, UT& U, int& code, Counters& cnt) {
    const VI t[3] = {{{a.x, a.y, a.z}, a.d, a.tri, {a.qx, a.qy, a.qz}},
                     {{b.x, b.y, b.z}, b.d, b.tri, {b.qx, b.qy, b.qz}},
                     {{c.x, c.y, c.z}, c.d, c.tri, {c.qx, c.qy, c.qz}}};
    auto own = [&](int i) { return t[i].d; };
    // slack is 0 in a pure FP64 run; in the certification phase of a MIXED run it is the
    // margin that covers the double rounding
    const double u = upper_bound_d(B, t, own, l - rp.slack, rp.order, rp.n_bounds, false, on, code, cnt.evals) + rp.slack;
    U = fmin(U, u);
  }
};

}  // namespace hd
