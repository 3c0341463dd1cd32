// twa_math.cuh -- FP32 device minimizers of the planning factors.
//
// Notation of Bento et al., "A message-passing algorithm for multi-agent
// trajectory planning" (NIPS 2013): n_lo / n_hi are the incoming messages of
// the two break-points of a segment, x_* the minimizer outputs.
//
// Collision and wall minimizers (Appendices C, D, I).  A segment [v_lo, v_hi]
// misses an open convex region iff a unit normal n separates them:
// <v_lo,n> >= h(n) and <v_hi,n> >= h(n), h the region's support function.
// For fixed n the cheapest v's are v = a + [h - <a,n>]_+ n, so the minimizer
// is min over directions of
//     E(n) = wl/2 [h - <a,n>]_+^2 + wh/2 [h - <b,n>]_+^2 .
// (Both hinges positive is the paper's tangent-slab configuration, one hinge
// at zero its compressed-spring configuration.)
//
// Disk of radius R at the origin (the collision minimizer through
// Eq. wall_min_goes_to_coll_min).  Let f(n) = wl (R - <a,n>)^2 +
// wh (R - <b,n>)^2 be the both-stretched piece, so E <= f/2 everywhere and
// E = f/2 where both hinges are positive.  Then
//     min E = min( E(n_f), m_a, m_b ),
// n_f the global minimiser of f on the unit circle, m_a the minimum of
// wl/2 [R - <a,n>]_+^2 over the arc <b,n> >= R (where the b hinge is zero)
// and m_b likewise: every piece of the circle is covered, and each of the
// three values is E at some direction.  n_f is a trust-region subproblem:
// with M = wl a a^T + wh b b^T = lambda1 e1 e1^T + lambda2 e2 e2^T and
// S = wl a + wh b, the global minimiser solves (M - mu I) n = R S with
// mu <= lambda1, i.e. t = lambda1 - mu >= 0 is the unique root of the
// decreasing secular function (R s1 / t)^2 + (R s2 / (d + t))^2 = 1,
// d = lambda2 - lambda1 (hard case: s1 = 0 and R |s2| < d gives t = 0).
// m_a / m_b are closed form: the arc point closest in angle to a (or b).
// Where that point is an end of the arc, <b, n> = R, the energy still falls on
// the arc's outside, so in exact arithmetic it is never below E(n_f); to
// rounding it ties with it, and is a candidate for that reason: which of two
// tying candidates wins is part of the FP32 results (see trs_global).
//
// Capsule (wall) regions use the same hinge energy with
// h(n) = max(<xL,n>, <xR,n>) + r, which is the disk energy of one end circle
// on each half-plane of directions.  The global minimum is at one of the two
// kink directions or at a local minimum of one end circle's energy: a local
// minimum of its both-stretched piece (global or local-nonglobal, both from
// the secular equation) or a single-hinge direction.  A circle whose
// half-plane cannot beat the kinks is skipped (capsule_end_dominated).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace twa {

// Host and device: the same FP32 code is also compiled into a host-side test
// harness (tests/minimizer_harness.cu) that compares it with the FP64 oracle.
// Everything is inlined, and candidate directions are written to fixed
// array slots only (unrolled loops), so that the minimizers keep
// their candidates in registers: a call or a dynamically indexed array puts
// them in local memory, whose latency sits on the minimizer's long dependent
// chain.
#define TWA_DEV __host__ __device__ __forceinline__
#define TWA_NOINLINE TWA_DEV
#ifndef TWA_ITER_HOOK
#define TWA_ITER_HOOK(kind)
#endif

TWA_DEV float2 mk(float x, float y) { return make_float2(x, y); }
TWA_DEV float2 operator+(float2 a, float2 b) { return mk(a.x + b.x, a.y + b.y); }
TWA_DEV float2 operator-(float2 a, float2 b) { return mk(a.x - b.x, a.y - b.y); }
TWA_DEV float2 operator-(float2 a) { return mk(-a.x, -a.y); }
TWA_DEV float2 operator*(float s, float2 a) { return mk(s * a.x, s * a.y); }
// The library is compiled without implicit multiply-add fusion: which pairs
// the compiler fuses depends on the code around an inlined function, and the
// same factor has to round alike in every kernel that computes it.  The fused
// operations are written out instead.
TWA_DEV float dot(float2 a, float2 b) { return fmaf(a.x, b.x, a.y * b.y); }
TWA_DEV float cross(float2 a, float2 b) { return fmaf(a.x, b.y, -(a.y * b.x)); }
TWA_DEV float2 axpy(float s, float2 a, float2 b) { return mk(fmaf(s, a.x, b.x), fmaf(s, a.y, b.y)); }  // s a + b
TWA_DEV float2 perp(float2 a) { return mk(-a.y, a.x); }
// a / |a|; dd: |a|^2, where the caller sums it in an order of its own.
TWA_DEV float2 normalized(float2 a, float dd) {
#ifdef __CUDA_ARCH__
  // one reciprocal square root (2 ulp) where |a|^2 is a normal float; the
  // directions are unit to a few ulp either way
  if (dd > 1e-30f && dd < 1e30f) {
    const float s = rsqrtf(dd);
    return mk(a.x * s, a.y * s);
  }
#endif
  float n = hypotf(a.x, a.y);
  return n > 0.f ? mk(a.x / n, a.y / n) : mk(1.f, 0.f);
}
TWA_DEV float2 normalized(float2 a) { return normalized(a, dot(a, a)); }

// Fast division (2 ulp for divisors of normal magnitude; every divisor here
// is a length, a curvature or a secular variable far from the float limits)
// and reciprocal square root, for the secular iterations and the direction
// arithmetic of the minimizers: fewer instructions on their long dependent
// chains.  The host build (test harness) uses the plain operations.
TWA_DEV float fdiv(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return a / b;
#endif
}
TWA_DEV float frsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.f / sqrtf(x);
#endif
}

// The power of two that scales a positive normal float into [1, 2).
TWA_DEV float pow2_inverse(float x) {
#ifdef __CUDA_ARCH__
  return __uint_as_float((254u - ((__float_as_uint(x) >> 23) & 0xffu)) << 23);
#else
  uint32_t u;
  memcpy(&u, &x, 4);
  u = (254u - ((u >> 23) & 0xffu)) << 23;
  memcpy(&x, &u, 4);
  return x;
#endif
}

// Angle of a unit vector in [0, 2 pi): the tie-break order of directions.
// Not inlined: it runs only on exact ties, and a copy at every tie-break
// would crowd the minimizers' instruction stream.
__host__ __device__ __noinline__ float angle_of(float2 n) {
  float t = atan2f(n.y, n.x);
  return t < 0.f ? t + 6.283185307179586f : t;
}
// a before b in the tie-break order
__host__ __device__ __noinline__ bool angle_less(float2 a, float2 b) {
  return angle_of(a) < angle_of(b);
}

// Squared distance from the origin to segment [p0, p1].  Interior projections
// use the cross product (absolute error ~ eps |p0|, no cancellation of
// |p0|^2 against the projection).
TWA_DEV float dist2_origin_segment(float2 p0, float2 p1) {
  float2 d = p1 - p0;
  float dd = dot(d, d);
  float t = -dot(p0, d);
  if (t <= 0.f || dd == 0.f) return dot(p0, p0);
  if (t >= dd) return dot(p1, p1);
  float c = cross(p0, d);
  return c * c / dd;
}

TWA_DEV float dist2_point_segment(float2 q, float2 p0, float2 p1) {
  return dist2_origin_segment(p0 - q, p1 - q);
}

// Keep the best (lowest E, then smallest angle) candidate direction.  tag
// records which kind of candidate won (read by the adjoint; dead otherwise).
struct Best {
  float2 n;
  float E;
  int tag;
  TWA_DEV void init() { n = mk(1.f, 0.f); E = INFINITY; tag = 0; }
  TWA_DEV void offer(float2 c, float e, int t = 0) {
    if (e < E || (e == E && angle_less(c, n))) { n = c; E = e; tag = t; }
  }
};

// ---------------------------------------------------------------------------
// Energy minimizer (Appendix E, Eq. energy_minimizer_output)
// ---------------------------------------------------------------------------
// pin_lo / pin_hi: that end's incoming weight is infinite (fixed endpoint).
TWA_DEV void energy_prox(float2 n_lo, float2 n_hi, float rho, bool pin_lo, bool pin_hi, float c,
                         float2& x_lo, float2& x_hi) {
  if (pin_lo && pin_hi) { x_lo = n_lo; x_hi = n_hi; return; }
  const float c2 = 2.f * c;
  if (pin_lo) {
    x_lo = n_lo;
    const float inv = 1.f / (c2 + rho);
    x_hi = inv * axpy(rho, n_hi, c2 * n_lo);
    return;
  }
  if (pin_hi) {
    x_hi = n_hi;
    const float inv = 1.f / (c2 + rho);
    x_lo = inv * axpy(rho, n_lo, c2 * n_hi);
    return;
  }
  // equal weights rho on both ends
  const float inv = 1.f / fmaf(4.f, c, rho);
  const float2 s = c2 * (n_lo + n_hi);
  x_lo = inv * axpy(rho, n_lo, s);
  x_hi = inv * axpy(rho, n_hi, s);
}

// ---------------------------------------------------------------------------
// Disk of radius R at the origin
// ---------------------------------------------------------------------------
TWA_DEV float hinge_E(float2 a, float2 b, float wl, float wh, float R, float2 n) {
  float ga = fmaxf(R - dot(a, n), 0.f), gb = fmaxf(R - dot(b, n), 0.f);
  return fmaf(0.5f * wl * ga, ga, 0.5f * wh * gb * gb);
}

// n1 e1 + n2 e2, e1 = perp(e2).
TWA_DEV float2 in_frame(float n1, float n2, float2 e2) {
  return mk(fmaf(n2, e2.x, -(n1 * e2.y)), fmaf(n1, e2.x, n2 * e2.y));
}

// Global minimiser(s) of f(n) = wl (R - <a,n>)^2 + wh (R - <b,n>)^2 on the
// unit circle.  Writes 1 or 2 directions (2 only for exact ties).
// The order of the operations, fused or not, is part of the results: where a
// candidate of another kind ties with the root to rounding, the last bit
// decides which one wins, and with it the branch that the adjoint
// differentiates (and, head on, the side on which the pair passes).  A form
// with a shorter chain (plain square roots, a climb without a bracket, no arc
// ends) took 4.2 us an iteration for 4.8 of the p = 4 circle's, but parted from
// these results by up to 2e-4 in 3 % of gradients of circle swaps, and by whole
// detours in one pass of 300.
TWA_NOINLINE int trs_global(float2 a, float2 b, float wl, float wh, float R,
                                       float2* out) {
  const float2 wa = wl * a, wb = wh * b;
  const float m11 = fmaf(wa.x, a.x, wb.x * b.x);
  const float m22 = fmaf(wa.y, a.y, wb.y * b.y);
  const float m12 = fmaf(wa.x, a.y, wb.x * b.y);
  const float2 S = wa + wb;
  const float hd = 0.5f * (m11 - m22);
  const float disc = hypotf(hd, m12);
  const float d = 2.f * disc;  // lambda2 - lambda1 >= 0
  const float q = fabsf(hd) + disc;
  const float2 e2 = (disc > 0.f) ? normalized((hd >= 0.f) ? mk(q, m12) : mk(m12, q), fmaf(m12, m12, q * q)) : mk(1.f, 0.f);
  const float2 e1 = perp(e2);
  const float s1 = cross(e2, S), s2 = dot(S, e2);
  const float Sn = hypotf(s1, s2);
  if (!(Sn > 0.f)) { out[0] = e1; out[1] = -e1; return 2; }
  const float A1 = R * fabsf(s1), A2 = R * fabsf(s2);
  if (A1 <= 1e-7f * R * Sn && A2 < d) {  // hard case: t = 0
    const float n2 = R * s2 / d;
    const float n1 = sqrtf(fmaxf(0.f, fmaf(-n2, n2, 1.f)));
    out[0] = in_frame(n1, n2, e2);
    out[1] = mk(fmaf(n1, e2.y, n2 * e2.x), fmaf(n2, e2.y, -(n1 * e2.x)));
    return 2;
  }
  // Root of h(t) = phi(t)^{-1/2} - 1 with phi = (A1/t)^2 + (A2/(d+t))^2.
  // 1/|n(t)| is concave and increasing (Moré-Sorensen), so Newton from the
  // left bracket end, where h <= 0, climbs monotonically to the root.
  float lo = fmaxf(fmaxf(A1, R * Sn - d), 0.f), hi = R * Sn;
  if (lo > hi) lo = hi;
  float t = lo > 0.f ? lo : 0.5f * hi;
#pragma unroll 1
  for (int it = 0; it < 40; ++it) {
    TWA_ITER_HOOK(0);
    const float it_ = fdiv(1.f, t), id = fdiv(1.f, d + t);
    const float q1 = A1 * it_, q2 = A2 * id;
    const float phi = q1 * q1 + q2 * q2;
    const float ip = frsqrt(phi);
    const float h = ip - 1.f;
    if (h > 0.f) hi = t; else lo = t;
    if (h == 0.f) break;
    const float dh = ip * ip * ip * fmaf(q1 * q1, it_, q2 * q2 * id);
    float tn = fmaf(-h, fdiv(1.f, dh), t);
    if (!(tn > lo && tn < hi)) tn = 0.5f * (lo + hi);
    // FP32 noise in h limits t to ~1e-7 relative; stop at 1e-6
    const bool done = fabsf(tn - t) <= 1e-6f * t || hi - lo <= 1e-6f * hi;
    t = tn;
    if (done) break;
  }
  // the smaller component from the root, the other from the unit length
  const float p1 = (t > 0.f) ? fdiv(R * s1, t) : copysignf(INFINITY, s1);
  const float p2 = fdiv(R * s2, d + t);
  const bool first = fabsf(p1) <= fabsf(p2);
  const float c = first ? p1 : p2;
  const float rest = copysignf(sqrtf(fmaxf(0.f, fmaf(-c, c, 1.f))), first ? s2 : s1);
  out[0] = normalized(first ? in_frame(p1, rest, e2) : in_frame(rest, p2, e2));
  return 1;
}

// The other local minimum of f, where there is one: mu in (lambda1, lambda2),
// where t = mu - lambda1 solves phi = (A1/t)^2 + (A2/(d - t))^2 = 1.  phi is
// convex on (0, d), so there are 0 or 2 roots; the curvature of f along the
// circle is (d - t) n1^2 - t n2^2, which has the sign of -dphi/dt, so the root
// left of phi's minimum is the local minimum (the other one a local maximum).
// Newton on 1/|n(t)| from the pole side, t = A1, where phi >= 1, climbs to it;
// when the climb passes phi's minimum (dphi/dt >= 0) there is no root.  With
// s2 = 0 the root is t = A1 < d; with s1 = 0 there is none left of the
// minimum.  Writes 0 or 1 direction; used by the wall minimizer, whose capsule
// restricts each end circle to a half-plane of directions.
TWA_NOINLINE int trs_local(float2 a, float2 b, float wl, float wh, float R, float2* out) {
  // lengths to R in [1, 2) and weights to [1, 2), by powers of two: the direction
  // is the same and the products below stay in range
  const float sc = pow2_inverse(R), sw = pow2_inverse(fmaxf(wl, wh));
  a = sc * a; b = sc * b; R *= sc;
  wl *= sw; wh *= sw;
  const float2 wa = wl * a, wb = wh * b;
  const float m11 = fmaf(wa.x, a.x, wb.x * b.x);
  const float m22 = fmaf(wa.y, a.y, wb.y * b.y);
  const float m12 = fmaf(wa.x, a.y, wb.x * b.y);
  const float2 S = wa + wb;
  const float hd = 0.5f * (m11 - m22);
  const float disc = hypotf(hd, m12);
  const float d = 2.f * disc;
  if (!(d > 0.f)) return 0;
  const float q = fabsf(hd) + disc;
  const float2 e2 = normalized((hd >= 0.f) ? mk(q, m12) : mk(m12, q));
  const float2 e1 = perp(e2);
  const float s1 = dot(S, e1), s2 = dot(S, e2);
  const float A1 = R * fabsf(s1), A2 = R * fabsf(s2);
  if (!(A1 > 0.f && A1 < d)) return 0;
  float t = A1;
  bool found = A2 == 0.f;
#pragma unroll 1
  for (int it = 0; it < 40 && !found; ++it) {
    TWA_ITER_HOOK(1);
    const float it_ = fdiv(1.f, t), id = fdiv(1.f, d - t);
    const float q1 = A1 * it_, q2 = A2 * id;
    const float w1 = q1 * q1, w2 = q2 * q2;
    const float phi = w1 + w2, slope = fmaf(w1, it_, -(w2 * id));
    if (!(slope > 0.f)) break;  // past the minimum of phi
    const float step = (phi * frsqrt(phi) - 1.f) * fdiv(phi, slope);
    t += step;
    if (!(t > 0.f && t < d)) break;
    found = fabsf(step) <= 1e-6f * t;
  }
  if (!found) return 0;
  // (n1, n2) = (-R s1 / t, R s2 / (d - t)) up to its length
  out[0] = normalized(axpy(-s1 * (d - t), e1, (s2 * t) * e2));
  return 1;
}

// Tangent normals n with <q, n> = R from a point q (|q| >= R).
TWA_DEV void tangent_normals(float2 q, float R, float2& t0, float2& t1) {
  float L2 = dot(q, q);
  float s = sqrtf(fmaxf(fmaf(-R, R, L2), 0.f));
  float inv = fdiv(1.f, L2);
  const float2 sp = s * perp(q);  // (fused in this order: see trs_global)
  t0 = inv * axpy(R, q, sp);
  t1 = inv * axpy(R, q, -sp);
}

// Direction in the arc {n : <q,n> >= R} (|q| >= R) maximising <w, n>.
// tangent: the answer is an end of the arc (<q,n> = R) rather than w / |w|.
TWA_DEV float2 arc_argmax(float2 q, float R, float2 w, bool& tangent) {
  float nw = hypotf(w.x, w.y);
  tangent = false;
  if (nw > 0.f && dot(q, w) >= R * nw) {
    const float inv = fdiv(1.f, nw);
    return mk(w.x * inv, w.y * inv);
  }
  tangent = true;
  float2 t0, t1;
  tangent_normals(q, R, t0, t1);
  float d0 = dot(w, t0), d1 = dot(w, t1);
  if (d0 > d1 || (d0 == d1 && angle_of(t0) <= angle_of(t1))) return normalized(t0);
  return normalized(t1);
}
TWA_DEV float2 arc_argmax(float2 q, float R, float2 w) {
  bool tangent;
  return arc_argmax(q, R, w, tangent);
}

// Kinds of winning direction of the free disk minimizer (Best::tag).
enum DiskTag {
  DISK_DEFAULT = 0,  // the (1, 0) fallback
  DISK_GLOBAL = 1,   // global minimiser n_f of the both-stretched piece f
  DISK_A_INNER = 2,  // a / |a| on the arc where b's hinge is zero
  DISK_A_TANGENT = 3,  // an end of that arc, <b, n> = R
  DISK_B_INNER = 4,  // b / |b| on the arc where a's hinge is zero
  DISK_B_TANGENT = 5   // an end of that arc, <a, n> = R
};

// Separating direction of the free disk minimizer and the kind of candidate
// it came from.
TWA_DEV float2 disk_dir_free(float2 a, float2 b, float wl, float wh, float R, int& tag) {
  Best best;
  best.init();
  best.offer(mk(1.f, 0.f), hinge_E(a, b, wl, wh, R, mk(1.f, 0.f)), DISK_DEFAULT);
  float2 c[2];
  int nc = trs_global(a, b, wl, wh, R, c);
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (k < nc) best.offer(c[k], hinge_E(a, b, wl, wh, R, c[k]), DISK_GLOBAL);
  // side 0: b's hinge can be zero, best a-term on that arc; side 1: the same
  // with a and b exchanged (one copy of the code, run twice)
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const float2 q = side ? a : b, w = side ? b : a;
    if (dot(q, q) >= R * R) {
      bool tg;
      float2 n = arc_argmax(q, R, w, tg);
      best.offer(n, hinge_E(a, b, wl, wh, R, n),
                 side ? (tg ? DISK_B_TANGENT : DISK_B_INNER) : (tg ? DISK_A_TANGENT : DISK_A_INNER));
    }
  }
  tag = best.tag;
  return best.n;
}

// Collision minimizer core: disk of radius R at the origin, finite equal or
// unequal weights, neither end pinned.  (a, b): targets; (vl, vh): result.
TWA_NOINLINE void disk_prox_free(float2 a, float2 b, float wl, float wh, float R,
                                            float2& vl, float2& vh) {
  int tag;
  float2 n = disk_dir_free(a, b, wl, wh, R, tag);
  vl = axpy(fmaxf(R - dot(a, n), 0.f), n, a);
  vh = axpy(fmaxf(R - dot(b, n), 0.f), n, b);
}

// One end pinned at q (weight infinite): the free end's target is w.  The
// separating direction ranges over the arc {<q,n> >= R}.
TWA_NOINLINE float2 disk_prox_pinned(float2 q, float2 w, float R) {
  float2 n = arc_argmax(q, R, w);
  return axpy(fmaxf(R - dot(w, n), 0.f), n, w);
}

// ---------------------------------------------------------------------------
// Capsule of radius r around the wall segment [c0, c1]
// ---------------------------------------------------------------------------
TWA_DEV float capsule_h(float2 c0, float2 c1, float r, float2 n) {
  return fmaxf(dot(c0, n), dot(c1, n)) + r;
}

TWA_DEV float capsule_E(float2 a, float2 b, float wl, float wh, float2 c0, float2 c1, float r,
                        float2 n) {
  float h = capsule_h(c0, c1, r, n);
  float ga = fmaxf(h - dot(a, n), 0.f), gb = fmaxf(h - dot(b, n), 0.f);
  return fmaf(0.5f * wl * ga, ga, 0.5f * wh * gb * gb);
}

// On the half-plane of directions where end circle ci gives the capsule's
// support (<c_ci - c_other, n> >= 0), the energy is that circle's disk
// energy.  Write n = c nu + s e (e the outward wall direction at that end, nu
// its normal, s >= 0) and beta_x, gamma_x for the coordinates of x - c_ci
// along nu and e.  With no target beyond the end (gamma <= 0) the hinge of
// target x is [r - c beta_x + s |gamma_x|]_+.
// (1) Both targets on one side of the wall's line (beta_a, beta_b of one
// sign): dropping s |gamma| gives a lower bound monotone in c.
// (2) Both in the quarter-turn cone behind the end (|beta_x| <= |gamma_x|):
// s >= 1 - |c| bounds the hinge from below by [r + |gamma_x| -
// |c| (|gamma_x| +- beta_x)]_+, which does not increase with |c|.
// Either way nothing in that half-plane is below the better kink (c = +-1,
// where the bounds are met), and the circle's candidates can be skipped; with
// one end pinned at a the constraint <a, n> >= h(n) asks for a's hinge to be
// zero, which holds at the kink if it holds anywhere on that side, so the rule
// is the same.  False for a zero-length wall.  The signs are decided in
// FP32, so each coordinate must clear a margin of 1e-6 |e| |x - c_ci| (a few
// units in the last place of the products): a target on the wall's line, on
// the perpendicular through the end or at the end centre keeps the circle's
// candidates (which are then computed exactly) instead of trusting a sign
// that rounding may have flipped.
TWA_DEV bool capsule_end_dominated(float2 a, float2 b, float2 c0, float2 c1, int ci) {
  const float2 e = c1 - c0;
  const float ee = dot(e, e);
  if (!(ee > 0.f)) return false;
  const float2 cc = ci ? c1 : c0;
  const float2 out = ci ? e : -e;
  const float2 nu = perp(e);
  const float2 da = a - cc, db = b - cc;
  const float ta = 1e-6f * sqrtf(ee * dot(da, da)), tb = 1e-6f * sqrtf(ee * dot(db, db));
  const float ga = dot(da, out), gb = dot(db, out);
  const float ba = dot(da, nu), bb = dot(db, nu);
  return ga < -ta && gb < -tb &&
         ((ba > ta && bb > tb) || (ba < -ta && bb < -tb) || (fabsf(ba) < -ga - ta && fabsf(bb) < -gb - tb));
}

// Kinds of winning capsule direction (Best::tag): 0 the (1, 0) fallback,
// 1 a kink, and per end circle ci: 2 + 4 ci a stationary point of its
// both-stretched piece (free) or a tangent from the fixed end (pinned),
// 3 + 4 ci the single-hinge direction of the lower (free) / free (pinned)
// end, 4 + 4 ci that of the upper end (free).
TWA_DEV float2 capsule_dir_free(float2 a, float2 b, float wl, float wh, float2 c0, float2 c1,
                                float r, int& tag) {
  Best best;
  best.init();
  best.offer(mk(1.f, 0.f), capsule_E(a, b, wl, wh, c0, c1, r, mk(1.f, 0.f)), 0);
  float2 e = c1 - c0;
  if (e.x != 0.f || e.y != 0.f) {  // kinks: both end circles give the same support
    float2 k0 = normalized(perp(e));
    best.offer(k0, capsule_E(a, b, wl, wh, c0, c1, r, k0), 1);
    best.offer(-k0, capsule_E(a, b, wl, wh, c0, c1, r, -k0), 1);
  }
#pragma unroll 1
  for (int ci = 0; ci < 2; ++ci) {
    if (capsule_end_dominated(a, b, c0, c1, ci)) continue;
    float2 cc = ci ? c1 : c0;
    float2 ac = a - cc, bc = b - cc;
    float2 t[2];
    const int nt = trs_global(ac, bc, wl, wh, r, t);
    bool mine = false;  // a global minimiser in this circle's half-plane
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (k < nt) {
        best.offer(t[k], capsule_E(a, b, wl, wh, c0, c1, r, t[k]), 2 + 4 * ci);
        mine |= (ci ? dot(e, t[k]) : -dot(e, t[k])) >= 0.f;
      }
    // (then nothing stretched in the half-plane is lower)
    if (!mine && trs_local(ac, bc, wl, wh, r, t))
      best.offer(t[0], capsule_E(a, b, wl, wh, c0, c1, r, t[0]), 2 + 4 * ci);
    if (dot(ac, ac) > 0.f) {
      float2 n = normalized(ac);
      best.offer(n, capsule_E(a, b, wl, wh, c0, c1, r, n), 3 + 4 * ci);
    }
    if (dot(bc, bc) > 0.f) {
      float2 n = normalized(bc);
      best.offer(n, capsule_E(a, b, wl, wh, c0, c1, r, n), 4 + 4 * ci);
    }
  }
  tag = best.tag;
  return best.n;
}

TWA_NOINLINE void capsule_prox_free(float2 a, float2 b, float wl, float wh, float2 c0,
                                               float2 c1, float r, float2& vl, float2& vh) {
  int tag;
  float2 n = capsule_dir_free(a, b, wl, wh, c0, c1, r, tag);
  float h = capsule_h(c0, c1, r, n);
  vl = axpy(fmaxf(h - dot(a, n), 0.f), n, a);
  vh = axpy(fmaxf(h - dot(b, n), 0.f), n, b);
}

#ifdef __CUDACC__
// capsule_prox_free by a whole warp (every lane calls it with the same
// arguments and gets the same result): the candidate directions of
// capsule_dir_free are shared out over 7 lanes (the fallback and kinks; per
// end circle the global and the local stationary point and the single-hinge
// directions), each lane keeps its best in the same order, and a
// warp reduction on (E, angle, position in the sequence) picks the candidate
// that the sequential scan keeps.  The secular solves then run side by side
// instead of one after another.
__device__ __forceinline__ void capsule_prox_free_warp(float2 a, float2 b, float wl, float wh,
                                                       float2 c0, float2 c1, float r, float2& vl,
                                                       float2& vh) {
  const int lane = threadIdx.x & 31;
  Best best;
  best.init();
  bool any = false;
  auto offer = [&](float2 c) {
    best.offer(c, capsule_E(a, b, wl, wh, c0, c1, r, c), 0);
    any = true;
  };
  if (lane == 0) {
    offer(mk(1.f, 0.f));
    float2 e = c1 - c0;
    if (e.x != 0.f || e.y != 0.f) {
      float2 k0 = normalized(perp(e));
      offer(k0);
      offer(-k0);
    }
  } else if (lane < 7 && !capsule_end_dominated(a, b, c0, c1, (lane - 1) / 3)) {
    const int ci = (lane - 1) / 3, task = (lane - 1) % 3;
    const float2 cc = ci ? c1 : c0;
    const float2 ac = a - cc, bc = b - cc;
    float2 t[2];
    int nt = 0;
    if (task == 0) nt = trs_global(ac, bc, wl, wh, r, t);
    else if (task == 1) nt = trs_local(ac, bc, wl, wh, r, t);
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (k < nt) offer(t[k]);
    if (task == 2) {
      if (dot(ac, ac) > 0.f) offer(normalized(ac));
      if (dot(bc, bc) > 0.f) offer(normalized(bc));
    }
  }
  // reduction: lower E, then smaller angle, then the earlier lane (whose
  // candidates come first in the sequential order)
  float E = any ? best.E : INFINITY;
  float2 n = best.n;
  int src = any ? lane : 32;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float E2 = __shfl_xor_sync(0xffffffffu, E, o);
    const float nx = __shfl_xor_sync(0xffffffffu, n.x, o), ny = __shfl_xor_sync(0xffffffffu, n.y, o);
    const int src2 = __shfl_xor_sync(0xffffffffu, src, o);
    bool take;
    if (src2 == 32) take = false;
    else if (src == 32) take = true;
    else if (E2 < E) take = true;
    else if (E2 == E) {
      const float g2 = angle_of(mk(nx, ny)), g = angle_of(n);
      take = g2 < g || (g2 == g && src2 < src);
    } else {
      // NaN energies never win in the sequential scan, and the fallback
      // (lane 0) is always offered first
      take = false;
    }
    if (take) { E = E2; n = mk(nx, ny); src = src2; }
  }
  const float h = capsule_h(c0, c1, r, n);
  vl = axpy(fmaxf(h - dot(a, n), 0.f), n, a);
  vh = axpy(fmaxf(h - dot(b, n), 0.f), n, b);
}
#endif

// One end pinned at q; free end target w.  Candidates: tangent directions
// from q to both end circles, the kinks, and the single-hinge directions;
// only directions that still separate q from the capsule are kept.
// Returns false if no candidate separates q (q inside the capsule).
TWA_DEV bool capsule_dir_pinned(float2 q, float2 w, float2 c0, float2 c1, float r, float2& dir,
                                int& tag) {
  float scale = fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)),
                      fmaxf(fmaxf(fabsf(c0.x), fabsf(c0.y)), fmaxf(fabsf(c1.x), fabsf(c1.y)))) + r;
  float tol = 4e-6f * scale;
  Best best;
  best.init();
  bool any = false;
  // candidates in a fixed order, each kept if it separates q
  auto offer = [&](float2 c, int t) {
    float h = capsule_h(c0, c1, r, c);
    if (dot(q, c) - h >= -tol) {
      float g = fmaxf(h - dot(w, c), 0.f);
      best.offer(c, 0.5f * g * g, t);
      any = true;
    }
  };
  float2 e = c1 - c0;
  if (e.x != 0.f || e.y != 0.f) {
    float2 k0 = normalized(perp(e));
    offer(k0, 1);
    offer(-k0, 1);
  }
#pragma unroll 1
  for (int ci = 0; ci < 2; ++ci) {
    if (any && capsule_end_dominated(q, w, c0, c1, ci)) continue;
    float2 cc = ci ? c1 : c0;
    float2 qc = q - cc;
    if (dot(qc, qc) >= r * r) {
      float2 t0, t1;
      tangent_normals(qc, r, t0, t1);
      offer(normalized(t0), 2 + 4 * ci);
      offer(normalized(t1), 2 + 4 * ci);
    }
    float2 wc = w - cc;
    if (dot(wc, wc) > 0.f) offer(normalized(wc), 3 + 4 * ci);
  }
  dir = best.n;
  tag = best.tag;
  return any;
}

TWA_NOINLINE bool capsule_prox_pinned(float2 q, float2 w, float2 c0, float2 c1, float r,
                                                 float2& vw) {
  float2 n;
  int tag;
  if (!capsule_dir_pinned(q, w, c0, c1, r, n, tag)) { vw = w; return false; }
  float h = capsule_h(c0, c1, r, n);
  vw = axpy(fmaxf(h - dot(w, n), 0.f), n, w);
  return true;
}

// ---------------------------------------------------------------------------
// Zero incoming weights (the feasibility problem, no kinetic factors)
// ---------------------------------------------------------------------------
// Weight classes of one end: 0 (zero), 1 (rho0), 2 (infinite: fixed end).
// One end's weight -> 0+ with the other finite has a lexicographic limit:
// the weighted end moves out of the region by the least amount (a segment
// shrunk to that point is feasible), then the zero-weight end solves the
// fixed-end problem against it.  Both zero are equal weights.

// Closest point to q outside the open disk of radius R at the origin.
TWA_DEV float2 disk_project_out(float2 q, float R) {
  const float L = hypotf(q.x, q.y);
  if (L >= R) return q;
  if (L > 0.f) return (R / L) * q;
  return mk(R, 0.f);
}

// Closest point to q outside the open capsule of radius r around [c0, c1]; a
// point on the axis leaves along the normal of smallest angle.
TWA_DEV float2 capsule_project_out(float2 q, float2 c0, float2 c1, float r) {
  const float2 e = c1 - c0;
  const float ee = dot(e, e);
  float t = ee > 0.f ? dot(q - c0, e) / ee : 0.f;
  t = fminf(1.f, fmaxf(0.f, t));
  const float2 c = axpy(t, e, c0);
  const float2 d = q - c;
  const float L = hypotf(d.x, d.y);
  if (L >= r) return q;
  if (L > 0.f) return axpy(r / L, d, c);
  if (!(ee > 0.f)) return c + mk(r, 0.f);
  const float2 n1 = normalized(perp(e));
  return axpy(r, (angle_of(n1) < angle_of(-n1)) ? n1 : -n1, c);
}

// Disk minimizer for weight classes (cl, ch) of the two ends of the relative
// segment (equal finite weights where both are 1).
TWA_DEV void disk_prox_classes(float2 a, float2 b, int cl, int ch, float R, float w, float2& vl,
                               float2& vh) {
  vl = a; vh = b;
  if (cl == 2 && ch == 2) return;
  if (cl == ch) { disk_prox_free(a, b, w, w, R, vl, vh); return; }  // both rho0 or both zero
  // one end fixed (class 2), or one end of zero weight, which first leaves
  // the disk by the least amount and is then held there: either way the other
  // end solves the fixed-end problem (one call site for the four cases)
  const bool lo_fixed = (cl == 2) || (cl == 1 && ch == 0);
  if (cl == 1 && ch == 0) vl = disk_project_out(a, R);
  if (cl == 0 && ch == 1) vh = disk_project_out(b, R);
  const float2 q = lo_fixed ? vl : vh, t = lo_fixed ? b : a;
  const float2 v = disk_prox_pinned(q, t, R);
  if (lo_fixed) vh = v; else vl = v;
}

// Capsule minimizer for weight classes; false if a fixed end lies inside.
TWA_DEV bool capsule_prox_classes(float2 a, float2 b, int cl, int ch, float2 c0, float2 c1, float r,
                                  float w, float2& vl, float2& vh) {
  vl = a; vh = b;
  if (cl == 2 && ch == 2) return true;
  if (cl == ch) { capsule_prox_free(a, b, w, w, c0, c1, r, vl, vh); return true; }  // equal weights
  // as disk_prox_classes: the other end solves the fixed-end problem
  const bool lo_fixed = (cl == 2) || (cl == 1 && ch == 0);
  if (cl == 1 && ch == 0) vl = capsule_project_out(a, c0, c1, r);
  if (cl == 0 && ch == 1) vh = capsule_project_out(b, c0, c1, r);
  return lo_fixed ? capsule_prox_pinned(vl, b, c0, c1, r, vh) : capsule_prox_pinned(vh, a, c0, c1, r, vl);
}

// ---------------------------------------------------------------------------
// Maximum / minimum velocity minimizers (Appendices F and G)
// ---------------------------------------------------------------------------
// |x_lo - x_hi| <= C (is_max) or >= C, from messages that violate it.  With
// equal finite weights the appendix's closed form keeps the midpoint and
// scales x_lo - x_hi to length C along n_lo - n_hi; an infinite weight (or a
// zero weight against a finite one) keeps the other end; both zero are equal
// weights.  Coincident ends (minimum velocity) separate along (1, 0).
TWA_DEV void velocity_prox(float2 n_lo, float2 n_hi, int cl, int ch, float C, float2& x_lo,
                           float2& x_hi) {
  x_lo = n_lo; x_hi = n_hi;
  if (cl == 2 && ch == 2) return;
  const float2 d = n_lo - n_hi;
  const float L = hypotf(d.x, d.y);
  const float2 u = L > 0.f ? (1.f / L) * d : mk(-1.f, 0.f);
  if (cl == 2 || (ch == 0 && cl != 0)) { x_hi = axpy(-C, u, n_lo); return; }
  if (ch == 2 || (cl == 0 && ch != 0)) { x_lo = axpy(C, u, n_hi); return; }
  const float2 m = 0.5f * (n_lo + n_hi);
  const float2 h = (0.5f * C) * u;  // rounded before it is added (the order of operations: see trs_global)
  x_lo = m + h;
  x_hi = m - h;
}

}  // namespace twa
