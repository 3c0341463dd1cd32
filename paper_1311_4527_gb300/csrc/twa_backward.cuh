// twa_backward.cuh -- the adjoint of one TWA iteration (Appendix B steps
// 1-7) with its branch choices frozen: which collision factors were active
// and which candidate direction each minimizer took.
//
// Forward iteration k (every weight rho0; u = 0 on edges that were not
// active and at fixed nodes):
//   n_e = z^k_node(e) - u^k_e;  x = g(n) per factor
//   z^{k+1}_v = (1 / c_v) sum over the c_v active edges e at v of (x_e + u^k_e)
//   u^{k+1}_e = u^k_e + alpha (x_e - z^{k+1}_v) on active edges at free nodes.
// Given zbar = dL/dz^{k+1} and ubar = dL/du^{k+1}, the adjoint step is
//   zhat_v = zbar_v - alpha sum_e ubar_e,   mbar_v = zhat_v / c_v
//   xbar_e = mbar_v + alpha ubar_e,          nbar = (dg/dn)^T xbar
//   dL/dz^k_v = sum_e nbar_e,   dL/du^k_e = ubar_e + mbar_v - nbar_e.
// One pass over the factors per iteration: whoever computes dL/du^k of an edge
// adds alpha times it to the sum that iteration k - 1 will read, if the edge
// was active in that one too (a flag of the tape; the kinetic edges always
// are), and mbar is formed where it is read, from the counts on the tape.  The
// sums and the adjoint of z go through three buffers: read, added to, cleared.
// At fixed nodes z is the start or goal, x is unused and u stays 0.  A
// collision edge's u^{k+1} matters only if the factor is active in both k and
// k+1 (else it is reset or unused), so its adjoint is kept with the iteration
// that wrote it (stamp) and read as 0 unless the stamp is k + 1.  Wall and
// velocity-limit factors are gated the same way and carried alike.
//
// Sums into nodes use FP64 atomics (order-dependent in the last bits only).
#pragma once
#include "twa_adjoint.cuh"
#include "twa_iter.cuh"

namespace {

// Flag of a tape entry: the factor was active in the iteration before too.
constexpr uint32_t WAS_ACTIVE = 0x80000000u;

struct AdjDev {
  int p, eta, ntp, k;       // k: iteration (kernels add *k0, the first one of their segment)
  float rho, alpha;
  const int2* tiles;
  const float* radius;
  const float* cost;        // [p][eta] c_{i,s}
  int nw, nv;               // wall kinds, then velocity-limit kinds (gated segment factors)
  int vo;                   // local planner epoch: no kinetic factor on segment 0
  unsigned vmin_mask;       // velocity kind v is a minimum
  const float4* walls;      // [nw]
  const float* vlim;        // [nv][p][eta]
  // the tape of iteration k
  const float2* z;          // z^k, [p][eta+1]
  const double* inv;        // 1 / active edges of a break-point (0 without one), [p][eta+1]
  const float4* ukin;       // u^k of the kinetic edges, [eta][p]
  const uint32_t* fid;      // collision slots active in iteration k (with WAS_ACTIVE)
  const float4* ucl;        // their u^k at the lower break-point: (u_i, u_j)
  const float4* uch;        // ... at the upper break-point
  const unsigned* count;    // how many
  const uint32_t* sidx;     // gated segment factors active in iteration k: (g eta + s) p + i (with WAS_ACTIVE)
  const float4* su;         // their u^k (lower, upper)
  const unsigned* scount;   // how many
  // adjoint state
  float4* ubk;              // kinetic u adjoints, [eta][p]: of u^{k+1} in, u^k out
  float4* ubl;              // collision u adjoints by slot (lower, upper)
  float4* ubh;
  const int* k0;
  int* stamp;               // the iteration whose u adjoint a slot holds
  float4* ubs;              // gated segment factor u adjoints, [(nw + nv) eta p]
  int* sstamp;              // ... and the iteration that wrote them
  const double2* zb_in;     // dL/dz^{k+1}
  double2* zb_out;          // dL/dz^k, accumulated
  double2* zb_clear;        // the next step's zb_out
  const double2* S_in;      // alpha * sum of u adjoints per node, for this iteration
  double2* S_out;           // ... for the one before it, accumulated
  double2* S_clear;
  float2* mbar;             // per node, where a pass before the factors' forms it (bw_run_kernel)
  double2* g_start;         // [p]
  double2* g_goal;          // [p]
  double* g_r;              // [p]
  double* g_c;              // [p][eta], adjoint of c_{i,s}
};

__device__ __forceinline__ void atomic_add2(double2* a, float2 v) {
  atomicAdd(&a->x, (double)v.x);
  atomicAdd(&a->y, (double)v.y);
}

__device__ __forceinline__ void decode_slot(const AdjDev& A, uint32_t f, int& s, int& i, int& j) {
  const uint32_t row = f >> 5, c = f & 31;
  const uint32_t blk = row >> 5, r = row & 31;
  s = (int)(blk / A.ntp);
  const int2 IJ = A.tiles[blk - (uint32_t)s * A.ntp];
  i = IJ.x * TILE + (int)r;
  j = IJ.y * TILE + (int)c;
}

// The u adjoint of pair slot f, 0 unless the iteration after this one wrote
// it.  Loaded beside the stamp, not after it (a slot never written holds
// anything, and is not used).
__device__ __forceinline__ float4 live_ub(const AdjDev& A, const float4* ub, uint32_t f) {
  const float4 v = ub[f];
  return A.stamp[f] == A.k + 1 ? v : make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __forceinline__ void scatter_edge(const AdjDev& A, double2* S, int i, int s, float2 ub) {
  atomic_add2(S + (size_t)i * (A.eta + 1) + s, mk(A.alpha * ub.x, A.alpha * ub.y));
}
// The two ends of one agent's segment s (nothing at fixed ends).
__device__ __forceinline__ void scatter_ends(const AdjDev& A, double2* S, int i, int s, float2 lo, float2 hi) {
  if (s > 0) scatter_edge(A, S, i, s, lo);
  if (s + 1 < A.eta) scatter_edge(A, S, i, s + 1, hi);
}

// The gated edges' part of S_in for the last iteration of a segment, whose
// activity was not known when the iteration behind it (the next segment's
// first) took its step.
__device__ __forceinline__ void bw_scatter_item(const AdjDev& A, unsigned t) {
  const unsigned ncoll = *A.count;
  double2* S = const_cast<double2*>(A.S_in);
  if (t >= ncoll) {  // a gated segment factor
    const uint32_t g = A.sidx[t - ncoll] & ~WAS_ACTIVE;
    const int i = (int)(g % A.p), s = (int)((g / A.p) % A.eta);
    if (A.sstamp[g] != A.k + 1) return;
    const float4 ub = A.ubs[g];
    scatter_ends(A, S, i, s, lo2(ub), hi2(ub));
    return;
  }
  const uint32_t f = A.fid[t] & ~WAS_ACTIVE;
  if (A.stamp[f] != A.k + 1) return;
  int s, i, j;
  decode_slot(A, f, s, i, j);
  const float4 bl = A.ubl[f], bh = A.ubh[f];
  scatter_ends(A, S, i, s, lo2(bl), lo2(bh));
  scatter_ends(A, S, j, s, hi2(bl), hi2(bh));
}

// Per break-point: the start / goal gradients at the fixed ends, and the
// buffers of the next step cleared.
__device__ __forceinline__ void bw_node(const AdjDev& A, int t) {
  const int E1 = A.eta + 1;
  const int i = t / E1, s = t - i * E1;
  if (s == 0 || s == A.eta) {
    const double2 zb = A.zb_in[t];
    double2* g = s == 0 ? A.g_start : A.g_goal;
    g[i].x += zb.x;
    g[i].y += zb.y;
  }
  A.S_clear[t] = make_double2(0.0, 0.0);
  A.zb_clear[t] = make_double2(0.0, 0.0);
}

// mbar of a free node.
__device__ __forceinline__ float2 node_mbar(const AdjDev& A, size_t node) {
  const double2 zb = A.zb_in[node], S = A.S_in[node];
  const double inv = A.inv[node];
  return mk((float)((zb.x - S.x) * inv), (float)((zb.y - S.y) * inv));
}

// Per edge: xbar, and the u adjoint once nbar is known.  MBAR: mbar was formed
// by a pass over the nodes.
template <bool MBAR>
__device__ __forceinline__ float2 edge_xbar(const AdjDev& A, bool fixed, int i, int s, float2 ub,
                                           float2& mb) {
  if (fixed) { mb = mk(0.f, 0.f); return mb; }
  const size_t node = (size_t)i * (A.eta + 1) + s;
  mb = MBAR ? A.mbar[node] : node_mbar(A, node);
  return axpy(A.alpha, ub, mb);
}
__device__ __forceinline__ float2 edge_ubar(bool fixed, float2 ub, float2 mb, float2 nb) {
  return fixed ? mk(0.f, 0.f) : mk(ub.x + mb.x - nb.x, ub.y + mb.y - nb.y);
}

// A wall or velocity-limit factor (gated like a collision factor).
template <bool MBAR>
__device__ __forceinline__ void bw_seg_item(const AdjDev& A, unsigned w) {
  const int E1 = A.eta + 1;
  const uint32_t entry = A.sidx[w], g = entry & ~WAS_ACTIVE;
  const int i = (int)(g % A.p), s = (int)((g / A.p) % A.eta);
  const int kind = (int)(g / ((uint32_t)A.p * A.eta));
  const bool pin_lo = (s == 0), pin_hi = (s == A.eta - 1);
  const float4 u = A.su[w];
  const float2 nl = A.z[(size_t)i * E1 + s] - lo2(u), nh = A.z[(size_t)i * E1 + s + 1] - hi2(u);
  const float4 ub = (A.sstamp[g] == A.k + 1) ? A.ubs[g] : make_float4(0.f, 0.f, 0.f, 0.f);
  float2 ml, mh;
  const float2 xl = edge_xbar<MBAR>(A, pin_lo, i, s, lo2(ub), ml);
  const float2 xh = edge_xbar<MBAR>(A, pin_hi, i, s + 1, hi2(ub), mh);
  float2 bl, bh;
  if (kind < A.nw) {
    const float4 W = A.walls[kind];
    float rb;
    wall_vjp(nl, nh, pin_lo, pin_hi, mk(W.x, W.y), mk(W.z, W.w), A.radius[i], A.rho, xl, xh, bl, bh, rb);
    atomicAdd(A.g_r + i, (double)rb);
  } else {
    const int v = kind - A.nw;
    velocity_vjp(nl, nh, pin_lo, pin_hi, A.vlim[((size_t)v * A.p + i) * A.eta + s], xl, xh, bl, bh);
  }
  atomic_add2(A.zb_out + (size_t)i * E1 + s, bl);
  atomic_add2(A.zb_out + (size_t)i * E1 + s + 1, bh);
  const float4 un = pack(edge_ubar(pin_lo, lo2(ub), ml, bl), edge_ubar(pin_hi, hi2(ub), mh, bh));
  A.ubs[g] = un;
  A.sstamp[g] = A.k;
  if (entry & WAS_ACTIVE) scatter_ends(A, A.S_out, i, s, lo2(un), hi2(un));
}

// The adjoint of one factor's minimizer (t past the break-points).
template <bool MBAR>
__device__ __forceinline__ void bw_factor_item(const AdjDev& A, unsigned t) {
  const int E1 = A.eta + 1;
  const unsigned nkin = (unsigned)(A.eta * A.p);
  const unsigned ncoll = *A.count;
  if (t >= nkin + ncoll) { bw_seg_item<MBAR>(A, t - nkin - ncoll); return; }
  if (t < nkin) {
    const int s = (int)(t / A.p), i = (int)(t - (unsigned)s * A.p);
    if (A.vo && s == 0) return;
    const bool pin_lo = (s == 0), pin_hi = (s == A.eta - 1);
    const float4 u = A.ukin[t];
    const float2 nl = A.z[(size_t)i * E1 + s] - lo2(u), nh = A.z[(size_t)i * E1 + s + 1] - hi2(u);
    const float4 ub = A.ubk[t];
    float2 ml, mh;
    const float2 xl = edge_xbar<MBAR>(A, pin_lo, i, s, lo2(ub), ml);
    const float2 xh = edge_xbar<MBAR>(A, pin_hi, i, s + 1, hi2(ub), mh);
    float2 bl, bh;
    float cb;
    energy_vjp(nl, nh, A.rho, pin_lo, pin_hi, A.cost[(size_t)i * A.eta + s], xl, xh, bl, bh, cb);
    atomic_add2(A.zb_out + (size_t)i * E1 + s, bl);
    atomic_add2(A.zb_out + (size_t)i * E1 + s + 1, bh);
    const float4 un = pack(edge_ubar(pin_lo, lo2(ub), ml, bl), edge_ubar(pin_hi, hi2(ub), mh, bh));
    A.ubk[t] = un;
    scatter_ends(A, A.S_out, i, s, lo2(un), hi2(un));
    A.g_c[(size_t)i * A.eta + s] += (double)cb;
    return;
  }
  const unsigned w = t - nkin;
  const uint32_t entry = A.fid[w], f = entry & ~WAS_ACTIVE;
  int s, i, j;
  decode_slot(A, f, s, i, j);
  const bool pin_lo = (s == 0), pin_hi = (s == A.eta - 1);
  const float4 a = A.ucl[w], b = A.uch[w];
  // n exactly as the forward minimizer pass formed it
  const float2 nil = A.z[(size_t)i * E1 + s] - lo2(a), nih = A.z[(size_t)i * E1 + s + 1] - lo2(b);
  const float2 njl = A.z[(size_t)j * E1 + s] - hi2(a), njh = A.z[(size_t)j * E1 + s + 1] - hi2(b);
  const float4 bl = live_ub(A, A.ubl, f), bh = live_ub(A, A.ubh, f);
  float2 mil, mjl, mih, mjh;
  const float2 xil = edge_xbar<MBAR>(A, pin_lo, i, s, lo2(bl), mil);
  const float2 xjl = edge_xbar<MBAR>(A, pin_lo, j, s, hi2(bl), mjl);
  const float2 xih = edge_xbar<MBAR>(A, pin_hi, i, s + 1, lo2(bh), mih);
  const float2 xjh = edge_xbar<MBAR>(A, pin_hi, j, s + 1, hi2(bh), mjh);
  float2 nbil, nbih, nbjl, nbjh;
  float Rb;
  coll_vjp(nil, nih, njl, njh, pin_lo, pin_hi, A.radius[i] + A.radius[j], A.rho, xil, xih, xjl,
           xjh, nbil, nbih, nbjl, nbjh, Rb);
  atomic_add2(A.zb_out + (size_t)i * E1 + s, nbil);
  atomic_add2(A.zb_out + (size_t)j * E1 + s, nbjl);
  atomic_add2(A.zb_out + (size_t)i * E1 + s + 1, nbih);
  atomic_add2(A.zb_out + (size_t)j * E1 + s + 1, nbjh);
  atomicAdd(A.g_r + i, (double)Rb);
  atomicAdd(A.g_r + j, (double)Rb);
  const float4 ul = pack(edge_ubar(pin_lo, lo2(bl), mil, nbil), edge_ubar(pin_lo, hi2(bl), mjl, nbjl));
  const float4 uh = pack(edge_ubar(pin_hi, lo2(bh), mih, nbih), edge_ubar(pin_hi, hi2(bh), mjh, nbjh));
  A.ubl[f] = ul;
  A.ubh[f] = uh;
  A.stamp[f] = A.k;
  if (entry & WAS_ACTIVE) {
    scatter_ends(A, A.S_out, i, s, lo2(ul), lo2(uh));
    scatter_ends(A, A.S_out, j, s, hi2(ul), hi2(uh));
  }
}

// Factors of an adjoint step.
__device__ __forceinline__ unsigned bw_factors(const AdjDev& A) {
  return (unsigned)(A.eta * A.p) + *A.count + *A.scount;
}

}  // namespace
