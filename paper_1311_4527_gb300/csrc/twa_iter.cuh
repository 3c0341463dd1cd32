// twa_iter.cuh -- the per-warp work of one TWA iteration (Appendix B steps
// 1-7 over the factor graph of Section 3.3 of Bento et al., NIPS 2013), shared
// by the single-planner kernels and the batched ones (both in plan.cu).
//
// Gated state (default): two launches.
//   Factor pass, collision_warp and segment_warp: every factor.  The pairs
//     that were active lately are on a worklist, 32 to a warp; a tile warp
//     looks through one (segment, agent tiles I <= J) block of 32 x 32 pairs
//     for others that collide; a segment warp takes one kinetic, wall or
//     velocity kind of one (segment, agent tile).  Whoever finds a factor
//     active runs its minimizer at once and adds m = x + u to the consensus
//     sums.
//   Node pass, consensus_warp: z = sum m / count per free break-point (step
//     5), and the per-segment records the next factor pass starts from.
// Dense state: test_block (every pair's u record streamed, lane = column
//   agent, then prox_item for the active ones) and segment_warp in one launch,
//   then the node pass.  (A batch runs prox_item over its worklists in a launch
//   of its own.)
//
// Step 7 needs z^{k+1}, which exists only after every factor ran, so x^{k+1}
// of the active factors is stored and u^{k+1} = u^k + alpha (x^{k+1} -
// z^{k+1}) is finished at the start of the next iteration.  Back weights
// (step 6) are rho0 at every interior node (the kinetic factors always send
// rho0 there) and infinity at the fixed ends; u on an edge whose forward
// weight was 0, or whose node is fixed, is 0.
//
// Collision-factor state lives in tile order: block blk = s * ntp + tp holds
// the 32 x 32 pair slots (row r = i - 32 I, column c = j - 32 J), so a warp
// streams one row as 32 consecutive float4 (512 B).  Per slot:
//   ulo[slot] = (u_i(s), u_j(s))       uhi[slot] = (u_i(s+1), u_j(s+1))
//   xlo / xhi = pending x^{k+1}, read and written only for active factors
//   bits[blk * 32 + r] bit c = forward weight rho0 in the last iteration.
// With the dense state the u record of every slot is read and written each
// iteration; otherwise only those of factors whose bit is set (every other u
// is 0 by the reset rule), which leaves 1 bit per factor of state traffic.
//
// Worklist of the gated state.  work[0 .. n) holds slots, bit 31 set where
// the pair was active in the last iteration; listed[row] bit c says that the
// pair is on it.  A pair joins when a tile warp finds it active, and stays on
// it after it turns inactive (a pair that left often comes back; its u is 0
// then), so the tile warps of an iteration can read `listed` while the list
// warps work: no pair leaves it meanwhile.  When more than half of the list is
// inactive, or an append did not fit, the next iteration builds it anew: the
// tile warps then take the pairs of `listed` too and the list warps nothing;
// a pair drops out if it was inactive and still is, which the test on z that a
// tile warp makes would also find.  `bits` and the slot records are the
// state, the list only an order of work, and any list gives the same
// iterates.  (An iteration that rebuilds goes through the tiles in the agents'
// own order, also where they are sorted, so that a block's listed pairs and
// its new ones are one warp's.)
//
// Sorted tiles (large single plans).  The tiles of the search are made of
// agents in the order of a Morton curve through their segments' midpoints,
// sorted anew now and then (perm / inv), with a box around each group of 32:
// two groups whose boxes do not meet hold no near pair.  The slots stay in
// agent order.  Boxes only grow between sorts (the node pass widens the box
// of an agent that left it), so they hold whatever the order's age.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "twa_math.cuh"

namespace {

using namespace twa;

constexpr int TILE = 32;
constexpr unsigned FULL = 0xffffffffu;

struct Dev {
  int p, eta, nw, nt, ntp;
  float rho, alpha;
  int dense, keep, admm;
  int nv;                // velocity-factor kinds after the walls (0..2)
  unsigned vmin_mask;    // bit v: velocity kind v is a minimum (else maximum)
  int noenergy;          // no kinetic factors (the feasibility problem)
  int vo;                // velocity-obstacle epoch (eta = 2): collision, wall and velocity
                         // factors on segment 0 only, the kinetic factor on segment 1 only
  const float* vlim;     // [nv][p][eta] velocity limits
  uint8_t* wnode;        // [p][eta+1] back-weight class when noenergy: 0 or 1
  const float2* z;       // z^k, [p][eta+1]
  float2* z_next;        // z^{k+1}; until the consensus pass writes it, z^{k-1}
  const float* radius;   // [p]
  const float* cost;     // [p][eta], kinetic coefficients c_{i,s}
  const float4* walls;   // [nw] (xL.x, xL.y, xR.x, xR.y)
  // uwall / xwall / wbits hold nw wall kinds followed by nv velocity kinds
  const int2* tiles;     // [ntp] (I, J), I <= J
  float4 *ulo, *uhi, *xlo, *xhi;
  uint32_t* bits;        // [eta * ntp * 32]
  float4 *ukin, *xkin;   // [eta][p]
  float4 *uwall, *xwall; // [nw][eta][p]
  uint32_t* wbits;       // [nw][eta][nt]
  float4* zseg;          // [eta][p] (z(s), z(s+1)) of z^k (gated state)
  float4* circ;          // [eta][p] bounding circle (m.x, m.y, b, -bounding_offset) of z^k, by
                         // place in the search order
  int sorted;            // sorted tiles (else the search order is the agents' own)
  int* perm;             // [eta][p] agent at a place of the search order
  int* inv;              // [eta][p] place of an agent
  int4* box;             // [eta][nt] box of the circles at 32 places (x, y least, x, y largest;
                         // floats as ordered integers)
  uint32_t* work;        // collision worklist (dense batches: the active slots of this iteration)
  unsigned cap;          // its capacity
  uint32_t* listed;      // [eta * ntp * 32] pairs on the worklist (gated state)
  unsigned* work_count;  // its length, by iteration parity: entries are appended here
  unsigned* work_count_prev;  // ... its length at the start of this iteration
  unsigned* ctl;         // gated state: [0] rebuild the worklist in this iteration, [1] entries
                         // of inactive pairs on it, [2] an append did not fit
  unsigned long long* accx;  // [p][eta+1] fixed-point sums of rho0-weighted m.x
  unsigned long long* accy;  //                                 ... of m.y
  unsigned* accc;        // [p][eta+1] number of rho0-weighted incoming edges
  const float* fix;      // fixed-point scale (a power of two) and |m| bound
  unsigned* res_cur;     // residual slot of this iteration (consensus part)
  unsigned* res_prev;    // residual slot of the previous iteration (primal part)
  unsigned* status;      // bit 0: a pinned wall minimizer had no separating direction;
                         // bit 1: a message out of the fixed-point range
};

// A descriptor whose sums are in shared memory (run_kernel): seven words per
// break-point, three limbs of m.x and of m.y and the count.
struct SoloDev : Dev {
  uint32_t sums;  // shared-memory address
};

// A descriptor whose node pass also notes 1 / counts for the backward pass.
template <class Base>
struct Taped : Base {
  double* inv;  // [p][eta+1]
};
__device__ __forceinline__ void note_count(const Dev&, size_t, unsigned) {}
template <class Base>
__device__ __forceinline__ void note_count(const Taped<Base>& P, size_t node, unsigned cnt) {
  P.inv[node] = cnt ? 1.0 / (double)cnt : 0.0;
}

__device__ __forceinline__ float maxabs2(float2 a) { return fmaxf(fabsf(a.x), fabsf(a.y)); }

// Step 7 of the previous iteration for one edge: u^k from the stored u^{k-1},
// the pending x^k and z^k.
__device__ __forceinline__ float2 finish_u(bool bprev, bool pinned, bool keep, float2 u_prev,
                                           float2 x_pend, float2 zk, float alpha, float& res) {
  if (pinned) return mk(0.f, 0.f);
  if (bprev) {
    float2 d = x_pend - zk;
    res = fmaxf(res, maxabs2(d));
    return axpy(alpha, d, u_prev);
  }
  return keep ? u_prev : mk(0.f, 0.f);
}

// Step 5's sums in 64-bit fixed point: each FP32 m is scaled by a power of
// two 2^e chosen from the layout's extent and rounded to an integer (an
// absolute error of at most 2^-(e+1), about 1e-13 at p = 1024 on the 40 x 40
// square, far below the FP32 ulp of m itself), then the integers are summed
// exactly; integer addition does not depend on the order of the atomics, so z
// is deterministic: the integer sum rounded once to FP32 and divided by the
// count in FP32 (within 1.5 units in the last place of the mean of the
// quantised messages).  A non-finite or out-of-range m sets status bit 1,
// which the consensus pass turns into a NaN residual.
__device__ __forceinline__ void contribute(const Dev& P, float scale, float bound, int i, int s,
                                           float2 m) {
  if (!(fabsf(m.x) <= bound && fabsf(m.y) <= bound)) {
    atomicOr(P.status, 2u);
    return;
  }
  const size_t node = (size_t)i * (P.eta + 1) + s;
  atomicAdd(P.accx + node, (unsigned long long)__float2ll_rn(m.x * scale));
  atomicAdd(P.accy + node, (unsigned long long)__float2ll_rn(m.y * scale));
  atomicAdd(P.accc + node, 1u);
}

// The same sums in shared memory, which has no 64-bit add: each integer goes
// in limbs of 22, 22 and 20 bits (the last one signed) into three 32-bit
// counters, which 1,024 messages cannot overflow, and nothing waits for the
// adds.  (64-bit atomics there are compare-and-swap loops.)
constexpr int SUM_WORDS = 7;
__device__ __forceinline__ void shared_add(uint32_t at, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t shared_take(uint32_t at) {  // read and clear
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(0u) : "memory");
  return v;
}
__device__ __forceinline__ void contribute(const SoloDev& P, float scale, float bound, int i, int s,
                                           float2 m) {
  if (!(fabsf(m.x) <= bound && fabsf(m.y) <= bound)) {
    atomicOr(P.status, 2u);
    return;
  }
  const uint32_t at = P.sums + 4u * SUM_WORDS * (uint32_t)(i * (P.eta + 1) + s);
  const long long x = __float2ll_rn(m.x * scale), y = __float2ll_rn(m.y * scale);
  constexpr uint32_t LIMB = (1u << 22) - 1u;
  shared_add(at, (uint32_t)x & LIMB);
  shared_add(at + 4, (uint32_t)(x >> 22) & LIMB);
  shared_add(at + 8, (uint32_t)(x >> 44));
  shared_add(at + 12, (uint32_t)y & LIMB);
  shared_add(at + 16, (uint32_t)(y >> 22) & LIMB);
  shared_add(at + 20, (uint32_t)(y >> 44));
  shared_add(at + 24, 1u);
}
template <class D>
__device__ __forceinline__ void contribute(const D& P, int i, int s, float2 m) {
  contribute(P, P.fix[0], P.fix[1], i, s, m);
}

// A break-point's sums and count, cleared for the next iteration.
__device__ __forceinline__ void take_sums(const Dev& P, size_t node, long long& sx, long long& sy, unsigned& cnt) {
  sx = (long long)P.accx[node];
  sy = (long long)P.accy[node];
  cnt = P.accc[node];
  P.accx[node] = 0ull;
  P.accy[node] = 0ull;
  P.accc[node] = 0u;
}
__device__ __forceinline__ void take_sums(const SoloDev& P, size_t node, long long& sx, long long& sy, unsigned& cnt) {
  const uint32_t at = P.sums + 4u * SUM_WORDS * (uint32_t)node;
  uint32_t w[SUM_WORDS];
#pragma unroll
  for (int q = 0; q < SUM_WORDS; ++q) w[q] = shared_take(at + 4 * q);
  auto whole = [](uint32_t a, uint32_t b, uint32_t c) {
    return (long long)((unsigned long long)a + ((unsigned long long)b << 22) + ((unsigned long long)(long long)(int)c << 44));
  };
  sx = whole(w[0], w[1], w[2]);
  sy = whole(w[3], w[4], w[5]);
  cnt = w[6];
}

// Standard-ADMM mode, a factor that was feasible in the previous iteration:
// its x^k was n^{k-1} = z^{k-1} - u^{k-1}, so step 7 needs no stored x.
__device__ __forceinline__ float2 finish_u_feasible(bool pinned, float2 u_prev, float2 z_prev,
                                                    float2 zk, float alpha, float& res) {
  if (pinned) return mk(0.f, 0.f);
  const float2 d = (z_prev - u_prev) - zk;
  res = fmaxf(res, maxabs2(d));
  return axpy(alpha, d, u_prev);
}

__device__ __forceinline__ float2 lo2(float4 v) { return mk(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return mk(v.z, v.w); }
__device__ __forceinline__ float4 pack(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

__device__ __forceinline__ void atomic_max_nonneg(unsigned* slot, float v) {
  atomicMax(slot, __float_as_uint(v));
}

// Four single-precision lanes as two pairs, and paired operations on them
// (one instruction for two multiply-adds).
__device__ __forceinline__ unsigned long long pair_of(float lo, float hi) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c) {
  unsigned long long v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ float lo_of(unsigned long long v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_of(unsigned long long v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

// Collision minimizer of one pair (Appendix C with equal weights rho on each
// end, or infinite at a fixed end).  n: (i lo, i hi, j lo, j hi).
__device__ __forceinline__ void coll_minimizer(float2 nil, float2 nih, float2 njl, float2 njh,
                                               bool pin_lo, bool pin_hi, float R, float rho,
                                               float2& xil, float2& xih, float2& xjl, float2& xjh) {
  float2 cl = njl - nil, ch = njh - nih;     // relative targets v = x_j - x_i
  float2 sl = nil + njl, sh = nih + njh;     // sum coordinates x_i + x_j
  xil = nil; xih = nih; xjl = njl; xjh = njh;
  if (pin_lo && pin_hi) return;
  if (pin_lo || pin_hi) {  // one call site for both fixed ends
    const float2 v = disk_prox_pinned(pin_lo ? cl : ch, pin_lo ? ch : cl, R);
    const float2 sm = pin_lo ? sh : sl;
    const float2 xi = 0.5f * (sm - v), xj = 0.5f * (sm + v);
    if (pin_lo) { xih = xi; xjh = xj; } else { xil = xi; xjl = xj; }
  } else {
    float2 vl, vh;
    float w = 0.5f * rho;  // rho rho / (rho + rho)
    disk_prox_free(cl, ch, w, w, R, vl, vh);
    xil = 0.5f * (sl - vl);
    xjl = 0.5f * (sl + vl);
    xih = 0.5f * (sh - vh);
    xjh = 0.5f * (sh + vh);
  }
}

// The collision minimizer with per-agent weight classes at each end (the
// feasibility problem; Appendix C's reduction with weights rho rho' / (rho +
// rho')): both agents at rho0 give relative weight rho0 / 2, a zero class on
// either gives relative weight 0 and the relative change goes to the
// zero-weight agent (split evenly when both are zero), a fixed end stays.
__device__ __forceinline__ void pair_end(float2 ni, float2 nj, int ci, int cj, float2 v, float2& xi,
                                         float2& xj) {
  if (ci == 2) { xi = ni; xj = nj; return; }
  if (ci == 0 && cj == 1) { xj = nj; xi = nj - v; return; }
  if (ci == 1 && cj == 0) { xi = ni; xj = ni + v; return; }
  const float2 sm = ni + nj;
  xi = 0.5f * (sm - v);
  xj = 0.5f * (sm + v);
}

__device__ __forceinline__ void coll_minimizer_classes(float2 nil, float2 nih, float2 njl,
                                                       float2 njh, int cil, int cih, int cjl,
                                                       int cjh, float R, float rho, float2& xil,
                                                       float2& xih, float2& xjl, float2& xjh) {
  const float2 cl = njl - nil, ch = njh - nih;
  const int rl = (cil == 2) ? 2 : ((cil == 1 && cjl == 1) ? 1 : 0);
  const int rh = (cih == 2) ? 2 : ((cih == 1 && cjh == 1) ? 1 : 0);
  float2 vl, vh;
  disk_prox_classes(cl, ch, rl, rh, R, 0.5f * rho, vl, vh);
  pair_end(nil, njl, cil, cjl, vl, xil, xjl);
  pair_end(nih, njh, cih, cjh, vh, xih, xjh);
}

// Collision test of the n-trajectories (Eq. f_coll_def): does the relative
// segment [cl, ch] pass closer than R to the origin?  Strict, so touching is
// inactive.  Division-free: for an interior closest point, dist^2 =
// cross(cl, d)^2 / |d|^2 is compared as cross^2 < R^2 |d|^2.
__device__ __forceinline__ bool collides(float2 cl, float2 ch, float R) {
  const float2 d = ch - cl;
  const float dd = dot(d, d);
  const float t = -dot(cl, d);
  const float R2 = R * R;
  const float c = cross(cl, d);
  // endpoints, or an interior closest point (0 < t < |d|^2)
  return (dot(cl, cl) < R2) | (dot(ch, ch) < R2) | ((t > 0.f) & (t < dd) & (c * c < R2 * dd));
}

// Do the segments [a0, a1] and [b0, b1] come closer than r (strict)?  They do
// if they cross, or if an end of one is that close to the other.
__device__ __forceinline__ bool within(float2 a0, float2 a1, float2 b0, float2 b1, float r) {
  const float2 da = a1 - a0, db = b1 - b0;
  const float2 p00 = b0 - a0, p01 = b1 - a0, p10 = b0 - a1, p11 = b1 - a1;
  const float d1 = cross(da, p00), d2 = cross(da, p01), d3 = -cross(db, p00), d4 = -cross(db, p10);
  const bool crossing = ((d1 < 0.f && d2 > 0.f) || (d1 > 0.f && d2 < 0.f)) &&
                        ((d3 < 0.f && d4 > 0.f) || (d3 > 0.f && d4 < 0.f));
  return crossing || collides(p00, p01, r) || collides(p10, p11, r) || collides(p00, p10, r) || collides(p01, p11, r);
}

// Kinetic factor (i, s): always active (it always sends rho0).  Finishes its
// pending dual update, runs the closed-form minimizer and stores x and u.
template <class D>
__device__ __forceinline__ void kinetic_factor(const D& P, int i, int s, float2 zl, float2 zh,
                                               bool pin_lo, bool pin_hi, float& res) {
  const size_t idx = (size_t)s * P.p + i;
  const float4 u4 = P.ukin[idx], x4 = P.xkin[idx];
  const float2 ul = finish_u(true, pin_lo, false, lo2(u4), lo2(x4), zl, P.alpha, res);
  const float2 uh = finish_u(true, pin_hi, false, hi2(u4), hi2(x4), zh, P.alpha, res);
  float2 xl, xh;
  energy_prox(zl - ul, zh - uh, P.rho, pin_lo, pin_hi, P.cost[(size_t)i * P.eta + s], xl, xh);
  P.xkin[idx] = pack(xl, xh);
  P.ukin[idx] = pack(ul, uh);
  if (!pin_lo) contribute(P, i, s, xl + ul);
  if (!pin_hi) contribute(P, i, s + 1, xh + uh);
}

// Back-weight classes of agent i's break-points s and s + 1: 2 at a fixed
// end, else rho0 (1) unless the feasibility problem left a node with only
// zero incoming weights (0).
__device__ __forceinline__ void end_classes(const Dev& P, int i, int s, bool pin_lo, bool pin_hi,
                                            int& cl, int& ch) {
  const size_t b = (size_t)i * (P.eta + 1) + s;
  cl = pin_lo ? 2 : (P.noenergy ? (int)P.wnode[b] : 1);
  ch = pin_hi ? 2 : (P.noenergy ? (int)P.wnode[b + 1] : 1);
}

// Gated segment factor w of (i, s): a wall (w < nw, Eq. wall_minimizer) or a
// maximum / minimum velocity factor (w >= nw, Eq. max_vel_min).  Forward
// weight rho0 when the n's violate it, else 0.  Called by a full warp (lane =
// agent of tile I).
template <class D>
__device__ __forceinline__ void wall_factor(const D& P, int w, int i, bool vi, int s, int I,
                                            float2 zl, float2 zh, float r, bool pin_lo,
                                            bool pin_hi, float& res) {
  const int lane = threadIdx.x & 31;
  const size_t widx = ((size_t)w * P.eta + s) * P.nt + I;
  const uint32_t word = P.wbits[widx];
  const bool bprev = vi && ((word >> lane) & 1u);
  const bool vel = w >= P.nw;
  float2 c0 = mk(0.f, 0.f), c1 = c0;
  if (!vel) {
    const float4 W = P.walls[w];
    c0 = mk(W.x, W.y); c1 = mk(W.z, W.w);
    // A wall none of the warp's agents was pushing against, and none can
    // reach: the segment lies in the disk of half its length about its
    // midpoint, so it is out of reach when the midpoint is farther than that
    // plus r from the wall (with a margin of 1e-4 of the radii and 1e-5 of
    // the coordinates, a hundred times the rounding).  Most walls of a warp
    // end here: the exact test costs about ten times as much.
    if (word == 0u && !P.dense) {
      const float2 m = 0.5f * (zl + zh), d = zh - zl;
      const float b = fmaf(0.5f, sqrtf(dot(d, d)), r);
      const float L = fmaxf(fmaxf(maxabs2(c0), maxabs2(c1)), maxabs2(m));
      const float reach = fmaf(1e-5f, L, 1.0001f * b);
      // (coordinates whose squares' products overflow: no wall is left out)
      if (!__any_sync(FULL, vi && !(L < 1e9f && dist2_point_segment(m, c0, c1) > reach * reach))) return;
    }
  }
  const size_t idx = ((size_t)w * P.eta + s) * P.p + i;
  float4 u4 = make_float4(0.f, 0.f, 0.f, 0.f), x4 = u4;
  if (vi && (P.dense || bprev)) u4 = P.uwall[idx];
  if (bprev) x4 = P.xwall[idx];
  float2 ul, uh;
  if (P.admm && vi && !bprev) {
    const int E1 = P.eta + 1;
    ul = finish_u_feasible(pin_lo, lo2(u4), P.z_next[(size_t)i * E1 + s], zl, P.alpha, res);
    uh = finish_u_feasible(pin_hi, hi2(u4), P.z_next[(size_t)i * E1 + s + 1], zh, P.alpha, res);
  } else {
    ul = finish_u(bprev, pin_lo, P.keep, lo2(u4), lo2(x4), zl, P.alpha, res);
    uh = finish_u(bprev, pin_hi, P.keep, hi2(u4), hi2(x4), zh, P.alpha, res);
  }
  const float2 nl = zl - ul, nh = zh - uh;
  bool act;
  float C = 0.f;
  if (vel) {
    const int v = w - P.nw;
    const bool vmin = (P.vmin_mask >> v) & 1u;
    if (vi) C = P.vlim[((size_t)v * P.p + i) * P.eta + s];
    const float2 d = nl - nh;
    const float d2 = dot(d, d);
    act = vi && (vmin ? d2 < C * C : d2 > C * C);
  } else {
    act = vi && within(nl, nh, c0, c1, r);
  }
  const uint32_t nw = __ballot_sync(FULL, act);
  if (lane == 0 && nw != word) P.wbits[widx] = nw;
  if (act) {
    float2 xl = nl, xh = nh;
    int cl, ch;
    end_classes(P, i, s, pin_lo, pin_hi, cl, ch);
    if (vel) {
      velocity_prox(nl, nh, cl, ch, C, xl, xh);
    } else if (!capsule_prox_classes(nl, nh, cl, ch, c0, c1, r, 0.5f * P.rho, xl, xh)) {
      atomicOr(P.status, 1u);
    }
    P.xwall[idx] = pack(xl, xh);
    P.uwall[idx] = pack(ul, uh);
    if (!pin_lo) contribute(P, i, s, xl + ul);
    if (!pin_hi) contribute(P, i, s + 1, xh + uh);
  } else if (vi && P.dense) {
    P.uwall[idx] = pack(ul, uh);
  }
}

// Kinetic, wall and velocity factors (steps 1-3 and the pending step 7): one
// warp per (kind f, segment s, agent tile I), lane = agent; item = (s nt + I)
// kinds + f, kind 0 the kinetic factor.
template <class D>
__device__ __forceinline__ void segment_warp(const D& P, int item) {
  const int kinds = 1 + P.nw + P.nv;
  const int sI = item / kinds, f = item - sI * kinds;
  const int s = sI / P.nt, I = sI - s * P.nt;
  if (P.vo && (f == 0) == (s == 0)) return;  // kinetic on segment 1 only, the rest on segment 0
  const int lane = threadIdx.x & 31, i = I * TILE + lane;
  const bool vi = i < P.p;
  const int E1 = P.eta + 1;
  const bool pin_lo = (s == 0), pin_hi = (s == P.eta - 1);
  float2 zl = mk(0.f, 0.f), zh = zl;
  float r = 0.f;
  if (vi) {
    if (P.dense) {
      zl = P.z[(size_t)i * E1 + s]; zh = P.z[(size_t)i * E1 + s + 1];
    } else {
      const float4 z4 = P.zseg[(size_t)s * P.p + i];
      zl = lo2(z4); zh = hi2(z4);
    }
    r = P.radius[i];
  }
  float res = 0.f;
  if (f == 0) {
    if (vi && !P.noenergy) kinetic_factor(P, i, s, zl, zh, pin_lo, pin_hi, res);
  } else {
    wall_factor(P, f - 1, i, vi, s, I, zl, zh, r, pin_lo, pin_hi, res);
  }
  if (__any_sync(FULL, res > 0.f)) {
    res = warp_max(res);
    if (lane == 0 && P.res_prev) atomic_max_nonneg(P.res_prev, res);
  }
}

__device__ __forceinline__ int tile_pair(int nt, int I, int J) {  // I <= J
  return I * nt - I * (I - 1) / 2 + (J - I);
}

// Slot of the pair (a, b), either order, on segment s.
__device__ __forceinline__ uint32_t pair_slot(const Dev& P, int s, int a, int b) {
  const int i = min(a, b), j = max(a, b);
  const uint32_t blk = (uint32_t)s * P.ntp + tile_pair(P.nt, i >> 5, j >> 5);
  return (blk * TILE + (i & 31)) * TILE + (j & 31);
}

// Inverse of tile_pair: the tiles (I, J), I <= J, of pair index t, without
// the table lookup (a square root, then an exact integer correction).
__device__ __forceinline__ void tile_of(int nt, int t, int& I, int& J) {
  const float b = 2.f * nt + 1.f;
  int i = (int)((b - sqrtf(fmaxf(b * b - 8.f * t, 0.f))) * 0.5f);
  i = max(0, min(i, nt - 1));
  while (i > 0 && tile_pair(nt, i, i) > t) --i;
  while (i + 1 < nt && tile_pair(nt, i + 1, i + 1) <= t) ++i;
  I = i;
  J = i + (t - tile_pair(nt, i, i));
}

// Dense state: the collision minimizer (Eq. coll_minimizer_problem through
// App. C/D/I) of an active pair, one thread.
__device__ __forceinline__ void prox_item(const Dev& P, uint32_t fid) {
  const int E1 = P.eta + 1;
  const uint32_t row = fid >> 5, c = fid & 31;
  const uint32_t blk = row >> 5, r = row & 31;
  const int s = (int)(blk / P.ntp);
  int I, J;
  tile_of(P.nt, (int)(blk - (uint32_t)s * P.ntp), I, J);
  const int i = I * TILE + r, j = J * TILE + c;
  const float scale = P.fix[0], bound = P.fix[1];  // loaded beside the minimizer
  const float4 a = P.ulo[fid], b = P.uhi[fid];
  const float2 nil = P.z[(size_t)i * E1 + s] - lo2(a), nih = P.z[(size_t)i * E1 + s + 1] - lo2(b);
  const float2 njl = P.z[(size_t)j * E1 + s] - hi2(a), njh = P.z[(size_t)j * E1 + s + 1] - hi2(b);
  float2 xil, xih, xjl, xjh;
  const bool pin_lo = (s == 0), pin_hi = (s == P.eta - 1);
  if (P.noenergy) {
    int cil, cih, cjl, cjh;
    end_classes(P, i, s, pin_lo, pin_hi, cil, cih);
    end_classes(P, j, s, pin_lo, pin_hi, cjl, cjh);
    coll_minimizer_classes(nil, nih, njl, njh, cil, cih, cjl, cjh, P.radius[i] + P.radius[j],
                           P.rho, xil, xih, xjl, xjh);
  } else {
    coll_minimizer(nil, nih, njl, njh, pin_lo, pin_hi, P.radius[i] + P.radius[j], P.rho,
                   xil, xih, xjl, xjh);
  }
  P.xlo[fid] = pack(xil, xjl);
  P.xhi[fid] = pack(xih, xjh);
  if (!pin_lo) {
    contribute(P, scale, bound, i, s, xil + lo2(a));
    contribute(P, scale, bound, j, s, xjl + hi2(a));
  }
  if (!pin_hi) {
    contribute(P, scale, bound, i, s + 1, xih + lo2(b));
    contribute(P, scale, bound, j, s + 1, xjh + hi2(b));
  }
}

// Dense state: one CTA of TILE / TROWS warps per (segment s, agent
// tiles I <= J) block of 32 x 32 collision factors; each warp takes TROWS
// rows (the launch shape the batched autotuner varies), lane = column agent j,
// and the row agents' data is broadcast from shared memory.  Per row, the warp
// streams the u records of its 32 pairs, finishes the pending dual update
// (step 7 of the previous iteration), forms n = z - u (step 1), runs the
// collision test (steps 2-3: weight rho0 or 0), stores the records and the
// row's activity bits and lists its active pairs.  A single plan's block then
// runs their minimizers itself (LOCAL, its own list in shared memory: a kernel
// of its own behind a global worklist cost 5 us of each iteration: 34.7 to 28.7
// us at p = 512, eta = 16, 19.2 to 10.0 at p = 40); a batch
// appends them to the members' worklists, which one launch shares out.
struct TestMem {
  float4 z[TILE], was[TILE];  // break-points of the row agents: z^k and (standard ADMM) z^{k-1}
  float r[TILE];
  uint32_t word[TILE];
  unsigned listed;
  uint16_t list[TILE * TILE];
};
template <int TROWS, int AHEAD, bool LOCAL>
__device__ __forceinline__ void test_block(const Dev& P, int blk, TestMem* M) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int E1 = P.eta + 1;
  float res = 0.f;
  const int s = blk / P.ntp;
  if (P.vo && s != 0) return;  // no collision factors between x and x_ref
  const int2 IJ = P.tiles[blk - s * P.ntp];
  const int I = IJ.x, J = IJ.y;
  const bool diag = (I == J);
  const bool pin_lo = (s == 0), pin_hi = (s == P.eta - 1);
  const int r0 = warp * TROWS;
  const int nrows = min(TROWS, P.p - I * TILE - r0);
  if (LOCAL) {
    if (threadIdx.x == 0) M->listed = 0u;
    __syncthreads();
  }
  if (nrows > 0) {  // warp-uniform
    // column agent of this lane
    const int j = J * TILE + lane;
    const bool vj = j < P.p, every = P.admm || P.keep;
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 zj = none, pj = none;
    float rj = 0.f;
    if (vj) {
      const size_t n = (size_t)j * E1 + s;
      zj = pack(P.z[n], P.z[n + 1]);
      if (P.admm) pj = pack(P.z_next[n], P.z_next[n + 1]);
      rj = P.radius[j];
    }
    if (lane < nrows) {
      const int i = I * TILE + r0 + lane;
      const size_t n = (size_t)i * E1 + s;
      M->z[r0 + lane] = pack(P.z[n], P.z[n + 1]);
      if (P.admm) M->was[r0 + lane] = pack(P.z_next[n], P.z_next[n + 1]);
      M->r[r0 + lane] = P.radius[i];
      M->word[r0 + lane] = P.bits[(size_t)blk * TILE + r0 + lane];
    }
    __syncwarp();
    for (int q0 = 0; q0 < nrows; q0 += AHEAD) {
      float4 ua[AHEAD], ub[AHEAD];
      // the group's records, all loads under way before the first is used
#pragma unroll
      for (int g = 0; g < AHEAD; ++g) {
        const int r = r0 + q0 + g;
        ua[g] = ub[g] = none;
        if (q0 + g < nrows && vj && (!diag || r < lane) && (every || ((M->word[r] >> lane) & 1u))) {
          const size_t fid = ((size_t)blk * TILE + r) * TILE + lane;
          ua[g] = P.ulo[fid];
          ub[g] = P.uhi[fid];
        }
      }
#pragma unroll
      for (int g = 0; g < AHEAD; ++g) {
        if (q0 + g >= nrows) break;  // warp-uniform
        const int r = r0 + q0 + g;
        const bool valid = vj && (!diag || r < lane);
        const size_t row = (size_t)blk * TILE + r, fid = row * TILE + lane;
        const float4 zi = M->z[r];
        const uint32_t word = M->word[r];
        const bool bprev = (word >> lane) & 1u;  // set only for valid pairs
        float2 uil = lo2(ua[g]), ujl = hi2(ua[g]), uih = lo2(ub[g]), ujh = hi2(ub[g]);
        if (bprev) {
          // finish step 7 of the previous iteration for this pair
          const float4 xa = P.xlo[fid], xb = P.xhi[fid];
          uil = finish_u(true, pin_lo, false, uil, lo2(xa), lo2(zi), P.alpha, res);
          ujl = finish_u(true, pin_lo, false, ujl, hi2(xa), lo2(zj), P.alpha, res);
          uih = finish_u(true, pin_hi, false, uih, lo2(xb), hi2(zi), P.alpha, res);
          ujh = finish_u(true, pin_hi, false, ujh, hi2(xb), hi2(zj), P.alpha, res);
        } else if (P.admm && valid) {
          // standard ADMM: the pair was feasible, so x^k = z^{k-1} - u^{k-1}
          const float4 pi = M->was[r];
          uil = finish_u_feasible(pin_lo, uil, lo2(pi), lo2(zi), P.alpha, res);
          ujl = finish_u_feasible(pin_lo, ujl, lo2(pj), lo2(zj), P.alpha, res);
          uih = finish_u_feasible(pin_hi, uih, hi2(pi), hi2(zi), P.alpha, res);
          ujh = finish_u_feasible(pin_hi, ujh, hi2(pj), hi2(zj), P.alpha, res);
        }
        // (reset rule: inactive edges carry u = 0, and were not loaded)
        if (pin_lo) { uil = mk(0.f, 0.f); ujl = uil; }
        if (pin_hi) { uih = mk(0.f, 0.f); ujh = uih; }
        const bool act = valid && collides((lo2(zj) - ujl) - (lo2(zi) - uil), (hi2(zj) - ujh) - (hi2(zi) - uih),
                                           M->r[r] + rj);
        if (valid) {
          P.ulo[fid] = pack(uil, ujl);
          P.uhi[fid] = pack(uih, ujh);
        }
        const uint32_t nword = __ballot_sync(FULL, act);
        if (nword != word && lane == 0) P.bits[row] = nword;
        if (nword) {
          unsigned base = 0;
          if (lane == 0) base = atomicAdd(LOCAL ? &M->listed : P.work_count, (unsigned)__popc(nword));
          base = __shfl_sync(FULL, base, 0) + __popc(nword & ((1u << lane) - 1u));
          if (act && LOCAL) M->list[base] = (uint16_t)(r * TILE + lane);
          if (act && !LOCAL) P.work[base] = (uint32_t)fid;
        }
      }
    }
  }
  res = warp_max(res);
  if (lane == 0 && res > 0.f && P.res_prev) atomic_max_nonneg(P.res_prev, res);
  if (LOCAL) {
    __syncthreads();
    const unsigned n = M->listed;
    for (unsigned t = threadIdx.x; t < n; t += blockDim.x) prox_item(P, (uint32_t)blk * TILE * TILE + M->list[t]);
  }
}

// Bounding-circle filter of the gated state.  Agent i's segment lies in the
// disk of centre m_i (its midpoint) and radius b_i (half its length plus
// r_i), so a pair can only collide when |m_i - m_j| <= b_i + b_j, i.e. when
//     m_i . m_j + b_i b_j >= Q_i / 2 + Q_j / 2,   Q = |m|^2 - b^2.
// With a_i = Q_i / 2 - 2e-6 (|m_i|^2 + b_i^2) the test is
// m_i . m_j + b_i b_j - a_i - a_j >= 0.  The margin, 4e-6 of the magnitudes
// involved, is about ten times the rounding of the expression and of the
// bounding radii, so the filter never drops a pair that the exact test would
// find colliding: the outcome is that of testing every pair exactly.
__device__ __forceinline__ float bounding_offset(float2 m, float b) {
  const float mm = dot(m, m), bb = b * b;
  return fmaf(-2e-6f, mm + bb, 0.5f * (mm - bb));
}

// Floats as integers of the same order, for integer atomics.
__device__ __forceinline__ int ordered(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
// The box of a bounding circle, a little wide (1e-5 of its size and place, a
// hundred times the rounding here and in the exact test): two agents that the
// exact test finds colliding have boxes that meet.  (One with an infinity or a
// NaN never passes that test, whatever its box.)
__device__ __forceinline__ int4 circle_box(float4 c) {
  const float ex = fmaf(1e-5f, fabsf(c.x) + c.z, c.z), ey = fmaf(1e-5f, fabsf(c.y) + c.z, c.z);
  return make_int4(ordered(c.x - ex), ordered(c.y - ey), ordered(c.x + ex), ordered(c.y + ey));
}
__device__ __forceinline__ float4 segment_circle(float2 zl, float2 zh, float r) {
  const float2 m = 0.5f * (zl + zh), d = zh - zl;
  const float b = fmaf(0.5f, sqrtf(dot(d, d)), r);
  return make_float4(m.x, m.y, b, -bounding_offset(m, b));
}

// The records the factor pass starts from (gated state), of agent i on
// segment s: both break-points together, and the bounding circle with the
// offset negated, at the agent's place in the search order.  Written by the
// node pass (and after z changed by other means), so that a tile warp loads
// 16 bytes per agent, coalesced, and derives nothing.
__device__ __forceinline__ void store_segment(const Dev& P, int i, int s, float2 zl, float2 zh) {
  const size_t so = (size_t)s * P.p;
  const float4 c = segment_circle(zl, zh, P.radius[i]);
  P.zseg[so + i] = pack(zl, zh);
  if (!P.sorted) { P.circ[so + i] = c; return; }
  const int at = P.inv[so + i];
  P.circ[so + at] = c;
  int4* box = P.box + (size_t)s * P.nt + (at >> 5);
  const int4 have = *box, need = circle_box(c);
  if (need.x < have.x) atomicMin(&box->x, need.x);
  if (need.y < have.y) atomicMin(&box->y, need.y);
  if (need.z > have.z) atomicMax(&box->z, need.z);
  if (need.w > have.w) atomicMax(&box->w, need.w);
}

// Position of the n-th set bit of w (n counted from 0, less than popc(w)).
__device__ __forceinline__ int nth_bit(uint32_t w, unsigned n) {
  int at = 0;
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) {
    const unsigned low = __popc(w & ((1u << k) - 1u));
    if (n >= low) { n -= low; w >>= k; at += k; }
  }
  return at;
}

// Shared memory of one tile warp: its 32 column agents' circles by component,
// their segments (by component with sorted tiles, where a pair of columns is
// one 8-byte load, else whole) and radii, their numbers, and the activity of
// the pairs of the current phase by row.
struct __align__(16) TileMem {
  float mx[32], my[32], b[32], na[32];
  union {
    float4 z[32];
    struct { float zlx[32], zly[32], zhx[32], zhy[32]; };
  };
  float r[32];
  int id[32];
  uint32_t act[32];
};

// collides() of a row agent (segment z, negated, and radius in both halves)
// with columns 2 k and 2 k + 1: the same operations, two at a time; bits 0 and
// 1 of the result.
struct RowPair { unsigned long long nlx, nly, nhx, nhy, r; };
__device__ __forceinline__ uint32_t collides2(const RowPair& A, const TileMem* M, int k) {
  auto at = [&](const float* v) { return reinterpret_cast<const unsigned long long*>(v)[k]; };
  const unsigned long long minus = pair_of(-1.f, -1.f);
  const unsigned long long lx = add2(at(M->zlx), A.nlx), ly = add2(at(M->zly), A.nly);
  const unsigned long long hx = add2(at(M->zhx), A.nhx), hy = add2(at(M->zhy), A.nhy);
  const unsigned long long R = add2(A.r, at(M->r)), R2 = mul2(R, R);
  const unsigned long long dx = fma2(lx, minus, hx), dy = fma2(ly, minus, hy);  // hx - lx, one rounding
  const unsigned long long dd = fma2(dx, dx, mul2(dy, dy)), ld = fma2(lx, dx, mul2(ly, dy));
  const unsigned long long c = fma2(lx, dy, mul2(mul2(ly, dx), minus));
  const unsigned long long ll = fma2(lx, lx, mul2(ly, ly)), hh = fma2(hx, hx, mul2(hy, hy));
  const unsigned long long cc = mul2(c, c), Rd = mul2(R2, dd);
  auto one = [](float ll, float hh, float ld, float dd, float cc, float R2, float Rd) {
    const float t = -ld;
    return (ll < R2) | (hh < R2) | ((t > 0.f) & (t < dd) & (cc < Rd));
  };
  return (one(lo_of(ll), lo_of(hh), lo_of(ld), lo_of(dd), lo_of(cc), lo_of(R2), lo_of(Rd)) ? 1u : 0u) |
         (one(hi_of(ll), hi_of(hh), hi_of(ld), hi_of(dd), hi_of(cc), hi_of(R2), hi_of(Rd)) ? 2u : 0u);
}

// A pair of one warp item: (i, j) on segment s with slot fid; prev: active in
// the last iteration.  Finishes its dual update, tests it and, when it is
// active, runs the minimizer, stores its record and adds its messages to the
// sums (steps 7, 1-4).  CLASSES: per-node back weights (the feasibility
// problem).
template <bool CLASSES, class D>
__device__ __forceinline__ bool pair_factor(const D& P, int s, int i, int j, uint32_t fid,
                                            bool prev, float& res) {
  const bool pin_lo = (s == 0), pin_hi = (s == P.eta - 1);
  const float4 zi = P.zseg[(size_t)s * P.p + i], zj = P.zseg[(size_t)s * P.p + j];
  const float R = P.radius[i] + P.radius[j];
  const float scale = P.fix[0], bound = P.fix[1];
  float2 uil = mk(0.f, 0.f), ujl = uil, uih = uil, ujh = uil;
  if (prev) {
    const float4 a = P.ulo[fid], b = P.uhi[fid], xa = P.xlo[fid], xb = P.xhi[fid];
    uil = finish_u(true, pin_lo, false, lo2(a), lo2(xa), lo2(zi), P.alpha, res);
    ujl = finish_u(true, pin_lo, false, hi2(a), hi2(xa), lo2(zj), P.alpha, res);
    uih = finish_u(true, pin_hi, false, lo2(b), lo2(xb), hi2(zi), P.alpha, res);
    ujh = finish_u(true, pin_hi, false, hi2(b), hi2(xb), hi2(zj), P.alpha, res);
  }
  const float2 nil = lo2(zi) - uil, nih = hi2(zi) - uih, njl = lo2(zj) - ujl, njh = hi2(zj) - ujh;
  if (!collides(njl - nil, njh - nih, R)) return false;
  float2 xil, xih, xjl, xjh;
  if (CLASSES) {
    int cil, cih, cjl, cjh;
    end_classes(P, i, s, pin_lo, pin_hi, cil, cih);
    end_classes(P, j, s, pin_lo, pin_hi, cjl, cjh);
    coll_minimizer_classes(nil, nih, njl, njh, cil, cih, cjl, cjh, R, P.rho, xil, xih, xjl, xjh);
  } else {
    coll_minimizer(nil, nih, njl, njh, pin_lo, pin_hi, R, P.rho, xil, xih, xjl, xjh);
  }
  P.ulo[fid] = pack(uil, ujl);
  P.uhi[fid] = pack(uih, ujh);
  P.xlo[fid] = pack(xil, xjl);
  P.xhi[fid] = pack(xih, xjh);
  if (!pin_lo) {
    contribute(P, scale, bound, i, s, xil + uil);
    contribute(P, scale, bound, j, s, xjl + ujl);
  }
  if (!pin_hi) {
    contribute(P, scale, bound, i, s + 1, xih + uih);
    contribute(P, scale, bound, j, s + 1, xjh + ujh);
  }
  return true;
}

// Activity flag of a worklist entry.  Problems of more than 2^31 slots keep no
// list (capacity 0: every iteration takes the rebuilding form).
constexpr uint32_t ACTIVE = 0x80000000u;

// Tile warps of a problem: one per 32 x 32 block on the last segment (early in
// a solve it spans each agent's whole way, nearly all its pairs take the exact
// test, and it goes first), `strip` blocks elsewhere (most of which the boxes
// rule out when the tiles are sorted), taken at equal distances so that the
// neighbouring groups, whose boxes meet, go to different warps (strips of 16
// consecutive blocks left one warp with all of them: 81 us at p = 4,095).
__host__ __device__ __forceinline__ int tile_warps(int nseg, int ntp, int strip) {
  return ntp + (nseg - 1) * ((ntp + strip - 1) / strip);
}

// Collision factors of the gated state, one warp.  item < nlist: list warp
// `item` of nlist takes the chunks of 32 worklist entries item, item + nlist,
// ...; else tile warp item - nlist takes one 32 x 32 block of pairs or a strip
// of them.
//
// Tile warp: lane = row agent.  The bounding circles of the 32 columns come
// from shared memory four columns at a time and are tested two columns per
// instruction; the sign of the result is shifted into the row's word, so a
// pair costs about four instructions (the scalar form with a compare and a
// select took seven).  Near pairs take the exact test, and those that collide
// and are not on the worklist are dealt over the whole warp, one pair per lane
// per round (row found by a shuffle binary search over the rows' prefix
// counts), to run the minimizer.  Both kinds of warp share one copy of that
// code (one loop, one call site): it is most of the kernel's instructions.
//
// mode FUSED is the above.  After a reset or an import nearly every active
// pair is new to the tile warps, which then run many rounds one after another
// where a layout is crowded (41 us for the p = 100 circle), so that iteration
// is two launches: LISTING (tile warps put every pair that was active or
// collides on the worklist) and LISTED (list warps only).
enum FactorMode { FUSED = 0, LISTING = 1, LISTED = 2 };

// Columns of a 32 x 32 block whose bounding circles (in M) come near the
// lane's row circle ci, as a word.
__device__ __forceinline__ uint32_t near_columns(const float4 ci, const TileMem* M) {
  const unsigned long long mx = pair_of(ci.x, ci.x), my = pair_of(ci.y, ci.y), b = pair_of(ci.z, ci.z),
                           na = pair_of(ci.w, ci.w);
  uint32_t far = 0u;
#pragma unroll
  for (int c = TILE - 4; c >= 0; c -= 4) {
    const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(M->mx + c);
    const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(M->my + c);
    const ulonglong2 B = *reinterpret_cast<const ulonglong2*>(M->b + c);
    const ulonglong2 A = *reinterpret_cast<const ulonglong2*>(M->na + c);
    const unsigned long long t1 = fma2(mx, X.y, fma2(my, Y.y, fma2(b, B.y, add2(na, A.y))));
    const unsigned long long t0 = fma2(mx, X.x, fma2(my, Y.x, fma2(b, B.x, add2(na, A.x))));
    // sign bits, highest column first
    far = __funnelshift_l((uint32_t)(t1 >> 32), far, 1);
    far = __funnelshift_l((uint32_t)t1, far, 1);
    far = __funnelshift_l((uint32_t)(t0 >> 32), far, 1);
    far = __funnelshift_l((uint32_t)t0, far, 1);
  }
  return ~far;
}

// Inclusive prefix sums over the warp.
__device__ __forceinline__ unsigned warp_inclusive(unsigned v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned w = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += w;
  }
  return v;
}

// Room for every lane's n worklist entries (one atomic): the lane's first.
__device__ __forceinline__ unsigned claim_entries(const Dev& P, unsigned n) {
  const unsigned incl = warp_inclusive(n);
  unsigned at = 0;
  if ((threadIdx.x & 31) == 31) {
    at = atomicAdd(P.work_count, incl);
    if ((unsigned long long)at + incl > P.cap) atomicOr(P.ctl + 2, 1u);
  }
  return __shfl_sync(FULL, at, 31) + (incl - n);
}

// A lane's worklist entry `entry` (position t): slot, segment, agents i < j.
__device__ __forceinline__ void entry_pair(const Dev& P, uint32_t entry, uint32_t& fid, int& s, int& i, int& j) {
  fid = entry & ~ACTIVE;
  const uint32_t row = fid >> 5, blk = row >> 5;
  s = (int)(blk / (uint32_t)P.ntp);
  int I, J;
  tile_of(P.nt, (int)(blk - (uint32_t)s * P.ntp), I, J);
  i = I * TILE + (int)(row & 31);
  j = J * TILE + (int)(fid & 31);
}

// A list warp's lane after its pair: the entry and the activity bit, where
// that changed.  Returns by how much the list's inactive entries grew.
__device__ __forceinline__ int entry_done(const Dev& P, unsigned long long t, uint32_t fid, bool prev, bool act) {
  if (act == prev) return 0;
  P.work[t] = fid | (act ? ACTIVE : 0u);
  const uint32_t bit = 1u << (fid & 31);
  if (act) atomicOr(P.bits + (fid >> 5), bit); else atomicAnd(P.bits + (fid >> 5), ~bit);
  return act ? -1 : 1;
}

// Pair g of a warp's pairs, dealt from the rows' words todo with inclusive
// prefix counts tincl and `total` in all: its row (the first whose count
// exceeds g) and column (0 past the end).
__device__ __forceinline__ void nth_pair(uint32_t todo, unsigned tincl, unsigned total, unsigned g, int& r, int& c) {
  r = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1)
    if (__shfl_sync(FULL, tincl, r + step - 1) <= g) r += step;
  const uint32_t w = __shfl_sync(FULL, todo, r);
  const unsigned first = __shfl_sync(FULL, tincl, r) - __popc(w);
  c = g < total ? nth_bit(w, g - first) : 0;
}

template <bool CLASSES, class D>
__device__ __forceinline__ void collision_warp(const D& P, int item, int nlist, TileMem* M, int mode) {
  const int lane = threadIdx.x & 31;
  const bool rebuild = mode == LISTED ? false : P.ctl[0] != 0u;
  const bool lister = item < nlist;
  float res = 0.f;
  // list warp
  unsigned n = 0, chunk = (unsigned)item;
  int gone = 0;  // entries turned inactive less entries turned active
  // tile warp
  int s = 0, I = 0, J = 0, blk = 0, phase = 0;
  size_t row = 0;
  uint32_t listed = 0u, todo = 0u, near = 0u;
  unsigned tincl = 0, total = 0, base = 0;
  if (lister) {
    if (rebuild || mode == LISTING) return;
    n = mode == LISTED ? *P.work_count : *P.work_count_prev;
  } else {
    const int nseg = P.vo ? 1 : P.eta;
    const int t = item - nlist;
    s = nseg - 1 - t / P.ntp;  // the last segment spans the longest way early in a solve: first
    const int tp = t - (nseg - 1 - s) * P.ntp;
    tile_of(P.nt, tp, I, J);
    blk = s * P.ntp + tp;
    const int i = I * TILE + lane, j = J * TILE + lane;
    const bool vi = i < P.p, vj = j < P.p;
    const size_t so = (size_t)s * P.p;
    const float4 none = make_float4(0.f, 0.f, 0.f, -INFINITY);
    const float4 ci = vi ? P.circ[so + i] : none, cj = vj ? P.circ[so + j] : none;
    row = (size_t)blk * TILE + lane;
    listed = (rebuild ? P.bits : P.listed)[row];
    M->mx[lane] = cj.x; M->my[lane] = cj.y; M->b[lane] = cj.z; M->na[lane] = cj.w;
    uint32_t valid = __ballot_sync(FULL, vj);  // (also orders the stores before the loads below)
    __syncwarp();
    if (!vi) valid = 0u;
    if (I == J) valid &= (lane == 31) ? 0u : (~0u << (lane + 1));  // pairs i < j
    near = near_columns(ci, M) & valid & ~listed;
    M->act[lane] = 0u;
    todo = rebuild ? listed : 0u;
    phase = mode == LISTING ? 2 : rebuild ? 0 : 1;
    if (__any_sync(FULL, near != 0u)) {
      float4 zi = make_float4(0.f, 0.f, 0.f, 0.f), zj = zi;
      float ri = 0.f, rj = 0.f;
      if (vi) { zi = P.zseg[so + i]; ri = P.radius[i]; }
      if (vj) { zj = P.zseg[so + j]; rj = P.radius[j]; }
      M->z[lane] = zj;
      M->r[lane] = rj;
      __syncwarp();
      // two columns a round: their chains overlap (on the segment that spans
      // the whole way nearly every pair is near)
      uint32_t hit = 0u;
      for (uint32_t w = near; w; ) {
        const int c = __ffs(w) - 1;
        w &= w - 1u;
        const int k = w ? __ffs(w) - 1 : c;
        w &= w - 1u;
        const float4 B = M->z[c], C = M->z[k];
        const bool h0 = collides(lo2(B) - lo2(zi), hi2(B) - hi2(zi), ri + M->r[c]);
        const bool h1 = collides(lo2(C) - lo2(zi), hi2(C) - hi2(zi), ri + M->r[k]);
        hit |= (h0 ? 1u << c : 0u) | (h1 ? 1u << k : 0u);
      }
      near = hit;
    }
    if (!rebuild && !__any_sync(FULL, near != 0u)) return;  // most tiles: nothing to run, nothing to note
    __syncwarp();
  }
  for (;;) {
    // the next 32 pairs
    int pi = 0, pj = 0, ps = 0, r = 0, c = 0;
    uint32_t fid = 0u;
    bool on = false, prev = false;
    const unsigned long long t = 32ull * chunk + lane;
    if (lister) {
      if (32ull * chunk >= n) break;  // warp-uniform
      on = t < n;
      if (on) {
        const uint32_t entry = P.work[t];
        prev = (entry & ACTIVE) != 0u;
        entry_pair(P, entry, fid, ps, pi, pj);
      }
    } else {
      if (base >= total) {  // start a phase: 0 the pairs active before (rebuild), 1 the new ones
        if (phase > 1) break;
        if (phase == 1) todo = near;
        ++phase;
        tincl = warp_inclusive(__popc(todo));
        total = __shfl_sync(FULL, tincl, 31);
        base = 0;
        if (total == 0) continue;
      }
      prev = phase == 1;  // (the phase was advanced as it started)
      const unsigned g = base + lane;
      base += 32;
      on = g < total;
      nth_pair(todo, tincl, total, g, r, c);
      ps = s;
      pi = I * TILE + r;
      pj = J * TILE + c;
      fid = (uint32_t)(((size_t)blk * TILE + r) * TILE + c);
    }
    bool act = false;
    if (on) act = pair_factor<CLASSES>(P, ps, pi, pj, fid, prev, res);
    if (lister) {
      if (on) gone += entry_done(P, t, fid, prev, act);
      chunk += (unsigned)nlist;
    } else if (act) {
      atomicOr(&M->act[r], 1u << c);
    }
  }
  if (lister) {
    if (__any_sync(FULL, gone != 0)) {
      gone = __reduce_add_sync(FULL, gone);
      if (lane == 0 && gone != 0) atomicAdd(P.ctl + 1, (unsigned)gone);
    }
  } else {
    __syncwarp();
    uint32_t nword = M->act[lane];
    const uint32_t flagged = mode == LISTING ? (rebuild ? listed : 0u) : ~0u;  // entries active so far
    if (mode == LISTING) {
      // (a reset leaves nothing active and `listed` clear; an import, rebuild)
      nword = near | flagged;
      P.listed[row] = nword;
      const int fresh = __reduce_add_sync(FULL, __popc(near));
      if (lane == 0 && fresh) atomicAdd(P.ctl + 1, (unsigned)fresh);
    } else if (rebuild) {
      if (nword != listed) P.bits[row] = nword;
      P.listed[row] = nword;
    } else if (nword) {
      atomicOr(P.bits + row, nword);
      P.listed[row] = listed | nword;
    }
    if (__any_sync(FULL, nword != 0u)) {
      unsigned at = claim_entries(P, __popc(nword));
      for (uint32_t w = nword; w; w &= w - 1u, ++at)
        if (at < P.cap) {
          const int bit = __ffs(w) - 1;
          P.work[at] = (uint32_t)(row * TILE + bit) | ((flagged >> bit) & 1u ? ACTIVE : 0u);
        }
    }
  }
  if (__any_sync(FULL, res > 0.f)) {  // only pairs active before have a residual
    res = warp_max(res);
    if (lane == 0 && P.res_prev) atomic_max_nonneg(P.res_prev, res);
  }
}

// Sorted tiles: pairs of tile t of segment s that collide with u = 0 and are
// not on the worklist, by row (lane) a word of columns.  sorted: the tile's
// agents come in the search order, else in their own (a rebuild).  rid: the
// lane's row agent.
__device__ __forceinline__ uint32_t tile_candidates(const Dev& P, int s, int t, int I, int J, bool sorted, TileMem* M,
                                                    int& rid) {
  const int lane = threadIdx.x & 31;
  const int ri = I * TILE + lane, cj = J * TILE + lane;
  const bool vi = ri < P.p, vj = cj < P.p;
  const size_t so = (size_t)s * P.p;
  const float4 none = make_float4(0.f, 0.f, 0.f, -INFINITY);
  rid = ri;
  int cid = cj, rat = ri, cat = cj;  // row and column agent, and the places of their circles
  if (sorted) {
    if (vi) rid = P.perm[so + ri];
    if (vj) cid = P.perm[so + cj];
  } else {
    if (vi) rat = P.inv[so + ri];
    if (vj) cat = P.inv[so + cj];
  }
  const float4 ci = vi ? P.circ[so + rat] : none, cc = vj ? P.circ[so + cat] : none;
  // with the agents' own order the block's listed pairs are known
  const uint32_t known = sorted ? 0u : P.listed[((size_t)s * P.ntp + t) * TILE + lane];
  __syncwarp();
  M->mx[lane] = cc.x; M->my[lane] = cc.y; M->b[lane] = cc.z; M->na[lane] = cc.w;
  M->id[lane] = cid;
  uint32_t valid = __ballot_sync(FULL, vj);
  __syncwarp();
  if (!vi) valid = 0u;
  if (I == J) valid &= (lane == 31) ? 0u : (~0u << (lane + 1));  // each pair once
  const uint32_t near = near_columns(ci, M) & valid & ~known;
  if (!__any_sync(FULL, near != 0u)) return 0u;
  float4 zi = make_float4(0.f, 0.f, 0.f, 0.f), zj = zi;
  float r = 0.f, rj = 0.f;
  if (vi) { zi = P.zseg[so + rid]; r = P.radius[rid]; }
  if (vj) { zj = P.zseg[so + cid]; rj = P.radius[cid]; }
  M->r[lane] = rj;
  M->zlx[lane] = zj.x; M->zly[lane] = zj.y; M->zhx[lane] = zj.z; M->zhy[lane] = zj.w;
  __syncwarp();
  uint32_t hit = 0u;
  if (__reduce_max_sync(FULL, __popc(near)) >= 12) {
    // near a third of the columns or more (the segment that spans the whole
    // way): every column, two an instruction (8.5 to 7.5 us a tile there)
    const RowPair A = {pair_of(-zi.x, -zi.x), pair_of(-zi.y, -zi.y), pair_of(-zi.z, -zi.z), pair_of(-zi.w, -zi.w),
                       pair_of(r, r)};
#pragma unroll 2
    for (int k = 0; k < TILE / 2; ++k) hit |= collides2(A, M, k) << (2 * k);
    hit &= near;
  } else {
    for (uint32_t w = near; w; w &= w - 1u) {
      const int c = __ffs(w) - 1;
      if (collides(mk(M->zlx[c], M->zly[c]) - lo2(zi), mk(M->zhx[c], M->zhy[c]) - hi2(zi), r + M->r[c]))
        hit |= 1u << c;
    }
  }
  if (sorted) {  // (those on the worklist are the list warps')
#pragma unroll 4
    for (uint32_t w = hit; w; w &= w - 1u) {
      const int c = __ffs(w) - 1;
      const uint32_t f = pair_slot(P, s, rid, M->id[c]);
      if ((P.listed[f >> 5] >> (f & 31)) & 1u) hit &= ~(1u << c);
    }
  }
  return hit;
}

// The same work with sorted tiles.  A tile warp goes through a strip of
// blocks, each in up to two phases (its listed pairs when the list is built
// anew, then the new ones); a separate function, because the state that takes
// costs the small plans 16% of a solve (261 us to 309 at p = 100).
template <bool CLASSES>
__device__ __forceinline__ void sorted_collision_warp(const Dev& P, int item, int nlist, int strip, TileMem* M, int mode) {
  const int lane = threadIdx.x & 31;
  const bool rebuild = mode == LISTED ? false : P.ctl[0] != 0u;
  const bool lister = item < nlist;
  const bool sorted = !rebuild;
  float res = 0.f;
  int idle = 0;  // inactive entries put on the list or left on it, less entries turned active
  // list warp
  unsigned n = 0, chunk = (unsigned)item;
  // tile warp: its blocks t0, t0 + step, ... (cnt of them) of segment s, the
  // current one q, those with near pairs; the current phase's pairs by row
  // (todo; was: those active before)
  int s = 0, t0 = 0, step = 0, cnt = 0, q = -1, I = 0, J = 0, rid = 0;
  uint32_t live = 0u, todo = 0u, was = 0u;
  unsigned tincl = 0, total = 0, base = 0;
  bool scan = false, next = true, open = false;
  if (lister) {
    if (rebuild || mode == LISTING) return;
    n = mode == LISTED ? *P.work_count : *P.work_count_prev;
  } else {
    const int nseg = P.vo ? 1 : P.eta, w = item - nlist;
    if (w < P.ntp) {
      s = nseg - 1; t0 = w; cnt = 1;
    } else {
      step = (P.ntp + strip - 1) / strip;
      const int v = w - P.ntp;
      s = nseg - 2 - v / step;
      t0 = v - (nseg - 2 - s) * step;
      cnt = (P.ntp - t0 + step - 1) / step;
    }
    bool meet = lane < cnt;
    if (sorted && meet) {
      int a, b;
      tile_of(P.nt, t0 + lane * step, a, b);
      const int4 A = P.box[(size_t)s * P.nt + a], B = P.box[(size_t)s * P.nt + b];
      meet = A.x <= B.z && B.x <= A.z && A.y <= B.w && B.y <= A.w;
    }
    live = __ballot_sync(FULL, meet);
    if (live == 0u) return;
  }
  for (;;) {
    // the next 32 pairs
    int pi = 0, pj = 0, ps = s, r = 0, c = 0;
    uint32_t fid = 0u;
    bool on = false, prev = false;
    const unsigned long long t = 32ull * chunk + lane;
    if (lister) {
      if (32ull * chunk >= n) break;  // warp-uniform
      on = t < n;
      if (on) {
        const uint32_t entry = P.work[t];
        prev = (entry & ACTIVE) != 0u;
        entry_pair(P, entry, fid, ps, pi, pj);
      }
    } else {
      uint32_t row = ((uint32_t)s * P.ntp + t0 + q * step) * TILE + lane;
      if (base >= total) {
        if (open) {  // end of a phase: activity, membership and entries of its pairs
          open = false;
          __syncwarp();
          const uint32_t acts = mode == LISTING ? (was & todo) : M->act[lane];
          const uint32_t keep = mode == LISTING ? todo : acts | (was & todo);
          if (scan) {  // (a rebuild: no list warp writes these words)
            if (acts != was) P.bits[row] = acts;
            P.listed[row] = keep;
          } else if (!sorted) {
            if (acts) atomicOr(P.bits + row, acts);
            if (keep) P.listed[row] |= keep;
          } else {
            for (uint32_t w = keep; w; w &= w - 1u) {
              const int k = __ffs(w) - 1;
              const uint32_t f = pair_slot(P, s, rid, M->id[k]);
              if ((acts >> k) & 1u) atomicOr(P.bits + (f >> 5), 1u << (f & 31));
              atomicOr(P.listed + (f >> 5), 1u << (f & 31));
            }
          }
          idle += __popc(keep & ~acts);
          if (__any_sync(FULL, keep != 0u)) {
            unsigned at = claim_entries(P, __popc(keep));
            for (uint32_t w = keep; w; w &= w - 1u, ++at) {
              const int k = __ffs(w) - 1;
              const uint32_t f = !scan && sorted ? pair_slot(P, s, rid, M->id[k]) : row * TILE + k;
              if (at < P.cap) P.work[at] = f | (((acts >> k) & 1u) ? ACTIVE : 0u);
            }
          }
        }
        // the next phase: a block's listed pairs (rebuild), then its tile's new ones
        base = total = 0;
        scan = next;
        if (next) {
          if (++q >= cnt) break;
          next = false;
          if (!rebuild) continue;
          row = ((uint32_t)s * P.ntp + t0 + q * step) * TILE + lane;
          todo = P.listed[row];
          was = P.bits[row];
          tile_of(P.nt, t0 + q * step, I, J);
        } else {
          next = true;
          was = 0u;
          if (!((live >> q) & 1u)) continue;
          tile_of(P.nt, t0 + q * step, I, J);
          todo = tile_candidates(P, s, t0 + q * step, I, J, sorted, M, rid);
        }
        if (!__any_sync(FULL, todo != 0u)) continue;
        open = true;
        if (mode == LISTING) continue;
        M->act[lane] = 0u;
        __syncwarp();
        tincl = warp_inclusive(__popc(todo));
        total = __shfl_sync(FULL, tincl, 31);
      }
      const unsigned g = base + lane;
      base += 32;
      on = g < total;
      nth_pair(todo, tincl, total, g, r, c);
      const uint32_t pw = __shfl_sync(FULL, was, r);
      prev = on && ((pw >> c) & 1u);
      pi = I * TILE + r;
      pj = J * TILE + c;
      fid = (row - lane + r) * TILE + c;
      const int ra = __shfl_sync(FULL, rid, r);
      if (sorted && on) {
        const int ca = M->id[c];
        pi = min(ra, ca);
        pj = max(ra, ca);
        fid = pair_slot(P, s, pi, pj);
      }
    }
    bool act = false;
    if (on) act = pair_factor<CLASSES>(P, ps, pi, pj, fid, prev, res);
    if (lister) {
      if (on) idle += entry_done(P, t, fid, prev, act);
      chunk += (unsigned)nlist;
    } else if (act) {
      atomicOr(&M->act[r], 1u << c);
    }
  }
  if (__any_sync(FULL, idle != 0)) {
    idle = __reduce_add_sync(FULL, idle);
    if (lane == 0 && idle != 0) atomicAdd(P.ctl + 1, (unsigned)idle);
  }
  if (__any_sync(FULL, res > 0.f)) {  // only pairs active before have a residual
    res = warp_max(res);
    if (lane == 0 && P.res_prev) atomic_max_nonneg(P.res_prev, res);
  }
}

// Steps 5-6 for one free break-point: z = sum(rho m) / sum(rho) from the
// fixed-point sums (every weight is rho0, so z is the mean of the incoming m;
// no incoming weight means z is unchanged).  Clears the sums for the next
// iteration.
template <class D>
__device__ __forceinline__ float2 consensus_node(const D& P, size_t node, float2 zo, unsigned status,
                                                 float& dz, bool& bad) {
  long long sx, sy;
  unsigned cnt;
  take_sums(P, node, sx, sy, cnt);
  note_count(P, node, cnt);
  float2 zn = zo;  // every incoming weight zero: treated as 1, which gives z unchanged
  if (P.admm) {
    // every edge is weighted; each feasible collision or wall factor sent
    // m = n + u = z^k, added here in the same exact fixed point
    const unsigned deg = 2u * (unsigned)(P.p - 1) + 2u + 2u * (unsigned)P.nw;
    const long long rest = (long long)(deg - cnt);
    const long long qx = __float2ll_rn(zo.x * P.fix[0]), qy = __float2ll_rn(zo.y * P.fix[0]);
    const float den = P.fix[0] * (float)deg;  // exact: a power of two times a small count
    zn = mk(__ll2float_rn(sx + rest * qx) / den, __ll2float_rn(sy + rest * qy) / den);
  } else if (cnt > 0u) {
    // the exact integer sum rounded once to FP32, then one FP32 division
    const float den = P.fix[0] * (float)cnt;
    zn = mk(__ll2float_rn(sx) / den, __ll2float_rn(sy) / den);
  }
  // step 6: the back weight is rho0 where some factor sent rho0, else 0
  if (P.noenergy) P.wnode[node] = cnt > 0u ? 1 : 0;
  P.z_next[node] = zn;
  const float2 d = zn - zo;
  const bool odd = (status & 2u) != 0u || !(fabsf(d.x) + fabsf(d.y) >= 0.f);
  bad |= odd;
  if (!odd) dz = fmaxf(dz, maxabs2(d));
  return zn;
}

// Warp-level end of the consensus pass: a NaN or overflow anywhere makes the
// residual NaN (reported as PLAN_ENUMERIC).  All 32 lanes must call it.
__device__ __forceinline__ void consensus_reduce(const Dev& P, float dz, bool bad) {
  dz = warp_max(dz);
  const bool anybad = __any_sync(FULL, bad);
  if ((threadIdx.x & 31) == 0) {
    if (anybad) atomicMax(P.res_cur, 0x7fc00000u);
    else if (dz > 0.f) atomic_max_nonneg(P.res_cur, dz);
  }
}

// Agents a node warp takes: as many whole agents as fit its 32 lanes.
__host__ __device__ __forceinline__ int agents_per_warp(int eta) { return eta + 1 <= 32 ? 32 / (eta + 1) : 1; }

// Node pass of one warp: every break-point of its agents, lane = break-point
// (consecutive in the [p][eta+1] arrays, so coalesced), longer agents in
// rounds of 32 from the far end.  A lane gets the next break-point's z from
// its neighbour and writes the segment records of the next factor pass.
template <class D>
__device__ __forceinline__ void consensus_warp(const D& P, int warp) {
  const int lane = threadIdx.x & 31, E1 = P.eta + 1, apw = agents_per_warp(P.eta);
  const unsigned status = *P.status;
  float dz = 0.f;
  bool bad = false;
  if (E1 <= 32) {
    const int a = lane / E1, s = lane - a * E1, i = warp * apw + a;
    const bool on = a < apw && i < P.p;
    float2 z = mk(0.f, 0.f);
    if (on) {
      const size_t node = (size_t)i * E1 + s;
      z = P.z[node];
      if (s > 0 && s < P.eta) z = consensus_node(P, node, z, status, dz, bad);
    }
    const float2 zh = mk(__shfl_down_sync(FULL, z.x, 1), __shfl_down_sync(FULL, z.y, 1));
    if (on && s < P.eta && !P.dense) store_segment(P, i, s, z, zh);
  } else if (warp < P.p) {
    float2 next = mk(0.f, 0.f);  // z of the round's far neighbour
    for (int s0 = (P.eta / 32) * 32; s0 >= 0; s0 -= 32) {
      const int s = s0 + lane;
      const size_t node = (size_t)warp * E1 + s;
      float2 z = mk(0.f, 0.f);
      if (s <= P.eta) {
        z = P.z[node];
        if (s > 0 && s < P.eta) z = consensus_node(P, node, z, status, dz, bad);
      }
      float2 zh = mk(__shfl_down_sync(FULL, z.x, 1), __shfl_down_sync(FULL, z.y, 1));
      if (lane == 31) zh = next;
      if (s < P.eta && !P.dense) store_segment(P, warp, s, z, zh);
      next = mk(__shfl_sync(FULL, z.x, 0), __shfl_sync(FULL, z.y, 0));
    }
  }
  consensus_reduce(P, dz, bad);
}

// Node warps of a problem.
__host__ __device__ __forceinline__ int node_warps(int p, int eta) {
  const int apw = agents_per_warp(eta);
  return (p + apw - 1) / apw;
}

// The worklist's length and mode for the next iteration, by one thread of
// the node pass.  frozen: the problem took no factor pass.
__device__ __forceinline__ void advance_worklist(const Dev& P, bool frozen) {
  unsigned n = *P.work_count;
  if (P.dense) n = 0u;  // the dense state's list is that of one iteration
  else if (!frozen) {
    // half of the list inactive (and more than a few warps' worth), or longer
    // than it fits, or slots that a list entry cannot hold
    const bool again = P.ctl[2] != 0u || 2u * P.ctl[1] > n + 1024u || P.cap == 0u;
    P.ctl[0] = again ? 1u : 0u;
    if (again) { n = 0u; P.ctl[1] = 0u; P.ctl[2] = 0u; }
  }
  *P.work_count_prev = n;  // the next iteration appends to the other parity's counter
}

}  // namespace
