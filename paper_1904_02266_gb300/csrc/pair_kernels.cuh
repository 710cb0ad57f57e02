// The CVO hot path on sm_103a: the cutoff-truncated all-pairs kernel
// reductions behind each gradient-ascent iteration, plus the FP64 tail, all in
// one persistent cooperative kernel per solve.
//
//  gradient pass  F = sum c_ij k(x_i, z~_j)                         (Eq. scalar)
//                 dF/domega = (1/ell^2) sum w_ij (z~_j x e_ij)      (Eq. 3_gradient,
//                 dF/dv     = (1/ell^2) sum w_ij e_ij                left-update signs)
//  step pass      S0..S4 = sum w_ij g^m_ij along xi                  (Eq. fourth)
//  tail (FP64)    xi = metric gradient (Eq. metric), t* = first maximiser of the
//                 quartic, P <- exp(t* xi) P (Eqs. newstep, step), lengthscale
//                 schedule and the Table 1 convergence test.
//
// One iteration (every block runs the same sequence; phases are separated by
// a grid barrier whose spin is bounded):
//  plan        (only when needed) one warp per source cluster (an octree node
//              of the source, at most 32 points): transform, bounding box, the
//              rows of target cells within the plan radius, stored as segments
//              of the cell-sorted target, and (clusters with at most
//              kFilterMax candidates) the count of candidates within the plan
//              radius of the box, per segment; the work of groups of 32
//              clusters is added up on the way (a queued solve's first plan and
//              a rebalance total it after a barrier).                   barrier
//              every block scans the group totals and places its own warps on
//              an even split of the work into pieces from all over the cloud,
//              cut at groups of four source points (no further barrier).
//  gradient    each warp walks its share of chunks of 32 filtered candidates:
//  pass        one lane per candidate target point against the cluster's
//              source points staged in shared memory (broadcast reads), the
//              distance tests of a chunk before its pair bodies. FP32 pairs,
//              two to a packed operation, one ex2.approx per kept pair,
//              per-lane FP32 sums, fixed-order reductions.             barrier
//  tail        every block adds all block partials (value-major) as aligned
//              64-bit integers and forms the same unit direction, so nothing
//              is published or broadcast.
//  step pass   as above along the unit direction.                      barrier
//  tail        step length, exponential-map update, next iteration: in FP64
//              at once, or, for small plain steps, the passes' pose in FP32
//              and the FP64 step behind the next gradient pass.
// The plan is reused while it still covers the cutoff: it is built with a
// radius 10% wider than the cutoff and rebuilt when the grid level changes,
// when the pose has drifted by more than that margin (a bound over the
// whole source cloud), or when it has become much wider than needed. A warp
// whose share of a reused plan fits its cache also lists, once per
// plan, the (candidate, source point) pairs of each cached cluster within the
// plan radius, and its passes evaluate the lists instead of whole chunks.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "cvo_internal.cuh"
#include "packed_f32.cuh"
#include "split_rule.h"

// Resident blocks per SM the solve kernel is compiled for (register budget).
#ifndef CVO_SOLVE_MIN_BLOCKS
#define CVO_SOLVE_MIN_BLOCKS 1
#endif

namespace cvo {

namespace {

constexpr float kFar = 1.0e18f;   // coordinate of padding points: never within any cutoff
constexpr unsigned kFull = 0xffffffffu;
constexpr double kSkin = 0.10;              // plan radius margin (fraction of the cutoff)
constexpr double kLoose = 1.25;             // replan when the plan radius exceeds this factor
constexpr int kFilterMax = 1024;            // candidates of a cluster the plan filters at most
constexpr int kActChunks = 32;              // chunks per cluster whose source-group activity is kept
// Teams of at most kSmallTeam blocks hold long shares. The streamed passes box-test
// the candidates of unfiltered clusters on the way in such teams, and wherever a
// warp's share is at least kCompactWork pair-test units; shorter shares of larger
// teams, whose split counts unfiltered candidates, come out more uneven than the
// test saves. Whole-GPU teams with every share tested, from 3000 units, and none:
// 20k room solve 5.55, 5.51, 5.51 ms, 100k evaluation 827, 820, 844 us, 16 served
// requests 95.6, 96.2, 98.1 ms
constexpr int kSmallTeam = 32;
constexpr int kCompactWork = 3000;
// Where the box test would drop hardly a candidate it only costs: the plan looks at 32
// candidates of each cluster with at least kDenseFrom of them, and where all pass the
// cluster goes without. Evaluations of 20k points in a blob of 0.4 m, cutoff 0.37 m: no
// test 1275 us, every cluster tested 1310, this rule 1261; 100k room points at
// lengthscale 0.05 600 and 594, planes at 0.35 17.6 and 17.5 ms. (Leaving targets of few cells
// untested: the blob 1263, planes at 0.2 to 0.35 4 to 7% slower.) Smaller clusters repay
// no look ahead.
constexpr int kDenseFrom = 4096;
// a warp's share of the work is cut into pieces taken from different parts of the
// cloud (split_work): one per kRangeWork pair-test units of it, at most
// kMaxRanges, from kRangeFrom units on. Whole-GPU teams, 100k room pair: up to 4
// pieces of 1500 units 46.9 ms, 8 of 1500 46.2, 8 of 700 45.4; at 20k points
// (about 1000 units a warp) a second piece costs a cluster and two ends more than
// it evens out. Small teams: two pieces from kSmallTeamFrom units on (64-pair batch:
// one piece 105.0 ms, two 104.0, up to eight 111.9). These lines, kCompactWork and
// kSpareWork count units of the caller's cost model (cost_chunk 48 and cost_cluster 32
// by default) and so move with it; with cost_chunk 16, 32, 96 and 256 and with
// cost_cluster 0, 128 and 1024 room solves of 2k to 100k points took 0.52 to 0.96 of
// their time before the lines were drawn
constexpr int kMaxRanges = 8;
constexpr int kRangeWork = 700;
constexpr int kRangeFrom = 2000;
constexpr int kSmallTeamFrom = 20000;
// shares below this many units leave the block's last warp out of the passes
// (split_work). Whole room solves without, from 400 and from 1500 units: 10k points
// 3.80, 3.68, 3.68 ms, 20k 5.65, 5.51, 5.57 ms, 28k 7.45, 7.44, 7.47 ms; the 2k planes
// pair, whose passes are the shortest, 825, 832, 832 us
constexpr int kSpareWork = 400;

// One feature value: FP32 planes, or BF16 planes widened to FP32 (FB).
template <bool FB>
__device__ __forceinline__ float load_feat(const float* planes, size_t idx) {
  if constexpr (FB) {
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(planes)[idx]);
  } else {
    return planes[idx];
  }
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int cell_floor(float v, float o, float inv_h, int n) {
  float q = floorf((v - o) * inv_h);
  q = fminf(fmaxf(q, -1.0f), (float)n);
  return (int)q;
}

// ---------------------------------------------------------------------------
// per-block iteration state (identical in every block of a team)
// ---------------------------------------------------------------------------

// The blocks that solve one pair together: the whole grid for a single
// solve, a contiguous run of claimed slots for a queued one.
struct Team {
  int rank, size;
};

// Scalars of the solve configuration that the FP64 tail reads every
// iteration, copied once per solve so that the tail issues no dependent
// global loads.
struct TailConst {
  double cX[3], cZ[3];
  double sigma2, inv_a2, inv_b2;
  double eps_pose, eps_grad, src_radius;
  int mode, step_order, max_iters;
  int reduce_fp32;   // precision study: block and cross-block sums in FP32
  unsigned wait_polls;                 // barrier polls before a block gives up
  unsigned long long join_limit_ns;    // longest wait of a queued team's join
  // FP32 copies for the FP32 parts of the tail
  float cXf[3], inv_a2f, inv_b2f, src_radius_f, eps_pose_f;
};

struct BlockCtx {
  TailConst tc;
  double P[16];           // current pose
  double xi[6];           // metric gradient (Eq. metric)
  double x0[6];           // its components before the metric factors (FP64 pair sums, centring
                          // back-map applied)
  double u64[6];          // xi / |xi|
  double xi_norm, xi_inv, F;
  double S[5];            // S0..S4 of the last step pass (formed when published)
  double s_raw[5];        // the step pass's sums along xi / |xi| (S_m = s_m sigma^2 |xi|^m)
  int small_grad;         // |xi| below the gradient threshold (or zero): no step, stop test
  double t, t_prev;
  IterConst ic;           // this iteration's constants
  double r_plan, plan_ell;
  int k, plan_level, plan_filter;
  int need_plan, done, converged, fallback, no_ascent, have_t_prev;
  int use_kept, collect_kept, rebalance;   // kept-pair weighting of the work split
  int use_act;                             // the split weighs active source groups by this (0: not)
  int cost_act;                            // what a rebalance of this plan will weigh them by
  int plan_no;                             // reused plans so far
  int check_fit;                           // a rebalance by more than kCostActive: see check_fits
  int cap;                                 // floats of a warp's cache
  SolveState* st;
  int compact;                             // streamed passes box-test unfiltered clusters
  int team_rank, team_size;                // this block's place in its team (read after a pass
                                           // from shared memory rather than kept in registers)
  unsigned long long nnz_total, cand_total, nnz_grad, cand_grad;
  float R[9], T[3];       // FP32 centred pose of the passes: z~' = R z' + T'
  float Rq[9], Tq[3];     // the same at the last plan
  // the centred FP64 pose in two FP32 parts (rounded, and what the rounding
  // left), for the FP32 step (quick_step)
  float Rb[9], Tb[3], Rl[9], Tl[3];
  int pending;            // P waits for the step of length pend_tau (refined in FP64) along u64
  float pend_tau;
  float om[3], vc[3];     // unit step direction (centred frame)
  float kw[3];            // (omega . v) omega / 6 l^2
  float c_del, c_eps, k_eps;   // -|omega|^2 / 3, -|omega|^2 / 12, -(omega . v)^2 / 48 l^2
  float rplan_f;
  // warp ranges (n_range of them per warp): from group g0 of chunk j0 of cluster
  // c0 up to (not including) group g1 of chunk j1 of cluster c1
  int n_range;
  int n_workers;          // warps that share the passes; with kWarps - 1 of them the last warp does
                          // the FP64 work of the iteration meanwhile
  int w_c0[kMaxRanges][kWarps], w_j0[kMaxRanges][kWarps], w_g0[kMaxRanges][kWarps];
  int w_c1[kMaxRanges][kWarps], w_j1[kMaxRanges][kWarps], w_g1[kMaxRanges][kWarps];
  // where the streamed rest of a partly cached share begins (c < 0: there is none)
  int rest_c[kWarps], rest_j[kWarps], rest_g[kWarps];
  int ring_floats;        // front of a warp's cache region that the streamed passes use
  double dR[9], V[9];     // tail scratch: exp map rotation and its V matrix
};

// ---- the FP64 tail, one warp wide -----------------------------------------
// On GB300 a warp's FP64 instruction holds the FP64 pipe about as long as a
// full warp's (about 64 cycles) whatever the number of active lanes, so the
// tail costs what its count of FP64 instructions costs. It runs on warp 0 of
// every block with independent components on separate lanes (the 3 x 4 pose
// product is three instructions, not thirty-six); scalar steps run on every
// lane at the cost of one. Lanes exchange values by shuffles, or through the
// block context (shared memory) between __syncwarp()s.

__device__ __forceinline__ double flip_sign(double v, bool neg) {
  return __longlong_as_double(__double_as_longlong(v) ^
                              (neg ? (long long)0x8000000000000000ull : 0ll));
}

// Conversions and power-of-two scalings by integer operations on the bit
// patterns. On GB300 every FP64 warp instruction (conversions and compares
// included) holds the FP64 pipe for about 64 cycles, so the tails keep their
// FP64 instruction count low and leave the rest to the integer and FP32 pipes.

// x 2^shift truncated to FP32 (toward zero); magnitudes below FP32's normal
// range give a signed zero, above it a signed infinity, a NaN stays a NaN.
__device__ __forceinline__ float f64_to_f32_shift(double x, int shift) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned sign = (unsigned)hi & 0x80000000u;
  const unsigned m = ((unsigned)(hi & 0xfffff) << 3) | (lo >> 29);
  if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (m != 0u || lo != 0u ? 0x400000u : 0u));
  const int e32 = e - 1023 + 127 + shift;
  if (e == 0 || e32 <= 0) return __uint_as_float(sign);
  if (e32 >= 255) return __uint_as_float(sign | 0x7f800000u);
  return __uint_as_float(sign | ((unsigned)e32 << 23) | m);
}

__device__ __forceinline__ float f64_to_f32(double x) { return f64_to_f32_shift(x, 0); }

// The exact FP64 value of an FP32 number (FP32 subnormals as zero).
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xffu;
  const unsigned sign = u & 0x80000000u;
  if (e == 0u) return __hiloint2double((int)sign, 0);
  const unsigned e64 = e == 0xffu ? 0x7ffu : e - 127u + 1023u;
  return __hiloint2double((int)(sign | (e64 << 20) | ((u & 0x7fffffu) >> 3)), (int)((u & 7u) << 29));
}

// x 2^k for k in [0, 8]: an exponent increment when x is normal and stays so.
__device__ __forceinline__ double mul_pow2(double x, int k) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  if (e > 0 && e + k < 0x7ff) return __hiloint2double(hi + (k << 20), __double2loint(x));
  return x * (double)(1 << k);
}

// x > 0 (false for zero, negative values and NaN), from the bit pattern.
__device__ __forceinline__ bool is_pos(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  if (hi < 0) return false;
  if (((hi >> 20) & 0x7ff) == 0x7ff && ((hi & 0xfffff) != 0 || lo != 0u)) return false;
  return hi != 0 || lo != 0u;
}

// The centred pose [R T'] of the FP64 pose in two FP32 parts, rounded to nearest,
// on lanes 0..11, element (r, c) = (l / 4, l % 4): R = the pose's rotation, T' = R cZ
// + T - cX. One warp.
__device__ __forceinline__ void split_pose(BlockCtx& b, int lane, float* hi_out) {
  const int l = min(lane, 11), r = l >> 2, c = l & 3;
  const double t3 = fma(b.P[4 * r + 2], b.tc.cZ[2],
                        fma(b.P[4 * r + 1], b.tc.cZ[1],
                            fma(b.P[4 * r], b.tc.cZ[0], b.P[4 * r + 3] - b.tc.cX[r])));
  const double v = c == 3 ? t3 : b.P[4 * r + c];
  const float hi = __double2float_rn(v);
  const float lo = f64_to_f32(v - f32_to_f64(hi));
  if (lane < 12) {
    if (c < 3) {
      b.Rb[3 * r + c] = hi;
      b.Rl[3 * r + c] = lo;
    } else {
      b.Tb[r] = hi;
      b.Tl[r] = lo;
    }
  }
  *hi_out = hi;
}

// Iteration k's constants, a word per lane: read ahead of their use, stored into
// the block's context when the iteration starts (one warp).
static_assert(sizeof(IterConst) == 64, "sixteen words");
__device__ __forceinline__ unsigned iter_word(const SolveCfg* cfg, int k, int lane) {
  return reinterpret_cast<const unsigned*>(cfg->iters + k)[lane & 15];
}
__device__ __forceinline__ void load_iter(BlockCtx& b, unsigned word, int lane) {
  if (lane < 16) reinterpret_cast<unsigned*>(&b.ic)[lane] = word;
  __syncwarp();
}

// The start of an iteration whose constants are in b.ic: the FP32 pose (from the
// FP64 pose, unless quick_step has formed it), and whether the traversal plan must
// be rebuilt. Warp 0, every lane.
__device__ __noinline__ void begin_iteration(BlockCtx& b, int lane) {
  const IterConst& ic = b.ic;
  const int l = min(lane, 11), r = l >> 2, c = l & 3;
  float v;
  if (b.pending) v = c == 3 ? b.T[r] : b.R[3 * r + c];
  else split_pose(b, lane, &v);
  // is the current plan still a superset of the pairs within the cutoff?
  const float need = ic.rprune;   // 1.001 r_c
  // reuse only at an unchanged lengthscale (the floor of the schedule): while
  // ell shrinks a fresh, tighter plan costs less than the extra candidates
  bool replan = b.need_plan || ic.level != b.plan_level ||
                __double_as_longlong(ic.ell) != __double_as_longlong(b.plan_ell);
  if (!replan) {
    // between the FP32 poses that the plan and the passes use; the 2e-5 relative
    // and 1e-6 r_c margins below cover the rounding
    const float d = v - (c == 3 ? b.Tq[r] : b.Rq[3 * r + c]);
    const float sq = lane < 12 ? d * d : 0.0f;
    float sr = c < 3 ? sq : 0.0f, st = c == 3 ? sq : 0.0f;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      sr += __shfl_xor_sync(kFull, sr, off);
      st += __shfl_xor_sync(kFull, st, off);
    }
    sr = __shfl_sync(kFull, sr, 0);
    st = __shfl_sync(kFull, st, 0);
    // |dR z + dT| <= |dR|_F |z| + |dT| for every source point, |z| <= r_src
    const float drift = fmaf(sqrtf(sr), b.tc.src_radius_f, sqrtf(st)) * (1.0f + 2e-5f) + 1e-6f * need;
    const float rp = b.rplan_f;
    replan = (need + drift > rp) || (rp > (float)kLoose * (need + drift));
  }
  __syncwarp();   // every lane has read the old poses
  if (lane < 12) {
    if (c < 3) b.R[3 * r + c] = v;
    else b.T[r] = v;
    if (replan) {
      if (c < 3) b.Rq[3 * r + c] = v;
      else b.Tq[r] = v;
    }
  }
  if (lane == 0) {
    if (replan) {
      b.need_plan = 1;
      b.plan_level = ic.level;
      b.plan_ell = ic.ell;
      b.plan_filter = ic.filter;
      // the radius is FP32 throughout: (float)(need (1 + skin)) is what the
      // plan and the passes use. A plan used for one iteration sees only
      // that iteration's pose (the pose moves at its end and the next
      // iteration re-plans at a new lengthscale), so it needs no skin
      b.r_plan = (double)need * (ic.filter ? 1.0 + kSkin : 1.0);
      b.rplan_f = (float)b.r_plan;
    }
  }
  __syncwarp();
}

// FP64 reciprocal from the FP32 one and a Newton step r <- r (2 - x r) (which
// squares the relative error: 1e-7 -> 1e-14). Finite, nonzero x within FP32
// range.
__device__ __forceinline__ double recip_refined(double x) {
  double r = (double)(1.0f / (float)x);
  r = r * fma(-x, r, 2.0);
  return r;
}

// FP64 reciprocal and square root of any finite x != 0 (x > 0): the
// refined FP32 forms inside FP32's range, the FP64 operations outside it.
__device__ __forceinline__ double rcp64(double x) {
  const double ax = fabs(x);
  return (ax > 1e-30 && ax < 1e30) ? recip_refined(x) : 1.0 / x;
}

__device__ __forceinline__ double sqrt64(double x) {
  if (!(x > 1e-30 && x < 1e30)) return sqrt(x);
  // y ~ 1/sqrt(x) from FP32, two FP64 Newton steps y <- y (1.5 - 0.5 x y^2)
  double y = (double)rsqrtf((float)x);
  y = y * fma(-0.5 * x, y * y, 1.5);
  y = y * fma(-0.5 * x, y * y, 1.5);
  return x * y;
}

// Smallest positive t at which G'(t) = c0 + c1 t + c2 t^2 + c3 t^3 changes sign
// from + to - (the first local maximum of the quartic model, Sec. 4 "Step
// size"), given c0 = S1 > 0. The coefficients are first scaled by a power of
// two (exact) so that the largest has magnitude in [0.5, 1). The critical
// points of G' (the real roots of G'' = c1 + 2 c2 t + 3 c3 t^2) cut t > 0 into
// pieces on which G' is monotone; the first piece whose right end has G' < 0
// (for the last piece, the sign of the leading coefficient) holds the answer,
// which a Newton iteration kept inside the shrinking bracket finds in FP64.
// Its start is the root of the closed-form cubic evaluated in FP32 (cbrt /
// acos / cos, no FP64 transcendentals), or the bracket's midpoint: a close
// start takes two steps; a far one (the FP32 form loses the small roots of a
// cubic whose roots differ by orders of magnitude) a few more.
//
// The start: a root of the cubic from the closed form, all in FP32 (f0..f3: the
// coefficients scaled so that the largest has magnitude in [0.5, 1); truncated:
// a start needs no more), refined by two FP32 Newton steps; a negligible cubic
// term is left out of the start only. Not positive if there is none.
__device__ __forceinline__ float cubic_start(float f0, float f1, float f2, float f3) {
  float ts = -1.0f;
  if (fabsf(f3) <= 1e-12f) {
    if (fabsf(f2) <= 1e-12f) {
      if (f1 < 0.0f) ts = -f0 / f1;
    } else {
      const float disc = fmaf(f1, f1, -4.0f * f2 * f0);
      if (disc >= 0.0f) {
        const float qf = -0.5f * (f1 + copysignf(sqrtf(disc), f1));
        const float ra = qf / f2, rb = f0 / qf;
        ts = (f2 < 0.0f) ? fmaxf(ra, rb) : fminf(ra, rb);
      }
    }
  } else {
    const float r3 = 1.0f / f3;
    const float B = f2 * r3, C = f1 * r3, D = f0 * r3;
    const float B3 = B * (1.0f / 3.0f);
    const float p = fmaf(-B, B3, C);
    const float q = fmaf((2.0f / 27.0f) * B * B, B, fmaf(-B3, C, D));
    const float disc = fmaf(0.25f * q, q, (1.0f / 27.0f) * p * p * p);
    if (disc > 0.0f) {
      const float u = -copysignf(cbrtf(0.5f * fabsf(q) + sqrtf(disc)), q);
      ts = (u != 0.0f ? u - p / (3.0f * u) : 0.0f) - B3;
    } else if (p < 0.0f) {
      // roots m cos(phi - 2 pi k / 3) - B/3: k = 0 largest, k = 1 middle, k = 2 smallest
      const float m = 2.0f * sqrtf(-p * (1.0f / 3.0f));
      const float arg = fminf(1.0f, fmaxf(-1.0f, 3.0f * q / (p * m)));
      const float phi = acosf(arg) * (1.0f / 3.0f);
      const float two_pi_3 = 2.09439510239319549f;
      // the hardware cosine is accurate enough for a start
      const float rk[3] = {m * __cosf(phi) - B3, m * __cosf(phi - two_pi_3) - B3,
                           m * __cosf(phi - 2.0f * two_pi_3) - B3};
      // the smallest positive one that G' crosses from + to - (as far as FP32 tells)
      for (int k = 0; k < 3; ++k) {
        const float tk = rk[k];
        if (tk > 0.0f && fmaf(fmaf(3.0f * f3, tk, 2.0f * f2), tk, f1) < 0.0f && (ts < 0.0f || tk < ts))
          ts = tk;
      }
    }
  }
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const float ff = fmaf(fmaf(fmaf(f3, ts, f2), ts, f1), ts, f0);
    const float fd = fmaf(fmaf(3.0f * f3, ts, 2.0f * f2), ts, f1);
    const float tn = ts - ff / fd;
    if (fd < 0.0f && tn > 0.0f && isfinite(tn)) ts = tn;
  }
  return ts;
}

// G' falls over all of [0, t]: G''(t) < 0 and the vertex test of a concave G'' in
// FP32 with a 1e-4 relative margin (their rounding is below 1e-6); G''(0) = c1 < 0
// is the caller's. Then t, if a root, is the first one and a + -> - crossing.
__device__ __forceinline__ bool falls_to(float f1, float f2, float f3, float ts, float* g2_out) {
  const float g2 = fmaf(fmaf(3.0f * f3, ts, 2.0f * f2), ts, f1);
  const float gmag = fabsf(f1) + fabsf(2.0f * f2 * ts) + fabsf(3.0f * f3 * ts * ts);
  const bool inside = f3 < 0.0f && f2 > 0.0f && f2 < -3.0f * f3 * ts * (1.0f + 1e-4f);
  const bool vertex_ok = !inside || 3.0f * f1 * f3 > f2 * f2 * (1.0f + 1e-4f);
  *g2_out = g2;
  return g2 < -1e-4f * gmag && vertex_ok;
}

__device__ bool first_maximiser(double c0, double c1, double c2, double c3, double* t_out) {
  // the largest exponent field among the coefficients (integer work: FP64
  // instructions are the scarce resource here)
  const int e_max = max(max((__double2hiint(c0) >> 20) & 0x7ff, (__double2hiint(c1) >> 20) & 0x7ff),
                        max((__double2hiint(c2) >> 20) & 0x7ff, (__double2hiint(c3) >> 20) & 0x7ff));
  if (e_max == 0x7ff) return false;   // an infinity or a NaN
  const int shift = 1022 - e_max;
  const float f0 = f64_to_f32_shift(c0, shift), f1 = f64_to_f32_shift(c1, shift);
  const float f2 = f64_to_f32_shift(c2, shift), f3 = f64_to_f32_shift(c3, shift);
  const float ts = cubic_start(f0, f1, f2, f3);
  const double t32 = f32_to_f64(ts);
  // fast path: one FP64 Newton step from that start on the unscaled
  // coefficients (the roots do not depend on a common scale), accepted when it
  // moves t by at most 2^-20 t (the step squares the start's error) and G' falls
  // from c0 > 0 over [0, t]; anything within the margins goes to the bracketed
  // search
  if (e_max >= 2 && ts > 0.0f && isfinite(ts) && __double2hiint(c1) < 0) {
    const double f = fma(fma(fma(c3, t32, c2), t32, c1), t32, c0);
    const double fp = fma(fma(3.0 * c3, t32, mul_pow2(c2, 1)), t32, c1);
    const int hfp = __double2hiint(fp), efp = (hfp >> 20) & 0x7ff;
    if (hfp < 0 && efp > 1023 - 120 && efp < 1023 + 120) {
      // 1/fp from FP32 and one FP64 Newton step
      double r = f32_to_f64(1.0f / f64_to_f32(fp));
      r = r * fma(-fp, r, 2.0);
      const double dt = -f * r;
      const double t = t32 + dt;
      const int ht = __double2hiint(t), hd = __double2hiint(dt);
      const int et = (ht >> 20) & 0x7ff, ed = (hd >> 20) & 0x7ff;
      const bool settled = ed <= et - 21;   // |dt| < 2^-20 t (dt = 0 has ed = 0)
      float g2;
      if (ht > 0 && et < 0x7ff && settled && falls_to(f1, f2, f3, ts, &g2)) {
        *t_out = t;
        return true;
      }
    }
  }
  // the bracketed search, on the coefficients scaled by a power of two
  double sc;
  if (e_max >= 2 && e_max <= 2044) {
    // 2^(1022 - e_max): the largest magnitude lands in [0.5, 1)
    sc = __hiloint2double((2045 - e_max) << 20, 0);
  } else {
    const double s = fmax(fmax(fabs(c0), fabs(c1)), fmax(fabs(c2), fabs(c3)));
    if (!(s > 0.0)) return false;
    // 2^-e with s = m 2^e, m in [0.5, 1) (subnormal s are scaled twice)
    sc = 1.0;
    double ss = s;
    if (ss < 0x1p-1000) {
      sc = 0x1p+1000;
      ss *= sc;
    }
    const int ex = min(1000, ((__double2hiint(ss) >> 20) & 0x7ff) - 1022);
    sc *= __hiloint2double((1023 - ex) << 20, 0);
  }
  c0 *= sc;
  c1 *= sc;
  c2 *= sc;
  c3 *= sc;
  if (fabs(c3) < 1e-30) c3 = 0.0;
  if (fabs(c2) < 1e-30) c2 = 0.0;
  // positive critical points of G', ascending
  double e0 = -1.0, e1 = -1.0;
  if (c3 != 0.0) {
    const double dd = fma(c2, c2, -3.0 * c1 * c3);   // discriminant of G'' over 4
    if (dd > 0.0) {
      const double qq = -(c2 + copysign(sqrt64(dd), c2));   // G'' roots: qq / (3 c3), c1 / qq
      double ra = qq * rcp64(3.0 * c3);
      double rb = qq != 0.0 ? c1 * rcp64(qq) : ra;
      if (ra > rb) {
        const double tmp = ra;
        ra = rb;
        rb = tmp;
      }
      if (ra > 0.0) {
        e0 = ra;
        if (rb > ra) e1 = rb;
      } else if (rb > 0.0) {
        e0 = rb;
      }
    }
  } else if (c2 != 0.0) {
    const double r = -c1 * rcp64(2.0 * c2);
    if (r > 0.0) e0 = r;
  }
  // the first monotone piece (lo, hi) on which G' falls below zero
  const double lead = c3 != 0.0 ? c3 : c2 != 0.0 ? c2 : c1;
  double lo = 0.0, hi = -1.0;   // hi < 0: unbounded
  bool found = false;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (found) break;
    const double b = k == 0 ? e0 : k == 1 ? e1 : -1.0;
    if (k < 2 && !(b > lo)) continue;   // no such critical point
    const double fb = b > 0.0 ? fma(fma(fma(c3, b, c2), b, c1), b, c0) : lead;
    if (fb < 0.0) {
      hi = b;
      found = true;
    } else if (b > 0.0) {
      lo = b;   // G' >= 0 at the end of this piece: no crossing in it
    } else {
      break;    // the last piece stays positive: no maximiser
    }
  }
  if (!found) return false;
  // Newton on G' inside [lo, hi] (G' > 0 at lo, < 0 at hi), bisection or
  // doubling when a step leaves the bracket; bounded. Start: the closed-form
  // root if it lies in the bracket, else the smallest point where a falling
  // term balances c0, (c0 / |c_k|)^(1/k), else the bracket's middle.
  const auto inside = [&](double x) { return isfinite(x) && x > lo && (hi < 0.0 || x < hi); };
  double t = t32;
  if (!inside(t)) {
    double tb = -1.0;
    if (c1 < 0.0) tb = c0 / -c1;
    if (c2 < 0.0) {
      const double r = (double)sqrtf((float)(c0 / -c2));
      if (r > 0.0 && (tb < 0.0 || r < tb)) tb = r;
    }
    if (c3 < 0.0) {
      const double r = (double)cbrtf((float)(c0 / -c3));
      if (r > 0.0 && (tb < 0.0 || r < tb)) tb = r;
    }
    t = inside(tb) ? tb : hi > 0.0 ? 0.5 * (lo + hi) : (lo > 0.0 ? 2.0 * lo : 1.0);
  }
  for (int it = 0; it < 64; ++it) {
    const double f = fma(fma(fma(c3, t, c2), t, c1), t, c0);
    if (f > 0.0) lo = t;
    else if (f < 0.0) hi = t;
    else break;
    const double fp = fma(fma(3.0 * c3, t, 2.0 * c2), t, c1);
    double tn = (fp < 0.0 && isfinite(fp)) ? fma(-f, rcp64(fp), t) : -1.0;
    if (tn > 0.0 && isfinite(tn) && fabs(tn - t) <= 1e-13 * tn) {
      t = tn;   // converged (the step is below the resolution of t)
      break;
    }
    if (!inside(tn)) {
      if (hi < 0.0) tn = 2.0 * fmax(t, lo);
      else if (lo > 0.0 && hi > 4.0 * lo) tn = sqrt64(lo * hi);
      else if (lo == 0.0) tn = 0.25 * hi;
      else tn = 0.5 * (lo + hi);
    }
    t = tn;
  }
  if (t > 0.0 && isfinite(t)) {
    *t_out = t;   // scaling all coefficients by one factor leaves the roots alone
    return true;
  }
  return false;
}

// Exp-map series (Eq. step): sin(th)/th, (1 - cos th)/th^2 and (th - sin th)/th^3
// as polynomials in x = th^2 (truncation error < 1e-16 for x < 0.25), one per
// lane 0..2.
__constant__ double kExpSeries[3][7] = {
    {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880, -1.0 / 39916800, 1.0 / 6227020800.0},
    {0.5, -1.0 / 24, 1.0 / 720, -1.0 / 40320, 1.0 / 3628800, -1.0 / 479001600,
     1.0 / 87178291200.0},
    {1.0 / 6, -1.0 / 120, 1.0 / 5040, -1.0 / 362880, 1.0 / 39916800, -1.0 / 6227020800.0,
     1.0 / 1307674368000.0}};

// Gradient tail, first part (warp 0, between the gradient barrier and the
// step pass): the unit step direction in the centred frame, in FP32, which is
// all the step pass needs. Lane a < 6 holds component a of the gradient before
// the metric factors, x0 = omega' + cX x v (rotation) or v (translation), in
// FP64 (the centring back-map may cancel); the common factor sigma^2 / ell^2
// drops out of the direction, so only 1/a^2 and 1/b^2 are applied. The FP64
// gradient itself (gradient_fp64) is formed while the block waits at the step
// pass's barrier.
__device__ void gradient_direction(BlockCtx& b, const double* sums, int lane) {
  const TailConst& tc = b.tc;
  const int a = lane % 3, a1 = a == 2 ? 0 : a + 1, a2 = a == 0 ? 2 : a - 1;
  const bool rot = lane < 3;
  const double cr = fma(tc.cX[a1], sums[4 + a2], -(tc.cX[a2] * sums[4 + a1]));
  const double x0 = sums[1 + min(lane, 5)] + (rot ? cr : 0.0);
  if (lane < 6) b.x0[lane] = x0;
  const float x = lane < 6 ? __double2float_rn(x0) * (rot ? tc.inv_a2f : tc.inv_b2f) : 0.0f;
  float nrm2 = x * x;
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) nrm2 += __shfl_xor_sync(kFull, nrm2, off);
  nrm2 = __shfl_sync(kFull, nrm2, 0);
  // 1/|x|: rsqrt and one Newton step (relative error about 1e-7)
  float inv = 0.0f;
  if (nrm2 > 0.0f && nrm2 < INFINITY) {
    inv = rsqrtf(nrm2);
    inv = inv * fmaf(-0.5f * nrm2, inv * inv, 1.5f);
  }
  // omega_a = x_a / |x|, v'_a = (v_a + (omega x cX)_a) / |x|
  const float xa1 = __shfl_sync(kFull, x, a1), xa2 = __shfl_sync(kFull, x, a2);
  const float xv = __shfl_sync(kFull, x, 3 + a);
  const float vc = (xv + fmaf(xa1, tc.cXf[a2], -(xa2 * tc.cXf[a1]))) * inv;
  if (lane < 3) {
    b.om[a] = x * inv;
    b.vc[a] = vc;
  }
  // the step pass's constants (chunk_bodies, list_pair): |omega|^2 and omega . v'
  const float om = x * inv;
  float ww = om * om, wv = om * vc;
  ww += __shfl_sync(kFull, ww, 1) + __shfl_sync(kFull, ww, 2);   // lane 0's is used
  wv += __shfl_sync(kFull, wv, 1) + __shfl_sync(kFull, wv, 2);
  const float kap = __shfl_sync(kFull, wv, 0) * b.ic.inv_l2f * (1.0f / 6.0f);
  if (lane < 3) b.kw[a] = kap * om;
  if (lane == 0) {
    b.c_del = -ww * (1.0f / 3.0f);
    b.c_eps = -ww * (1.0f / 12.0f);
    b.k_eps = -wv * wv * b.ic.inv_l2f * (1.0f / 48.0f);
  }
  __syncwarp();
}

// In the first iteration of a rebalance that weighed active groups by more than
// kCostActive, behind its gradient pass (every block has filled its cache before that
// pass's barrier, so all read the same): if a warp of the team could not cache its share,
// the next iteration rebalances again, by kCostActive. One warp of 2280 that streams its
// rest in every pass of a plan holds up the team by 10% of the solve (active_weight has
// the figures). One lane.
__device__ __forceinline__ void check_fits(BlockCtx& b) {
  b.check_fit = 0;
  if (__ldcg(&b.st->spilled) != b.plan_no) return;
  b.cost_act = kCostActive;
  b.rebalance = 1;
}

// Gradient tail, second part (one warp, while the block waits at the step pass's
// barrier): the metric gradient xi (Eq. metric), |xi|,
// xi / |xi| in FP64, F and the gradient pass's counts.
__device__ void gradient_fp64(BlockCtx& b, const double* sums, int lane) {
  const TailConst& tc = b.tc;
  const double x = lane < 6 ? b.x0[lane] * (lane < 3 ? b.ic.kf_rot : b.ic.kf_tr) : 0.0;
  double nrm2 = x * x;
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) nrm2 += __shfl_xor_sync(kFull, nrm2, off);
  nrm2 = __shfl_sync(kFull, nrm2, 0);
  // |xi| and 1/|xi|: FP32 rsqrt refined by an FP64 Newton step
  // y <- y (1.5 - 0.5 x y^2) (relative error 1e-7 -> 1e-14)
  double inv = 0.0, nrm = 0.0;
  const int e2 = (__double2hiint(nrm2) >> 20) & 0x7ff;
  if (__double2hiint(nrm2) >= 0 && e2 > 1023 - 100 && e2 < 1023 + 100) {
    inv = f32_to_f64(rsqrtf(f64_to_f32(nrm2)));
    inv = inv * fma(-0.5 * nrm2, inv * inv, 1.5);
    nrm = nrm2 * inv;
  } else if (nrm2 > 0.0) {
    nrm = sqrt(nrm2);
    inv = 1.0 / nrm;
  }
  if (lane < 6) {
    b.xi[lane] = x;
    b.u64[lane] = x * inv;
  }
  if (lane == 0) {
    b.xi_norm = nrm;
    b.xi_inv = inv;
    b.small_grad = (!(nrm > 0.0) || nrm < tc.eps_grad) ? 1 : 0;
    b.F = tc.sigma2 * sums[0];
    b.nnz_grad = (unsigned long long)__double_as_longlong(sums[7]);
    b.cand_grad = (unsigned long long)__double_as_longlong(sums[8]);
    if (b.check_fit) check_fits(b);
  }
  __syncwarp();
}

// S0..S4 of the last step pass (Eq. fourth along xi): the pass summed along
// xi / |xi|, so S_m = s_m sigma^2 |xi|^m. Formed for the published results
// only. Any thread.
__device__ __forceinline__ void form_step_sums(BlockCtx& b) {
  double pw = b.tc.sigma2;
  for (int m = 0; m < 5; ++m) {
    b.S[m] = b.s_raw[m] * pw;
    pw *= b.xi_norm;
  }
}

// P <- exp(tau xi / |xi|) P in FP64 (Eqs. newstep, step), one warp.
__device__ void apply_step(BlockCtx& b, double tau, int lane) {
  // twist tau xi / |xi|: rotation phi (lanes 0..2), translation rho (lanes 3..5)
  const double tw = tau * b.u64[min(lane, 5)];
  const double p0 = __shfl_sync(kFull, tw, 0), p1 = __shfl_sync(kFull, tw, 1);
  const double p2 = __shfl_sync(kFull, tw, 2);
  const double r0 = __shfl_sync(kFull, tw, 3), r1 = __shfl_sync(kFull, tw, 4);
  const double r2 = __shfl_sync(kFull, tw, 5);
  const double x = fma(p0, p0, fma(p1, p1, p2 * p2));
  // A = sin(th)/th, B = (1 - cos th)/th^2, C = (th - sin th)/th^3 on lanes 0, 1, 2.
  // The series alternate with falling terms, so the first term left out
  // bounds the error: 1 term below x = 1e-16, 2 below 1e-8, 3 below 1e-5, 4
  // below 1e-3 (errors below 1e-17 relative), all 7 below 0.25.
  double coef;
  if (x < 0.25) {
    const double* k = kExpSeries[min(lane, 2)];
    const int n = x < 1e-16 ? 0 : x < 1e-8 ? 1 : x < 1e-5 ? 2 : x < 1e-3 ? 3 : 6;
    coef = k[n];
    for (int i = n - 1; i >= 0; --i) coef = fma(coef, x, k[i]);
  } else {
    const double th = sqrt(x);
    const double sn = sin(th), hs = sin(0.5 * th);
    coef = lane == 0 ? sn / th : lane == 1 ? 2.0 * hs * hs / x : (th - sn) / (x * th);
  }
  const double A = __shfl_sync(kFull, coef, 0), B = __shfl_sync(kFull, coef, 1);
  const double C = __shfl_sync(kFull, coef, 2);
  // M = I + c1 W + c2 W^2 (W = hat(phi), W^2 = phi phi^T - |phi|^2 I): lanes 0..8
  // give dR = I + A W + B W^2, lanes 9..17 V = I + B W + C W^2 (Eq. step)
  const int q = lane % 9, i = q / 3, j = q % 3;
  const double pi = i == 0 ? p0 : i == 1 ? p1 : p2;
  const double pj = j == 0 ? p0 : j == 1 ? p1 : p2;
  const int kk = 3 - i - j;   // the third index when i != j
  const double pk = kk == 0 ? p0 : kk == 1 ? p1 : p2;
  const double w = i == j ? 0.0 : flip_sign(pk, (j - i + 3) % 3 == 1);
  const double w2 = fma(pi, pj, i == j ? -x : 0.0);
  const bool first = lane < 9;
  const double mv = fma(first ? A : B, w, fma(first ? B : C, w2, i == j ? 1.0 : 0.0));
  if (lane < 9) b.dR[q] = mv;
  else if (lane < 18) b.V[q] = mv;
  __syncwarp();
  // dT = V rho on lanes 0..2
  const int rr = lane % 3;
  const double dt = fma(b.V[3 * rr], r0, fma(b.V[3 * rr + 1], r1, b.V[3 * rr + 2] * r2));
  // P <- [dR dT] P on lanes 0..11, element (r, c) = (l / 4, l % 4)
  const int l = min(lane, 11), r = l >> 2, c = l & 3;
  const double dtr = __shfl_sync(kFull, dt, r);
  const double pn = fma(b.dR[3 * r], b.P[c],
                        fma(b.dR[3 * r + 1], b.P[4 + c],
                            fma(b.dR[3 * r + 2], b.P[8 + c], c == 3 ? dtr : 0.0)));
  __syncwarp();   // every lane has read the old pose
  if (lane < 12) b.P[lane] = pn;
  if (lane == 0) {
    const double t = tau * b.xi_inv;
    b.t = t;
    b.t_prev = t;
    b.have_t_prev = 1;
  }
  __syncwarp();
}

// The step of the iteration in FP32, for the passes of the next one, when it is
// small and plain: everything an iteration waits for between its step pass and
// the next gradient pass, with no FP64 instruction in it. The FP64 step
// (pending_step) follows while the block waits at the next barrier. The pose is
// base + (base's rounding rest + the step's change), the change good to about
// 1e-7 of itself, so for the steps taken here (tau up to 2^-8 / kappa, kappa the
// condition of the root) the passes' pose is the FP64 pose rounded with 0.02 of
// an ulp more error; the FP64 pose itself is not touched by it. Returns false,
// with nothing changed, for anything else: larger steps, a step within 1e-4 of
// the stop test's, the last iteration, no ascent, fallback, second order. Warp 0.
__device__ bool quick_step(BlockCtx& b, const double* sums, int lane) {
  const TailConst& tc = b.tc;
  if (b.small_grad || tc.step_order != 4 || b.k + 1 >= tc.max_iters || !is_pos(sums[1])) return false;
  // G'(tau) = f0 + f1 tau + f2 tau^2 + f3 tau^3 from the sums' bits (truncated to
  // FP32; magnitudes well inside its range, else the FP64 tail)
  float f[4];
  bool plain = __double2hiint(sums[2]) < 0;   // G'' < 0 at 0
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const unsigned hi = (unsigned)__double2hiint(sums[m + 1]), lo = (unsigned)__double2loint(sums[m + 1]);
    plain = plain && ((hi >> 20) & 0x7ffu) - 948u < 150u;   // 2^-75 .. 2^75
    f[m] = (float)(m + 1) * __uint_as_float((hi & 0x80000000u) |
                                            (((hi & 0x7fffffffu) << 3 | lo >> 29) - (896u << 23)));
  }
  if (!plain) return false;
  const float f0 = f[0], f1 = f[1], f2 = f[2], f3 = f[3];
  // Newton from the root of the linear part, which the steps taken here are near
  float ts = __fdividef(-f0, f1);
#pragma unroll
  for (int it = 0; it < 4; ++it)
    ts -= __fdividef(fmaf(fmaf(fmaf(f3, ts, f2), ts, f1), ts, f0),
                     fmaf(fmaf(3.0f * f3, ts, 2.0f * f2), ts, f1));
  float g2;
  if (!(ts > 0.0f && ts < 0.00390625f) || !falls_to(f1, f2, f3, ts, &g2)) return false;
  // the root's error is |G'(ts)| / |G''| plus rounding of about 2^-22 mag / |G''|
  const float mag = f0 + fabsf(f1 * ts) + fabsf(f2 * ts * ts) + fabsf(f3 * ts * ts * ts);
  const float res = fabsf(fmaf(fmaf(fmaf(f3, ts, f2), ts, f1), ts, f0));
  if (!(mag <= -g2 * 0.00390625f && res <= 4.8e-7f * mag)) return false;
  if (b.ic.at_floor && !(ts > tc.eps_pose_f * (1.0f + 1e-4f))) return false;   // may stop: FP64 decides
  // in the centred frame the unit twist is (omega, v') as the step pass used it;
  // lanes 0..11 take element (r, c) = (l / 4, l % 4), r1 and r2 the axes after r
  const int l = min(lane, 11), r = l >> 2, c = l & 3;
  const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;
  const float p0 = ts * b.om[r], p1 = ts * b.om[r1], p2 = ts * b.om[r2];
  const float x = fmaf(p0, p0, fmaf(p1, p1, p2 * p2));   // below 2^-16
  const float A = fmaf(x, -1.0f / 6.0f, 1.0f), B = fmaf(x, -1.0f / 24.0f, 0.5f);
  // row r of (c1 W + c2 W^2) y, W = hat(phi): W y = phi x y, W^2 y = phi (phi . y) - x y
  const auto apply = [&](float y0, float y1, float y2, float c1, float c2) {
    const float dot = fmaf(p0, y0, fmaf(p1, y1, p2 * y2));
    return fmaf(c1, fmaf(p1, y2, -(p2 * y1)), c2 * fmaf(p0, dot, -(x * y0)));
  };
  const float* base = c == 3 ? b.Tb : b.Rb + c;
  const int st = c == 3 ? 1 : 3;
  const float y0 = base[st * r], y1 = base[st * r1], y2 = base[st * r2];
  float d = apply(y0, y1, y2, A, B);
  const float v0 = ts * b.vc[r], v1 = ts * b.vc[r1], v2 = ts * b.vc[r2];
  if (c == 3) d += v0 + apply(v0, v1, v2, B, 1.0f / 6.0f);
  const float v = y0 + ((c == 3 ? b.Tl[r] : b.Rl[3 * r + c]) + d);
  if (lane < 12) {
    if (c < 3) b.R[3 * r + c] = v;
    else b.T[r] = v;
  }
  if (lane == 0) {
    b.pending = 1;
    b.pend_tau = ts;
    b.k += 1;
  }
  __syncwarp();
  return true;
}

// The FP64 part of a quick step: the root refined by FP64 Newton steps from the
// FP32 one (quick_step has shown that G' falls over [0, tau]), the pose, and its
// parts for the next quick step. One warp, while the block waits at a barrier.
__device__ __noinline__ void pending_step(BlockCtx& b, int lane) {
  const double c0 = b.s_raw[1], c1 = mul_pow2(b.s_raw[2], 1), c2 = 3.0 * b.s_raw[3],
               c3 = mul_pow2(b.s_raw[4], 2);
  const double c2x2 = mul_pow2(c2, 1), c3x3 = 3.0 * c3;
  double tau = f32_to_f64(b.pend_tau);
  for (int it = 0; it < 4; ++it) {
    const double f = fma(fma(fma(c3, tau, c2), tau, c1), tau, c0);
    const double fp = fma(fma(c3x3, tau, c2x2), tau, c1);
    double r = (double)(1.0f / (float)fp);
    r = r * fma(-fp, r, 2.0);
    const double dt = -f * r;
    tau += dt;
    // settled: |dt| < 2^-20 tau, so that the next step would change nothing
    if (((__double2hiint(dt) >> 20) & 0x7ff) <= ((__double2hiint(tau) >> 20) & 0x7ff) - 21) break;
  }
  apply_step(b, tau, lane);
  float hi;
  split_pose(b, lane, &hi);
  if (lane == 0) b.pending = 0;
  __syncwarp();
}

// Step tail: step length, pose update P <- exp(t xi) P, stop test. Warp 0.
// The step length is found in tau = |xi| t, the step along xi / |xi|: G'(t) =
// sum_m m S_m t^(m-1) = sigma^2 |xi| sum_m m s_m tau^(m-1), so the quartic of
// the pass's own sums has the same roots in tau (no powers of |xi| needed),
// and the twist is tau (xi / |xi|).
__device__ void finish_step(BlockCtx& b, const double* sums, int lane) {
  const TailConst& tc = b.tc;
  if (lane < 5) b.s_raw[lane] = sums[lane];
  if (lane == 0) {
    b.nnz_total += b.nnz_grad + (unsigned long long)__double_as_longlong(sums[5]);
    b.cand_total += b.cand_grad + (unsigned long long)__double_as_longlong(sums[6]);
  }
  if (tc.mode == kModeEval) {
    __syncwarp();
    if (lane == 0) {
      form_step_sums(b);
      b.done = 1;
    }
    __syncwarp();
    return;
  }
  if (quick_step(b, sums, lane)) return;
  // the step length (the same scalar work on every lane)
  double tau;
  int no_ascent = 0, fallback = 0;
  // no step along a gradient below the stop test's threshold (at rounding
  // level S1 can still be positive, and the quartic's root is then arbitrary);
  // S1 > 0 exactly when s1 > 0
  if (b.small_grad || !is_pos(sums[1])) {
    tau = 0.0;
    no_ascent = 1;
  } else {
    bool ok;
    if (tc.step_order == 2) {
      ok = sums[2] < 0.0;
      tau = ok ? -sums[1] / mul_pow2(sums[2], 1) : 0.0;
    } else {
      ok = first_maximiser(sums[1], mul_pow2(sums[2], 1), 3.0 * sums[3], mul_pow2(sums[4], 2),
                           &tau);
    }
    if (!ok) {
      fallback = 1;
      // half the previous step, or 1e-3 / |xi| on the first one (tau = 1e-3)
      tau = b.have_t_prev ? 0.5 * b.t_prev * b.xi_norm : 1e-3;
    }
  }
  apply_step(b, tau, lane);
  if (lane == 0) {
    b.no_ascent += no_ascent;
    b.fallback += fallback;
    // Table 1: |t xi| = |tau| below eps_pose, or |xi| below eps_grad, at the floor
    const bool conv = b.ic.at_floor && (fabs(tau) < tc.eps_pose || b.small_grad);
    b.k += 1;
    if (conv || b.k >= tc.max_iters) {
      b.done = 1;
      b.converged = conv ? 1 : 0;
    }
  }
  __syncwarp();
}


// The team barrier counts arrivals on one counter that is never reset during
// a launch: generation g is complete when (g + 1) * nblk blocks have arrived.
// Thread 0 of each block adds its arrival with an acquire-release atomic after
// the block's __syncthreads (so every write the block made before the barrier
// is ordered before it) that returns the count before it: the block whose
// arrival completes the generation goes on at once, the others poll the
// counter with acquire loads. No block has to release the others.
__device__ __forceinline__ unsigned barrier_arrive_count(SolveState* st) {
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
               : "=r"(old)
               : "l"(&st->bar_count)
               : "memory");
  return old;
}

// An error bit of the solve, also where the host reads its result from.
__device__ __forceinline__ void raise_status(SolveState* st, int bits) {
  atomicOr(&st->status, bits);
  if (st->host) atomicOr_system(&st->host->status, bits);
}

// Wait until `target` arrivals (thread 0). A block that polls `limit` times
// raises kStatusTimeout and returns false; its team then leaves the solve loop
// when the other blocks' own waits run out at the next barrier, which the
// timed-out block never reaches (an error path, bounded).
__device__ __forceinline__ bool barrier_wait(SolveState* st, unsigned target, unsigned limit) {
  unsigned spins = 0;
  while (ld_acquire(&st->bar_count) < target) {
    if (++spins > limit) {
      raise_status(st, (int)kStatusTimeout);
      return false;
    }
    // the first polls follow one another: most waits end within them, and a sleep
    // is as long as the whole wait
    if (spins > 64u) __nanosleep(32);
  }
  return true;
}

// Bounded barrier of the team's nblk blocks. Every block calls it the same
// number of times; all blocks are resident (cooperative launch).
__device__ bool grid_sync(SolveState* st, unsigned& gen, int* s_flag, int nblk, unsigned limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = (gen + 1) * (unsigned)nblk;
    const bool last = barrier_arrive_count(st) + 1 == target;
    *s_flag = (last || barrier_wait(st, target, limit)) ? 1 : 0;
  }
  gen += 1;
  __syncthreads();
  return *s_flag != 0;
}

// Sum over a warp of 64-bit integers of magnitude below 2^62 / 32: three 32-bit
// reductions of its parts (26 + 26 low bits, the signed rest).
__device__ __forceinline__ long long warp_sum_i64(long long v) {
  const unsigned lo = __reduce_add_sync(kFull, (unsigned)v & 0x3ffffffu);
  const unsigned mid = __reduce_add_sync(kFull, (unsigned)(v >> 26) & 0x3ffffffu);
  const int hi = __reduce_add_sync(kFull, (int)(v >> 52));
  return ((long long)hi << 52) + ((long long)mid << 26) + (long long)lo;
}

// The sum of the nblk values at p (one warp, every lane gets it): exact up to a
// truncation of each value 52 bits below the largest. The block partials are FP32 sums
// widened to FP64 (run_pass), so that only values 2^29 times smaller than the largest lose
// bits at all, no more than FP64 additions take from them (theirs round at the size of the
// running sum; values of 53 bits would fare worse here). The mantissas are
// aligned to the largest exponent and added as integers, in any order with the
// same result: on GB300 an FP64 instruction holds its scheduler's FP64 pipe for
// about 64 cycles, and the ten dependent additions per value (two values to a
// scheduler) were half of the reduction. Values out of the range in which the
// aligned sum is a normal number, infinities and NaNs take FP64 additions.
template <int PER>
__device__ __forceinline__ double sum_partials(const double* p, int nblk, int lane) {
  double v[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int blk = lane + 32 * k;
    v[k] = blk < nblk ? __ldcg(&p[blk]) : 0.0;
  }
  unsigned e_max = 0u;
#pragma unroll
  for (int k = 0; k < PER; ++k)
    e_max = max(e_max, ((unsigned)__double2hiint(v[k]) >> 20) & 0x7ffu);
  e_max = __reduce_max_sync(kFull, e_max);
  if (e_max == 0u) return 0.0;   // zeros (a subnormal is no sum of FP32 products)
  if (e_max < 100u || e_max > 2000u) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < PER; ++k) acc += v[k];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(kFull, acc, off);
    return acc;
  }
  long long acc = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const long long bits = __double_as_longlong(v[k]);
    const unsigned e = (unsigned)(bits >> 52) & 0x7ffu;
    const unsigned shift = min(e_max - e, 63u);
    // 53-bit mantissa, aligned; 512 of them stay below 2^62
    const long long m = ((bits & 0xfffffffffffffll) | 0x10000000000000ll) >> shift;
    acc += e == 0u ? 0ll : bits < 0 ? -m : m;
  }
  acc = warp_sum_i64(acc);
  if (acc == 0) return 0.0;
  // acc 2^(e_max - 1075): the conversion, then the exponent field
  const double d = (double)acc;
  return __hiloint2double(__double2hiint(d) + (((int)e_max - 1075) << 20), __double2loint(d));
}

// Fixed-order sum of the nblk block partials (nvals <= 9 values each,
// value-major; the last two are counts, held as 64-bit integers in the
// doubles' bits), by one block: warp w < nvals - 2 sums value w, one contiguous
// run of nblk doubles, lane l those of blocks l, l + 32, ... (all loads issued
// first); the last two warps add a count each. Results land in out[] (shared).
// Every thread of the block calls it.
template <int PER, class Smem>
__device__ void reduce_partials_of(const double* partials, int nvals, double* out, int nblk,
                                   Smem& sm) {
  static_assert(kWarps >= 9, "seven FP values and the two counts need nine warps");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nf = nvals - 2;     // FP values; nf <= 7
  if (warp < nf) {
    const double* p = partials + (size_t)warp * nblk;
    double acc;
    if (sm.b.tc.reduce_fp32 != 0) {
      float accf = 0.f;
      for (int blk = lane; blk < nblk; blk += 32) accf += (float)__ldcg(&p[blk]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) accf += __shfl_xor_sync(kFull, accf, off);
      acc = (double)accf;
    } else {
      acc = sum_partials<PER>(p, nblk, lane);
    }
    if (lane == 0) out[warp] = acc;
  } else if (warp >= kWarps - 2) {
    const int c = warp - (kWarps - 2);
    const double* p = partials + (size_t)(nf + c) * nblk;
    unsigned long long v[PER], n = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int blk = lane + 32 * k;
      v[k] = blk < nblk ? (unsigned long long)__double_as_longlong(__ldcg(&p[blk])) : 0ull;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) n += v[k];
    // counts stay below n m = 2^44 over the team
    n = (unsigned long long)warp_sum_i64((long long)n);
    if (lane == 0) out[nf + c] = __longlong_as_double((long long)n);
  }
  __syncthreads();
}

template <class Smem>
__device__ __forceinline__ void reduce_partials(const double* partials, int nvals, double* out,
                                                int nblk, Smem& sm) {
  if (nblk <= 160) reduce_partials_of<5>(partials, nvals, out, nblk, sm);
  else reduce_partials_of<16>(partials, nvals, out, nblk, sm);   // nblk <= 512
}

// Barrier that also reduces the pass: every block adds its arrival (a release
// reduction after the block's partials are written), waits for the
// generation's last arrival with acquire loads, and then adds all block
// partials itself (reduce_partials), so that no block has to
// publish totals and release the others. A block reads the partials of
// generation g only before it arrives at generation g + 1, and the next
// writes to the same partial buffer (two generations later) come after that
// arrival, so one buffer per pass kind is enough. Every thread of every block
// gets the totals in sums[]. Bounded like grid_sync.
// `meanwhile` runs on one warp of the block between its arrival and the reduction:
// FP64 work that nothing needs before the pass's tail.
template <class Smem, class Meanwhile>
__device__ bool grid_sync_reduce(SolveState* st, unsigned& gen, Smem& sm, const double* partials,
                                 int nvals, int nblk, Meanwhile meanwhile) {
  const unsigned g = gen;
  gen += 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = (g + 1) * (unsigned)nblk;
    const bool last = barrier_arrive_count(st) + 1 == target;
    sm.flag = (last || barrier_wait(st, target, sm.b.tc.wait_polls)) ? 1 : 0;
  }
  if (threadIdx.x >> 5 == kWarps / 2 + 1) meanwhile((int)(threadIdx.x & 31));
  __syncthreads();
  if (!sm.flag) return false;
  reduce_partials(partials, nvals, sm.sums, nblk, sm);
  return true;
}

// Start of a queued solve: wait until every block of the team has claimed its
// slot. Blocks of a team come free at different times (each finishes the pair
// it held), so this wait can last as long as one pair's solve; it is bounded
// by join_limit_ns of the global timer (SolveCfg), after which the pair fails
// with kStatusTimeout.
template <class Smem>
__device__ bool team_join(SolveState* st, int team_size, Smem& sm) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    atomicAdd(&st->join_count, 1u);
    const unsigned long long t_start = globaltimer();
    unsigned polls = 0;
    while (ld_acquire(&st->join_count) < (unsigned)team_size) {
      if ((++polls & 255u) == 0 && globaltimer() - t_start > sm.b.tc.join_limit_ns) {
        ok = 0;
        raise_status(st, (int)kStatusTimeout);
        break;
      }
      __nanosleep(256);
    }
    __threadfence();
    if (ld_acquire((const unsigned*)&st->status) & kStatusTimeout) ok = 0;
    sm.flag = ok;
  }
  __syncthreads();
  return sm.flag != 0;
}

// Squared distance from x to the box [lo, hi] (zero inside), the one form the
// plan and every pass evaluate, so that they agree on each candidate.
__device__ __forceinline__ float box_dist2(float4 x, float4 lo, float4 hi) {
  const float dx = fmaxf(fmaxf(lo.x - x.x, x.x - hi.x), 0.f);
  const float dy = fmaxf(fmaxf(lo.y - x.y, x.y - hi.y), 0.f);
  const float dz = fmaxf(fmaxf(lo.z - x.z, x.z - hi.z), 0.f);
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Work of a cluster of cs points with fc filtered candidates, in pair-test units
// (cluster_work without what only a pass can tell).
__device__ __forceinline__ long long plan_work(const SolveCfg* cfg, int cs, int fc) {
  const int nch = (fc + 31) >> 5;
  return nch > 0 ? (long long)cfg->cost_cluster +
                       (long long)nch * (((cs + 3) & ~3) + cfg->cost_chunk)
                 : 0ll;
}

// Plan of one cluster (one warp): transform its points, bounding box, cell
// rows within the plan radius -> segments, candidate count; then the
// candidates themselves are read once and those farther than the plan radius
// from the bounding box are filtered out (they cannot come within the cutoff
// of any of the cluster's points while the plan is valid: a point within r_c
// at the current pose lies within r_c + drift < plan radius of its plan-pose
// position, which is inside the box). Per segment, the number of candidates
// that pass gives the filtered offsets the work split and the passes use.
// s_xs, s_pf, s_cnt: the warp's shared arrays (kMaxSeg + 1 entries). agg (may be
// NULL): the work totals of the groups of 32 clusters, to which the cluster's is
// added (integers: the same total in any order).
__device__ void plan_cluster(const SolveCfg* cfg, const BlockCtx& b, SolveState* st, int c,
                             int lane, int* s_xs, int* s_pf, int* s_cnt, long long* agg) {
  const GridView& g = cfg->grids[b.ic.level];
  const ClusterView& cv = cfg->clusters[b.ic.level];
  __syncwarp();   // the shared arrays of the warp's previous cluster are free
  const int p0 = cv.cstart[c];
  const int cs = cv.cstart[c + 1] - p0;
  const bool zv = lane < cs;
  float zx = 0.f, zy = 0.f, zz = 0.f;
  if (zv) {
    const float4 p = cfg->src.xyz[p0 + lane];
    zx = fmaf(b.R[0], p.x, fmaf(b.R[1], p.y, fmaf(b.R[2], p.z, b.T[0])));
    zy = fmaf(b.R[3], p.x, fmaf(b.R[4], p.y, fmaf(b.R[5], p.z, b.T[1])));
    zz = fmaf(b.R[6], p.x, fmaf(b.R[7], p.y, fmaf(b.R[8], p.z, b.T[2])));
  }
  float blo[3] = {zv ? zx : INFINITY, zv ? zy : INFINITY, zv ? zz : INFINITY};
  float bhi[3] = {zv ? zx : -INFINITY, zv ? zy : -INFINITY, zv ? zz : -INFINITY};
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      blo[a] = fminf(blo[a], __shfl_xor_sync(kFull, blo[a], off));
      bhi[a] = fmaxf(bhi[a], __shfl_xor_sync(kFull, bhi[a], off));
    }
  }
  const float rp = b.rplan_f;
  const float rp2 = rp * rp;
  const int cx0 = max(0, cell_floor(blo[0] - rp, g.ox, g.inv_h, g.nx));
  const int cx1 = min(g.nx - 1, cell_floor(bhi[0] + rp, g.ox, g.inv_h, g.nx));
  const int cy0 = max(0, cell_floor(blo[1] - rp, g.oy, g.inv_h, g.ny));
  const int cy1 = min(g.ny - 1, cell_floor(bhi[1] + rp, g.oy, g.inv_h, g.ny));
  const int cz0 = max(0, cell_floor(blo[2] - rp, g.oz, g.inv_h, g.nz));
  const int cz1 = min(g.nz - 1, cell_floor(bhi[2] + rp, g.oz, g.inv_h, g.nz));
  const int nyr = cy1 - cy0 + 1, nzr = cz1 - cz0 + 1;
  const int nrows = (cx0 <= cx1 && nyr > 0 && nzr > 0) ? nyr * nzr : 0;
  int* sxs = cfg->seg_xs + (size_t)c * kMaxSeg;
  int* spf = cfg->seg_pref + (size_t)c * kMaxSeg;
  const unsigned lt = (1u << lane) - 1u;
  int nseg = 0, total = 0;
  bool overflow = false;
  for (int rb = 0; rb < nrows; rb += 32) {
    const int r = rb + lane;
    int len = 0, xs = 0;
    if (r < nrows) {
      const int cy = cy0 + r % nyr, cz = cz0 + r / nyr;
      const float ylo = g.oy + cy * g.h, yhi = ylo + g.h;
      const float zlo = g.oz + cz * g.h, zhi = zlo + g.h;
      const float dy = fmaxf(0.f, fmaxf(ylo - bhi[1], blo[1] - yhi));
      const float dz = fmaxf(0.f, fmaxf(zlo - bhi[2], blo[2] - zhi));
      const float rem = rp2 - dy * dy - dz * dz;
      if (rem >= 0.f) {
        const float rx = sqrtf(rem);
        const int a0 = max(cx0, cell_floor(blo[0] - rx, g.ox, g.inv_h, g.nx));
        const int a1 = min(cx1, cell_floor(bhi[0] + rx, g.ox, g.inv_h, g.nx));
        if (a0 <= a1) {
          const int base = g.nx * (cy + g.ny * cz);
          xs = g.cell_start[base + a0];
          len = g.cell_start[base + a1 + 1] - xs;
        }
      }
    }
    const unsigned m = __ballot_sync(kFull, len > 0);
    const int idx = nseg + __popc(m & lt);
    const int keep = (len > 0 && idx < kMaxSeg) ? len : 0;
    if (len > 0 && idx >= kMaxSeg) overflow = true;
    int incl = keep;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += v;
    }
    if (keep > 0) {
      sxs[idx] = xs;
      spf[idx] = total + incl - keep;
      s_xs[idx] = xs;
      s_pf[idx] = total + incl - keep;
    }
    nseg += __popc(m);
    total += __shfl_sync(kFull, incl, 31);
  }
  if (__any_sync(kFull, overflow) && lane == 0) raise_status(st, (int)kStatusSegOverflow);
  nseg = min(nseg, kMaxSeg);
  if (lane == 0) s_pf[nseg] = total;
  for (int i = lane; i < nseg; i += 32) s_cnt[i] = 0;
  __syncwarp();
  // the filter: every candidate read once, four rounds of 32 loads in flight.
  // Only a plan that will be reused (the next iteration keeps the lengthscale)
  // is filtered, and only its clusters of at most kFilterMax candidates; the
  // others get the whole space as their box (every candidate passes): a plan
  // used for one iteration does not repay the extra read
  const bool filt = b.plan_filter != 0 && total <= kFilterMax;
  const float4 lo4 = filt ? make_float4(blo[0], blo[1], blo[2], 0.f)
                          : make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
  const float4 hi4 = filt ? make_float4(bhi[0], bhi[1], bhi[2], 0.f)
                          : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
  bool dense = false;
  if (!filt) {
    for (int i = lane; i < nseg; i += 32) s_cnt[i] = s_pf[i + 1] - s_pf[i];
    if (total >= kDenseFrom) {
      // 32 candidates spread over the segments through the box test (kDenseFrom)
      const int q = (int)((unsigned)lane * (unsigned)(total >> 5));
      int at = 0;
      while (s_pf[at + 1] <= q) ++at;
      const float4 x = g.xyz[s_xs[at] + (q - s_pf[at])];
      dense = __all_sync(kFull, box_dist2(x, make_float4(blo[0], blo[1], blo[2], 0.f),
                                          make_float4(bhi[0], bhi[1], bhi[2], 0.f)) <= rp2);
    }
  }
  int seg = 0;
  for (int u0 = 0; filt && u0 < total; u0 += 128) {
    float4 xq[4];
    int sq[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = u0 + 32 * k + lane;
      sq[k] = -1 - lane;   // distinct for every lane past the end
      xq[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q < total) {
        while (s_pf[seg + 1] <= q) ++seg;
        sq[k] = seg;
        xq[k] = g.xyz[s_xs[seg] + (q - s_pf[seg])];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool pass = sq[k] >= 0 && box_dist2(xq[k], lo4, hi4) <= rp2;
      const unsigned m = __ballot_sync(kFull, pass);
      const unsigned grp = __match_any_sync(kFull, sq[k]);
      const int n = __popc(grp & m);
      if (sq[k] >= 0 && lane == __ffs(grp) - 1 && n > 0) atomicAdd(&s_cnt[sq[k]], n);
    }
  }
  __syncwarp();
  // filtered offsets of the segments (exclusive prefix over at most 64)
  const int n0 = lane < nseg ? s_cnt[lane] : 0;
  const int n1 = lane + 32 < nseg ? s_cnt[lane + 32] : 0;
  int i0 = n0, i1 = n1;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v0 = __shfl_up_sync(kFull, i0, off);
    const int v1 = __shfl_up_sync(kFull, i1, off);
    if (lane >= off) {
      i0 += v0;
      i1 += v1;
    }
  }
  const int t0 = __shfl_sync(kFull, i0, 31);
  const int t1 = __shfl_sync(kFull, i1, 31);
  int* sff = cfg->seg_fpref + (size_t)c * kMaxSeg;
  if (lane < nseg) sff[lane] = i0 - n0;
  if (lane + 32 < nseg) sff[lane + 32] = t0 + i1 - n1;
  cfg->ch_act[(size_t)c * kActChunks + lane] = 0u;
  if (lane == 0) {
    cfg->cl_act[c] = 0;
    cfg->cl_nseg[c] = nseg;
    cfg->cl_cand[c] = total;
    cfg->cl_fcand[c] = t0 + t1;
    cfg->cl_kept[c] = 0;
    if (agg) {
      const long long w = plan_work(cfg, cs, t0 + t1);
      if (w) atomicAdd(reinterpret_cast<unsigned long long*>(agg + (c >> 5)), (unsigned long long)w);
    }
    // the box at the plan pose, whether or not the plan filtered (w = 1: the
    // segment offsets count the candidates within the plan radius of it; 2: a box
    // test would hardly drop a candidate)
    cfg->cl_box[2 * (size_t)c] = make_float4(blo[0], blo[1], blo[2], filt ? 1.f : dense ? 2.f : 0.f);
    cfg->cl_box[2 * (size_t)c + 1] = make_float4(bhi[0], bhi[1], bhi[2], 0.f);
  }
}

// Work of cluster c under the current plan, in pair-test units: staging the
// cluster costs cost_cluster, each chunk of 32 filtered candidates its cs4
// pair tests per lane (cluster size padded to a multiple of 4) plus
// cost_chunk of per-chunk overhead, plus (use_kept, once the plan's first
// gradient pass has counted them) cost_kept per kept pair of the cluster,
// spread evenly over its chunks. Chunk j starts at offset cost_cluster + j * k,
// k = the per-chunk cost; within a chunk, the overhead and the first group of
// four source points come first, then one group (4 tests) after another.
// With act > 0 (a reused plan, once its first gradient pass has recorded
// which source groups of which chunks kept a pair), each such group costs
// act more (its pair bodies); chunks beyond the recorded ones count
// every group as active.
__device__ __forceinline__ long long cluster_work(const SolveCfg* cfg, const ClusterView& cv,
                                                  int c, int* k_out, int* cs4_out, int* nch_out,
                                                  bool use_kept, int act) {
  const int tc = __ldcg(&cfg->cl_fcand[c]);
  const int cs4 = ((cv.cstart[c + 1] - cv.cstart[c]) + 3) & ~3;
  const int nch = (tc + 31) >> 5;
  *cs4_out = cs4;
  *nch_out = nch;
  int k = cs4 + cfg->cost_chunk;
  if (use_kept && nch > 0)
    k += (int)(cfg->cost_kept * (float)__ldcg(&cfg->cl_kept[c]) / (float)nch);
  *k_out = k;
  if (nch <= 0) return 0;
  long long w = (long long)cfg->cost_cluster + (long long)nch * k;
  if (act)
    w += (long long)act * ((long long)__ldcg(&cfg->cl_act[c]) +
                                   (long long)max(0, nch - kActChunks) * (cs4 >> 2));
  return w;
}

// Entries of a warp's pair list (build_lists), per padded feature width (640 at 5 feature
// planes, 448 at 3 and 8, 400 without features). They are static shared memory, so each
// takes two bytes a warp from the plan cache, which packs clusters and chunks; the
// counts are those that cost no 32-point slot when the cache was made of slots. The room
// pair of 20k points lists 250 a warp.
template <int DPS>
__host__ __device__ constexpr int list_max() {
  return DPS == 5 ? 640 : DPS == 1 ? 400 : 448;
}
constexpr int kListShift = 22;   // cache_cl of a listed cluster slot: cluster | length << 22
static_assert(kMaxPoints <= (1 << kListShift), "cluster index must fit below the list length");

// Per warp: the cell-row segments of the cluster being staged from the plan
// (plan, cache fill, streamed passes), or, for a warp whose share is cached
// from a plan that will be reused, its pair list (the segments are not needed
// once the cache is filled, and a cached warp never streams).
struct WarpSeg {
  int xs[kMaxSeg];
  int pf[kMaxSeg + 1];
  int fpf[kMaxSeg + 1];   // filtered offsets (the plan: per-segment counts)
};
template <int DPS>
union WarpScratch {
  WarpSeg seg;
  unsigned short list[list_max<DPS>()];
};

// Per block: the work split.
struct SplitScratch {
  long long scan[kThreads];
  long long wsum[kWarps];
  // per end of a warp's range: its position in the work, and the group of
  // clusters that holds it with the position where that group starts
  long long at[2 * kWarps * kMaxRanges], base[2 * kWarps * kMaxRanges];
  int group[2 * kWarps * kMaxRanges];
};

// Shared memory of the solve kernel.
template <int DPS, int NU>
struct SolveSmem {
  // staged cluster, local: (-2 z_l, |z_l|^2), see stage_cluster: float4 rows for a listed
  // cluster, four planes of kClusterMax floats for the chunk path
  float4 z[kWarps][kClusterMax];
  float4 zo[kWarps];                // origin of each warp's staged cluster (centred frame)
  float zf[kWarps][DPS][kClusterMax];
  float4 u[kWarps][NU][kClusterMax];   // step vectors of a listed cluster's points (stage_cluster)
  float zw[kWarps][kClusterMax];       // step pass: -z_l . kw
  union {
    WarpScratch<DPS> ws[kWarps];    // cell-row segments of the staged cluster, or the pair list
    SplitScratch split;             // between the plan and the cache fill, when neither is live
  };
  float red[kWarps][10];
  double sums[10];
  int flag;
  long long q_slot;                 // queue: claimed slot (-1: none left)
  int q_entry;                      //        entry that slot belongs to
  short cache_n[kWarps];            // slots cached per warp (-1: streamed)
  unsigned short cache_hdr[kWarps][32];
  int cache_cl[kWarps][32];         // cluster of each cached cluster slot (a listed one: | list
                                    //   length << kListShift), chunk index of a chunk slot
  BlockCtx b;
};

// (cluster, chunk, group) of the first unit of work that starts at or after
// s, for s inside group-of-clusters `group` whose work starts at `base` (one
// warp). Units of a cluster whose work starts at e0: its staging
// [e0, e0 + cost_cluster), then per chunk j (starting at e = e0 +
// cost_cluster + j k) the unit of source group 0 at e (it carries the chunk's
// overhead oh = k - cs4) and the unit of source group g > 0 at e + oh + 4 g.
// The chunk may equal the cluster's chunk count, which means the next
// cluster's first chunk.
__device__ void locate(const SolveCfg* cfg, const ClusterView& cv, int group, long long base,
                       long long s, int lane, int* c_out, int* j_out, int* g_out,
                       bool use_kept, int act) {
  const int c = group * 32 + lane;
  long long w = 0;
  int kk = 4, cs4_l = 4, nch_l = 0;
  if (c < cv.ncl) w = cluster_work(cfg, cv, c, &kk, &cs4_l, &nch_l, use_kept, act);
  long long incl = w;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const long long v = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += v;
  }
  const long long excl = base + incl - w;
  const unsigned m = __ballot_sync(kFull, c < cv.ncl && w > 0 && s >= excl && s < excl + w);
  if (m) {
    const int src = __ffs(m) - 1;
    const int cc = group * 32 + src;
    const long long e = __shfl_sync(kFull, excl, src) + cfg->cost_cluster;
    const int k4 = __shfl_sync(kFull, kk, src);
    const int cs4 = __shfl_sync(kFull, cs4_l, src);
    const int oh = k4 - cs4;
    const int G = cs4 >> 2;
    const int nch = __shfl_sync(kFull, nch_l, src);
    int j = 0, gq = 0;
    if (act && s > e) {
      // chunk j costs k4 + act x (its active groups; all of them past
      // the recorded chunks); lane j holds chunk j's mask
      const unsigned gm = (1u << G) - 1u;
      long long cum = 0;   // end of the chunks before this round, relative to e
      for (int j0 = 0;; j0 += 32) {
        const int jj = j0 + lane;
        unsigned mj = gm;
        if (jj < nch && jj < kActChunks) mj = __ldcg(&cfg->ch_act[(size_t)cc * kActChunks + jj]) & gm;
        const long long kj = jj < nch ? (long long)k4 + (long long)act * __popc(mj) : 0;
        long long in = kj;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const long long v = __shfl_up_sync(kFull, in, off);
          if (lane >= off) in += v;
        }
        // the chunk whose end lies beyond s (s - e < cum + in)
        const unsigned hit = __ballot_sync(kFull, jj < nch && s - e < cum + in);
        if (hit) {
          const int src2 = __ffs(hit) - 1;
          const long long start = e + cum + __shfl_sync(kFull, in - kj, src2);
          const unsigned m = __shfl_sync(kFull, mj, src2);
          j = j0 + src2;
          if (s > start) {
            // units of the chunk: group 0 at start (with the overhead), group
            // g at start + oh + sum over g' < g of (4 + act a_g')
            long long u = start + oh + 4 + act * (long long)(m & 1u);
            gq = G;
            for (int g = 1; g < G; ++g) {
              if (u >= s) {
                gq = g;
                break;
              }
              u += 4 + act * (long long)((m >> g) & 1u);
            }
            if (gq >= G) {
              ++j;
              gq = 0;
            }
          }
          break;
        }
        cum += __shfl_sync(kFull, in, 31);
        if (j0 + 32 >= nch) {   // past the last chunk (cannot happen: s < end)
          j = nch;
          break;
        }
      }
    } else if (s > e) {
      const long long r = s - e;
      j = (int)(r / k4);
      const int rr = (int)(r - (long long)j * k4);
      if (rr > 0) {
        gq = max(1, (rr - oh + 3) >> 2);   // the first g >= 1 with oh + 4 g >= rr
        if (gq >= (cs4 >> 2)) {
          ++j;
          gq = 0;
        }
      }
    }
    *c_out = cc;
    *j_out = j;
    *g_out = gq;
  } else {
    *c_out = min(group * 32 + 32, cv.ncl);
    *j_out = 0;
    *g_out = 0;
  }
}

// Place the block's warps on an even split of the plan's work into NR x NW pieces
// (NW warps in the team): a piece owns the units (a chunk's source group) whose
// work starts in [floor(p TW / (NR NW)), floor((p + 1) TW / (NR NW))). Warp w of nw
// of block r takes the pieces p = (k nw + w) size + r, k < NR: the share of the
// tests that keep a pair, which the plan does not know, varies smoothly over the
// cloud, so a block whose warps take pieces from all over it ends its pass at
// about the time the other blocks do, where one contiguous run of the work per
// block left the slowest block 1.2 to 1.3 times the mean. Each further piece costs
// its warp a cluster to stage and two ends to locate.
template <int DPS, int NU>
__device__ __noinline__ void split_work(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int tid, Team team,
                           const long long* agg) {
  const ClusterView& cv = cfg->clusters[sm.b.ic.level];
  const int lane = tid & 31, warp = tid >> 5;
  const int ng = (cv.ncl + 31) / 32;
  const int per = (ng + kThreads - 1) / kThreads;
  const int g0 = min(ng, tid * per), g1 = min(ng, g0 + per);
  long long local = 0;
  for (int gi = g0; gi < g1; ++gi) local += __ldcg(&agg[gi]);
  // inclusive scan over the block's threads: within warps, then the warp totals
  long long incl = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const long long v = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) sm.split.wsum[warp] = incl;
  __syncthreads();
  long long TW = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if (w < warp) incl += sm.split.wsum[w];
    TW += sm.split.wsum[w];
  }
  sm.split.scan[tid] = incl;
  // short shares leave the last warp out: its FP64 work (pending_step,
  // gradient_fp64: 2.3 and 0.6 us) then hides behind the passes instead of
  // lengthening the waits at their barriers, for a fifteenth more work per warp
  const int nw = TW < (long long)team.size * kWarps * kSpareWork ? kWarps - 1 : kWarps;
  const long long NW = (long long)team.size * nw;
  const long long share = TW / NW;
  const bool small = team.size <= kSmallTeam;
  const int nr = share < (small ? kSmallTeamFrom : kRangeFrom) ? 1
                 : small ? 2 : (int)min((long long)kMaxRanges, share / kRangeWork);
  __syncthreads();
  // end h of the k-th piece of warp w on thread (k nw + w) 2 + h: the thread
  // whose run of groups holds it, by binary search, then the group
  if (tid < 2 * nw * nr) {
    const long long piece = (long long)(tid >> 1) * team.size + team.rank + (tid & 1);
    const long long at = TW > 0 ? (piece * TW) / (NW * nr) : 0;
    int group = -1;
    long long base = 0;
    if (at < TW) {
      int lo = 0, hi = kThreads - 1;   // the first thread whose inclusive sum is beyond `at`
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sm.split.scan[mid] > at) hi = mid;
        else lo = mid + 1;
      }
      base = lo > 0 ? sm.split.scan[lo - 1] : 0;
      const int ge = min(ng, (lo + 1) * per);
      for (int gi = lo * per; gi < ge; ++gi) {
        const long long w = __ldcg(&agg[gi]);
        if (at < base + w) {
          group = gi;
          break;
        }
        base += w;
      }
    }
    sm.split.group[tid] = group;
    sm.split.base[tid] = base;
    sm.split.at[tid] = at;
  }
  if (tid == 0) {
    sm.b.n_range = nr;
    // (a plan used once has no rebalance: its chain of round trips is shorter without)
    if (!sm.b.use_act && sm.b.plan_filter) {
      sm.b.plan_no += 1;
      sm.b.cost_act = active_weight(TW, NW, cv.ncl, cfg->src.m, cfg->cost_chunk, cfg->cost_cluster,
                                    DPS > 1 ? 4 + DPS : 4, sm.b.cap);
    }
    sm.b.check_fit = sm.b.use_act > kCostActive ? 1 : 0;
    sm.b.n_workers = nw;
    sm.b.compact = small || share >= kCompactWork ? 1 : 0;
  }
  __syncthreads();
  for (int k = 0; k < nr; ++k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = 2 * (k * nw + warp) + h;
      int c = cv.ncl, jj = 0, gg = 0;   // past the end: no chunk
      if (warp < nw && sm.split.group[q] >= 0)
        locate(cfg, cv, sm.split.group[q], sm.split.base[q], sm.split.at[q], lane, &c, &jj, &gg,
               sm.b.use_kept != 0, sm.b.use_act);
      if (lane == 0) {
        if (h == 0) {
          sm.b.w_c0[k][warp] = c;
          sm.b.w_j0[k][warp] = jj;
          sm.b.w_g0[k][warp] = gg;
        } else {
          sm.b.w_c1[k][warp] = c;
          sm.b.w_j1[k][warp] = jj;
          sm.b.w_g1[k][warp] = gg;
        }
      }
    }
  }
  __syncthreads();
}

// Stage one cluster for a warp: lane j < cs holds the cluster's centred
// source point p and its features. The transformed point z~' = R p + T is
// stored relative to the cluster's origin o (lane 0's transformed point) as
// (-2 z_l, |z_l|^2), z_l = z~' - o, so that a candidate x_l = x' - o tests
// its squared distance as |x_l|^2 + x_l . (-2 z_l) + |z_l|^2: three FMAs
// with x_l and |x_l|^2 formed once per chunk. The cluster is small (an
// octree cell of the plan's level), so |x_l| and |z_l| stay within a few
// cutoff radii and the expansion loses no more than a few bits to
// cancellation. Padding slots hold (0, 0, 0, +inf): beyond every cutoff,
// zero weight. The chunk path reads four consecutive points of one component
// at a time, so it gets the components as planes; a cluster with a pair list
// (`listed`) is read point by point, so it gets rows, and for the step pass
// the points' step vectors go to the warp's slots as well, their fourth
// components holding the per-point constants that turn x_l . U_k into the term.
template <bool STEP, int DP, int DPS, int NU>
__device__ __forceinline__ void stage_cluster(SolveSmem<DPS, NU>& sm, int warp, int lane, bool zv,
                                              float4 p, const float pf[DPS], bool listed) {
  const BlockCtx& b = sm.b;
  float zt[3] = {0.f, 0.f, 0.f};
  if (zv) {
    zt[0] = fmaf(b.R[0], p.x, fmaf(b.R[1], p.y, fmaf(b.R[2], p.z, b.T[0])));
    zt[1] = fmaf(b.R[3], p.x, fmaf(b.R[4], p.y, fmaf(b.R[5], p.z, b.T[1])));
    zt[2] = fmaf(b.R[6], p.x, fmaf(b.R[7], p.y, fmaf(b.R[8], p.z, b.T[2])));
  }
  // lane 0 holds a point of every staged cluster (cs >= 1)
  const float ox = __shfl_sync(kFull, zt[0], 0), oy = __shfl_sync(kFull, zt[1], 0),
              oz = __shfl_sync(kFull, zt[2], 0);
  const float lx = zv ? zt[0] - ox : 0.f, ly = zv ? zt[1] - oy : 0.f, lz = zv ? zt[2] - oz : 0.f;
  const float4 row = zv ? make_float4(-2.f * lx, -2.f * ly, -2.f * lz,
                                      fmaf(lx, lx, fmaf(ly, ly, lz * lz)))
                        : make_float4(0.f, 0.f, 0.f, INFINITY);
  if (listed) {
    sm.z[warp][lane] = row;
  } else {
    float* pl = reinterpret_cast<float*>(sm.z[warp]);
    pl[lane] = row.x;
    pl[kClusterMax + lane] = row.y;
    pl[2 * kClusterMax + lane] = row.z;
    pl[3 * kClusterMax + lane] = row.w;
  }
  if (lane == 0) sm.zo[warp] = make_float4(ox, oy, oz, 0.f);
#pragma unroll
  for (int d = 0; d < DP; ++d) sm.zf[warp][d][lane] = zv ? pf[d] : 0.f;
  if (STEP) {
    sm.zw[warp][lane] = -fmaf(lx, b.kw[0], fmaf(ly, b.kw[1], lz * b.kw[2]));
    if (listed) {
      const float* om = b.om;
      const float c1 = 0.5f * b.ic.inv_l2f, c2 = 0.25f * b.ic.inv_l2f;
      const float u1[3] = {om[1] * zt[2] - om[2] * zt[1] + b.vc[0],
                           om[2] * zt[0] - om[0] * zt[2] + b.vc[1],
                           om[0] * zt[1] - om[1] * zt[0] + b.vc[2]};
      const float u2[3] = {om[1] * u1[2] - om[2] * u1[1], om[2] * u1[0] - om[0] * u1[2],
                           om[0] * u1[1] - om[1] * u1[0]};
      const float u11 = fmaf(u1[0], u1[0], fmaf(u1[1], u1[1], u1[2] * u1[2]));
      const float4 U1 = make_float4(u1[0] * c1, u1[1] * c1, u1[2] * c1, 0.f);
      const float4 U2 = make_float4(u2[0] * c2, u2[1] * c2, u2[2] * c2, 0.f);
      const auto zl_dot = [&](const float4& U) { return fmaf(lx, U.x, fmaf(ly, U.y, lz * U.z)); };
      sm.u[warp][0][lane] = make_float4(U1.x, U1.y, U1.z, -zl_dot(U1));
      sm.u[warp][1 % NU][lane] = make_float4(U2.x, U2.y, U2.z, -zl_dot(U2) - c2 * u11);
    }
  }
}

// The step pass (Eq. fourth). Along P <- exp(t xi) P, xi = (omega, v) a unit
// direction, a source point moves by u_1 = omega x z~' + v, u_2 = omega x u_1,
// and Rodrigues' formula closes the series: u_3 = (omega . v) omega -
// |omega|^2 u_1, u_4 = -|omega|^2 u_2, with u_1 . u_2 = 0, u_1 . u_3 = -|u_2|^2
// and |u_2|^2 = |omega|^2 |u_1|^2 - (omega . v)^2. With e = x' - z~' the exponent's
// coefficients are then
//   beta  = e . u_1 / l^2
//   gamma = (e . u_2 - |u_1|^2) / 2 l^2
//   delta = (e . u_3 / 6 - u_1 . u_2 / 2) / l^2
//         = (omega . v) (e . omega) / 6 l^2 - |omega|^2 beta / 6
//   eps   = (e . u_4 / 24 - u_1 . u_3 / 6 - |u_2|^2 / 8) / l^2
//         = -|omega|^2 gamma / 12 - (omega . v)^2 / 24 l^2
// so a pair needs three inner products (beta, gamma, e . omega) where the printed
// form takes four. The same holds seen from the target point: |x' - exp(t xi) z~'|
// = |exp(-t xi) x' - z~'|, so with a_1 = omega x x' + v and a_2 = omega x a_1,
// beta = e . a_1 / l^2 and gamma = (-e . a_2 - |a_1|^2) / 2 l^2: linear in e with
// vectors that belong to the candidate alone. In the cluster's frame e = x_l + m / 2
// (m = -2 z_l), each is c + m . V; V and c are formed once per chunk and stay in
// the lane's registers, where vectors of the source point are shared loads per
// pair. Halved terms (beta / 2, gamma / 2) keep factors of two out of the bodies;
// the sums are scaled back, exactly, once per chunk.
struct StepVectors {
  f32x2 v1[3], v2[3], c1, c2, cw;
};

__device__ __forceinline__ StepVectors step_vectors(const BlockCtx& b, float x, float y, float z,
                                                    float xl, float yl, float zl) {
  const float w0 = b.om[0], w1 = b.om[1], w2 = b.om[2];
  const float k1 = 0.5f * b.ic.inv_l2f, k2 = -0.25f * b.ic.inv_l2f;
  const float a0 = w1 * z - w2 * y + b.vc[0], a1 = w2 * x - w0 * z + b.vc[1],
              a2 = w0 * y - w1 * x + b.vc[2];
  const float p0 = a0 * k1, p1 = a1 * k1, p2 = a2 * k1;
  const float q0 = (w1 * a2 - w2 * a1) * k2, q1 = (w2 * a0 - w0 * a2) * k2,
              q2 = (w0 * a1 - w1 * a0) * k2;
  StepVectors s;
  s.v1[0] = dup2(0.5f * p0);
  s.v1[1] = dup2(0.5f * p1);
  s.v1[2] = dup2(0.5f * p2);
  s.v2[0] = dup2(0.5f * q0);
  s.v2[1] = dup2(0.5f * q1);
  s.v2[2] = dup2(0.5f * q2);
  s.c1 = dup2(fmaf(xl, p0, fmaf(yl, p1, zl * p2)));
  s.c2 = dup2(fmaf(k2, fmaf(a0, a0, fmaf(a1, a1, a2 * a2)), fmaf(xl, q0, fmaf(yl, q1, zl * q2))));
  s.cw = dup2(fmaf(xl, b.kw[0], fmaf(yl, b.kw[1], zl * b.kw[2])));
  return s;
}

// A candidate against the cluster staged for the warp.
struct ChunkLane {
  f32x2 X, Y, Z;          // x_l
  float xl, yl, zl, x2, thr;
};

__device__ __forceinline__ ChunkLane chunk_lane(float4 xp, float4 o, float rc2) {
  ChunkLane k;
  k.xl = xp.x - o.x;
  k.yl = xp.y - o.y;
  k.zl = xp.z - o.z;
  k.x2 = fmaf(k.xl, k.xl, fmaf(k.yl, k.yl, k.zl * k.zl));
  k.thr = rc2 - k.x2;   // about -3e36 for a padding candidate: never kept
  k.X = dup2(k.xl);
  k.Y = dup2(k.yl);
  k.Z = dup2(k.zl);
  return k;
}

// Four staged source points as planes, two packed pairs.
struct SourceGroup {
  ulonglong2 x, y, z, w;
};

__device__ __forceinline__ SourceGroup source_group(const float* pl, int j0) {
  SourceGroup g;
  g.x = *reinterpret_cast<const ulonglong2*>(pl + j0);
  g.y = *reinterpret_cast<const ulonglong2*>(pl + kClusterMax + j0);
  g.z = *reinterpret_cast<const ulonglong2*>(pl + 2 * kClusterMax + j0);
  g.w = *reinterpret_cast<const ulonglong2*>(pl + 3 * kClusterMax + j0);
  return g;
}

__device__ __forceinline__ void group_tests(const SourceGroup& g, const ChunkLane& k, f32x2 t[2]) {
  t[0] = fma2(k.X, g.x.x, fma2(k.Y, g.y.x, fma2(k.Z, g.z.x, g.w.x)));
  t[1] = fma2(k.X, g.x.y, fma2(k.Y, g.y.y, fma2(k.Z, g.z.y, g.w.y)));
}

// The lane keeps one of the group's four pairs.
__device__ __forceinline__ bool group_kept(const SourceGroup& g, const ChunkLane& k) {
  f32x2 t[2];
  group_tests(g, k, t);
  float t0, t1, t2, t3;
  unpack2(t[0], t0, t1);
  unpack2(t[1], t2, t3);
  return fminf(fminf(t0, t1), fminf(t2, t3)) <= k.thr;
}

// The source groups in [jlo, jhi) of which any lane keeps a pair with its candidate
// (bit g: group g), the same in every lane.
template <int DPS, int NU>
__device__ __forceinline__ unsigned chunk_groups(const SolveSmem<DPS, NU>& sm, int warp,
                                                 const ChunkLane& k, int jlo, int jhi) {
  const float* pl = reinterpret_cast<const float*>(sm.z[warp]);
  unsigned mine = 0u;
#pragma unroll 2
  for (int j0 = jlo; j0 < jhi; j0 += 4)
    if (group_kept(source_group(pl, j0), k)) mine |= 1u << (j0 >> 2);
  return __reduce_or_sync(kFull, mine);
}

// The same for two chunks at once over all groups: the tests are bound by their
// 16-byte broadcast loads (eight cycles of a scheduler each with all four
// loading), which two candidates share. Queued solves only (TWO): their passes are
// mostly these chunks (64-pair batch 103.9 -> 102.2 ms, 16 served requests 95.7 ->
// 94.5); in single solves the registers it takes cost the cached floor passes more
// (2k pair 819 -> 847 us, 20k 5.49 -> 5.54 ms) than large shares gain (100k 45.3 ->
// 44.2 ms).
template <int DPS, int NU>
__device__ __forceinline__ void chunk_groups2(const SolveSmem<DPS, NU>& sm, int warp, float4 xa,
                                              float4 xb, int jhi, float rc2, unsigned active[2]) {
  const ChunkLane ka = chunk_lane(xa, sm.zo[warp], rc2), kb = chunk_lane(xb, sm.zo[warp], rc2);
  const float* pl = reinterpret_cast<const float*>(sm.z[warp]);
  unsigned ma = 0u, mb = 0u;
#pragma unroll 2
  for (int j0 = 0; j0 < jhi; j0 += 4) {
    const SourceGroup g = source_group(pl, j0);
    if (group_kept(g, ka)) ma |= 1u << (j0 >> 2);
    if (group_kept(g, kb)) mb |= 1u << (j0 >> 2);
  }
  active[0] = __reduce_or_sync(kFull, ma);
  active[1] = __reduce_or_sync(kFull, mb);
}

// The pair bodies of a chunk's active groups.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ __forceinline__ void chunk_bodies(SolveSmem<DPS, NU>& sm, int warp, float4 xp,
                                             const ChunkLane& lane_k, const float xf[DPS],
                                             unsigned active, float A, float acc[7],
                                             unsigned& nnz) {
  if (active == 0u) return;
  const float xl = lane_k.xl, yl = lane_k.yl, zl = lane_k.zl, x2 = lane_k.x2, thr = lane_k.thr;
  const float* pl = reinterpret_cast<const float*>(sm.z[warp]);
  const f32x2 q0 = dup2(A * x2), A2 = dup2(A);
  f32x2 F[DPS];
#pragma unroll
  for (int d = 0; d < DP; ++d) F[d] = dup2(xf[d]);
  StepVectors sv;
  f32x2 c_del, c_eps, k_eps;
  if (STEP) {
    // a padding candidate takes the origin, so that its step terms stay finite
    const bool pad = xp.w != 0.f;
    sv = step_vectors(sm.b, pad ? 0.f : xp.x, pad ? 0.f : xp.y, pad ? 0.f : xp.z, pad ? 0.f : xl,
                      pad ? 0.f : yl, pad ? 0.f : zl);
    c_del = dup2(sm.b.c_del);
    c_eps = dup2(sm.b.c_eps);
    k_eps = dup2(sm.b.k_eps);
  }
  // gradient: W, M (3); step: the five sums, halved or quartered
  f32x2 s[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
  for (unsigned rem = active; rem != 0u; rem &= rem - 1u) {
    const int j0 = 4 * (__ffs(rem) - 1);
    const SourceGroup g = source_group(pl, j0);
    f32x2 t[2];
    group_tests(g, lane_k, t);
    f32x2 q[2] = {q0, q0};
    f32x2 cdot[2] = {0ull, 0ull};
#pragma unroll
    for (int d = 0; d < DP; ++d) {
      const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(&sm.zf[warp][d][j0]);
      if (color_of(MODE) == kColorKernel) {
        const f32x2 d0 = sub2(F[d], f.x), d1 = sub2(F[d], f.y);
        q[0] = fma2(d0, d0, q[0]);
        q[1] = fma2(d1, d1, q[1]);
      } else if (color_of(MODE) == kColorDot) {
        cdot[0] = fma2(F[d], f.x, cdot[0]);
        cdot[1] = fma2(F[d], f.y, cdot[1]);
      }
    }
    ulonglong2 zw;
    if (STEP) zw = *reinterpret_cast<const ulonglong2*>(&sm.zw[warp][j0]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const f32x2 mx = h ? g.x.y : g.x.x, my = h ? g.y.y : g.y.x, mz = h ? g.z.y : g.z.x;
      float t0, t1, e0, e1, w0, w1;
      unpack2(t[h], t0, t1);
      const bool k0 = t0 <= thr, k1 = t1 <= thr;
      unpack2(fma2(A2, t[h], q[h]), e0, e1);
      w0 = ex2_approx(-e0);
      w1 = ex2_approx(-e1);
      if (color_of(MODE) == kColorDot) {
        float c0, c1;
        unpack2(cdot[h], c0, c1);
        w0 *= c0;
        w1 *= c1;
      }
      const f32x2 w = pack2(k0 ? w0 : 0.f, k1 ? w1 : 0.f);
      nnz += (k0 ? 1u : 0u) + (k1 ? 1u : 0u);
      s[0] = add2(s[0], w);
      if (!STEP) {
        // m = (-2 z_l, .) is finite, so a zero weight adds exactly zero
        s[1] = fma2(w, mx, s[1]);
        s[2] = fma2(w, my, s[2]);
        s[3] = fma2(w, mz, s[3]);
      } else {
        float b0, b1;
        unpack2(fma2(mx, sv.v1[0], fma2(my, sv.v1[1], fma2(mz, sv.v1[2], sv.c1))), b0, b1);
        const f32x2 beta = pack2(k0 ? b0 : 0.f, k1 ? b1 : 0.f);
        const f32x2 gam = fma2(mx, sv.v2[0], fma2(my, sv.v2[1], fma2(mz, sv.v2[2], sv.c2)));
        const f32x2 del = fma2(c_del, beta, add2(sv.cw, h ? zw.y : zw.x));
        const f32x2 eps = fma2(c_eps, gam, k_eps);
        // with b = beta / 2, c = gamma / 2: g2 = 2 (b^2 + c), g3 = 4 (b (b^2 / 3 + c) +
        // delta / 4), g4 = 2 (b^2 (b^2 / 3 + c) + c (b^2 + c) + b delta + eps / 2)
        const f32x2 b2 = mul2(beta, beta);
        const f32x2 u = fma2(b2, dup2(1.0f / 3.0f), gam);
        const f32x2 g2 = add2(b2, gam);
        const f32x2 g3 = fma2(beta, u, mul2(dup2(0.25f), del));
        const f32x2 g4 = fma2(b2, u, fma2(gam, g2, fma2(beta, del, eps)));
        s[1] = fma2(w, beta, s[1]);
        s[2] = fma2(w, g2, s[2]);
        s[3] = fma2(w, g3, s[3]);
        s[4] = fma2(w, g4, s[4]);
      }
    }
  }
  if (!STEP) {
    // E_i = sum_j w e_ij = x_l W - sum_j w z_l = x_l W + M / 2; x' fixed per
    // lane: sum_j w (z~'_j x e_ij) = x' x E_i. A padding lane has W = M = 0
    // and a finite x_l.
    const float W = sum2(s[0]);
    const float Ex = fmaf(xl, W, 0.5f * sum2(s[1]));
    const float Ey = fmaf(yl, W, 0.5f * sum2(s[2]));
    const float Ez = fmaf(zl, W, 0.5f * sum2(s[3]));
    acc[0] += W;
    acc[1] += xp.y * Ez - xp.z * Ey;
    acc[2] += xp.z * Ex - xp.x * Ez;
    acc[3] += xp.x * Ey - xp.y * Ex;
    acc[4] += Ex;
    acc[5] += Ey;
    acc[6] += Ez;
  } else {
    acc[0] += sum2(s[0]);
    acc[1] = fmaf(2.0f, sum2(s[1]), acc[1]);
    acc[2] = fmaf(2.0f, sum2(s[2]), acc[2]);
    acc[3] = fmaf(4.0f, sum2(s[3]), acc[3]);
    acc[4] = fmaf(2.0f, sum2(s[4]), acc[4]);
  }
}

// One 32-candidate chunk against the staged cluster: lane = candidate x'
// (xp, features xf; padding points lie beyond every cutoff and carry w = 1),
// over the cluster's points [jlo, jhi) (multiples of 4, at most the cluster
// size rounded up to 4; padding slots lie beyond the cutoff too). FP32 pair
// arithmetic, one ex2.approx per pair. Distances are taken relative to the
// cluster's origin (stage_cluster): t = x_l . (-2 z_l) + |z_l|^2 equals
// d^2 - |x_l|^2, so a pair is kept when t <= r_c^2 - |x_l|^2, and the
// exponent A d^2 is A t + A |x_l|^2.
// Points are taken four at a time, as two packed pairs: the staged planes give
// both halves of each operand with one 16-byte broadcast load per four points
// and component. First the distance tests of every group of four, each lane
// noting the groups in which it keeps a pair; one reduction over the warp then
// gives the groups to evaluate, whose bodies run without votes or branches (a
// rejected pair contributes exactly nothing: its weight is selected to zero, and
// its beta, whose fourth power would be the first of its step terms to
// overflow). Testing all groups first keeps the chain of loads, test, vote and
// branch out of the bodies, which repeat the test's six packed FMAs instead.
// Returns the active groups.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ __forceinline__ unsigned chunk_pairs(SolveSmem<DPS, NU>& sm, int warp, float4 xp,
                                                const float xf[DPS], int jlo, int jhi, float rc2,
                                                float A, float acc[7], unsigned& nnz) {
  const ChunkLane k = chunk_lane(xp, sm.zo[warp], rc2);
  const unsigned active = chunk_groups<DPS, NU>(sm, warp, k, jlo, jhi);
  chunk_bodies<STEP, DP, MODE, DPS, NU>(sm, warp, xp, k, xf, active, A, acc, nnz);
  return active;
}

// A warp's k-th range of work (BlockCtx::w_*).
struct WarpRange {
  int c0, j0, g0, c1, j1, g1;
};

__device__ __forceinline__ WarpRange warp_range(const BlockCtx& b, int warp, int k) {
  return WarpRange{b.w_c0[k][warp], b.w_j0[k][warp], b.w_g0[k][warp],
                   b.w_c1[k][warp], b.w_j1[k][warp], b.w_g1[k][warp]};
}

// Chunks [jb, je] of cluster c (nch chunks) that hold work of the range.
__device__ __forceinline__ bool range_chunks(const WarpRange& r, int c, int nch, int& jb, int& je) {
  if (c < r.c0 || c > r.c1) return false;
  jb = c == r.c0 ? r.j0 : 0;
  je = nch - 1;
  if (c == r.c1) je = min(je, r.g1 > 0 ? r.j1 : r.j1 - 1);
  return jb <= je;
}

// Source groups [glo, ghi) of chunk j of cluster c (G groups) in the range.
__device__ __forceinline__ void range_groups(const WarpRange& r, int c, int j, int G, int& glo,
                                             int& ghi) {
  glo = (c == r.c0 && j == r.j0) ? r.g0 : 0;
  ghi = (c == r.c1 && j == r.j1) ? min(r.g1, G) : G;
}

// The nseg segments of cluster c into the warp's shared arrays: first target
// index, candidate offset (then tc) and filtered offset (then fc) of each segment.
template <int DPS, int NU>
__device__ __forceinline__ void load_segments(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int warp,
                                              int lane, int c, int nseg, int tc, int fc) {
  static_assert(kMaxSeg == 64, "two segments per lane");
  const size_t at = (size_t)c * kMaxSeg + lane;
  int v[2][3];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool have = lane + 32 * h < nseg;
    v[h][0] = have ? __ldcg(&cfg->seg_xs[at + 32 * h]) : 0;
    v[h][1] = have ? __ldcg(&cfg->seg_pref[at + 32 * h]) : 0;
    v[h][2] = have ? __ldcg(&cfg->seg_fpref[at + 32 * h]) : 0;
  }
  WarpSeg& seg = sm.ws[warp].seg;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (lane + 32 * h >= nseg) continue;
    seg.xs[lane + 32 * h] = v[h][0];
    seg.pf[lane + 32 * h] = v[h][1];
    seg.fpf[lane + 32 * h] = v[h][2];
  }
  if (lane == 0) {
    seg.pf[nseg] = tc;
    seg.fpf[nseg] = fc;
  }
  __syncwarp();
}

// Position of candidate q of the staged cluster (-1 beyond tc), advancing seg.
template <int DPS, int NU>
__device__ __forceinline__ int candidate_at(const SolveSmem<DPS, NU>& sm, int warp, int q, int tc,
                                            int& seg) {
  if (q >= tc) return -1;
  const WarpSeg& sg = sm.ws[warp].seg;
  while (sg.pf[seg + 1] <= q) ++seg;
  return sg.xs[seg] + (q - sg.pf[seg]);
}

// Features of target point xi (zeros for -1).
template <int DP, int DPS, bool FB>
__device__ __forceinline__ void load_features(const GridView& g, int xi, float xf[DPS]) {
#pragma unroll
  for (int d = 0; d < DPS; ++d) xf[d] = 0.f;
  if (xi < 0) return;
#pragma unroll
  for (int d = 0; d < DP; ++d) xf[d] = load_feat<FB>(g.feat, (size_t)d * g.n_pad + xi);
}

// Candidate q of the staged cluster (padding beyond tc), advancing seg.
template <int DP, int DPS, int NU, bool FB>
__device__ __forceinline__ float4 load_candidate(const GridView& g, SolveSmem<DPS, NU>& sm, int warp,
                                                 int q, int tc, int& seg, float xf[DPS]) {
  const int xi = candidate_at<DPS, NU>(sm, warp, q, tc, seg);
  load_features<DP, DPS, FB>(g, xi, xf);
  return xi >= 0 ? g.xyz[xi] : make_float4(-kFar, -kFar, -kFar, 1.f);
}

// The same without its features, its position in place of w.
template <int DPS, int NU>
__device__ __forceinline__ float4 load_point(const GridView& g, const SolveSmem<DPS, NU>& sm, int warp,
                                             int q, int tc, int& seg) {
  const int xi = candidate_at<DPS, NU>(sm, warp, q, tc, seg);
  float4 p = xi >= 0 ? g.xyz[xi] : make_float4(-kFar, -kFar, -kFar, 0.f);
  p.w = __int_as_float(xi);
  return p;
}

// Cursor over the filtered candidates of the cluster whose segments are
// staged: the next block of 32 candidates starts at candidate u; `skip`
// filtered candidates are still to be dropped (they precede the range); seg
// is this lane's segment; made counts the filtered candidates produced.
struct FCursor {
  int u, skip, seg, made;
};

// Cursor at filtered candidate f0 (< fc): the last segment whose filtered
// offset is <= f0 (a segment that filters to nothing shares its offset with
// the next one), from its first candidate.
template <int DPS, int NU>
__device__ __forceinline__ FCursor fcursor_at(const SolveSmem<DPS, NU>& sm, int warp, int nseg,
                                              int f0) {
  int lo = 0, hi = nseg;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (sm.ws[warp].seg.fpf[mid] <= f0) lo = mid;
    else hi = mid;
  }
  FCursor cur;
  cur.u = sm.ws[warp].seg.pf[lo];
  cur.skip = f0 - sm.ws[warp].seg.fpf[lo];
  cur.seg = lo;
  cur.made = 0;
  return cur;
}

// The block of candidates at cur.u (this lane's is xp) through the plan's
// filter: the filtered index (counted from the cursor's start) of this lane's
// candidate, or -1; the cursor moves to the next block.
__device__ __forceinline__ int fplace(FCursor& cur, float4 xp, float4 lo, float4 hi, float rp2,
                                      int lane, int tc) {
  const bool pass = cur.u + lane < tc && box_dist2(xp, lo, hi) <= rp2;
  const unsigned m = __ballot_sync(kFull, pass);
  const int r = __popc(m & ((1u << lane) - 1u));
  const int n = __popc(m);
  const int d = min(cur.skip, n);
  cur.skip -= d;
  const int o = (pass && r >= d) ? cur.made + r - d : -1;
  cur.made += n - d;
  cur.u += 32;
  return o;
}

// Kept pairs of cluster c counted by this warp, added to the plan's
// per-cluster totals (one atomic per warp and cluster).
__device__ __forceinline__ void add_kept(const SolveCfg* cfg, int c, unsigned kept, int lane) {
  unsigned k = kept;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) k += __shfl_down_sync(kFull, k, off);
  if (lane == 0 && c >= 0 && k) atomicAdd(&cfg->cl_kept[c], (int)k);
}

// Source groups of chunk j of cluster c that kept a pair, recorded by the
// plan's first gradient pass (lane 0; the mask is warp-uniform).
__device__ __forceinline__ void add_active(const SolveCfg* cfg, int c, int j, unsigned active,
                                           int lane) {
  if (lane == 0 && active && c >= 0 && j < kActChunks) {
    atomicOr(&cfg->ch_act[(size_t)c * kActChunks + j], active);
    atomicAdd(&cfg->cl_act[c], __popc(active));
  }
}

// Stage the cluster of cs points from p0 on for the warp from global memory (raw
// centred source points and features, transformed by stage_cluster), and its
// segments, whose loads are issued with the points'.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ __forceinline__ void stage_from_global(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int c,
                                                  int p0, int cs, int nseg, int tc, int fc, int warp,
                                                  int lane) {
  const bool zv = lane < cs;
  float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
  float pf[DPS];
#pragma unroll
  for (int d = 0; d < DPS; ++d) pf[d] = 0.f;
  if (zv) {
    p = cfg->src.xyz[p0 + lane];
#pragma unroll
    for (int d = 0; d < DP; ++d)
      pf[d] = load_feat<bf16_of(MODE)>(cfg->src.feat, (size_t)d * cfg->src.m_pad + p0 + lane);
  }
  load_segments<DPS, NU>(cfg, sm, warp, lane, c, nseg, tc, fc);
  stage_cluster<STEP, DP, DPS, NU>(sm, warp, lane, zv, p, pf, false);
  __syncwarp();
}

// Entries of the streamed passes' ring (a power of two), float4 each.
template <bool TWO>
__host__ __device__ constexpr int ring_size() {
  return TWO ? 128 : 64;
}

// One range of a warp's share of a pair pass, streamed from global memory (L2): lane
// sums in acc, counts in nnz / cand. The filtered candidates of each chunk
// are gathered through a ring of entries (position and coordinates) in the
// warp's (otherwise unused) cache region, with the next block of 32 candidates
// loading while the current chunk runs; their features are read once they are
// known to pass, ahead of the chunk's distance tests, which do not need them.
// Lane l holds the numbers of cluster base + l, read 32 clusters at a time, so
// that a cluster waits for one round trip to L2 (its points, segments and box)
// instead of four.
template <bool STEP, int DP, int MODE, int DPS, int NU, bool TWO>
__device__ void pass_stream(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int warp, int lane,
                            WarpRange r, float* ring, float acc[7], unsigned& nnz,
                            unsigned& cand) {
  const BlockCtx& b = sm.b;
  const GridView& g = cfg->grids[b.ic.level];
  const ClusterView& cv = cfg->clusters[b.ic.level];
  const float rc2 = b.ic.rc2, A = b.ic.A;
  const float rp2 = b.rplan_f * b.rplan_f;
  const bool collect = !STEP && b.collect_kept;
  constexpr int kRing = ring_size<TWO>();
  float4* rxyz = reinterpret_cast<float4*>(ring);
  const int c_end = min(r.c1, cv.ncl - 1);
  int l_tc = 0, l_fc = 0, l_p0 = 0, l_cs = 0, l_nseg = 0;
  for (int c = r.c0; c <= c_end; ++c) {
    const int li = (c - r.c0) & 31;
    if (li == 0 && c + lane <= c_end) {
      l_tc = __ldcg(&cfg->cl_cand[c + lane]);
      l_fc = __ldcg(&cfg->cl_fcand[c + lane]);
      l_nseg = __ldcg(&cfg->cl_nseg[c + lane]);
      l_p0 = cv.cstart[c + lane];
      l_cs = cv.cstart[c + lane + 1] - l_p0;
    }
    const int tc = __shfl_sync(kFull, l_tc, li), fc = __shfl_sync(kFull, l_fc, li);
    int jb, je;
    if (!range_chunks(r, c, (fc + 31) >> 5, jb, je)) continue;
    const int cs = __shfl_sync(kFull, l_cs, li), nseg = __shfl_sync(kFull, l_nseg, li);
    const int cs4 = (cs + 3) & ~3;
    const float4 lo = __ldcg(&cfg->cl_box[2 * (size_t)c]);
    const float4 hi = __ldcg(&cfg->cl_box[2 * (size_t)c + 1]);
    __syncwarp();   // every lane is done with the previous cluster
    stage_from_global<STEP, DP, MODE, DPS, NU>(cfg, sm, c, __shfl_sync(kFull, l_p0, li), cs, nseg, tc,
                                               fc, warp, lane);
    FCursor cur = fcursor_at<DPS, NU>(sm, warp, nseg, jb * 32);
    const int want = min(fc, 32 * (je + 1)) - 32 * jb;
    const unsigned nnz0 = nnz;
    if (lo.w == 0.f && !collect && b.compact) {
      // a cluster the plan did not filter (a plan used for one iteration):
      // the candidates of the range's chunks go through the box test here
      // and the survivors are compacted through the ring into full chunks
      // of all source groups. A chunk the range shares with the neighbouring
      // warp (it starts or ends at a source group inside it) runs unfiltered
      // with its own groups, as the plan's numbering of chunks assigns it.
      const int G = cs4 >> 2;
      int glo_b, ghi_b, glo_e, ghi_e;
      range_groups(r, c, jb, G, glo_b, ghi_b);
      range_groups(r, c, je, G, glo_e, ghi_e);
      const bool head = glo_b > 0 || ghi_b < G;
      const bool tail = je != jb && ghi_e < G;
      const auto raw_chunk = [&](int j, int glo, int ghi) {
        FCursor cj = fcursor_at<DPS, NU>(sm, warp, nseg, j * 32);
        float xf[DPS];
        const float4 xp =
            load_candidate<DP, DPS, NU, bf16_of(MODE)>(g, sm, warp, j * 32 + lane, tc, cj.seg, xf);
        if (glo < ghi) {
          const int jlo = 4 * glo, jhi = min(cs4, 4 * ghi);
          if (j * 32 + lane < tc) cand += (unsigned)max(0, min(cs, jhi) - jlo);
          chunk_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, xp, xf, jlo, jhi, rc2, A, acc, nnz);
        }
      };
      if (head) raw_chunk(jb, glo_b, ghi_b);
      const int j0 = head ? jb + 1 : jb, j1 = tail ? je - 1 : je;
      if (j0 <= j1) {
        const int uend = min(tc, 32 * (j1 + 1));
        // a cursor at raw candidate 32 j0 (its segment from the offsets, which
        // count every candidate here), nothing to skip
        FCursor cf = fcursor_at<DPS, NU>(sm, warp, nseg, j0 * 32);
        cf.u = j0 * 32;
        cf.skip = 0;
        float4 xpn = load_point<DPS, NU>(g, sm, warp, cf.u + lane, uend, cf.seg);
        int used = 0;
        constexpr int kTake = TWO ? 64 : 32;   // candidates taken at a time
        for (;;) {
          // place blocks of 32 until those are there or the range is done (at
          // most kTake + 31 entries are unread, so the ring never overwrites one)
          while (cf.made - used < kTake && cf.u < uend) {
            const int o = fplace(cf, xpn, lo, hi, rp2, lane, uend);
            if (o >= 0) rxyz[o & (kRing - 1)] = xpn;
            if (cf.u < uend) xpn = load_point<DPS, NU>(g, sm, warp, cf.u + lane, uend, cf.seg);
          }
          const int cnt = min(kTake, cf.made - used);
          if (cnt <= 0) break;
          __syncwarp();
          // this lane's candidate of the first (h = 0) or second chunk
          const auto take = [&](int h, int& xi) {
            float4 xp = make_float4(-kFar, -kFar, -kFar, 1.f);
            xi = -1;
            if (lane + 32 * h < cnt) {
              xp = rxyz[(used + 32 * h + lane) & (kRing - 1)];
              xi = __float_as_int(xp.w);
              xp.w = 0.f;
            }
            return xp;
          };
          int xi;
          float xf[DPS];
          if constexpr (TWO) {
            const float4 xb = take(1, xi);
            float4 xp = take(0, xi);
            load_features<DP, DPS, bf16_of(MODE)>(g, xi, xf);
            unsigned active[2];
            chunk_groups2<DPS, NU>(sm, warp, xp, xb, cs4, rc2, active);
            cand += (unsigned)cs * ((lane < cnt ? 1u : 0u) + (lane + 32 < cnt ? 1u : 0u));
            for (int h = 0; h < 2; ++h) {
              chunk_bodies<STEP, DP, MODE, DPS, NU>(sm, warp, xp, chunk_lane(xp, sm.zo[warp], rc2),
                                                    xf, active[0], A, acc, nnz);
              if (h == 1 || active[1] == 0u) break;
              active[0] = active[1];
              xp = take(1, xi);
              load_features<DP, DPS, bf16_of(MODE)>(g, xi, xf);
            }
          } else {
            const float4 xp = take(0, xi);
            load_features<DP, DPS, bf16_of(MODE)>(g, xi, xf);
            cand += lane < cnt ? (unsigned)cs : 0u;
            chunk_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, xp, xf, 0, cs4, rc2, A, acc, nnz);
          }
          __syncwarp();   // read before the next placement reuses the entries
          used += cnt;
        }
      }
      if (tail) raw_chunk(je, glo_e, ghi_e);
      continue;
    }
    if (lo.w != 1.f) {
      // an unfiltered cluster whose first gradient pass records which source
      // groups kept pairs, chunk by chunk: chunk j holds candidates 32 j ..
      // 32 j + 31, loaded straight into registers, the next chunk's while this
      // one runs
      float xfn[DPS];
      float4 xpn = load_candidate<DP, DPS, NU, bf16_of(MODE)>(g, sm, warp, jb * 32 + lane, tc,
                                                              cur.seg, xfn);
      for (int j = jb; j <= je; ++j) {
        const float4 xp = xpn;
        float xf[DPS];
#pragma unroll
        for (int d = 0; d < DPS; ++d) xf[d] = xfn[d];
        if (j < je)
          xpn = load_candidate<DP, DPS, NU, bf16_of(MODE)>(g, sm, warp, (j + 1) * 32 + lane, tc,
                                                           cur.seg, xfn);
        int glo, ghi;
        range_groups(r, c, j, cs4 >> 2, glo, ghi);
        if (glo < ghi) {
          const int jlo = 4 * glo, jhi = min(cs4, 4 * ghi);
          if (j * 32 + lane < tc) cand += (unsigned)max(0, min(cs, jhi) - jlo);
          const unsigned act =
              chunk_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, xp, xf, jlo, jhi, rc2, A, acc, nnz);
          if (collect) add_active(cfg, c, j, act, lane);
        }
      }
      if (collect) add_kept(cfg, c, nnz - nnz0, lane);
      continue;
    }
    float4 xpn = load_point<DPS, NU>(g, sm, warp, cur.u + lane, tc, cur.seg);
    int used = 0;
    for (int j = jb; j <= je; ++j) {
      const int cnt = min(32, want - used);
      // place blocks until the chunk is complete (at most 63 entries are
      // unread, so the ring never overwrites one)
      while (cur.made - used < cnt && cur.u < tc) {
        const int o = fplace(cur, xpn, lo, hi, rp2, lane, tc);
        if (o >= 0) rxyz[o & (kRing - 1)] = xpn;
        if (cur.u < tc) xpn = load_point<DPS, NU>(g, sm, warp, cur.u + lane, tc, cur.seg);
      }
      __syncwarp();
      float4 xp = make_float4(-kFar, -kFar, -kFar, 1.f);
      int xi = -1;
      const bool have = lane < cnt && used + lane < cur.made;
      if (have) {
        xp = rxyz[(used + lane) & (kRing - 1)];
        xi = __float_as_int(xp.w);
        xp.w = 0.f;
      }
      float xf[DPS];
      load_features<DP, DPS, bf16_of(MODE)>(g, xi, xf);
      __syncwarp();   // read before the next placement reuses the entries
      int glo, ghi;
      range_groups(r, c, j, cs4 >> 2, glo, ghi);
      if (glo < ghi) {
        const int jlo = 4 * glo, jhi = min(cs4, 4 * ghi);
        if (have) cand += (unsigned)max(0, min(cs, jhi) - jlo);
        const unsigned act =
            chunk_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, xp, xf, jlo, jhi, rc2, A, acc, nnz);
        if (collect) add_active(cfg, c, j, act, lane);
      }
      used += cnt;
    }
    if (collect) add_kept(cfg, c, nnz - nnz0, lane);
  }
}

// Shared-memory cache of a warp's share of the plan (cap floats): chunk slots
// from the front, each the 32 candidates of a chunk (float4 xyz, then DP
// feature planes of 32 floats; padding points beyond every cutoff), and the raw
// centred source points of the clusters from the back, each cluster just as
// large as it is (float4 rows, then DP planes, of its size rounded up to 4: a
// cluster of the floor holds 5.5 points of the room pair on average, and a
// 32-point slot for each took about a third of the cache). The items follow in
// order in cache_hdr: a cluster (kSlotCluster | its size), then its chunks
// (number of valid candidates | first source group << 6 | end source group
// << 10). Filled once per plan, so that the passes of every iteration that reuses
// the plan (at the lengthscale floor, most of the solve) read no global memory. A
// share of a reused plan that is too large is cached as far as it goes, with the
// front left to the streamed pass's ring for the rest of it (BlockCtx::rest_c).
constexpr int kCacheSlots = 32;                 // items per warp
constexpr unsigned short kSlotCluster = 0x8000;
constexpr unsigned short kSlotList = 0x4000;      // cluster whose pairs are listed

template <int DP>
__device__ __forceinline__ constexpr int slot_floats() {
  return 32 * (4 + DP);
}

// Floats a cluster of cs points takes in the cache.
template <int DP>
__device__ __forceinline__ int cluster_floats(int cs) {
  return ((cs + 3) & ~3) * (4 + DP);
}

// Pair lists of a plan that will be reused (Verlet-style): for each cached
// cluster, the (candidate, source point) pairs of its cached chunks within
// the plan radius at the plan pose, in slot order and, within a chunk, source
// point by source point. While the plan is valid every source point stays
// within the skin of where it was at the plan pose (the drift test of
// begin_iteration), so these pairs are a superset of the pairs within the
// cutoff, and the passes evaluate only them (each with the exact cutoff test)
// instead of every candidate against every source group. An entry is
// candidate lane | chunk slot << 5 | source point << 10; the lists live in the
// warp's shared scratch (list_max entries). A cluster whose list would not
// fit keeps the chunk-by-chunk evaluation.
template <int DP, int DPS, int NU>
__device__ __noinline__ void build_lists(SolveSmem<DPS, NU>& sm, int warp, int lane, const float* base,
                            int cap, int n) {
  unsigned short* pl = sm.ws[warp].list;
  constexpr int kCap = list_max<DPS>();
  const BlockCtx& b = sm.b;
  float R[9], T[3];
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = b.Rq[i];
#pragma unroll
  for (int i = 0; i < 3; ++i) T[i] = b.Tq[i];
  const float rp2 = b.rplan_f * b.rplan_f;
  const unsigned lt = (1u << lane) - 1u;
  int run = 0, coff = cap, k = 0;
  for (int s = 0; s < n; ++s) {
    const unsigned h = sm.cache_hdr[warp][s];
    const int cs = (int)(h & 0x3f);
    coff -= cluster_floats<DP>(cs);
    const float4 p = reinterpret_cast<const float4*>(base + coff)[min(lane, cs - 1)];
    const float zx = fmaf(R[0], p.x, fmaf(R[1], p.y, fmaf(R[2], p.z, T[0])));
    const float zy = fmaf(R[3], p.x, fmaf(R[4], p.y, fmaf(R[5], p.z, T[1])));
    const float zz = fmaf(R[6], p.x, fmaf(R[7], p.y, fmaf(R[8], p.z, T[2])));
    const int start = run;
    bool fits = true;
    int t = s + 1;
    for (; t < n && !(sm.cache_hdr[warp][t] & kSlotCluster); ++t, ++k) {
      const unsigned hc = sm.cache_hdr[warp][t];
      const int cnt = (int)(hc & 0x3f);
      const int jlo = 4 * (int)((hc >> 6) & 0xf), jhi = min(cs, 4 * (int)((hc >> 10) & 0xf));
      const float4 xp =
          reinterpret_cast<const float4*>(base + (size_t)k * slot_floats<DP>())[lane];
      const bool valid = lane < cnt;
      for (int j = jlo; j < jhi && fits; ++j) {
        const float dx = xp.x - __shfl_sync(kFull, zx, j);
        const float dy = xp.y - __shfl_sync(kFull, zy, j);
        const float dz = xp.z - __shfl_sync(kFull, zz, j);
        const bool in = valid && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= rp2;
        const unsigned m = __ballot_sync(kFull, in);
        if (run + __popc(m) > kCap) {
          fits = false;   // warp-uniform
        } else {
          if (in) pl[run + __popc(m & lt)] = (unsigned short)(lane | (k << 5) | (j << 10));
          run += __popc(m);
        }
      }
    }
    if (!fits) run = start;
    if (lane == 0 && fits) {
      sm.cache_hdr[warp][s] = (unsigned short)(h | kSlotList);
      sm.cache_cl[warp][s] |= (run - start) << kListShift;
    }
    s = t - 1;
  }
  __syncwarp();
}

template <int DP, int MODE, int DPS, int NU>
__device__ __noinline__ void fill_cache(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int warp, int lane,
                           float* cache, int cap) {
  const BlockCtx& b = sm.b;
  const GridView& g = cfg->grids[b.ic.level];
  const ClusterView& cv = cfg->clusters[b.ic.level];
  const WarpRange r = warp_range(b, warp, 0);
  const float rp2 = b.rplan_f * b.rplan_f;
  // the numbers of cluster c + lane and its chunks in the range (none: live false),
  // read together so that the fill waits for two round trips to L2 per cluster
  // (these, then its points, segments and box) instead of six
  const int c_end = min(r.c1, cv.ncl - 1);
  int l_tc = 0, l_fc = 0, l_p0 = 0, l_cs = 0, l_nseg = 0, l_jb = 0, l_je = -1, at = -1;
  bool live = false;
  const auto read = [&](int c) {
    at = c;
    live = false;
    if (c + lane > c_end) return;
    l_tc = __ldcg(&cfg->cl_cand[c + lane]);
    l_fc = __ldcg(&cfg->cl_fcand[c + lane]);
    l_nseg = __ldcg(&cfg->cl_nseg[c + lane]);
    l_p0 = cv.cstart[c + lane];
    l_cs = cv.cstart[c + lane + 1] - l_p0;
    live = range_chunks(r, c + lane, (l_fc + 31) >> 5, l_jb, l_je);
  };
  // what the share needs (one in several pieces is too large for the cache)
  int need = 0, items = b.n_range > 1 ? kCacheSlots + 1 : 0;
  for (int c = r.c0; c <= c_end && need <= cap && items <= kCacheSlots; c += 32) {
    read(c);
    // (a lane's count may be large, the sum is capped)
    const int nc = live ? min(1 + l_je - l_jb, kCacheSlots) : 0;
    need += __reduce_add_sync(kFull, live ? cluster_floats<DP>(l_cs) + nc * slot_floats<DP>() : 0);
    items += __reduce_add_sync(kFull, live ? 1 + nc : 0);
  }
  const bool part = need > cap || items > kCacheSlots;
  if (part && lane == 0 && b.use_act > kCostActive) atomicMax(&b.st->spilled, b.plan_no);
  if (part && (b.n_range > 1 || !b.plan_filter)) {
    if (lane == 0) sm.cache_n[warp] = -1;
    __syncwarp();
    return;
  }
  float* base = cache + (size_t)warp * cap;
  if (part) base += b.ring_floats;
  int room = part ? cap - b.ring_floats : cap;
  int n = 0, k = 0, coff = room;   // items, chunk slots, where the clusters begin
  int rest_c = -1, rest_j = 0, rest_g = 0;
  for (int cb = r.c0; cb <= c_end && rest_c < 0; cb += 32) {
    if (cb != at) read(cb);
    for (unsigned todo = __ballot_sync(kFull, live); todo && rest_c < 0; todo &= todo - 1u) {
      const int li = __ffs(todo) - 1, c = cb + li;
      const int tc = __shfl_sync(kFull, l_tc, li), fc = __shfl_sync(kFull, l_fc, li);
      const int p0 = __shfl_sync(kFull, l_p0, li), nseg = __shfl_sync(kFull, l_nseg, li);
      const int cs = __shfl_sync(kFull, l_cs, li), cs4 = (cs + 3) & ~3;
      const int jb = __shfl_sync(kFull, l_jb, li);
      int je = __shfl_sync(kFull, l_je, li);
      room -= cluster_floats<DP>(cs);
      if (part) {
        // the chunks of this cluster that still fit; the rest is streamed
        const int fit = min(kCacheSlots - n - 1, room < 0 ? 0 : room / slot_floats<DP>());
        if (1 + je - jb > fit) {
          rest_c = c;
          rest_j = jb + max(fit, 0);
          rest_g = c == r.c0 && rest_j == r.j0 ? r.g0 : 0;
          je = rest_j - 1;
          if (je < jb) break;
        }
      }
      room -= (1 + je - jb) * slot_floats<DP>();
      coff -= cluster_floats<DP>(cs);
      float4 lo = __ldcg(&cfg->cl_box[2 * (size_t)c]);
      float4 hi = __ldcg(&cfg->cl_box[2 * (size_t)c + 1]);
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
      float pf[DPS];
      if (lane < cs) {
        p = cfg->src.xyz[p0 + lane];
#pragma unroll
        for (int d = 0; d < DP; ++d)
          pf[d] = load_feat<bf16_of(MODE)>(cfg->src.feat, (size_t)d * cfg->src.m_pad + p0 + lane);
      }
      load_segments<DPS, NU>(cfg, sm, warp, lane, c, nseg, tc, fc);
      float* sl = base + coff;
      if (lane < cs) {
        reinterpret_cast<float4*>(sl)[lane] = p;
#pragma unroll
        for (int d = 0; d < DP; ++d) sl[(4 + d) * cs4 + lane] = pf[d];
      }
      if (lane == 0) {
        sm.cache_hdr[warp][n] = (unsigned short)(kSlotCluster | cs);
        sm.cache_cl[warp][n] = c;
      }
      ++n;
      if (lo.w != 1.f) {   // not filtered by the plan: every candidate of the range is cached
        lo = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
        hi = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
      }
      FCursor cur = fcursor_at<DPS, NU>(sm, warp, nseg, jb * 32);
      const int want = min(fc, 32 * (je + 1)) - 32 * jb;
      float* s0 = base + (size_t)k * slot_floats<DP>();
      while (cur.made < want && cur.u < tc) {
        float xf[DPS];
        const float4 xp =
            load_candidate<DP, DPS, NU, bf16_of(MODE)>(g, sm, warp, cur.u + lane, tc, cur.seg, xf);
        const int o = fplace(cur, xp, lo, hi, rp2, lane, tc);
        if (o >= 0 && o < want) {
          float* sk = s0 + (size_t)(o >> 5) * slot_floats<DP>();
          reinterpret_cast<float4*>(sk)[o & 31] = xp;
#pragma unroll
          for (int d = 0; d < DP; ++d) sk[128 + d * 32 + (o & 31)] = xf[d];
        }
      }
      const int nchk = je - jb + 1;
      for (int o = min(cur.made, want) + lane; o < 32 * nchk; o += 32) {   // padding
        float* sk = s0 + (size_t)(o >> 5) * slot_floats<DP>();
        reinterpret_cast<float4*>(sk)[o & 31] = make_float4(-kFar, -kFar, -kFar, 1.f);
#pragma unroll
        for (int d = 0; d < DP; ++d) sk[128 + d * 32 + (o & 31)] = 0.f;
      }
      if (lane <= je - jb) {
        const int j = jb + lane;
        int glo, ghi;
        range_groups(r, c, j, cs4 >> 2, glo, ghi);
        const int cnt = min(32, want - 32 * lane);
        sm.cache_hdr[warp][n + lane] = (unsigned short)(cnt | (glo << 6) | (ghi << 10));
        sm.cache_cl[warp][n + lane] = j;   // a chunk slot keeps its chunk index
      }
      n += nchk;
      k += nchk;
      __syncwarp();   // the segment arrays are reused by the next cluster
    }
  }
  if (lane == 0) {
    sm.cache_n[warp] = (short)n;
    sm.b.rest_c[warp] = rest_c;
    sm.b.rest_j[warp] = rest_j;
    sm.b.rest_g[warp] = rest_g;
  }
  __syncwarp();
  // (the segments of a streamed rest take the place of the lists)
  if (b.plan_filter && !part) build_lists<DP, DPS, NU>(sm, warp, lane, base, cap, n);
}

// One entry of a cluster's pair list (build_lists) against the staged
// cluster: lane = one (candidate, source point) pair, with the same FP32
// arithmetic as chunk_pairs (the same cutoff test on the same values, so the
// same pairs are kept, and the same weight), the gradient sums formed per pair
// (e = x_l - z_l, z~' x e = x' x e). Returns the kept flag.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ __forceinline__ bool list_pair(SolveSmem<DPS, NU>& sm, int warp, const float* base,
                                          float4 o, unsigned e, bool valid, float rc2, float A,
                                          float acc[7], unsigned& nnz) {
  const int k = (int)(e & 31u), t = (int)((e >> 5) & 31u), j = (int)(e >> 10);
  const float* sl = base + (size_t)t * slot_floats<DP>();
  const float4 xp = reinterpret_cast<const float4*>(sl)[k];
  const float4 m = sm.z[warp][j];
  const float xl = xp.x - o.x, yl = xp.y - o.y, zl = xp.z - o.z;
  const float x2 = fmaf(xl, xl, fmaf(yl, yl, zl * zl));
  const float thr = rc2 - x2;
  const float q0 = A * x2;
  const float tt = fmaf(xl, m.x, fmaf(yl, m.y, fmaf(zl, m.z, m.w)));
  const bool keep = valid && tt <= thr;
  float w;
  if (color_of(MODE) == kColorKernel) {
    float qf = q0;
#pragma unroll
    for (int d = 0; d < DP; ++d) {
      const float df = sl[128 + d * 32 + k] - sm.zf[warp][d][j];
      qf = fmaf(df, df, qf);
    }
    w = ex2_approx(-fmaf(A, tt, qf));
  } else if (color_of(MODE) == kColorDot) {
    float cdot = 0.f;
#pragma unroll
    for (int d = 0; d < DP; ++d) cdot = fmaf(sl[128 + d * 32 + k], sm.zf[warp][d][j], cdot);
    w = ex2_approx(-fmaf(A, tt, q0)) * cdot;
  } else {
    w = ex2_approx(-fmaf(A, tt, q0));
  }
  w = keep ? w : 0.f;
  nnz += keep ? 1u : 0u;
  if (!STEP) {
    // e = x_l - z_l = x_l + m / 2; every term is finite, so w = 0 adds zero
    const float ex = fmaf(0.5f, m.x, xl), ey = fmaf(0.5f, m.y, yl), ez = fmaf(0.5f, m.z, zl);
    acc[0] += w;
    acc[1] = fmaf(w, xp.y * ez - xp.z * ey, acc[1]);
    acc[2] = fmaf(w, xp.z * ex - xp.x * ez, acc[2]);
    acc[3] = fmaf(w, xp.x * ey - xp.y * ex, acc[3]);
    acc[4] = fmaf(w, ex, acc[4]);
    acc[5] = fmaf(w, ey, acc[5]);
    acc[6] = fmaf(w, ez, acc[6]);
  } else {
    // beta / 2, gamma / 2 and the terms of chunk_pairs' step body
    const float4 U1 = sm.u[warp][0][j], U2 = sm.u[warp][1 % NU][j];
    const float* kw = sm.b.kw;
    float beta = fmaf(xl, U1.x, fmaf(yl, U1.y, fmaf(zl, U1.z, U1.w)));
    beta = keep ? beta : 0.f;
    const float gam = fmaf(xl, U2.x, fmaf(yl, U2.y, fmaf(zl, U2.z, U2.w)));
    const float ew = fmaf(xl, kw[0], fmaf(yl, kw[1], fmaf(zl, kw[2], sm.zw[warp][j])));
    const float del = fmaf(sm.b.c_del, beta, ew);
    const float eps = fmaf(sm.b.c_eps, gam, sm.b.k_eps);
    const float b2 = beta * beta;
    const float u = fmaf(b2, 1.0f / 3.0f, gam);
    const float g2 = b2 + gam;
    const float g3 = fmaf(beta, u, 0.25f * del);
    const float g4 = fmaf(b2, u, fmaf(gam, g2, fmaf(beta, del, eps)));
    acc[0] += w;
    acc[1] = fmaf(w, 2.0f * beta, acc[1]);
    acc[2] = fmaf(w, 2.0f * g2, acc[2]);
    acc[3] = fmaf(w, 4.0f * g3, acc[3]);
    acc[4] = fmaf(w, 2.0f * g4, acc[4]);
  }
  return keep;
}

// A listed cluster (staged): its nl pairs, 64 per round (two per lane, whose
// chains overlap), the next round's entries loading while this one runs. In
// the plan's first gradient pass (collect) the source groups of each chunk that
// kept a pair are gathered per chunk slot: lane t holds slot t's mask in act.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ void list_pairs(SolveSmem<DPS, NU>& sm, int warp, int lane, const float* base,
                           const unsigned short* pl, int nl, float rc2, float A, float acc[7],
                           unsigned& nnz, unsigned& cand, bool collect, unsigned& act) {
  const float4 o = sm.zo[warp];
  unsigned e0 = lane < nl ? pl[lane] : 0u, e1 = lane + 32 < nl ? pl[lane + 32] : 0u;
  for (int r = 0; r < nl; r += 64) {
    const bool v0 = r + lane < nl, v1 = r + 32 + lane < nl;
    const unsigned c0 = e0, c1 = e1;
    e0 = r + 64 + lane < nl ? pl[r + 64 + lane] : 0u;
    e1 = r + 96 + lane < nl ? pl[r + 96 + lane] : 0u;
    cand += (v0 ? 1u : 0u) + (v1 ? 1u : 0u);
    const bool k0 = list_pair<STEP, DP, MODE, DPS, NU>(sm, warp, base, o, c0, v0, rc2, A, acc, nnz);
    const bool k1 = list_pair<STEP, DP, MODE, DPS, NU>(sm, warp, base, o, c1, v1, rc2, A, acc, nnz);
    if (collect) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool kk = h ? k1 : k0;
        const unsigned ee = h ? c1 : c0;
        const int ts = (int)((ee >> 5) & 31u);
        const unsigned bit = 1u << (ee >> 12);   // source group j / 4
        unsigned pend = __ballot_sync(kFull, kk);
        while (pend) {
          const int sl = __shfl_sync(kFull, ts, __ffs(pend) - 1);
          const bool mine = kk && ts == sl;
          const unsigned bits = __reduce_or_sync(kFull, mine ? bit : 0u);
          if (lane == sl) act |= bits;
          pend &= ~__ballot_sync(kFull, mine);
        }
      }
    }
  }
}

// The same share as pass_stream, from the warp's cache.
template <bool STEP, int DP, int MODE, int DPS, int NU>
__device__ void pass_cached(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int warp, int lane,
                            const float* cache, int cap, float acc[7], unsigned& nnz,
                            unsigned& cand) {
  const float rc2 = sm.b.ic.rc2, A = sm.b.ic.A;
  const bool collect = !STEP && sm.b.collect_kept;
  const float* base = cache + (size_t)warp * cap;
  if (sm.b.rest_c[warp] >= 0) {   // the front is the ring of the streamed rest
    base += sm.b.ring_floats;
    cap -= sm.b.ring_floats;
  }
  const unsigned short* pl = sm.ws[warp].list;
  const int n = sm.cache_n[warp];
  int cs = 0, cs4 = 0, cur = -1, loff = 0, k = 0, coff = cap;
  unsigned nnz0 = nnz;
  for (int s = 0; s < n; ++s) {
    const unsigned h = sm.cache_hdr[warp][s];
    if (h & kSlotCluster) {
      if (collect) {
        add_kept(cfg, cur, nnz - nnz0, lane);
        nnz0 = nnz;
      }
      cur = sm.cache_cl[warp][s] & ((1 << kListShift) - 1);
      cs = (int)(h & 0x3f);
      cs4 = (cs + 3) & ~3;
      coff -= cluster_floats<DP>(cs);
      const float* sl = base + coff;
      const int i = min(lane, cs - 1);
      const float4 p = reinterpret_cast<const float4*>(sl)[i];
      float f[DPS];
#pragma unroll
      for (int d = 0; d < DPS; ++d) f[d] = d < DP ? sl[(4 + d) * cs4 + i] : 0.f;
      __syncwarp();   // every lane is done with the previous cluster
      stage_cluster<STEP, DP, DPS, NU>(sm, warp, lane, lane < cs, p, f, (h & kSlotList) != 0);
      __syncwarp();
      if (h & kSlotList) {
        // the cluster's chunks through its pair list, then past its chunks
        int t = s + 1;
        while (t < n && !(sm.cache_hdr[warp][t] & kSlotCluster)) ++t;
        const int nl = (int)((unsigned)sm.cache_cl[warp][s] >> kListShift);
        unsigned act = 0u;
        list_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, lane, base, pl + loff, nl, rc2, A, acc, nnz,
                                            cand, collect, act);
        loff += nl;
        const int nk = t - s - 1;   // its chunk slots: k .. k + nk - 1, items s + 1 .. t - 1
        if (collect && lane >= k && lane < k + nk && act && cur >= 0) {
          const int j = sm.cache_cl[warp][s + 1 + lane - k];
          if (j < kActChunks) {
            atomicOr(&cfg->ch_act[(size_t)cur * kActChunks + j], act);
            atomicAdd(&cfg->cl_act[cur], __popc(act));
          }
        }
        k += nk;
        s = t - 1;
      }
    } else {
      const float* sl = base + (size_t)k * slot_floats<DP>();
      const float4 p = reinterpret_cast<const float4*>(sl)[lane];
      float f[DPS];
#pragma unroll
      for (int d = 0; d < DPS; ++d) f[d] = d < DP ? sl[128 + d * 32 + lane] : 0.f;
      ++k;
      const int cnt = (int)(h & 0x3f);
      const int jlo = 4 * (int)((h >> 6) & 0xf), jhi = min(cs4, 4 * (int)((h >> 10) & 0xf));
      if (lane < cnt) cand += (unsigned)max(0, min(cs, jhi) - jlo);
      const unsigned act =
          chunk_pairs<STEP, DP, MODE, DPS, NU>(sm, warp, p, f, jlo, jhi, rc2, A, acc, nnz);
      if (collect) add_active(cfg, cur, sm.cache_cl[warp][s], act, lane);
    }
  }
  if (collect) add_kept(cfg, cur, nnz - nnz0, lane);
}

template <bool STEP, int DP, int MODE, int DPS, int NU, bool TWO>
__device__ __forceinline__ void pass_warp(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, int warp,
                                          int lane, float* cache, int cap, float acc[7],
                                          unsigned& nnz, unsigned& cand) {
  const BlockCtx& b = sm.b;
  int streamed = b.n_range;
  WarpRange r = warp_range(b, warp, 0);
  if (sm.cache_n[warp] >= 0) {
    pass_cached<STEP, DP, MODE, DPS, NU>(cfg, sm, warp, lane, cache, cap, acc, nnz, cand);
    streamed = b.rest_c[warp] >= 0 ? 1 : 0;
    r.c0 = b.rest_c[warp];
    r.j0 = b.rest_j[warp];
    r.g0 = b.rest_g[warp];
  }
  for (int k = 0; k < streamed; ++k) {
    if (k > 0) r = warp_range(b, warp, k);
    pass_stream<STEP, DP, MODE, DPS, NU, TWO>(cfg, sm, warp, lane, r, cache + (size_t)warp * cap, acc,
                                         nnz, cand);
  }
}

// One pass over the block's warps, then the block partial (fixed order).
template <bool STEP, int DP, int MODE, int DPS, int NU, bool TWO>
__device__ void run_pass(const SolveCfg* cfg, SolveSmem<DPS, NU>& sm, double* partials,
                         float* cache, int cap) {
  constexpr int NACC = STEP ? 5 : 7;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float acc[7];
#pragma unroll
  for (int i = 0; i < 7; ++i) acc[i] = 0.f;
  unsigned nnz = 0, cand = 0;
  if (warp == kWarps - 1 && sm.b.n_workers < kWarps) {
    if (STEP) gradient_fp64(sm.b, sm.sums, lane);
    else if (sm.b.pending) pending_step(sm.b, lane);
  }
  pass_warp<STEP, DP, MODE, DPS, NU, TWO>(cfg, sm, warp, lane, cache, cap, acc, nnz, cand);
  __syncwarp();
  // the warp's sums: halves of the warp exchange half of the values, then quarters,
  // eighths, so that lane 4 i ends with the sum of value i (nine shuffles, not 35)
  float v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = i < NACC ? acc[i < 7 ? i : 6] : 0.f;
#pragma unroll
  for (int half = 4, off = 16; half > 0; half >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float keep = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
      v[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
  }
  v[0] += __shfl_xor_sync(kFull, v[0], 2);
  v[0] += __shfl_xor_sync(kFull, v[0], 1);
  if ((lane & 3) == 0 && (lane >> 2) < NACC) sm.red[warp][lane >> 2] = v[0];
  const unsigned wn = __reduce_add_sync(kFull, nnz), wc = __reduce_add_sync(kFull, cand);
  if (lane == 0) {
    sm.red[warp][NACC] = __uint_as_float(wn);
    sm.red[warp][NACC + 1] = __uint_as_float(wc);
  }
  __syncthreads();
  if (warp == 0 && lane < NACC + 2) {
    double s = 0.0;
    if (lane < NACC) {
      // the block's sixteen warp sums in FP32 (fixed order); FP64 starts with the
      // cross-block reduction
      float f = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) f += sm.red[w][lane];
      s = (double)f;
    } else {
      unsigned long long n = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) n += __float_as_uint(sm.red[w][lane]);
      s = __longlong_as_double((long long)n);   // a count: its bits, summed as an integer
    }
    partials[(size_t)lane * sm.b.team_size + sm.b.team_rank] = s;
  }
}

__device__ void publish(SolveState* st, const BlockCtx& b) {
  for (int i = 0; i < 16; ++i) st->P[i] = b.P[i];
  for (int i = 0; i < 6; ++i) st->xi[i] = b.xi[i];
  for (int i = 0; i < 5; ++i) st->S[i] = b.S[i];
  st->xi_norm = b.xi_norm;
  st->F = b.F;
  st->t = b.t;
  st->ell = b.ic.ell;
  st->level = b.ic.level;
  st->iter = b.k;
  st->done = b.done;
  st->converged = b.converged;
  st->fallback_steps = b.fallback;
  st->no_ascent_steps = b.no_ascent;
  st->nnz_total = b.nnz_total;
  st->cand_total = b.cand_total;
  st->nnz_eval = b.nnz_grad;
  st->cand_eval = b.cand_grad;
}

// The whole solve of one pair (or one evaluation) by one team of blocks.
template <int DP, int MODE, int DPS, int NU, bool TWO>
__device__ void solve_pair(const SolveCfg* __restrict__ cfg, SolveState* __restrict__ st,
                           double* __restrict__ partials, IterRecord* __restrict__ records,
                           Team team, SolveSmem<DPS, NU>& sm, bool join, float* cache,
                           int cap) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned gen = 0;
  double* part_g = partials;
  double* part_s = partials + (size_t)team.size * kPartialStride;
  const long long NW = (long long)team.size * kWarps;
  const long long gw = (long long)team.rank * kWarps + warp;

  if (tid == 0) {
    BlockCtx& b = sm.b;
    TailConst& tc = b.tc;
    for (int a = 0; a < 3; ++a) {
      tc.cX[a] = cfg->cX[a];
      tc.cZ[a] = cfg->cZ[a];
    }
    tc.sigma2 = cfg->sigma2;
    tc.inv_a2 = 1.0 / cfg->a2;
    tc.inv_b2 = 1.0 / cfg->b2;
    tc.eps_pose = cfg->eps_pose;
    tc.eps_grad = cfg->eps_grad;
    tc.src_radius = cfg->src_radius;
    tc.mode = cfg->mode;
    tc.step_order = cfg->step_order;
    tc.max_iters = cfg->max_iters;
    tc.reduce_fp32 = cfg->reduce_fp32;
    tc.wait_polls = cfg->wait_polls;
    tc.join_limit_ns = cfg->join_limit_ns;
    for (int a = 0; a < 3; ++a) tc.cXf[a] = (float)cfg->cX[a];
    tc.inv_a2f = (float)(1.0 / cfg->a2);
    tc.inv_b2f = (float)(1.0 / cfg->b2);
    tc.src_radius_f = (float)cfg->src_radius * (1.0f + 1e-6f);
    tc.eps_pose_f = (float)cfg->eps_pose;
    for (int i = 0; i < 16; ++i) b.P[i] = st->P0[i];
    b.k = 0;
    b.team_rank = team.rank;
    b.team_size = team.size;
    b.plan_level = -1;
    b.plan_filter = 0;
    b.need_plan = 1;
    b.done = cfg->max_iters <= 0 ? 1 : 0;
    b.converged = b.fallback = b.no_ascent = b.have_t_prev = 0;
    b.use_kept = b.collect_kept = b.rebalance = b.use_act = 0;
    b.plan_no = b.check_fit = 0;
    b.cap = cap;
    b.st = st;
    b.t = b.t_prev = 0.0;
    b.pending = 0;
    b.ring_floats = 4 * ring_size<TWO>();
    b.nnz_total = b.cand_total = b.nnz_grad = b.cand_grad = 0;
    b.F = b.xi_norm = 0.0;
    for (int i = 0; i < 6; ++i) b.xi[i] = 0.0;
    for (int i = 0; i < 5; ++i) b.S[i] = 0.0;
    b.r_plan = 0.0;
    b.plan_ell = 0.0;
  }
  __syncthreads();
  if (warp == 0) {
    load_iter(sm.b, iter_word(cfg, 0, lane), lane);
    if (!sm.b.done) begin_iteration(sm.b, lane);
  }
  __syncthreads();
  if (join && !team_join(st, team.size, sm)) {
    if (tid == 0) sm.b.done = 1;   // a team that never assembled runs no iteration
    __syncthreads();
  }
  if (team.rank == 0 && tid == 0) st->t_begin_ns = globaltimer();

  int plans = 0;               // plans built by this solve
  long long* agg = nullptr;    // group totals of the current plan
  while (!sm.b.done) {
    unsigned long long t0 = 0, t1 = 0, t2 = 0, tg1 = 0, tg2 = 0, ts1 = 0, ts2 = 0;
    const bool stamp = records != nullptr && team.rank == 0 && tid == 0;
    if (stamp) t0 = globaltimer();
    const int replan = sm.b.need_plan;
    // a new plan, or the one rebalance of a plan that is being reused: its
    // work split redone with what its first gradient pass recorded (the source
    // groups that kept pairs; with cost_kept > 0 the kept pairs per cluster)
    const int rebalance = !replan && sm.b.rebalance;
    if (replan || rebalance) {
      const ClusterView& cv = cfg->clusters[sm.b.ic.level];
      const int ng = (cv.ncl + 31) / 32;
      if (replan) {
        // the plan's own group totals are added up while its clusters are planned,
        // in one of two buffers in turn; the other is zeroed for the next plan
        // (every block has long read it). The first plan of a solve finds its
        // buffer as the last solve left it and forms the totals after a barrier
        // of their own, as a rebalance does
        agg = cfg->group_agg + (size_t)(plans & 1) * cfg->agg_stride;
        long long* other = cfg->group_agg + (size_t)((plans + 1) & 1) * cfg->agg_stride;
        for (long long i = gw * 32 + lane; i < cfg->agg_stride; i += NW * 32) other[i] = 0;
        for (long long c = gw; c < cv.ncl; c += NW)
          plan_cluster(cfg, sm.b, st, (int)c, lane, sm.ws[warp].seg.xs, sm.ws[warp].seg.pf,
                       sm.ws[warp].seg.fpf, plans > 0 ? agg : nullptr);
        if (!grid_sync(st, gen, &sm.flag, team.size, sm.b.tc.wait_polls)) break;
      }
      if (tid == 0) {
        sm.b.use_kept = rebalance && cfg->cost_kept > 0.f;
        sm.b.use_act = rebalance && sm.b.plan_filter ? sm.b.cost_act : 0;
      }
      __syncthreads();
      if (rebalance || plans == 0) {
        for (long long gi = gw; gi < ng; gi += NW) {
          const int c = (int)gi * 32 + lane;
          int kk, cs4, nch;
          long long w = c < cv.ncl ? cluster_work(cfg, cv, c, &kk, &cs4, &nch, sm.b.use_kept != 0, sm.b.use_act)
                                   : 0;
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(kFull, w, off);
          if (lane == 0) agg[gi] = w;
        }
        if (!grid_sync(st, gen, &sm.flag, team.size, sm.b.tc.wait_polls)) break;
      }
      if (replan) ++plans;
      split_work<DPS, NU>(cfg, sm, tid, team, agg);
      fill_cache<DP, MODE, DPS, NU>(cfg, sm, warp, lane, cache, cap);
      if (tid == 0) {
        sm.b.need_plan = 0;
        sm.b.collect_kept = replan && (cfg->cost_kept > 0.f || sm.b.plan_filter);
        sm.b.rebalance = sm.b.collect_kept;
        if (rebalance) sm.b.rebalance = 0;
      }
      __syncthreads();
    }
    if (stamp) t1 = globaltimer();
    // ---- gradient pass ----
    run_pass<false, DP, MODE, DPS, NU, TWO>(cfg, sm, part_g, cache, cap);
    if (stamp) tg1 = globaltimer();
    if (!grid_sync_reduce(st, gen, sm, part_g, 9, team.size, [&](int ln) {
          if (sm.b.n_workers == kWarps && sm.b.pending) pending_step(sm.b, ln);
        }))
      break;
    if (stamp) tg2 = globaltimer();
    if (warp == 0) {
      if (lane == 0) sm.b.collect_kept = 0;
      gradient_direction(sm.b, sm.sums, lane);
    }
    __syncthreads();
    if (stamp) t2 = globaltimer();
    // ---- step pass ----
    run_pass<true, DP, MODE, DPS, NU, TWO>(cfg, sm, part_s, cache, cap);
    if (stamp) ts1 = globaltimer();
    // the next iteration's constants, on their way while the block waits
    const unsigned icw = iter_word(cfg, min(sm.b.k + 1, sm.b.tc.max_iters - 1), lane);
    // (the gradient's totals stay in sm.sums until the reduction)
    if (!grid_sync_reduce(st, gen, sm, part_s, 7, team.size,
                          [&](int ln) {
                            if (sm.b.n_workers == kWarps) gradient_fp64(sm.b, sm.sums, ln);
                          }))
      break;
    if (stamp) ts2 = globaltimer();
    if (warp == 0) {
      BlockCtx& b = sm.b;
      const int k = b.k;
      const unsigned long long pairs_before = b.nnz_total;
      finish_step(b, sm.sums, lane);
      if (stamp && k < b.tc.max_iters) {
        IterRecord& r = records[k];
        r.ell = b.ic.ell;
        r.t_plan_ns = (float)(t1 - t0);
        r.t_grad_ns = (float)(t2 - t1);
        r.t_step_ns = (float)(globaltimer() - t2);
        r.t_grad_pass_ns = (float)(tg1 - t1);
        r.t_grad_sync_ns = (float)(tg2 - t1);
        r.t_step_pass_ns = (float)(ts1 - t2);
        r.t_step_sync_ns = (float)(ts2 - t2);
        r.replanned = replan;
        r.grad_pairs = (long long)b.nnz_grad;
        r.step_pairs = (long long)(b.nnz_total - pairs_before - b.nnz_grad);
        r.grad_candidates = (long long)b.cand_grad;
      }
      __syncwarp();
      if (!b.done) {
        load_iter(b, icw, lane);
        begin_iteration(b, lane);
      }
    }
    __syncthreads();
  }
  if (team.rank == 0 && tid == 0) {
    form_step_sums(sm.b);
    // a single solve's result goes straight to the host's pinned copy
    SolveState* out = st->host ? st->host : st;
    publish(out, sm.b);
    out->t_begin_ns = st->t_begin_ns;
    out->t_end_ns = globaltimer();
  }
  __syncthreads();
}

// The whole solve (or one evaluation) in one cooperative launch: the grid is
// one team.
template <int DP, int MODE>
__global__ void __launch_bounds__(kThreads, CVO_SOLVE_MIN_BLOCKS)
solve_kernel(const SolveCfg* __restrict__ cfg, SolveState* __restrict__ st,
             double* __restrict__ partials, IterRecord* __restrict__ records, int cache_cap) {
  constexpr int DPS = DP > 0 ? DP : 1;
  constexpr int NU = 2;
  __shared__ SolveSmem<DPS, NU> sm;
  extern __shared__ float4 dyn_smem[];
  solve_pair<DP, MODE, DPS, NU, false>(cfg, st, partials, records, Team{(int)blockIdx.x, (int)gridDim.x},
                                sm, false, reinterpret_cast<float*>(dyn_smem), cache_cap);
}

__device__ __forceinline__ unsigned long long ld_acquire_sys_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed_sys_u64(const void* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_sys_s32(int* p, int v) {
  asm volatile("st.release.sys.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Entry fields read at system scope: the entries of a served queue live in
// host memory that the host appends to while the kernel runs.
__device__ QueueEntry load_entry(const QueueEntry* e) {
  static_assert(sizeof(QueueEntry) == 40, "QueueEntry layout");
  QueueEntry r;
  unsigned long long w[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) w[i] = ld_relaxed_sys_u64(reinterpret_cast<const unsigned long long*>(e) + i);
  memcpy(&r, w, sizeof(r));
  return r;
}

// Claim the next slot (thread 0): slots are handed out in order, so every
// slot of an entry is claimed before any slot of a later one. A team whose
// first blocks start before the rest have claimed their slots waits at its
// first barrier; the entries ahead of it never wait on later ones, so the
// blocks they hold come free in bounded time and staff it.
__device__ void claim_slot(const QueueEntry* entries, const QueueCtl* ctl,
                           unsigned long long* head, int* kstatus,
                           unsigned long long idle_limit_ns, long long* slot_out,
                           int* entry_out) {
  const unsigned long long t_start = globaltimer();
  unsigned polls = 0;
  for (;;) {
    const unsigned long long tail = ld_acquire_sys_u64(&ctl->tail);
    const unsigned long long h = atomicAdd(head, 0ull);
    if (h < tail) {
      if (atomicCAS(head, h, h + 1) != h) continue;
      // the entry holding slot h: the last one whose first slot is <= h
      const unsigned long long ne = ld_relaxed_sys_u64(&ctl->n_entries);
      long long lo = 0, hi = (long long)ne;   // invariant: entry lo starts at or before h
      while (hi - lo > 1) {
        const long long mid = (lo + hi) >> 1;
        const QueueEntry em = load_entry(entries + mid);
        if ((unsigned long long)em.slot0 <= h) lo = mid;
        else hi = mid;
      }
      *slot_out = (long long)h;
      *entry_out = (int)lo;
      return;
    }
    if (ld_acquire_sys_u64(&ctl->stop) != 0) break;
    if ((++polls & 63u) == 0 && globaltimer() - t_start > idle_limit_ns) {
      atomicOr(kstatus, (int)kStatusIdleTimeout);
      break;
    }
    __nanosleep(1024);
  }
  *slot_out = -1;
  *entry_out = -1;
}

// Solve results for the host, read at L2 (the team's first block published
// them), the done flag last (release at system scope).
__device__ void write_result(const SolveState* st, PairResult* out) {
  for (int i = 0; i < 16; ++i) out->P[i] = __ldcg(&st->P[i]);
  out->F = __ldcg(&st->F);
  out->t = __ldcg(&st->t);
  out->ell = __ldcg(&st->ell);
  out->device_ms = (double)(__ldcg(&st->t_end_ns) - __ldcg(&st->t_begin_ns)) * 1e-6;
  out->pair_evals = (long long)__ldcg(&st->nnz_total);
  out->candidates = (long long)__ldcg(&st->cand_total);
  out->iters = __ldcg(&st->iter);
  out->converged = __ldcg(&st->converged);
  out->fallback_steps = __ldcg(&st->fallback_steps);
  out->no_ascent_steps = __ldcg(&st->no_ascent_steps);
  out->status = __ldcg(&st->status);
  __threadfence_system();
  st_release_sys_s32(&out->done, 1);
}

// Many pairs in one persistent cooperative launch. Blocks claim slots of a
// queue of entries; the blocks holding the slots of one entry form its team.
template <int DP, int MODE>
__global__ void __launch_bounds__(kThreads, CVO_SOLVE_MIN_BLOCKS)
queue_kernel(const QueueEntry* __restrict__ entries, const QueueCtl* __restrict__ ctl,
             unsigned long long* __restrict__ head, int* __restrict__ kstatus,
             unsigned long long idle_limit_ns, int cache_cap) {
  constexpr int DPS = DP > 0 ? DP : 1;
  constexpr int NU = 2;
  __shared__ SolveSmem<DPS, NU> sm;
  extern __shared__ float4 dyn_smem[];
  for (;;) {
    if (threadIdx.x == 0) {
      long long slot;
      int e;
      claim_slot(entries, ctl, head, kstatus, idle_limit_ns, &slot, &e);
      sm.q_slot = slot;
      sm.q_entry = e;
    }
    __syncthreads();
    if (sm.q_slot < 0) break;
    const QueueEntry en = load_entry(entries + sm.q_entry);
    const Team team{(int)(sm.q_slot - en.slot0), en.team};
    solve_pair<DP, MODE, DPS, NU, true>(en.cfg, en.st, en.partials, nullptr, team, sm, true,
                                  reinterpret_cast<float*>(dyn_smem), cache_cap);
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned left = atomicAdd(&en.st->leave_count, 1u);
      if (left == (unsigned)en.team - 1 && en.out) {
        __threadfence();
        write_result(en.st, en.out);
      }
    }
    __syncthreads();
  }
}

// Dynamic shared memory of the plan cache: what CVO_SOLVE_MIN_BLOCKS blocks
// per SM leave of the SM's shared memory after their static shared memory,
// in equal shares of whole 64 bytes per warp (set once per kernel instantiation).
struct CacheCfg {
  int bytes = 0, cap = 0;   // cap: floats per warp
  cudaError_t err = cudaSuccess;
};

template <int DP, int MODE>
const CacheCfg& cache_cfg() {
  static const CacheCfg cfg = [] {
    CacheCfg c;
    int dev = 0, smem_sm = 0, reserved = 0;
    cudaFuncAttributes fa{};
    c.err = cudaGetDevice(&dev);
    if (c.err == cudaSuccess)
      c.err = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (c.err == cudaSuccess)
      c.err = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (c.err == cudaSuccess) c.err = cudaFuncGetAttributes(&fa, solve_kernel<DP, MODE>);
    if (c.err != cudaSuccess) return c;
    const int slot = 32 * (4 + DP);   // slot_floats
    const int avail = smem_sm / CVO_SOLVE_MIN_BLOCKS - reserved - (int)fa.sharedSizeBytes;
    c.cap = std::max(0, std::min(kCacheSlots * slot, avail / kWarps / 64 * 16));
    if (c.cap < 4 * 128) {   // ring_size, twice a single solve's
      c.err = cudaErrorInvalidConfiguration;
      return c;
    }
    c.bytes = c.cap * kWarps * (int)sizeof(float);
    if (c.bytes > 0) {
      c.err = cudaFuncSetAttribute(solve_kernel<DP, MODE>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, c.bytes);
      if (c.err == cudaSuccess)
        c.err = cudaFuncSetAttribute(queue_kernel<DP, MODE>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, c.bytes);
    }
    return c;
  }();
  return cfg;
}

template <int DP, int MODE>
cudaError_t launch_solve_t(int nblocks, const SolveCfg* cfg, SolveState* st, double* partials,
                           IterRecord* records, cudaStream_t s) {
  const CacheCfg& cc = cache_cfg<DP, MODE>();
  if (cc.err != cudaSuccess) return cc.err;
  int cap = cc.cap;
  void* args[] = {(void*)&cfg, (void*)&st, (void*)&partials, (void*)&records, (void*)&cap};
  return cudaLaunchCooperativeKernel((const void*)solve_kernel<DP, MODE>, dim3(nblocks),
                                     dim3(kThreads), args, (size_t)cc.bytes, s);
}

template <int DP, int MODE>
cudaError_t launch_queue_t(int nblocks, const QueueEntry* entries, const QueueCtl* ctl,
                           unsigned long long* head, int* kstatus, unsigned long long idle_ns,
                           cudaStream_t s) {
  const CacheCfg& cc = cache_cfg<DP, MODE>();
  if (cc.err != cudaSuccess) return cc.err;
  int cap = cc.cap;
  void* args[] = {(void*)&entries, (void*)&ctl,     (void*)&head,
                  (void*)&kstatus, (void*)&idle_ns, (void*)&cap};
  return cudaLaunchCooperativeKernel((const void*)queue_kernel<DP, MODE>, dim3(nblocks),
                                     dim3(kThreads), args, (size_t)cc.bytes, s);
}

template <int DP, int MODE>
int blocks_per_sm_t() {
  const CacheCfg& cc = cache_cfg<DP, MODE>();
  if (cc.err != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, solve_kernel<DP, MODE>, kThreads,
                                                    (size_t)cc.bytes) != cudaSuccess)
    return 0;
  return n;
}

// Launchers of one feature layout (explicitly instantiated, one translation
// unit per feature width, so that the variants compile in parallel).
template <int DP>
cudaError_t launch_solve_dp(int color_mode, int nblocks, const SolveCfg* cfg, SolveState* st,
                            double* partials, IterRecord* records, cudaStream_t s) {
  if constexpr (DP == 0) {
    return launch_solve_t<0, kColorNone>(nblocks, cfg, st, partials, records, s);
  } else {
    switch (color_mode) {
      case kColorKernel:
        return launch_solve_t<DP, kColorKernel>(nblocks, cfg, st, partials, records, s);
      case kColorDot:
        return launch_solve_t<DP, kColorDot>(nblocks, cfg, st, partials, records, s);
      case kColorKernel | kFeatBf16:
        return launch_solve_t<DP, kColorKernel | kFeatBf16>(nblocks, cfg, st, partials, records, s);
      case kColorDot | kFeatBf16:
        return launch_solve_t<DP, kColorDot | kFeatBf16>(nblocks, cfg, st, partials, records, s);
      default:
        return cudaErrorInvalidValue;
    }
  }
}

template <int DP>
cudaError_t launch_queue_dp(int color_mode, int nblocks, const QueueEntry* entries,
                            const QueueCtl* ctl, unsigned long long* head, int* kstatus,
                            unsigned long long idle_limit_ns, cudaStream_t s) {
  if constexpr (DP == 0) {
    return launch_queue_t<0, kColorNone>(nblocks, entries, ctl, head, kstatus, idle_limit_ns, s);
  } else {
    switch (color_mode) {
      case kColorKernel:
        return launch_queue_t<DP, kColorKernel>(nblocks, entries, ctl, head, kstatus,
                                                idle_limit_ns, s);
      case kColorDot:
        return launch_queue_t<DP, kColorDot>(nblocks, entries, ctl, head, kstatus, idle_limit_ns,
                                             s);
      case kColorKernel | kFeatBf16:
        return launch_queue_t<DP, kColorKernel | kFeatBf16>(nblocks, entries, ctl, head, kstatus,
                                                            idle_limit_ns, s);
      case kColorDot | kFeatBf16:
        return launch_queue_t<DP, kColorDot | kFeatBf16>(nblocks, entries, ctl, head, kstatus,
                                                         idle_limit_ns, s);
      default:
        return cudaErrorInvalidValue;
    }
  }
}

template <int DP>
int blocks_per_sm_dp(int color_mode) {
  if constexpr (DP == 0) {
    return blocks_per_sm_t<0, kColorNone>();
  } else {
    switch (color_mode) {
      case kColorKernel: return blocks_per_sm_t<DP, kColorKernel>();
      case kColorDot: return blocks_per_sm_t<DP, kColorDot>();
      case kColorKernel | kFeatBf16: return blocks_per_sm_t<DP, kColorKernel | kFeatBf16>();
      case kColorDot | kFeatBf16: return blocks_per_sm_t<DP, kColorDot | kFeatBf16>();
      default: return 0;
    }
  }
}

}  // namespace

}  // namespace cvo
