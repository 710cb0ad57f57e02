// Gradient pass without any device allocation: the all-pairs form of the
// gradient pass (every target point against every source point, same cutoff
// test and same FP32 pair arithmetic as the solve kernel), whose block
// partials live in a fixed, file-scope device array instead of memory the
// library allocates. For callers that must not allocate device memory during
// a call: code running where cudaMalloc is not allowed or not wanted (inside
// a real-time loop with a frozen memory footprint, or a host that owns all
// device memory through its own pool).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/cvo.h"
#include "cvo_internal.cuh"
#include "packed_f32.cuh"

namespace {

using namespace cvo;

constexpr int kNaThreads = 128;
constexpr int kNaSrc = 2 * kNaThreads; // source points of a work item, two per thread
constexpr int kNaTile = 256;           // its target points at most
constexpr int kNaMaxBlocks = 608;      // partial slots in the static scratch
constexpr int kNaGrid = 4 * 152;       // blocks of a full launch: four to each of GB300's SMs
constexpr int kNaQueue = 2048;         // pairs a warp appends to its queue at once
constexpr int kNaStride = 8;           // F, omega'(3), v(3), kept pairs
constexpr int kNaMaxDevices = 64;
constexpr int kNaFlush = 256;          // pairs a lane adds in FP32 before its sums go to FP64
                                       //   (tested once a round, which may add 128 more)
constexpr int kNaSample = 8192;        // source points from which a launch samples the clouds, and
constexpr int kNaDense = 20;           //   the kept pairs of 128 from which it evaluates in place
constexpr float kNaFar = 1e18f;        // coordinate of the slots past the ends
constexpr float kNaWild = 1e15f;       // in place, coordinates from here on go pair by pair

// Scratch shared by every call on a device: kNaMaxBlocks block partials
// (38 KB). Held by every GPU that loads the library until the process exits.
__device__ __align__(256) double g_na_partials[kNaMaxBlocks * kNaStride];

static_assert(kNaGrid <= kNaMaxBlocks, "one partial slot per block");
static_assert(kNaSrc <= 256 && kNaTile <= 256, "a queued pair packs both indices in 16 bits");

std::mutex g_na_mu;
double* g_na_addr[kNaMaxDevices] = {};  // device address of g_na_partials per device
thread_local std::string g_na_err;

struct NaArgs {
  double R[9], T[3];       // pose P = [R T]
  float A;                 // log2(e) / (2 ell^2)
  float rc2;               // cutoff radius squared
  float fscale;            // feature pre-scale
  int n, m, D;
  int tile;                // target points of a work item, a multiple of 32
};

template <int DP>
struct NaSmem {
  alignas(16) float z[3 + DP][kNaSrc];     // transformed source points and scaled features
  alignas(16) float x[3 + DP][kNaTile];    // target points relative to the first one, features
  unsigned short queue[kNaThreads / 32][32 + kNaQueue];   // kept pairs: target | source << 8
  double red[7][kNaThreads];
  unsigned long long cnt[kNaThreads / 32];
  float R[9], T[3], x0[3], z0[3];
};

// One kept pair: target t against source s of the staged tiles.
template <int DP, int MODE>
__device__ __forceinline__ void na_pair(const NaSmem<DP>& sm, int t, int s, float A, float acc[7]) {
  const float zx = sm.z[0][s], zy = sm.z[1][s], zz = sm.z[2][s];
  const float ex = sm.x[0][t] - zx, ey = sm.x[1][t] - zy, ez = sm.x[2][t] - zz;
  const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
  float w;
  if (MODE == kColorKernel) {
    float q = 0.f;
#pragma unroll
    for (int d = 0; d < DP; ++d) {
      const float df = sm.x[3 + d][t] - sm.z[3 + d][s];
      q = fmaf(df, df, q);
    }
    w = ex2_approx(-fmaf(A, d2, q));
  } else if (MODE == kColorDot) {
    float c = 0.f;
#pragma unroll
    for (int d = 0; d < DP; ++d) c = fmaf(sm.x[3 + d][t], sm.z[3 + d][s], c);
    w = ex2_approx(-A * d2) * c;
  } else {
    w = ex2_approx(-A * d2);
  }
  const float vx = w * ex, vy = w * ey, vz = w * ez;
  acc[0] += w;
  acc[1] += zy * vz - zz * vy;   // omega' += z~' x w e, v += w e
  acc[2] += zz * vx - zx * vz;
  acc[3] += zx * vy - zy * vx;
  acc[4] += vx;
  acc[5] += vy;
  acc[6] += vz;
}

// A warp's part of a work item in place: the lane's two source points against every
// target, two to a packed operation, the weight of a pair that is not kept selected to
// zero. Its products are then zero as long as the coordinates are below kNaWild, and the
// slots past the ends are beyond a cutoff below kNaWild; an item with larger ones, or a
// NaN, goes pair by pair. Adds the lane's sums F, omega', v to acc64 and returns its kept
// pairs.
template <int DP, int MODE>
__device__ __forceinline__ unsigned na_dense(const NaSmem<DP>& sm, int warp, int lane, int tn, int ms,
                                             float rc2, float A, double acc64[7]) {
  const int s0 = warp * 64 + lane;
  bool wild = !(rc2 < kNaWild * kNaWild);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    wild = wild || (s0 < ms && !(fabsf(sm.z[c][s0]) < kNaWild)) ||
           (s0 + 32 < ms && !(fabsf(sm.z[c][s0 + 32]) < kNaWild));
    for (int t = lane; t < tn; t += 32) wild = wild || !(fabsf(sm.x[c][t]) < kNaWild);
  }
  if (__any_sync(0xffffffffu, wild)) {
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    unsigned cnt = 0;
    for (int s = s0; s < min(ms, s0 + 64); s += 32) {
      for (int t = 0; t < tn; ++t) {
        const float ex = sm.x[0][t] - sm.z[0][s], ey = sm.x[1][t] - sm.z[1][s],
                    ez = sm.x[2][t] - sm.z[2][s];
        if (!(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= rc2)) continue;
        ++cnt;
        na_pair<DP, MODE>(sm, t, s, A, acc);
      }
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) acc64[k] += (double)acc[k];
    return cnt;
  }
  f32x2 Z[2][3 + DP];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int c = 0; c < 3 + DP; ++c) Z[h][c] = dup2(sm.z[c][s0 + 32 * h]);
  }
  float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const f32x2 A2 = dup2(A);
  f32x2 sum[2][4] = {{0ull, 0ull, 0ull, 0ull}, {0ull, 0ull, 0ull, 0ull}};
  unsigned cnt = 0;
  for (int t = 0; t < tn; t += 4) {
    ulonglong2 X[3 + DP];
#pragma unroll
    for (int c = 0; c < 3 + DP; ++c) X[c] = *reinterpret_cast<const ulonglong2*>(&sm.x[c][t]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const f32x2 ex = sub2(p ? X[0].y : X[0].x, Z[h][0]);
        const f32x2 ey = sub2(p ? X[1].y : X[1].x, Z[h][1]);
        const f32x2 ez = sub2(p ? X[2].y : X[2].x, Z[h][2]);
        const f32x2 d2 = fma2(ex, ex, fma2(ey, ey, mul2(ez, ez)));
        f32x2 q = 0ull;   // appearance: sum of squared differences, or inner product
#pragma unroll
        for (int d = 0; d < DP; ++d) {
          const f32x2 f = p ? X[3 + d].y : X[3 + d].x;
          if (MODE == kColorKernel) {
            const f32x2 df = sub2(f, Z[h][3 + d]);
            q = fma2(df, df, q);
          } else if (MODE == kColorDot) {
            q = fma2(f, Z[h][3 + d], q);
          }
        }
        float d20, d21, e0, e1;
        unpack2(d2, d20, d21);
        const bool k0 = d20 <= rc2, k1 = d21 <= rc2;
        unpack2(MODE == kColorKernel ? fma2(A2, d2, q) : mul2(A2, d2), e0, e1);
        float w0 = ex2_approx(-e0), w1 = ex2_approx(-e1);
        if (MODE == kColorDot) {
          float c0, c1;
          unpack2(q, c0, c1);
          w0 *= c0;
          w1 *= c1;
        }
        const f32x2 w = pack2(k0 ? w0 : 0.f, k1 ? w1 : 0.f);
        cnt += (k0 ? 1u : 0u) + (k1 ? 1u : 0u);
        sum[h][0] = add2(sum[h][0], w);
        sum[h][1] = fma2(w, ex, sum[h][1]);
        sum[h][2] = fma2(w, ey, sum[h][2]);
        sum[h][3] = fma2(w, ez, sum[h][3]);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {   // omega' += z~' x E, v += E, E = sum w e
    const float zx = sm.z[0][s0 + 32 * h], zy = sm.z[1][s0 + 32 * h], zz = sm.z[2][s0 + 32 * h];
    const float Ex = sum2(sum[h][1]), Ey = sum2(sum[h][2]), Ez = sum2(sum[h][3]);
    acc[0] += sum2(sum[h][0]);
    acc[1] += zy * Ez - zz * Ey;
    acc[2] += zz * Ex - zx * Ez;
    acc[3] += zx * Ey - zy * Ex;
    acc[4] += Ex;
    acc[5] += Ey;
    acc[6] += Ez;
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) acc64[k] += (double)acc[k];
  return cnt;
}

// The all-pairs gradient pass. A work item is 256 source points against a tile
// of at most 256 target points; blocks take items in turn and keep one partial
// sum each, so that small clouds spread over many SMs (a thread per source point
// with every target in turn ran 3 blocks for 600 points and 79 for 20000).
// Most pairs are out of range and the points come in no particular order, so
// testing and evaluating are kept apart: a lane holds two source points, tests
// them against 64 targets (broadcast from shared memory, two per packed
// operation: bound by the FMA pipe at six cycles of a scheduler for 32 tests)
// and notes the kept ones in masks; the warp appends the pairs to its queue
// and evaluates 32 queued pairs at a time, one per lane, whatever points they
// belong to: F, sum w z~ x e and sum w e need no order. Evaluating in place
// would run a body for every group of tests in which any lane keeps a pair,
// which at 1% kept is nearly all of them. 20000 x 20000 points at 1.3% kept: 160
// us against 1274 us before (the tests alone are 60 us of the FMA pipe, the queued
// pairs' scattered shared loads about 30).
// Where most pairs are kept the queue is the dearer way (20000 x 20000 points, five
// features, all kept: 2220 us, against 1660 of a thread per source point), so a launch
// samples the clouds first and evaluates every item in place from a sixth kept on: 335 us
// whatever is kept, which the queue passes at 14% (328 us; 23%: 471). The choice is the
// launch's, not an item's: a choice within the items, by a sample, the first round or the
// item before, cost the queue 1 to 5% in registers and code. Below kNaSample source
// points nothing is sampled (it takes 1 us): a kept pair costs the queue 5.5 ps, and a
// thread per source point took 83 ns per target, so the queue loses from 15000 on.
// Coordinates are taken relative to the first target point x0 (one rounding of
// the difference), so FP32 pair arithmetic never subtracts large coordinates.
template <int DP, int MODE>
__global__ void __launch_bounds__(kNaThreads, 4)
na_grad_kernel(const float* __restrict__ x, const float* __restrict__ fx,
               const float* __restrict__ z, const float* __restrict__ fz, NaArgs a,
               double* __restrict__ partials) {
  __shared__ NaSmem<DP> sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    if (tid != r) continue;
    double tr = a.T[r] - (double)x[r];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sm.R[3 * r + c] = (float)a.R[3 * r + c];
      tr += a.R[3 * r + c] * (double)z[c];
    }
    sm.T[r] = (float)tr;   // z~' = R (z - z0) + T', T' = R z0 + T - x0
    sm.x0[r] = x[r];
    sm.z0[r] = z[r];
  }
  unsigned short* queue = sm.queue[warp];
  float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  double acc64[7] = {0, 0, 0, 0, 0, 0, 0};
  // kept pairs: up to n x m = 2^44 over a block, so 64-bit
  unsigned long long cnt = 0;
  int added = 0;
  const auto evaluate = [&](unsigned e) {
    na_pair<DP, MODE>(sm, (int)(e & 255u), (int)(e >> 8), a.A, acc);
  };
  const int nS = (a.m + kNaSrc - 1) / kNaSrc, nT = (a.n + a.tile - 1) / a.tile;
  const long long items = (long long)nS * nT;
  // The item's source points from j0 on and target points from i0 on.
  const auto stage = [&](int j0, int i0) {
    for (int k = tid; k < kNaSrc; k += kNaThreads) {
      const int j = j0 + k;
      float zx = -kNaFar, zy = -kNaFar, zz = -kNaFar;   // past the end: beyond every cutoff
      if (j < a.m) {
        const float px = z[3 * (size_t)j] - sm.z0[0], py = z[3 * (size_t)j + 1] - sm.z0[1],
                    pz = z[3 * (size_t)j + 2] - sm.z0[2];
        const float *R = sm.R, *T = sm.T;
        zx = fmaf(R[0], px, fmaf(R[1], py, fmaf(R[2], pz, T[0])));
        zy = fmaf(R[3], px, fmaf(R[4], py, fmaf(R[5], pz, T[1])));
        zz = fmaf(R[6], px, fmaf(R[7], py, fmaf(R[8], pz, T[2])));
      }
      sm.z[0][k] = zx;
      sm.z[1][k] = zy;
      sm.z[2][k] = zz;
#pragma unroll
      for (int d = 0; d < DP; ++d)
        sm.z[3 + d][k] = j < a.m && d < a.D ? fz[(size_t)a.D * j + d] * a.fscale : 0.f;
    }
    for (int k = tid; k < a.tile; k += kNaThreads) {
      const int i = i0 + k;
#pragma unroll
      for (int c = 0; c < 3; ++c)
        sm.x[c][k] = i < a.n ? x[3 * (size_t)i + c] - sm.x0[c] : kNaFar;
#pragma unroll
      for (int d = 0; d < DP; ++d)
        sm.x[3 + d][k] = i < a.n && d < a.D ? fx[(size_t)a.D * i + d] * a.fscale : 0.f;
    }
  };
  // A sample of 128 pairs from all over the clouds, the same for every block: where a
  // sixth or more are kept, every item is evaluated in place.
  int sample = 0;
  if (a.m >= kNaSample) {
    __syncthreads();   // R and T are there
    const long long si = (long long)(tid * 37 & 127) * a.n >> 7, sj = (long long)tid * a.m >> 7;
    float e[3], p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) p[c] = z[3 * sj + c] - sm.z0[c];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      e[c] = x[3 * si + c] - sm.x0[c] -
             fmaf(sm.R[3 * c], p[0], fmaf(sm.R[3 * c + 1], p[1], fmaf(sm.R[3 * c + 2], p[2], sm.T[c])));
    sample = __syncthreads_count(fmaf(e[0], e[0], fmaf(e[1], e[1], e[2] * e[2])) <= a.rc2);
  }
  const bool in_place = sample >= kNaDense;
  if (in_place) {
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
      const int j0 = (int)(it / nT) * kNaSrc, i0 = (int)(it % nT) * a.tile;
      __syncthreads();   // the tiles of the previous item are free
      stage(j0, i0);
      __syncthreads();
      if (j0 + warp * 64 < a.m)
        cnt += na_dense<DP, MODE>(sm, warp, lane, min(a.tile, a.n - i0), a.m - j0, a.rc2, a.A, acc64);
    }
  }
  for (long long it = in_place ? items : blockIdx.x; it < items; it += gridDim.x) {
    const int j0 = (int)(it / nT) * kNaSrc, i0 = (int)(it % nT) * a.tile;
    const int tn = min(a.tile, a.n - i0);
    __syncthreads();   // the tiles of the previous item are free (and R, T are there)
    stage(j0, i0);
    __syncthreads();
    if (j0 + warp * 64 >= a.m) continue;   // a warp past the last source point
    f32x2 Z[2][3];
    bool zv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = warp * 64 + 32 * h + lane;
      zv[h] = j0 + k < a.m;
#pragma unroll
      for (int c = 0; c < 3; ++c) Z[h][c] = dup2(sm.z[c][k]);
    }
    int queued = 0;   // the same in every lane
    for (int t0 = 0; t0 < tn; t0 += 64) {
      // the lane's kept pairs: bit k of keep[h][w] is source h, target t0 + 32 w + k
      unsigned keep[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        if (t0 + 32 * w >= tn) break;
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          const int t = t0 + 32 * w + k;
          const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(&sm.x[0][t]);
          const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(&sm.x[1][t]);
          const ulonglong2 W = *reinterpret_cast<const ulonglong2*>(&sm.x[2][t]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const f32x2 ex = sub2(p ? X.y : X.x, Z[h][0]);
              const f32x2 ey = sub2(p ? Y.y : Y.x, Z[h][1]);
              const f32x2 ez = sub2(p ? W.y : W.x, Z[h][2]);
              const f32x2 d2 = fma2(ex, ex, fma2(ey, ey, mul2(ez, ez)));
              float d20, d21;
              unpack2(d2, d20, d21);
              if (d20 <= a.rc2) keep[h][w] |= 1u << (k + 2 * p);
              if (d21 <= a.rc2) keep[h][w] |= 1u << (k + 2 * p + 1);
            }
          }
        }
        // points past the ends never count, whatever the cutoff
        const int left = tn - t0 - 32 * w;
        const unsigned valid = left < 32 ? (1u << left) - 1u : 0xffffffffu;
        keep[0][w] &= zv[0] ? valid : 0u;
        keep[1][w] &= zv[1] ? valid : 0u;
      }
      const int n0 = __popc(keep[0][0]) + __popc(keep[1][0]);
      const int n1 = __popc(keep[0][1]) + __popc(keep[1][1]);
      cnt += (unsigned)(n0 + n1);
      const int total = __reduce_add_sync(0xffffffffu, n0 + n1);
      if (total == 0) continue;
      // both words at once, or, should they not fit the queue, one after the other
      const bool both = total <= kNaQueue;
      for (int w0 = 0; w0 < 2; ++w0) {
        const int mine = both ? n0 + n1 : w0 ? n1 : n0;
        int pos = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, pos, off);
          if (lane >= off) pos += v;
        }
        const int end = queued + __shfl_sync(0xffffffffu, pos, 31);
        pos += queued - mine;
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          if (!both && w != w0) continue;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const unsigned src = (unsigned)(warp * 64 + 32 * h + lane) << 8 | (unsigned)(t0 + 32 * w);
            for (unsigned m = keep[h][w]; m != 0u; m &= m - 1u)
              queue[pos++] = (unsigned short)(src + (unsigned)(__ffs(m) - 1));
          }
        }
        queued = end;
        __syncwarp();
        while (queued >= 32) {   // full rounds from the end of the queue; fewer than 32 pairs stay
          queued -= 32;
          evaluate(queue[queued + lane]);
          ++added;
        }
        __syncwarp();
        if (both) break;
      }
      if (added >= kNaFlush) {
#pragma unroll
        for (int k = 0; k < 7; ++k) {
          acc64[k] += (double)acc[k];
          acc[k] = 0.f;
        }
        added = 0;
      }
    }
    if (lane < queued) evaluate(queue[lane]);
    ++added;
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) sm.red[k][tid] = acc64[k] + (double)acc[k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
  if (lane == 0) sm.cnt[warp] = cnt;
  __syncthreads();
  // 16 threads per value, 8 lanes' sums each, in a fixed order
  const int k = tid >> 4, part = tid & 15;
  double v = 0.0;
  if (k < 7) {
#pragma unroll
    for (int q = 0; q < kNaThreads / 16; ++q) v += sm.red[k][q * 16 + part];
  }
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off, 16);
  if (part == 0) {
    if (k == 7) {
      unsigned long long c = 0;
      for (int w = 0; w < kNaThreads / 32; ++w) c += sm.cnt[w];
      v = (double)c;
    }
    partials[(size_t)blockIdx.x * kNaStride + k] = v;
  }
}

// Fixed-order reduction of the block partials (one warp per value: on GB300 an
// FP64 instruction costs a warp the same with one lane or 32, and one thread
// adding 79 x 8 partials in turn took longer than the pass over 2000 points)
// and the metric gradient.
__global__ void __launch_bounds__(32 * kNaStride)
na_finish_kernel(const double* __restrict__ partials, int nblocks, const float* __restrict__ x,
                 double sigma2, double inv_l2, double a2, double b2, double* __restrict__ out) {
  __shared__ double s[kNaStride];
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  double v = 0.0;
  for (int b = lane; b < nblocks; b += 32) v += partials[(size_t)b * kNaStride + k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if (lane == 0) s[k] = v;
  __syncthreads();
  const int i = threadIdx.x;
  if (i == 0) out[0] = sigma2 * s[0];
  if (i == 7) out[7] = s[7];
  if (i >= 1 && i < 4) {
    const int c1 = i % 3, c2 = (i + 1) % 3;   // the two axes after axis i - 1
    const double cxv = (double)x[c1] * s[4 + c2] - (double)x[c2] * s[4 + c1];
    out[i] = sigma2 * (s[i] + cxv) * inv_l2 / a2;
  }
  if (i >= 4 && i < 7) out[i] = sigma2 * s[i] * inv_l2 / b2;
}

template <int DP, int MODE>
cudaError_t na_launch(int nblocks, const float* x, const float* fx, const float* z, const float* fz,
                      const NaArgs& a, double* partials, cudaStream_t s) {
  na_grad_kernel<DP, MODE><<<nblocks, kNaThreads, 0, s>>>(x, fx, z, fz, a, partials);
  return cudaGetLastError();
}

int na_fail(int code, const char* msg) {
  g_na_err = msg;
  return code;
}

}  // namespace

extern "C" int cvo_eval_gradient_static(const float* d_x, const float* d_fx, int64_t n,
                                        const float* d_z, const float* d_fz, int64_t m,
                                        const cvo_params* params, const double P[16], double ell,
                                        double* d_out, void* stream) {
  g_na_err.clear();
  if (!d_x || !d_z || !d_out || !params || !P)
    return na_fail(CVO_ERR_INVALID_ARG, "NULL pointer argument");
  if (n < 1 || m < 1 || n > kMaxPoints || m > kMaxPoints)
    return na_fail(CVO_ERR_INVALID_ARG, "point count outside [1, 2^22]");
  const cvo_params& p = *params;
  if (!(ell > 0.0) || !std::isfinite(ell) || !(p.kcut > 0.0 && p.kcut < 1.0) || !(p.sigma > 0.0) ||
      !(p.a2 > 0.0) || !(p.b2 > 0.0) || p.feat_dim < 0 || p.feat_dim > CVO_MAX_FEAT)
    return na_fail(CVO_ERR_INVALID_ARG, "invalid parameters");
  if (p.color_mode != CVO_COLOR_NONE && p.color_mode != CVO_COLOR_KERNEL &&
      p.color_mode != CVO_COLOR_DOT)
    return na_fail(CVO_ERR_INVALID_ARG, "color_mode must be CVO_COLOR_NONE, _KERNEL or _DOT");
  if (p.color_mode == CVO_COLOR_KERNEL && p.feat_dim > 0 &&
      !(p.ell_color > 0.0 && std::isfinite(p.ell_color)))
    return na_fail(CVO_ERR_INVALID_ARG, "ell_color must be finite and > 0");
  if (p.color_mode == CVO_COLOR_DOT && p.feat_dim > 0 &&
      !(p.color_scale > 0.0 && std::isfinite(p.color_scale)))
    return na_fail(CVO_ERR_INVALID_ARG, "color_scale must be finite and > 0");
  for (int i = 0; i < 16; ++i)
    if (!std::isfinite(P[i])) return na_fail(CVO_ERR_INVALID_ARG, "pose has a non-finite entry");
  int mode = p.color_mode;
  int D = p.feat_dim;
  if (mode == CVO_COLOR_NONE || D == 0) {
    mode = CVO_COLOR_NONE;
    D = 0;
  } else if (!d_fx || !d_fz) {
    return na_fail(CVO_ERR_INVALID_ARG, "NULL feature pointer");
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices)
    return na_fail(CVO_ERR_CUDA, "no usable current device");
  double* partials = nullptr;
  {
    // one-time set-up per device: the device address of the static scratch
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_addr[dev]) {
      void* ptr = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&ptr, g_na_partials);
      if (e != cudaSuccess) return na_fail(CVO_ERR_CUDA, cudaGetErrorString(e));
      g_na_addr[dev] = static_cast<double*>(ptr);
    }
    partials = g_na_addr[dev];
  }
  NaArgs a{};
  for (int r = 0; r < 3; ++r) {
    for (int c = 0; c < 3; ++c) a.R[3 * r + c] = P[4 * r + c];
    a.T[r] = P[4 * r + 3];
  }
  const double ell2 = ell * ell;
  a.A = (float)(1.4426950408889634 / (2.0 * ell2));
  a.rc2 = (float)(2.0 * ell2 * std::log(1.0 / p.kcut));
  a.fscale = mode == CVO_COLOR_KERNEL
                 ? (float)std::sqrt(1.4426950408889634 / (2.0 * p.ell_color * p.ell_color))
                 : mode == CVO_COLOR_DOT ? (float)std::sqrt(p.color_scale) : 1.0f;
  a.n = (int)n;
  a.m = (int)m;
  a.D = D;
  // the smallest tile whose items fit one wave, so that a small call spreads over
  // as many blocks as it has items; larger calls take the largest tile, which
  // stages the points least often
  const int64_t nS = (m + kNaSrc - 1) / kNaSrc;
  a.tile = 32;
  while (a.tile < kNaTile && nS * ((n + a.tile - 1) / a.tile) > kNaGrid) a.tile *= 2;
  const int nblocks = (int)std::min<int64_t>(nS * ((n + a.tile - 1) / a.tile), kNaGrid);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e;
  const int dp = D == 0 ? 0 : D <= 3 ? 3 : D <= 5 ? 5 : 8;
  if (mode == CVO_COLOR_NONE) e = na_launch<0, kColorNone>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s);
  else if (mode == CVO_COLOR_KERNEL)
    e = dp == 3 ? na_launch<3, kColorKernel>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s)
      : dp == 5 ? na_launch<5, kColorKernel>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s)
                : na_launch<8, kColorKernel>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s);
  else
    e = dp == 3 ? na_launch<3, kColorDot>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s)
      : dp == 5 ? na_launch<5, kColorDot>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s)
                : na_launch<8, kColorDot>(nblocks, d_x, d_fx, d_z, d_fz, a, partials, s);
  if (e != cudaSuccess) return na_fail(CVO_ERR_CUDA, cudaGetErrorString(e));
  na_finish_kernel<<<1, 32 * kNaStride, 0, s>>>(partials, nblocks, d_x, p.sigma * p.sigma, 1.0 / ell2, p.a2,
                                    p.b2, d_out);
  e = cudaGetLastError();
  if (e != cudaSuccess) return na_fail(CVO_ERR_CUDA, cudaGetErrorString(e));
  return CVO_OK;
}

// Detail message of the last failed context-free call on this host thread.
const char* cvo_static_last_error() { return g_na_err.c_str(); }
