// Semi-dense front end on the GPU (Sec. 5: the points are the pixels with a
// high intensity gradient, back-projected from the depth image). From a depth
// image and an HSV image it selects, back-projects and describes the points
// the solver aligns, with every step in these kernels:
//
//   pixels     validity (depth in range), intensity gradient of the V channel
//              (central differences, one-sided at the border) and its
//              magnitude, FP32 with one rounding per operation
//   threshold  the linear-interpolation percentile of the valid magnitudes, in
//              FP64, from its two order statistics, which a radix select on the
//              bit patterns finds (non-negative floats order as integers): three
//              histograms of 11, 11 and 10 bits, each of the magnitudes that
//              share the digits found so far
//   keep       valid and magnitude > threshold; kept pixels are counted per
//              block, ranked in raster order from the counts before their
//              block; above max_points the ranks floor(k m / max_points) are
//              kept
//   points     z = depth, x = ((u - cx) / fx) z, y = ((v - cy) / fy) z and the
//              features H, S, V, clip(gx / s), clip(gy / s), FP32
//
// Pixel selection is index work: the kept set and its order are exact, the
// same on any run. Five launches and one wait: at 640 x 480 every kernel is a few
// microseconds of latency, so what counts is how few there are (sorting the
// magnitudes to read two of them took 12 of the 23 launches, and their count had
// to visit the host): 279 -> 75 us per frame, of which the call's host side, with
// its allocation, wait and read-back, is about half.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "runtime.h"

namespace cvo {

namespace {

constexpr int kScanBlock = 1024;

__device__ __forceinline__ float intensity(const float* hsv, int W, int x, int y) {
  return hsv[3 * ((size_t)y * W + x) + 2];
}

// Intensity gradient of pixel (x, y).
__device__ __forceinline__ void fe_gradient(const float* hsv, int W, int H, int x, int y, float& gx,
                                            float& gy) {
  if (x == 0) gx = __fsub_rn(intensity(hsv, W, 1, y), intensity(hsv, W, 0, y));
  else if (x == W - 1) gx = __fsub_rn(intensity(hsv, W, W - 1, y), intensity(hsv, W, W - 2, y));
  else gx = __fmul_rn(0.5f, __fsub_rn(intensity(hsv, W, x + 1, y), intensity(hsv, W, x - 1, y)));
  if (y == 0) gy = __fsub_rn(intensity(hsv, W, x, 1), intensity(hsv, W, x, 0));
  else if (y == H - 1) gy = __fsub_rn(intensity(hsv, W, x, H - 1), intensity(hsv, W, x, H - 2));
  else gy = __fmul_rn(0.5f, __fsub_rn(intensity(hsv, W, x, y + 1), intensity(hsv, W, x, y - 1)));
}

// Device scratch of a selection, zeroed before each run.
struct FeCounts {
  unsigned hist[3][2048];     // digit counts: top 11 bits, next 11, last 10
  unsigned above;             // ~(smallest key beyond the first two digits found)
  int kept[kScanBlock];       // kept pixels per block of kScanBlock pixels
};

// The key of a pixel without a valid depth: no magnitude has it (a NaN result
// is 0x7fffffff).
constexpr unsigned kNoKey = 0xffffffffu;

// Adds the block's shared digit counts to the device's.
__device__ __forceinline__ void fe_flush(const unsigned* s_hist, unsigned* hist) {
  __syncthreads();
  for (int i = threadIdx.x; i < 2048; i += kScanBlock)
    if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
}

__global__ void __launch_bounds__(kScanBlock)
fe_pixels_kernel(const float* __restrict__ depth, const float* __restrict__ hsv, int W, int H,
                 float dmin, float dmax, unsigned* __restrict__ keys, FeCounts* __restrict__ c) {
  __shared__ unsigned s_hist[2048];
  for (int i = threadIdx.x; i < 2048; i += kScanBlock) s_hist[i] = 0u;
  __syncthreads();
  const int p = blockIdx.x * kScanBlock + threadIdx.x;
  if (p < W * H) {
    const int y = p / W, x = p - y * W;
    float gx, gy;
    fe_gradient(hsv, W, H, x, y, gx, gy);
    const float mag = __fsqrt_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)));
    const float d = depth[p];
    const bool valid = isfinite(d) && d >= dmin && d <= dmax;
    const unsigned key = valid ? __float_as_uint(mag) : kNoKey;
    keys[p] = key;
    if (valid) atomicAdd(&s_hist[key >> 21], 1u);
  }
  fe_flush(s_hist, c->hist[0]);
}

// 2048 digit counts, two per thread of a block of kScanBlock, with the counts up to
// and including this thread's and the total. Every thread of the block calls it.
struct FeScan {
  unsigned a, b, incl, total;
};

__device__ FeScan fe_scan(const unsigned* hist) {
  __shared__ unsigned s_warp[kScanBlock / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint2 v = __ldcg(reinterpret_cast<const uint2*>(hist) + t);
  FeScan f{v.x, v.y, v.x + v.y, 0u};
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, f.incl, off);
    if (lane >= off) f.incl += u;
  }
  __syncthreads();   // the shared words of an earlier call have been read
  if (lane == 31) s_warp[warp] = f.incl;
  __syncthreads();
  const unsigned w = s_warp[lane];
  f.total = __reduce_add_sync(0xffffffffu, w);
  f.incl += __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
  return f;
}

// Where rank r falls: the digit and the rank left within it (digit 2047, rank 0, when
// r is at or beyond the total). Every thread of the block calls it.
struct FeDigit {
  unsigned digit, left;
};

__device__ FeDigit fe_locate(const FeScan& f, unsigned rank) {
  __shared__ FeDigit s_found;
  const unsigned before = f.incl - f.a - f.b;
  __syncthreads();   // an earlier call's answer has been read
  if (threadIdx.x == 0 && rank >= f.total) s_found = FeDigit{2047u, 0u};
  if (rank >= before && rank < f.incl) {
    const bool second = rank >= before + f.a;
    s_found = FeDigit{2u * threadIdx.x + (second ? 1u : 0u), rank - before - (second ? f.a : 0u)};
  }
  __syncthreads();
  return s_found;
}

// The valid pixels, the lower order statistic's rank at percentile q among them and
// the FP64 position it comes from (numpy's 'linear' method), and the digits of that
// statistic found so far: the top one (level 1), and the next (level 2).
struct FePrefix {
  unsigned n, rank, d0, d1, left;
  double h;
};

__device__ FePrefix fe_prefix(const FeCounts* c, double q, int level) {
  __shared__ unsigned s_rank;
  __shared__ double s_h;
  FePrefix f;
  const FeScan top = fe_scan(c->hist[0]);
  f.n = top.total;
  if (threadIdx.x == 0) {   // FP64 on one thread of one warp
    const double h = f.n > 0u ? (double)(int)(f.n - 1u) * (q / 100.0) : 0.0;
    s_rank = (unsigned)(int)floor(h);
    s_h = h;
  }
  __syncthreads();
  f.rank = s_rank;
  f.h = s_h;
  FeDigit d = fe_locate(top, f.rank);
  f.d0 = d.digit;
  f.left = d.left;
  f.d1 = 0u;
  if (level > 1) {
    d = fe_locate(fe_scan(c->hist[1]), f.left);
    f.d1 = d.digit;
    f.left = d.left;
  }
  return f;
}

// Digit counts of the keys that share the digits found so far; at the last
// level also the smallest key beyond them (where the upper order statistic lies
// when the lower one is the last of its prefix).
__global__ void __launch_bounds__(kScanBlock)
fe_digits_kernel(const unsigned* __restrict__ keys, int n, double q, int level,
                 FeCounts* __restrict__ c) {
  __shared__ unsigned s_hist[2048];
  __shared__ unsigned s_above;
  for (int i = threadIdx.x; i < 2048; i += kScanBlock) s_hist[i] = 0u;
  if (threadIdx.x == 0) s_above = 0u;
  const FePrefix f = fe_prefix(c, q, level);
  __syncthreads();
  const int p = blockIdx.x * kScanBlock + threadIdx.x;
  if (p < n) {
    const unsigned key = keys[p];
    if (key != kNoKey) {
      if (level == 1) {
        if (key >> 21 == f.d0) atomicAdd(&s_hist[(key >> 10) & 2047u], 1u);
      } else {
        const unsigned pre = f.d0 << 11 | f.d1;
        if (key >> 10 == pre) atomicAdd(&s_hist[key & 1023u], 1u);
        else if (key >> 10 > pre && ~key > s_above) atomicMax(&s_above, ~key);
      }
    }
  }
  fe_flush(s_hist, c->hist[level]);
  if (level == 2 && threadIdx.x == 0 && s_above) atomicMax(&c->above, s_above);
}

// The percentile, from its two order statistics, in FP64.
__device__ double fe_threshold(const FeCounts* c, double q) {
  __shared__ double s_thr;
  const FePrefix f = fe_prefix(c, q, 2);
  const FeScan last = fe_scan(c->hist[2]);
  const FeDigit lo = fe_locate(last, f.left), hi = fe_locate(last, f.left + 1u);
  if (threadIdx.x == 0) {
    const unsigned pre = (f.d0 << 11 | f.d1) << 10;
    const unsigned ka = pre | lo.digit;
    // the next rank: in the same prefix, beyond it, or (the last rank) the same
    const unsigned kb = f.rank + 1u >= f.n ? ka : f.left + 1u < last.total ? pre | hi.digit
                                                                         : ~__ldcg(&c->above);
    const double t = f.h - (double)(int)f.rank;
    const double a = (double)__uint_as_float(ka), b = (double)__uint_as_float(kb);
    const double d = b - a;
    s_thr = f.n > 0u ? (t < 0.5 ? a + d * t : b - d * (1.0 - t)) : 0.0;
  }
  __syncthreads();
  return s_thr;
}

__device__ __forceinline__ bool fe_kept(unsigned key, double thr) {
  return key != kNoKey && (double)__uint_as_float(key) > thr;
}

// Kept pixels per block; block 0 leaves the threshold for the next kernel.
__global__ void __launch_bounds__(kScanBlock)
fe_count_kernel(const unsigned* __restrict__ keys, int n, double q, FeCounts* __restrict__ c,
                double* __restrict__ thr_out) {
  const double thr = fe_threshold(c, q);
  const int p = blockIdx.x * kScanBlock + threadIdx.x;
  const int m = __syncthreads_count(p < n && fe_kept(keys[p], thr));
  if (threadIdx.x == 0) {
    c->kept[blockIdx.x] = m;
    if (blockIdx.x == 0) *thr_out = thr;
  }
}

// Kept pixel of rank r goes to output slot r, or, when m > cap, to the slot k
// with floor(k m / cap) == r (if any). Nothing is written when more points than
// `room` would be (room 0: there is room for every pixel). totals: valid pixels,
// kept pixels.
__global__ void __launch_bounds__(kScanBlock)
fe_emit_kernel(const float* __restrict__ depth, const float* __restrict__ hsv,
               const unsigned* __restrict__ keys, const FeCounts* __restrict__ c,
               const double* __restrict__ thr, int W, int H, long long cap, long long room,
               float fx, float fy, float cx, float cy, float gs, float* __restrict__ out_xyz,
               float* __restrict__ out_feat, int* __restrict__ out_pix, int* __restrict__ totals) {
  __shared__ int s_before[kScanBlock / 32], s_total[kScanBlock / 32], s_warp[kScanBlock / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // kept pixels in the blocks before this one, and in all of them
  const int v = t < (int)gridDim.x ? __ldcg(&c->kept[t]) : 0;
  const int vb = __reduce_add_sync(0xffffffffu, t < (int)blockIdx.x ? v : 0);
  const int va = __reduce_add_sync(0xffffffffu, v);
  const int p = blockIdx.x * kScanBlock + t;
  const bool keep = p < W * H && fe_kept(keys[p], *thr);
  const unsigned mask = __ballot_sync(0xffffffffu, keep);
  if (lane == 0) {
    s_before[warp] = vb;
    s_total[warp] = va;
    s_warp[warp] = __popc(mask);
  }
  __syncthreads();
  long long m = 0, r = __popc(mask & ((1u << lane) - 1u));
  for (int w = 0; w < kScanBlock / 32; ++w) {
    m += s_total[w];
    r += s_before[w] + (w < warp ? s_warp[w] : 0);
  }
  if (blockIdx.x == 0) {
    const unsigned valid = fe_scan(c->hist[0]).total;
    if (t == 0) {
      totals[0] = (int)valid;
      totals[1] = (int)m;
    }
  }
  const long long n_emit = cap > 0 && m > cap ? cap : m;
  if (!keep || (room > 0 && n_emit > room)) return;
  long long k = r;
  if (cap > 0 && m > cap) {
    k = (r * cap + m - 1) / m;   // smallest k with k m / cap >= r
    if (k >= cap || (k * m) / cap != r) return;
  }
  const int y = p / W, x = p - y * W;
  const float z = depth[p];
  out_xyz[3 * k + 0] = __fmul_rn(__fdiv_rn(__fsub_rn((float)x, cx), fx), z);
  out_xyz[3 * k + 1] = __fmul_rn(__fdiv_rn(__fsub_rn((float)y, cy), fy), z);
  out_xyz[3 * k + 2] = z;
  if (out_feat) {
    float gx, gy;
    fe_gradient(hsv, W, H, x, y, gx, gy);
    out_feat[5 * k + 0] = hsv[3 * (size_t)p + 0];
    out_feat[5 * k + 1] = hsv[3 * (size_t)p + 1];
    out_feat[5 * k + 2] = hsv[3 * (size_t)p + 2];
    out_feat[5 * k + 3] = fminf(fmaxf(__fdiv_rn(gx, gs), -1.0f), 1.0f);
    out_feat[5 * k + 4] = fminf(fmaxf(__fdiv_rn(gy, gs), -1.0f), 1.0f);
  }
  if (out_pix) out_pix[k] = p;
}

inline int nblocks(long long n, int t) { return (int)((n + t - 1) / t); }

// The selection into caller-visible device buffers (context lock held).
// out_xyz / out_feat / out_pix have room for cap points (cap > 0) or for
// every pixel (cap == 0).
int frontend_run(cvo_ctx* ctx, const float* depth, const float* hsv, int W, int H,
                 const cvo_frontend_params& fp, bool on_dev, cudaStream_t us, long long cap,
                 float* out_xyz, float* out_feat, int* out_pix, int64_t* n_out) {
  const long long npix = (long long)W * H;
  if (W < 2 || H < 2 || npix > (long long)kScanBlock * kScanBlock)
    return fail(ctx, CVO_ERR_INVALID_ARG, "image must be at least 2 x 2 and at most 2^20 pixels");
  if (!(fp.fx > 0) || !(fp.fy > 0) || !std::isfinite(fp.cx) || !std::isfinite(fp.cy) ||
      !(fp.depth_min <= fp.depth_max) || !(fp.percentile >= 0.0 && fp.percentile <= 100.0) ||
      !(fp.grad_scale > 0) || fp.max_points < 0)
    return fail(ctx, CVO_ERR_INVALID_ARG, "bad front-end parameters");
  cudaStream_t s = ctx->stream;
  const int n = (int)npix;
  const int nb = nblocks(n, kScanBlock);
  // one scratch allocation carved into 256-byte aligned pieces, sized with the
  // same rounding the carving uses: counts, threshold, totals, the images (when
  // they come from the host) and the keys
  auto round_up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t pix4 = round_up(sizeof(float) * (size_t)n);
  const size_t bytes = round_up(sizeof(FeCounts)) + round_up(sizeof(double)) +
                       round_up(sizeof(int) * 2) +
                       (on_dev ? 0 : pix4 + round_up(sizeof(float) * 3 * (size_t)n)) + pix4;
  char* scratch = nullptr;
  if (cudaMallocFromPoolAsync((void**)&scratch, bytes, ctx->pool, s) != cudaSuccess)
    return fail(ctx, CVO_ERR_CUDA, "front-end scratch allocation failed");
  char* cur = scratch;
  auto take = [&](size_t b) {
    char* r = cur;
    cur += round_up(b);
    return r;
  };
  FeCounts* counts = (FeCounts*)take(sizeof(FeCounts));
  double* thr = (double*)take(sizeof(double));
  int* totals = (int*)take(sizeof(int) * 2);   // valid pixels, kept pixels
  const float* d_depth = depth;
  const float* d_hsv = hsv;
  cudaError_t e = cudaSuccess;
  if (!on_dev) {
    float* dd = (float*)take(sizeof(float) * (size_t)n);
    float* dh = (float*)take(sizeof(float) * (size_t)n * 3);
    e = cudaMemcpyAsync(dd, depth, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(dh, hsv, sizeof(float) * (size_t)n * 3, cudaMemcpyHostToDevice, s);
    d_depth = dd;
    d_hsv = dh;
  } else if (us && us != s) {
    cudaEvent_t ev;
    e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev, us);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev, 0);
    cudaEventDestroy(ev);
  }
  unsigned* keys = (unsigned*)take(sizeof(unsigned) * (size_t)n);
  if ((size_t)(cur - scratch) > bytes) {   // the sizing above must cover the carving
    cudaFreeAsync(scratch, s);
    return fail(ctx, CVO_ERR_INTERNAL, "front-end scratch sizing");
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, sizeof(FeCounts), s);
  if (e == cudaSuccess) {
    fe_pixels_kernel<<<nb, kScanBlock, 0, s>>>(d_depth, d_hsv, W, H, (float)fp.depth_min,
                                               (float)fp.depth_max, keys, counts);
    fe_digits_kernel<<<nb, kScanBlock, 0, s>>>(keys, n, fp.percentile, 1, counts);
    fe_digits_kernel<<<nb, kScanBlock, 0, s>>>(keys, n, fp.percentile, 2, counts);
    fe_count_kernel<<<nb, kScanBlock, 0, s>>>(keys, n, fp.percentile, counts, thr);
    fe_emit_kernel<<<nb, kScanBlock, 0, s>>>(
        d_depth, d_hsv, keys, counts, thr, W, H, fp.max_points, cap, (float)fp.fx, (float)fp.fy,
        (float)fp.cx, (float)fp.cy, (float)fp.grad_scale, out_xyz, out_feat, out_pix, totals);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ctx->h_int, totals, sizeof(int) * 2, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(scratch, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  const int n_valid = e == cudaSuccess ? ctx->h_int[0] : 0;
  const long long m = e == cudaSuccess ? ctx->h_int[1] : 0;
  long long n_emit = m;
  if (fp.max_points > 0 && m > fp.max_points) n_emit = fp.max_points;
  if (e == cudaSuccess && cap > 0 && n_emit > cap)
    return fail(ctx, CVO_ERR_INVALID_ARG, "output buffers too small for the selected points");
  if (e != cudaSuccess) return fail(ctx, CVO_ERR_CUDA, std::string("front end: ") + cudaGetErrorString(e));
  if (n_valid == 0) return fail(ctx, CVO_ERR_INVALID_ARG, "no pixel has a depth in range");
  *n_out = n_emit;
  return CVO_OK;
}

}  // namespace

}  // namespace cvo

using namespace cvo;

extern "C" {

void cvo_frontend_params_default(cvo_frontend_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->fx = p->fy = 525.0;
  p->cx = 319.5;
  p->cy = 239.5;
  p->depth_min = 0.5;
  p->depth_max = 5.0;
  p->percentile = 80.0;
  p->grad_scale = 0.05;
  p->max_points = 0;
}

int cvo_frontend_select(cvo_ctx* ctx, const float* depth, const float* hsv, int width, int height,
                        const cvo_frontend_params* params, uint32_t flags, void* stream,
                        float* out_xyz, float* out_feat, int32_t* out_pixel, int64_t capacity,
                        int64_t* n_out) {
  if (!ctx) return CVO_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (!depth || !hsv || !params || !out_xyz || !n_out || capacity <= 0)
    return fail(ctx, CVO_ERR_INVALID_ARG, "NULL pointer or capacity <= 0");
  if (serve_active(ctx))
    return fail(ctx, CVO_ERR_BUSY, "the request loop is running (cvo_serve_stop ends it)");
  CK(cudaSetDevice(ctx->device));
  return frontend_run(ctx, depth, hsv, width, height, *params, (flags & CVO_DEVICE_PTR) != 0,
                      (cudaStream_t)stream, capacity, out_xyz, out_feat, out_pixel, n_out);
}

int cvo_frontend_cloud(cvo_ctx* ctx, const float* depth, const float* hsv, int width, int height,
                       const cvo_frontend_params* params, uint32_t flags, void* stream,
                       int32_t* handle_out, int64_t* n_out) {
  if (!ctx) return CVO_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (!depth || !hsv || !params || !handle_out)
    return fail(ctx, CVO_ERR_INVALID_ARG, "NULL pointer");
  const int D = ctx->prm.color_mode == CVO_COLOR_NONE ? 0 : ctx->prm.feat_dim;
  if (D != 0 && D != 5)
    return fail(ctx, CVO_ERR_INVALID_ARG, "the front end makes 5 features (feat_dim must be 5)");
  if (serve_active(ctx))
    return fail(ctx, CVO_ERR_BUSY, "the request loop is running (cvo_serve_stop ends it)");
  CK(cudaSetDevice(ctx->device));
  const long long npix = (long long)width * height;
  long long cap = params->max_points > 0 ? std::min<long long>(params->max_points, npix) : npix;
  if (width < 2 || height < 2) return fail(ctx, CVO_ERR_INVALID_ARG, "image must be at least 2 x 2");
  float* buf = nullptr;
  if (cudaMallocFromPoolAsync((void**)&buf, sizeof(float) * 8 * (size_t)cap, ctx->pool,
                              ctx->stream) != cudaSuccess)
    return fail(ctx, CVO_ERR_CUDA, "front-end output allocation failed");
  int64_t n = 0;
  int rc = frontend_run(ctx, depth, hsv, width, height, *params, (flags & CVO_DEVICE_PTR) != 0,
                        (cudaStream_t)stream, cap, buf, buf + 3 * cap, nullptr, &n);
  if (rc == CVO_OK && n == 0) rc = fail(ctx, CVO_ERR_INVALID_ARG, "no pixel passes the threshold");
  Cloud* c = nullptr;
  if (rc == CVO_OK)
    rc = create_cloud(ctx, buf, D > 0 ? buf + 3 * cap : nullptr, n, true, ctx->stream, &c);
  cudaFreeAsync(buf, ctx->stream);
  cudaStreamSynchronize(ctx->stream);
  if (rc != CVO_OK) return rc;
  *handle_out = add_cloud(ctx, c);
  if (n_out) *n_out = n;
  return CVO_OK;
}

}  // extern "C"
