// The step tail of one iteration, alone, one warp a case: the state that the solve kernel holds
// at an iteration's start, its gradient and step sums in, the passes' next pose and the FP64
// pose out.
#include "../paper_1904_02266_gb300/csrc/pair_kernels.cuh"

namespace {

struct Case {
  double P[16], cX[3], cZ[3];
  double grad[9];     // F, omega'(3), v(3), two counts
  double s[7];        // S0..S4 along xi / |xi|, two counts
  double ell, eps_pose;
  long long at_floor;
};

struct Result {
  double P[16], tau, quick;
  float R[9], T[3];   // the passes' next pose
};

__global__ void step_kernel(const Case* in, Result* out) {
  using namespace cvo;
  __shared__ BlockCtx b;
  const Case& c = in[blockIdx.x];
  const int lane = threadIdx.x;
  if (lane == 0) {
    memset(&b, 0, sizeof(b));
    for (int a = 0; a < 3; ++a) {
      b.tc.cX[a] = c.cX[a];
      b.tc.cZ[a] = c.cZ[a];
      b.tc.cXf[a] = (float)c.cX[a];
    }
    b.tc.sigma2 = b.tc.inv_a2 = b.tc.inv_b2 = 1.0;
    b.tc.inv_a2f = b.tc.inv_b2f = 1.0f;
    b.tc.eps_pose = c.eps_pose;
    b.tc.eps_pose_f = (float)c.eps_pose;
    b.tc.mode = kModeAlign;
    b.tc.step_order = 4;
    b.tc.max_iters = 100;
    for (int i = 0; i < 16; ++i) b.P[i] = c.P[i];
    b.ic.ell = c.ell;
    b.ic.inv_l2 = 1.0 / (c.ell * c.ell);
    b.ic.inv_l2f = (float)b.ic.inv_l2;
    b.ic.kf_rot = b.ic.kf_tr = b.ic.inv_l2;
    b.ic.rprune = (float)c.ell;
    b.ic.at_floor = (int)c.at_floor;
    b.need_plan = 1;
    b.plan_level = -1;
  }
  __syncwarp();
  begin_iteration(b, lane);
  gradient_direction(b, c.grad, lane);
  gradient_fp64(b, c.grad, lane);
  finish_step(b, c.s, lane);
  const bool quick = b.pending != 0;
  if (quick) {
    begin_iteration(b, lane);
    pending_step(b, lane);
  } else {
    begin_iteration(b, lane);
  }
  if (lane == 0) {
    Result& r = out[blockIdx.x];
    for (int i = 0; i < 16; ++i) r.P[i] = b.P[i];
    for (int i = 0; i < 9; ++i) r.R[i] = b.R[i];
    for (int i = 0; i < 3; ++i) r.T[i] = b.T[i];
    r.tau = b.t * b.xi_norm;
    r.quick = quick ? 1.0 : 0.0;
  }
}

}  // namespace

extern "C" int run_steps(const void* in, void* out, int n) {
  Case* d_in = nullptr;
  Result* d_out = nullptr;
  cudaError_t e = cudaMalloc(&d_in, sizeof(Case) * n);
  if (e == cudaSuccess) e = cudaMalloc(&d_out, sizeof(Result) * n);
  if (e == cudaSuccess) e = cudaMemcpy(d_in, in, sizeof(Case) * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    step_kernel<<<n, 32>>>(d_in, d_out);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, d_out, sizeof(Result) * n, cudaMemcpyDeviceToHost);
  cudaFree(d_in);
  cudaFree(d_out);
  return (int)e;
}
