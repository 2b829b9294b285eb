// Filter line-search primal-dual interior-point driver (paper Introduction:
// the NLP is solved by "a filter line-search interior point solver"; the
// algorithm statement followed is Waechter & Biegler, 2006) with every
// iterate resident on the device.
//
// The host runs only scalar control (filter, barrier and inertia-correction
// decisions); vectors never leave the GPU.  Per iteration the host reads one
// small block of scalars after each phase.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "problem.cuh"

namespace collo {

constexpr int IBS = 256;

template <int BS>
__device__ double bsum(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int s = BS / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] += sh[t + s];
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}
template <int BS>
__device__ double bmax(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int s = BS / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] = fmax(sh[t], sh[t + s]);
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}
template <int BS>
__device__ double bmin(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int s = BS / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] = fmin(sh[t], sh[t + s]);
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

__global__ void k_axpy(double* __restrict__ y, const double* __restrict__ x, double a, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    y[i] += a * x[i];
}

cudaError_t launch_axpy(double* y, const double* x, double a, size_t n, cudaStream_t st) {
  int g = (int)std::min<size_t>((n + 255) / 256, 4096);
  count_launch();
  k_axpy<<<std::max(g, 1), 256, 0, st>>>(y, x, a, n);
  return cudaGetLastError();
}

// ---- batched IPM kernels (one block per instance unless stated) ------------------

// theta0 pushed into the bounds (Waechter & Biegler 2006, Sec. 3.6), bound
// duals 1.
__global__ void k_init_point_b(const DevInst* __restrict__ insts, const int* __restrict__ act,
                               double kappa1, double kappa2) {
  const DevInst& I = insts[act[blockIdx.x]];
  const DevProb& P = I.P;
  const size_t nz = (size_t)P.N * P.np * P.n;
  for (int q = threadIdx.x; q < P.p; q += blockDim.x) {
    const double lo = P.theta_lo[q], hi = P.theta_hi[q];
    const double pl = fmin(kappa1 * fmax(1.0, fabs(lo)), kappa2 * (hi - lo));
    const double pu = fmin(kappa1 * fmax(1.0, fabs(hi)), kappa2 * (hi - lo));
    I.x[nz + q] = fmin(fmax(I.th0[q], lo + pl), hi - pu);
    I.zl[q] = 1.0;
    I.zu[q] = 1.0;
  }
}

// Parameter-space quantities for barrier parameter mu:
//   sigma_theta = zl/sl + zu/su (into sigma[nz..]); bar = mu/sl - mu/su;
//   zlmzu = zl - zu; out: max / min of (sl zl, su zu), sum zl + zu,
//   sum log sl + log su.
__global__ void __launch_bounds__(IBS)
k_theta_prep_b(const DevInst* __restrict__ insts, const int* __restrict__ act,
               const InstParams* __restrict__ prm) {
  __shared__ double sh[IBS];
  const DevInst& I = insts[act[blockIdx.x]];
  const DevProb& P = I.P;
  const double mu = prm[blockIdx.x].mu;
  const size_t nz = (size_t)P.N * P.np * P.n;
  double wmax = 0.0, wmin = 1e300, zs = 0.0, lg = 0.0;
  for (int q = threadIdx.x; q < P.p; q += IBS) {
    const double th = I.x[nz + q];
    const double sl = th - P.theta_lo[q], su = P.theta_hi[q] - th;
    I.sigma[nz + q] = I.zl[q] / sl + I.zu[q] / su;
    I.bar[q] = mu / sl - mu / su;
    I.zlmzu[q] = I.zl[q] - I.zu[q];
    wmax = fmax(wmax, fmax(sl * I.zl[q], su * I.zu[q]));
    wmin = fmin(wmin, fmin(sl * I.zl[q], su * I.zu[q]));
    zs += I.zl[q] + I.zu[q];
    lg += log(sl) + log(su);
  }
  wmax = bmax<IBS>(wmax, sh);
  wmin = bmin<IBS>(wmin, sh);
  zs = bsum<IBS>(zs, sh);
  lg = bsum<IBS>(lg, sh);
  if (threadIdx.x == 0) {
    I.out[O_WMAX] = wmax; I.out[O_WMIN] = wmin; I.out[O_ZSUM] = zs; I.out[O_LOG] = lg;
  }
}

// |lambda|_1 (which = 0) or grad^T kb over the primal entries (which = 1).
__global__ void __launch_bounds__(IBS)
k_vec_reduce_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int which) {
  __shared__ double sh[IBS];
  const DevInst& I = insts[act[blockIdx.x]];
  double v = 0.0;
  if (which == 0)
    for (long long i = threadIdx.x; i < I.n_c; i += IBS) v += fabs(I.lam[i]);
  else
    for (long long i = threadIdx.x; i < I.n_x; i += IBS) v += I.E.grad[i] * I.kb[i];
  v = bsum<IBS>(v, sh);
  if (threadIdx.x == 0) I.out[which == 0 ? O_LAM1 : O_GDX] = v;
}

// Bound-dual steps, fraction-to-boundary step sizes and the barrier part of
// grad(phi_mu)^T dx.
__global__ void __launch_bounds__(IBS)
k_theta_step_b(const DevInst* __restrict__ insts, const int* __restrict__ act,
               const InstParams* __restrict__ prm) {
  __shared__ double sh[IBS];
  const DevInst& I = insts[act[blockIdx.x]];
  const DevProb& P = I.P;
  const double mu = prm[blockIdx.x].mu, tau = prm[blockIdx.x].tau;
  const size_t nz = (size_t)P.N * P.np * P.n;
  double amax = 1.0, az = 1.0, g = 0.0;
  for (int q = threadIdx.x; q < P.p; q += IBS) {
    const double th = I.x[nz + q], d = I.kb[nz + q];
    const double sl = th - P.theta_lo[q], su = P.theta_hi[q] - th;
    const double dzl = mu / sl - I.zl[q] - (I.zl[q] / sl) * d;
    const double dzu = mu / su - I.zu[q] + (I.zu[q] / su) * d;
    I.dz[q] = dzl;
    I.dz[P.p + q] = dzu;
    if (d < 0) amax = fmin(amax, -tau * sl / d);
    if (-d < 0) amax = fmin(amax, tau * su / d);
    if (dzl < 0) az = fmin(az, -tau * I.zl[q] / dzl);
    if (dzu < 0) az = fmin(az, -tau * I.zu[q] / dzu);
    g += (-mu / sl + mu / su) * d;
  }
  amax = bmin<IBS>(amax, sh);
  az = bmin<IBS>(az, sh);
  g = bsum<IBS>(g, sh);
  if (threadIdx.x == 0) { I.out[O_AMAX] = amax; I.out[O_AZ] = az; I.out[O_GPHI] = g; }
}

// Barrier log terms at the trial point theta + alpha dtheta.
__global__ void __launch_bounds__(IBS)
k_trial_barrier_b(const DevInst* __restrict__ insts, const int* __restrict__ act,
                  const InstParams* __restrict__ prm) {
  __shared__ double sh[IBS];
  const DevInst& I = insts[act[blockIdx.x]];
  const DevProb& P = I.P;
  const double alpha = prm[blockIdx.x].alpha;
  const size_t nz = (size_t)P.N * P.np * P.n;
  double lg = 0.0, bad = 0.0;
  for (int q = threadIdx.x; q < P.p; q += IBS) {
    const double th = I.x[nz + q] + alpha * I.kb[nz + q];
    const double sl = th - P.theta_lo[q], su = P.theta_hi[q] - th;
    if (!(sl > 0) || !(su > 0)) bad = 1.0;
    else lg += log(sl) + log(su);
  }
  lg = bsum<IBS>(lg, sh);
  bad = bmax<IBS>(bad, sh);
  if (threadIdx.x == 0) { I.out[O_TLOG] = lg; I.out[O_TOK] = bad > 0 ? 0.0 : 1.0; }
}

// Grid-stride over the n_x + n_c entries of every active instance (prefix
// pre): mode 0 accepts the step (x += alpha dx, lambda += alpha dlambda,
// bound duals += alpha_z dz then reset into [mu/(kS s), kS mu/s]); mode 1
// adds the refinement correction (kb += kc); mode 2 zeroes lambda.
__global__ void k_update_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int A,
                           const long long* __restrict__ pre, const InstParams* __restrict__ prm,
                           int mode) {
  const long long total = pre[A];
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int lo = 0, hi = A;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (pre[mid] <= t) lo = mid; else hi = mid;
    }
    const int k = lo;
    const DevInst& I = insts[act[k]];
    const long long j = t - pre[k];
    if (mode == 1) { I.kb[j] += I.kc[j]; continue; }
    if (mode == 2) { if (j < I.n_c) I.lam[j] = 0.0; continue; }
    const InstParams pr = prm[k];
    const long long nz = I.n_x - I.P.p;
    if (j >= nz && j < I.n_x) {
      // parameter entry q: the same thread moves theta_q and its bound duals
      const DevProb& P = I.P;
      const int q = (int)(j - nz);
      const double th = I.x[j] + pr.alpha * I.kb[j];
      I.x[j] = th;
      const double sl = th - P.theta_lo[q], su = P.theta_hi[q] - th;
      double a = I.zl[q] + pr.alpha_z * I.dz[q];
      double b = I.zu[q] + pr.alpha_z * I.dz[P.p + q];
      a = fmax(fmin(a, pr.ksig * pr.mu / sl), pr.mu / (pr.ksig * sl));
      b = fmax(fmin(b, pr.ksig * pr.mu / su), pr.mu / (pr.ksig * su));
      I.zl[q] = a;
      I.zu[q] = b;
    } else if (j < I.n_x) {
      I.x[j] += pr.alpha * I.kb[j];
    } else {
      I.lam[j - I.n_x] += pr.alpha * I.kb[j];
    }
  }
}

// ---- batched launchers -------------------------------------------------------------
cudaError_t launch_init_point_b(const DevInst* insts, const int* act, int A, double k1, double k2,
                                cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  count_launch();
  k_init_point_b<<<A, 128, 0, st>>>(insts, act, k1, k2);
  return cudaGetLastError();
}

cudaError_t launch_theta_prep_b(const DevInst* insts, const int* act, int A, const InstParams* prm,
                                cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  count_launch();
  k_theta_prep_b<<<A, IBS, 0, st>>>(insts, act, prm);
  return cudaGetLastError();
}

cudaError_t launch_vec_reduce_b(const DevInst* insts, const int* act, int A, int which,
                                cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  count_launch();
  k_vec_reduce_b<<<A, IBS, 0, st>>>(insts, act, which);
  return cudaGetLastError();
}

cudaError_t launch_theta_step_b(const DevInst* insts, const int* act, int A, const InstParams* prm,
                                cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  count_launch();
  k_theta_step_b<<<A, IBS, 0, st>>>(insts, act, prm);
  return cudaGetLastError();
}

cudaError_t launch_trial_barrier_b(const DevInst* insts, const int* act, int A,
                                   const InstParams* prm, cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  count_launch();
  k_trial_barrier_b<<<A, IBS, 0, st>>>(insts, act, prm);
  return cudaGetLastError();
}

cudaError_t launch_update_b(const DevInst* insts, const int* act, int A, const long long* pre,
                            long long total, const InstParams* prm, int mode, cudaStream_t st) {
  if (A == 0 || total == 0) return cudaSuccess;
  int g = (int)std::min<long long>((total + 255) / 256, 8192);
  count_launch();
  k_update_b<<<std::max(g, 1), 256, 0, st>>>(insts, act, A, pre, prm, mode);
  return cudaGetLastError();
}

}  // namespace collo
