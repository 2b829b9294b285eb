// Structured FP64 KKT products and residual norms of one instance, shared by
// the evaluation kernels and the fused refinement kernel.  The reductions are
// fixed trees (sums) or maxima, so a result does not depend on which kernel or
// block size computes it.
#pragma once
#include "collo_internal.cuh"

namespace collo {

constexpr int EVAL_BS = 128;
constexpr int RED_BS = 256;
constexpr int TH_BS = 1024;   // threads of the per-instance reductions over elements
// Doubles of shared memory they use: column_sums, and block_max3 behind it.
constexpr int TH_SH = 32 * 33 + 3 * TH_BS / 32;

// |v| as bits that order like the values, a value that is not a number as zero
// (fmax passes over one).  Comparing them costs integer instructions; an FP64
// one holds its pipe for 64 cycles per warp.
__device__ inline unsigned long long abs_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return b > 0x7ff0000000000000ull ? 0ull : b;
}
__device__ inline unsigned long long max_bits(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}
// Block-wide maxima of three such values, valid on warp 0; sh: 3 (BS / 32)
// words.  The values are maxima: their order does not matter.
template <int BS>
__device__ inline void block_max3(unsigned long long& a, unsigned long long& b,
                                  unsigned long long& c, unsigned long long* sh) {
  constexpr int NW = BS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto shuffle = [&](unsigned long long& v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max_bits(v, __shfl_xor_sync(0xffffffffu, v, o));
  };
  shuffle(a); shuffle(b); shuffle(c);
  if (lane == 0) { sh[warp] = a; sh[NW + warp] = b; sh[2 * NW + warp] = c; }
  __syncthreads();
  if (warp == 0) {
    a = lane < NW ? sh[lane] : 0ull;
    b = lane < NW ? sh[NW + lane] : 0ull;
    c = lane < NW ? sh[2 * NW + lane] : 0ull;
    shuffle(a); shuffle(b); shuffle(c);
  }
}
// Column sums of v[N][L] for the 32 columns from q0 on, by TH_BS threads: per
// column 32 partial sums over i = l, l + 32, ... in that order, then a fixed tree;
// warp w returns the sum of column q0 + w.  A warp reads 32
// neighbouring columns of a row, so the loads are whole lines (one warp per column
// read a sector per lane: 50 species, 2000 elements 225 us for all columns on one
// SM, 37 us on p / 32 of them).  One barrier: the tree over a column's partial sums
// is a warp's.  sh: TH_SH doubles, the first 32 x 33.
__device__ inline double column_sums(const double* __restrict__ v, int N, int L, int q0,
                                     double* sh) {
  const int ql = threadIdx.x & 31, l = threadIdx.x >> 5, q = q0 + ql;
  double y = 0.0;
  if (q < L)
    for (int i0 = l; i0 < N; i0 += 256) {
      double t[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) t[j] = i0 + 32 * j < N ? v[(size_t)(i0 + 32 * j) * L + q] : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i0 + 32 * j < N) y += t[j];
    }
  sh[l * 33 + ql] = y;
  __syncthreads();
  y = sh[ql * 33 + l];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
  return y;
}
// Blocks of an instance's reductions: the scalars, and 32 columns each.
__host__ __device__ inline int theta_blocks(int p) { return 1 + (p + 31) / 32; }

// Deterministic block reductions (fixed tree over a fixed thread order).
template <int BS>
__device__ inline double block_sum(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
#pragma unroll
  for (int s = BS / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] += sh[t + s];
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

template <int BS>
__device__ inline double block_max(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
#pragma unroll
  for (int s = BS / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] = fmax(sh[t], sh[t + s]);
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

// The sums of a and b and the maximum of c over the first RED_BS threads of a larger
// block (all its threads call), in block_sum's order; valid on thread 0.  One
// barrier: a lane of the first warp adds its column of the tree, then shuffles
// (three trees in shared memory, nine barriers of 32 warps each: the reductions of a
// two-species evaluation 12.4 -> 8.0 us).  sh: 3 RED_BS doubles.
__device__ inline void first_sums(double& a, double& b, double& c, double* sh) {
  const int t = threadIdx.x;
  if (t < RED_BS) { sh[t] = a; sh[RED_BS + t] = b; sh[2 * RED_BS + t] = c; }
  __syncthreads();
  if (t >= 32) return;
  auto tree = [&](const double* s, auto op) {
    double v[RED_BS / 32];
#pragma unroll
    for (int k = 0; k < RED_BS / 32; ++k) v[k] = s[t + 32 * k];
#pragma unroll
    for (int h = RED_BS / 64; h > 0; h >>= 1)
#pragma unroll
      for (int k = 0; k < h; ++k) v[k] = op(v[k], v[k + h]);
    double y = v[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) y = op(y, __shfl_xor_sync(0xffffffffu, y, o));
    return y;
  };
  auto add = [](double x, double y) { return x + y; };
  a = tree(sh, add);
  b = tree(sh + RED_BS, add);
  c = tree(sh + 2 * RED_BS, [](double x, double y) { return fmax(x, y); });
}

// Structured FP64 product y = K v of the regularised KKT matrix
//   [ W + diag(sigma) + dw I   J^T  ] [vx]
//   [ J                       -dc I ] [vl]
// and r = b - y (b may be null: r = -y).  The derivative blocks are visited
// only at their structural nonzeros (the pattern lists of DevProb, ascending,
// so each sum keeps the order of the dense loop; the skipped terms are exact
// zeros).  One block per element computes the
// element's 2 (K + 1) n rows and its contribution to the p parameter rows; norms per
// element go to npart[i][0..2] (max |r_x|, max |r_c|, max |b| over the
// element's rows).  The first element clears norms[0..2] for resid_theta_one.
template <int BS = EVAL_BS>
__device__ inline void resid_elem(const DevProb& P, const DevEval& E, const double* __restrict__ sigma,
                           double dw, double dc, const double* __restrict__ vx,
                           const double* __restrict__ vl, const double* __restrict__ bx,
                           double bxs, const double* __restrict__ bc, double bcs,
                           double* __restrict__ rout, double* __restrict__ thpart,
                           double* __restrict__ npart, int i, unsigned long long* red,
                           double* __restrict__ norms) {
  const int n = P.n, p = P.p, N = P.N, K = P.K, np = P.np;
  const int tid = threadIdx.x;
  const size_t nz = (size_t)N * np * n, nx = nz + p;
  const size_t zoff = (size_t)i * np * n;
  const double* vz = vx;
  const double* vt = vx ? vx + nz : nullptr;
  const size_t nn = (size_t)n * n, np_ = (size_t)n * p;
  const double* JZ = E.JZ + (size_t)i * K * nn;
  const double* JT = E.JT + (size_t)i * K * np_;
  const double* Wzz = E.Wzz + (size_t)i * K * nn;
  const double* Wzt = E.Wzt + (size_t)i * K * np_;
  const double* Wob = E.Wobj + (size_t)i * n * np * np;
  const bool next = chain_next(P, i);
  if (i == 0 && tid < 3) norms[tid] = 0.0;
  unsigned long long mx = 0, mc = 0, mb = 0;
  for (int idx = tid; idx < np * n; idx += BS) {
    const int j = idx / n, s = idx - j * n;
    // primal row z[i][j][s]
    double y = 0.0;
    if (vz) {
      if (P.obs_sp[s])
        for (int l = 0; l < np; ++l) y += Wob[(s * np + j) * np + l] * vz[zoff + l * n + s];
      if (j >= 1) {
        const double* wr = Wzz + (size_t)(j - 1) * nn + (size_t)s * n;
        for (int e = P.wzr_ptr[s]; e < P.wzr_ptr[s + 1]; ++e) {
          const int t = P.wzr_i[e];
          y += wr[t] * vz[zoff + j * n + t];
        }
        const double* wt = Wzt + (size_t)(j - 1) * np_ + (size_t)s * p;
        for (int e = P.wtr_ptr[s]; e < P.wtr_ptr[s + 1]; ++e) {
          const int q = P.wtr_i[e];
          y += wt[q] * vt[q];
        }
      }
      y += ((sigma ? sigma[zoff + idx] : 0.0) + dw) * vz[zoff + idx];
    }
    if (vl) {
      if (j >= 1) {
        const double* jz = JZ + (size_t)(j - 1) * nn;
        for (int e = P.jzc_ptr[s]; e < P.jzc_ptr[s + 1]; ++e) {
          const int t = P.jzc_i[e];
          y += jz[(size_t)t * n + s] * vl[zoff + j * n + t];
        }
      }
      for (int k = 1; k < np; ++k) y += P.D[k][j] * vl[zoff + k * n + s];
      if (j == 0) y += vl[zoff + s];
      // the next element's continuity row: -b_j (Radau: -1 at j = K)
      if (next && P.bw[j] != 0.0) {
        if (P.gauss) y -= P.bw[j] * vl[zoff + np * n + s];
        else y -= vl[zoff + np * n + s];
      }
    }
    if (bx) mb = max_bits(mb, abs_bits(bx[zoff + idx]));
    if (bc) mb = max_bits(mb, abs_bits(bc[zoff + idx]));
    double rr = (bx ? bxs * bx[zoff + idx] : 0.0) - y;
    if (rout) rout[zoff + idx] = rr;
    mx = max_bits(mx, abs_bits(rr));
    // dual row c[i][j][s]
    double yc = 0.0;
    if (vz) {
      if (j == 0) {
        double prev = 0.0;
        if (!chain_start(P, i)) {
          if (!P.gauss) {
            prev = vz[zoff - n + s];
          } else {
            const size_t po = zoff - (size_t)np * n + s;
            for (int l = 0; l < np; ++l) prev += P.bw[l] * vz[po + (size_t)l * n];
          }
        }
        yc = vz[zoff + s] - prev;
      } else {
        for (int l = 0; l < np; ++l) yc += P.D[j][l] * vz[zoff + l * n + s];
        const double* jz = JZ + (size_t)(j - 1) * nn + (size_t)s * n;
        for (int e = P.jzr_ptr[s]; e < P.jzr_ptr[s + 1]; ++e) {
          const int t = P.jzr_i[e];
          yc += jz[t] * vz[zoff + j * n + t];
        }
        const double* jt = JT + (size_t)(j - 1) * np_ + (size_t)s * p;
        for (int e = P.jtr_ptr[s]; e < P.jtr_ptr[s + 1]; ++e) {
          const int q = P.jtr_i[e];
          yc += jt[q] * vt[q];
        }
      }
    }
    if (vl) yc -= dc * vl[zoff + idx];
    double rc = (bc ? bcs * bc[zoff + idx] : 0.0) - yc;
    if (rout) rout[nx + zoff + idx] = rc;
    mc = max_bits(mc, abs_bits(rc));
  }
  // this element's part of the parameter rows
  for (int q = tid; q < p; q += BS) {
    double y = 0.0;
    for (int k = 1; k < np; ++k)
      for (int e = P.thq_ptr[q]; e < P.thq_ptr[q + 1]; ++e) {
        const int s = P.thq_i[e];
        if (vz) y += Wzt[(size_t)(k - 1) * np_ + (size_t)s * p + q] * vz[zoff + k * n + s];
        if (vl) y += JT[(size_t)(k - 1) * np_ + (size_t)s * p + q] * vl[zoff + k * n + s];
      }
    thpart[(size_t)i * p + q] = y;
  }
  block_max3<BS>(mx, mc, mb, red);
  if (tid == 0) {
    npart[i * 3 + 0] = __longlong_as_double((long long)mx);
    npart[i * 3 + 1] = __longlong_as_double((long long)mc);
    npart[i * 3 + 2] = __longlong_as_double((long long)mb);
  }
}

// Residual modes of the batched product (which vectors of the instance):
//   R_DUAL: r_x = -(grad + J^T lambda - zl + zu)   (dual infeasibility)
//   R_RHS:  Newton right-hand side -[grad phi_mu + J^T lambda; c] into ka
//   R_IR:   r = ka - K kb with the factorization's sigma / delta_w / delta_c into kr
enum ResidMode { R_DUAL = 0, R_RHS = 1, R_IR = 2 };

struct ResidArgs {
  const double *sigma, *vx, *vl, *bx, *bc, *th_extra;
  double bxs, bcs, dw, dc;
  double* rout;
};

__device__ inline ResidArgs resid_args(const DevInst& I, const InstParams& pr, int mode) {
  ResidArgs a{};
  if (mode == R_DUAL) {
    a.vl = I.lam; a.bx = I.E.grad; a.bxs = -1.0; a.th_extra = I.zlmzu;
  } else if (mode == R_RHS) {
    a.vl = I.lam; a.bx = I.E.grad; a.bxs = -1.0; a.bc = I.E.c; a.bcs = -1.0;
    a.th_extra = I.bar; a.rout = I.ka;
  } else {
    a.sigma = I.sigma; a.vx = I.kb; a.vl = I.kb + I.n_x; a.bx = I.ka; a.bxs = 1.0;
    a.bc = I.ka + I.n_x; a.bcs = 1.0; a.dw = pr.dw; a.dc = pr.dc; a.rout = I.kr;
  }
  return a;
}

// Parameter rows of r = b - K v, and the global norms:
// out[0] = max|r_x|, out[1] = max|r_c|, out[2] = max|b| (b may be null).
// Block 0 of the instance's theta_blocks takes the norms of the elements, block b
// the parameters from 32 (b - 1) on (column_sums of thpart[N][p]); all raise
// out[0..2] (cleared by resid_elem) to their maxima.  TH_BS threads.
__device__ inline void resid_theta_one(const DevProb& P, const DevEval& E,
                                const double* __restrict__ sigma, double dw,
                                const double* __restrict__ vx, const double* __restrict__ bx,
                                double bxs, const double* __restrict__ bc,
                                double* __restrict__ rout, const double* __restrict__ thpart,
                                const double* __restrict__ npart,
                                const double* __restrict__ th_extra, double* __restrict__ out,
                                int block, double* sh) {
  const int tid = threadIdx.x, p = P.p, N = P.N;
  const size_t nz = (size_t)N * P.np * P.n;
  unsigned long long mx = 0, mc = 0, mb = 0;
  if (block == 0) {
    for (int i = tid; i < N; i += TH_BS) {
      mx = max_bits(mx, abs_bits(npart[i * 3 + 0]));
      mc = max_bits(mc, abs_bits(npart[i * 3 + 1]));
      mb = max_bits(mb, abs_bits(npart[i * 3 + 2]));
    }
    if (bx)
      for (int q = tid; q < p; q += TH_BS) mb = max_bits(mb, abs_bits(bx[nz + q]));
  } else {
    const int q0 = 32 * (block - 1), q = q0 + (tid >> 5);
    const bool mine = (tid & 31) == 0 && q < p;
    // asked for before the sum
    double w = 0.0, v = 0.0, ex = 0.0, b = 0.0;
    if (mine) {
      if (vx) { w = E.wtt[q] + (sigma ? sigma[nz + q] : 0.0) + dw; v = vx[nz + q]; }
      if (th_extra) ex = th_extra[q];
      if (bx) b = bx[nz + q];
    }
    double y = column_sums(thpart, N, p, q0, sh);
    if (mine) {
      if (vx) y += w * v;
      if (th_extra) y -= ex;
      const double rr = (bx ? bxs * b : 0.0) - y;
      if (rout) rout[nz + q] = rr;
      mx = abs_bits(rr);
    }
  }
  block_max3<TH_BS>(mx, mc, mb, reinterpret_cast<unsigned long long*>(sh + 32 * 33));
  if (tid == 0) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(out);
    atomicMax(o, mx);
    atomicMax(o + 1, mc);
    atomicMax(o + 2, mb);
  }
}

}  // namespace collo
