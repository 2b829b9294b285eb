// Collocation forward sweep (paper Section "Optimization framework
// configurations": initial guesses from a forward solve at theta0): for each
// element in turn, Newton's method on the K collocation equations in the
// element's interior states, one CUDA block per problem.
//
// Bound: latency.  The elements depend on one another, so a problem's sweep is
// a chain of small dense solves on one SM; what counts is the number of
// dependent steps per element, not their arithmetic.  Hence
//  * the Newton matrix is inverted (FP32, Gauss-Jordan with partial pivoting)
//    and kept, in registers, across iterations and elements; an iteration is
//    then a residual (FP64), one matrix-vector product and a convergence test,
//    three barriers instead of two per matrix column.  The matrix is inverted
//    again at the current point when the correction shrinks by less than
//    CHORD_RATE per iteration;
//  * an element starts from the previous element's collocation polynomial
//    extrapolated over it.
// An element takes this short way only when it is plainly the easy case: the
// first correction is small and every further one contracts fast, after at
// most one new inverse.  Otherwise, and at the start of a chain, the element
// is solved the plain way, which alone decides which solution is followed and
// which elements are given up: above 32 unknowns Newton's method from the
// constant guess, a new inverse in every iteration; up to 32 unknowns from the
// previous element's stage increments, a new inverse when the contraction is
// slow.
// Residual, update and stopping test are FP64; the FP32 inverse only decides
// how fast the iteration contracts.  The short way's contraction is linear, and
// what it leaves behind adds up along the chain: it goes on until the remainder,
// from the slowest contraction seen with this inverse, is below SHORT_REST of the
// largest state, or the correction is at rounding level.  Ending at 2e-16 and at the
// contraction of the last step alone left the sweep of 27 species, 120 elements
// 2.3e-13 from the 64-bit solution and that of 50 species, 400 elements 3.4e-14; now
// 7e-16 and 1e-15, as with an LU in every iteration.
//
// Measured on a GB300 against Newton's method with an FP32 LU in every
// iteration (one warp up to 32 unknowns, one block above): 10 species, 400
// elements 18.4 -> 2.4 ms; 27 species, 415 elements 181 -> 4.0 ms (the remainder
// above costs a third: 1.7 and 2.9 ms with the shorter stop); 50 species, 400 elements
// 455 -> 6.8 ms.  On meshes so coarse that every element
// goes the plain way: 27 species 563 -> 32 us an element, 100 species 14.5 -> 11.5 ms.
#include <algorithm>
#include <map>
#include <mutex>

#include "problem.cuh"
#include "subst.cuh"

namespace collo {

constexpr int SWEEP_MAXIT = 30;
constexpr float CHORD_RATE = 0.25f;   // contraction per iteration below which an inverse is kept
constexpr float EASY_STEP = 0.05f;      // largest first correction of the short way, against max |Z|
constexpr float SHORT_REST = 1e-18f;    // remainder at which the short way ends, against max |Z|
constexpr int SWEEP_MAX_THREADS = 512;
constexpr int SWEEP_REG_DIM = 192;    // largest K n whose inverse is held in registers

// Threads of a problem's sweep: few warps for small systems (a barrier costs
// less), 16 otherwise.
__host__ __device__ inline int sweep_threads(int dim) {
  return dim <= 32 ? 128 : (dim <= 64 ? 256 : SWEEP_MAX_THREADS);
}

// Dynamic shared memory of one problem, in the order of SweepMem.
__host__ __device__ inline int sweep_pad(int dim) { return (dim + 31) & ~31; }
__host__ __device__ inline size_t sweep_mem_bytes(const DevProb& P, bool mat_in_smem) {
  const size_t dim = (size_t)P.K * P.n, dp = sweep_pad((int)dim), r = P.r;
  size_t b = sizeof(double) * (2 * (size_t)P.n + 2 * (size_t)P.K * (P.n + 1) + P.K * r + 4 * r);
  b += sizeof(float) * 4 * dp;                              // b, two columns, pivot row
  b += sizeof(int) * (2 * r + 4 * r + P.n + 1 + dp);
  if (dim <= SWEEP_REG_DIM) b += sizeof(float) * dim * P.n;   // df/dz blocks
  else if (mat_in_smem) b += sizeof(float) * dim * dim;
  return (b + 15) & ~size_t(15);
}

struct SweepMem {
  double* z0[2];    // [n] state at the element's start (this element's and the next one's)
  double* Z[2];     // [K][n + 1] interior states, each row ended by 1.0 (see mon)
  double* mon;      // [K][r] monomials
  double* coef;     // [nnz] h nu k_r of the species' reaction lists
  float* b;         // residual in elimination order
  float* col[2];    // pivot column
  float* row;       // pivot row
  float* jz;        // [K n][n] h df/dz (register inverse) or the matrix itself
  int* react;       // [r][2] reactants, the absent second one = n
  int* lst;         // [nnz] reactions of the species' lists
  int* ptr;         // [n + 1] list bounds
  int* step;        // [K n] elimination step of each equation
};

__device__ inline SweepMem sweep_mem(const DevProb& P, double* sm) {
  const int n = P.n, K = P.K, r = P.r, dp = sweep_pad(K * n);
  SweepMem m;
  m.z0[0] = sm; m.z0[1] = sm + n;
  m.Z[0] = m.z0[1] + n; m.Z[1] = m.Z[0] + K * (n + 1);
  m.mon = m.Z[1] + K * (n + 1);
  m.coef = m.mon + K * r;
  m.b = reinterpret_cast<float*>(m.coef + 4 * r);
  m.col[0] = m.b + dp; m.col[1] = m.col[0] + dp;
  m.row = m.col[1] + dp;
  m.react = reinterpret_cast<int*>(m.row + dp);
  m.lst = m.react + 2 * r;
  m.ptr = m.lst + 4 * r;
  m.step = m.ptr + n + 1;
  m.jz = reinterpret_cast<float*>(m.step + dp);
  return m;
}

// Barrier over the NW warps of a problem's sweep (the block may be larger: the
// other warps have left).
template <int NW>
__device__ inline void sweep_bar() {
  asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory");
}

// Entry (row, col) of the collocation equations' matrix without its df/dz part.
__device__ inline float colloc_entry(const double (*D)[NPMAX], int n, int row, int col) {
  const int k = row / n, s = row - k * n, j = col / n, t = col - j * n;
  return s == t ? (float)D[k + 1][j + 1] : 0.f;
}

// The index (0 .. dim-1) and value of the largest |col[i]| over the rows not
// yet used (bit q of `used`: row lane + 32 q), the same on every warp; -1 when
// it is zero or not finite.
template <int CPL>
__device__ inline int sweep_pivot(const float* col, int dim, unsigned used) {
  const int lane = threadIdx.x & 31;
  unsigned best = 0;
  int bi = 0;
#pragma unroll
  for (int q = 0; q < CPL; ++q) {
    const int i = lane + 32 * q;
    // the absolute value's bits order like the values; not-a-number above all
    const unsigned v = (i < dim && !((used >> q) & 1u)) ? (__float_as_uint(col[i]) & 0x7fffffffu) : 0u;
    if (v > best) { best = v; bi = i; }
  }
  const unsigned top = __reduce_max_sync(0xffffffffu, best);
  if (top == 0u || top >= 0x7f800000u) return -1;
  const unsigned who = __ballot_sync(0xffffffffu, best == top);
  return __shfl_sync(0xffffffffu, bi, __ffs(who) - 1);
}

// In-place Gauss-Jordan inversion with partial pivoting by rows, the matrix in
// registers: warp w, lane l hold rows w + NW k (k < RPW) and columns
// l + 32 c (c < CPL).  Rows are not exchanged: step[i] is the step at which row
// i was the pivot row; afterwards row i gives unknown step[i], and column c
// multiplies the right-hand side of the equation whose step is c.  Two
// barriers per step: the pivot column's owners publish it, every warp finds
// the same pivot in it, the pivot row's owner publishes that row scaled, all
// update.  False (on every thread) when a pivot is zero or not finite.
template <int NW, int RPW, int CPL>
__device__ bool sweep_invert(float (&m)[RPW][CPL], int dim, const SweepMem& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned used = 0;
#pragma unroll
  for (int cc = 0; cc < CPL; ++cc)
    for (int ln = 0; ln < 32; ++ln) {
      const int c = 32 * cc + ln;
      if (c >= dim) break;
      float* col = s.col[c & 1];
      if (lane == ln)
#pragma unroll
        for (int k = 0; k < RPW; ++k)
          if (warp + NW * k < dim) col[warp + NW * k] = m[k][cc];
      sweep_bar<NW>();
      const int p = sweep_pivot<CPL>(col, dim, used);
      if (p < 0) return false;
      if (lane == (p & 31)) used |= 1u << (p >> 5);
      const float inv = __fdividef(1.f, col[p]);
      if (warp == p % NW) {
#pragma unroll
        for (int k = 0; k < RPW; ++k)
          if (warp + NW * k == p)
#pragma unroll
            for (int q = 0; q < CPL; ++q)
              s.row[lane + 32 * q] = (q == cc && lane == ln) ? inv : m[k][q] * inv;
        if (lane == 0) s.step[p] = c;
      }
      sweep_bar<NW>();
      float rv[CPL];
#pragma unroll
      for (int q = 0; q < CPL; ++q) rv[q] = s.row[lane + 32 * q];
#pragma unroll
      for (int k = 0; k < RPW; ++k) {
        const float f = col[warp + NW * k];   // zero past the last row
        if (lane == ln) m[k][cc] = 0.f;
#pragma unroll
        for (int q = 0; q < CPL; ++q) m[k][q] = fmaf(-f, rv[q], m[k][q]);
      }
      if (warp == p % NW)   // the pivot row is the published one
#pragma unroll
        for (int k = 0; k < RPW; ++k)
          if (warp + NW * k == p)
#pragma unroll
            for (int q = 0; q < CPL; ++q) m[k][q] = rv[q];
    }
  return true;
}

// The same inversion with the matrix [dim][dim] in memory (systems above
// SWEEP_REG_DIM).
template <int NW>
__device__ bool sweep_invert_mem(float* m, int dim, const SweepMem& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  for (int i = tid; i < dim; i += NW * 32) s.step[i] = -1;
  for (int c = 0; c < dim; ++c) {
    float* col = s.col[c & 1];
    for (int i = tid; i < dim; i += NW * 32) col[i] = m[(size_t)i * dim + c];
    sweep_bar<NW>();
    unsigned best = 0;
    int bi = 0;
    for (int i = lane; i < dim; i += 32) {
      const unsigned v = s.step[i] < 0 ? (__float_as_uint(col[i]) & 0x7fffffffu) : 0u;
      if (v > best) { best = v; bi = i; }
    }
    const unsigned top = __reduce_max_sync(0xffffffffu, best);
    if (top == 0u || top >= 0x7f800000u) return false;
    const unsigned who = __ballot_sync(0xffffffffu, best == top);
    const int p = __shfl_sync(0xffffffffu, bi, __ffs(who) - 1);
    const float inv = __fdividef(1.f, col[p]);
    for (int j = tid; j < dim; j += NW * 32)
      s.row[j] = j == c ? inv : m[(size_t)p * dim + j] * inv;
    sweep_bar<NW>();
    if (tid == 0) s.step[p] = c;
    for (int i = warp; i < dim; i += NW) {
      const float f = i == p ? -1.f : col[i];
      float* mi = m + (size_t)i * dim;
      for (int j = lane; j < dim; j += 32)
        mi[j] = fmaf(-f, s.row[j], (i == p || j == c) ? 0.f : mi[j]);
    }
    sweep_bar<NW>();
  }
  return true;
}

// CPL > 0: the inverse in registers (RPW x CPL per thread); CPL = 0: in memory
// (gmat, or shared memory when null).  LPR: threads that share a residual row.
// An FP64 instruction holds its SM quarter's pipe for 64 cycles whatever its
// active lanes (measured), so the residual's terms are spread over at least
// four warps: LPR = 4 up to 32 rows, 2 up to 64, then 1.
template <int NW, int RPW, int CPL, int LPR>
__device__ void sweep_one(const DevProb& P, double* __restrict__ x, int* __restrict__ fails,
                          float* __restrict__ gmat, double* sm) {
  constexpr int NT = NW * 32;
  constexpr int MR = CPL > 0 ? RPW : 1, MC = CPL > 0 ? CPL : 1;
  __shared__ double D[NPMAX][NPMAX], ext[NPMAX][NPMAX];
  __shared__ unsigned wmax[2][2][NW];
  const int n = P.n, r = P.r, K = P.K, np = P.np, dim = K * n, zl = n + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SweepMem s = sweep_mem(P, sm);
  float* mat = CPL > 0 ? nullptr : (gmat ? gmat : s.jz);
  const size_t nz = (size_t)P.N * np * n;
  float m[MR][MC];
  for (int t = tid; t < np * np; t += NT) {
    const int k = t / np, j = t - k * np;
    D[k][j] = P.D[k][j];
    // l_j(1 + tau_k): the element's polynomial at the next element's points;
    // row 0: the state at the element's end (Eq. 2c: Radau z_K, Gauss sum_j b_j z_j)
    double v = 1.0;
    for (int l = 0; l < np; ++l)
      if (l != j) v *= (1.0 + P.tau[k] - P.tau[l]) / (P.tau[j] - P.tau[l]);
    ext[k][j] = k > 0 ? v : (P.gauss ? P.bw[j] : (j == K ? 1.0 : 0.0));
  }
  for (int j = tid; j < r; j += NT) {
    const int b2 = P.react[2 * j + 1];
    s.react[2 * j] = P.react[2 * j];
    s.react[2 * j + 1] = b2 < 0 ? n : b2;
  }
  for (int t = tid; t <= n; t += NT) s.ptr[t] = P.nu_ptr[t];
  for (int t = tid; t < 2 * K; t += NT) s.Z[t & 1][(t >> 1) * zl + n] = 1.0;
  for (int t = tid; t < sweep_pad(dim); t += NT)
    s.b[t] = s.row[t] = s.col[0][t] = s.col[1][t] = 0.f;
  sweep_bar<NW>();
  const int nnz = s.ptr[n];
  for (int e = tid; e < nnz; e += NT) s.lst[e] = P.nu_r[e];
  // this thread's places, found once (integer divisions): its monomial, its
  // residual row and part, its entry of the element's end
  const int mk = tid / r, mj = tid - mk * r;
  const int mon_a = mk < K ? mk * zl + s.react[2 * mj] : 0;
  const int mon_b = mk < K ? mk * zl + s.react[2 * mj + 1] : 0;
  const int g_row = tid / LPR, g_part = tid - g_row * LPR;
  const int g_k = g_row / n, g_q = g_row - g_k * n;
  const bool g_on = g_row < dim;
  const int g_e0 = g_on ? s.ptr[g_q] : 0, g_e1 = g_on ? s.ptr[g_q + 1] : 0;
  const int e_k = tid / n, e_q = tid - e_k * n;
  int my_z = -1, my_step = 0;   // register inverse: place in Z of this lane's sum, step[g_row]
  int nfail = 0;
  bool have = false;            // an inverse is held
  float rate = 0.f;             // ... its slowest contraction so far
  int least = SWEEP_MAXIT, excess = 0;   // iterations since it was made (below)
  const int excess_max = 8 + dim / 6;
  int cur = 0;
  for (int i = 0; i < P.N; ++i, cur ^= 1) {
    double* z0 = s.z0[cur];
    double* Z = s.Z[cur];
    const bool first = chain_start(P, i);
    if (first) {               // a condition's first element: its rates and x0
      const int c = i / P.Nch;
      sweep_bar<NW>();         // the previous element's readers of coef are done
      for (int e = tid; e < nnz; e += NT) {
        const int j = P.nu_r[e], q = P.pidx[j];
        double k = q < 0 ? P.kfix[j] : (P.logscale ? exp10(x[nz + q]) : x[nz + q]);
        if (P.kscale) k *= P.kscale[(size_t)c * r + j];
        s.coef[e] = P.h * P.nu_v[e] * k;
      }
      for (int t = tid; t < n; t += NT) z0[t] = P.x0[(size_t)c * n + t];
    }
    sweep_bar<NW>();
    bool ok = false;
    int its = 0;
    // attempt 0: the short way; attempt 1: the plain way
    for (int attempt = first ? 1 : 0; attempt < 2 && !ok; ++attempt) {
      if (attempt == 1) {
        const double* zp = s.z0[cur ^ 1];   // the previous element's states
        const double* Zp = s.Z[cur ^ 1];
        for (int t = tid; t < dim; t += NT) {
          const int k = t / n, q = t - k * n;
          Z[k * zl + q] = z0[q] + (CPL == 1 && !first ? Zp[k * zl + q] - zp[q] : 0.0);
        }
        have = false;
        sweep_bar<NW>();
      }
      float prev = INFINITY;
      bool made = false;        // an inverse was made for this element
      for (its = 0; its < SWEEP_MAXIT; ++its) {
        if (!have) {
          // matrix at the current point: D[k][j] delta_st - delta_kj h df_s/dz_t
          float* jz = CPL > 0 ? s.jz : mat;
          const int jl = CPL > 0 ? n : dim;
          if (CPL > 0) {
            for (int t = tid; t < dim * n; t += NT) jz[t] = 0.f;
          } else {
            for (int t = tid; t < dim * dim; t += NT) {
              const int row = t / dim;
              jz[t] = colloc_entry(D, n, row, t - row * dim);
            }
          }
          sweep_bar<NW>();
          for (int row = tid; row < dim; row += NT) {
            const int k = row / n, q = row - k * n;
            const double* zk = Z + k * zl;
            float* jr = jz + (size_t)row * jl + (CPL > 0 ? 0 : k * n);
            for (int e = s.ptr[q]; e < s.ptr[q + 1]; ++e) {
              const int rr = s.lst[e], a = s.react[2 * rr], b = s.react[2 * rr + 1];
              const float c = (float)s.coef[e];
              jr[a] -= c * (float)zk[b];
              if (b < n) jr[b] -= c * (float)zk[a];
            }
          }
          sweep_bar<NW>();
          bool good;
          if constexpr (CPL > 0) {
#pragma unroll
            for (int k = 0; k < RPW; ++k)
#pragma unroll
              for (int c = 0; c < CPL; ++c) {
                const int row = warp + NW * k, col = lane + 32 * c;
                float v = 0.f;
                if (row < dim && col < dim) {
                  v = colloc_entry(D, n, row, col);
                  const int kb = row / n;
                  if (col / n == kb) v += jz[row * n + col - kb * n];
                }
                m[k][c] = v;
              }
            good = sweep_invert<NW, RPW, CPL>(m, dim, s);
          } else {
            good = sweep_invert_mem<NW>(mat, dim, s);
          }
          if (!good) { sweep_bar<NW>(); break; }
          have = true;
          made = true;
          if (attempt == 0) prev = INFINITY;   // the next correction is this inverse's first
          rate = 0.f;
          least = SWEEP_MAXIT;
          excess = 0;
          sweep_bar<NW>();   // step[] is complete
          if constexpr (CPL > 0) {
            constexpr int SH = RPW <= 8 ? 2 : 1;   // see warp_rows_sum
            const int row = warp + NW * (lane >> SH);
            my_z = -1;
            if ((lane & ((1 << SH) - 1)) == 0 && (lane >> SH) < RPW && row < dim) {
              const int v = s.step[row], k = v / n;
              my_z = k * zl + v - k * n;
            }
            my_step = g_on ? s.step[g_row] : 0;
          }
        }
        if (mk < K) s.mon[tid] = Z[mon_a] * Z[mon_b];
        for (int t = tid + NT; t < K * r; t += NT) {
          const int k = t / r, j = t - k * r;
          s.mon[t] = Z[k * zl + s.react[2 * j]] * Z[k * zl + s.react[2 * j + 1]];
        }
        sweep_bar<NW>();
        if constexpr (CPL > 0) {
          double g = 0.0;
          if (g_on) {
            const double* Dk = D[g_k + 1];
            // the products with D nearly cancel: all in one chain of multiply-adds
            // (rounded apart by several threads they tripled the sweep's error)
            if (g_part == 0) {
              g = Dk[0] * z0[g_q];
              for (int j = 1; j < np; ++j) g = fma(Dk[j], Z[(j - 1) * zl + g_q], g);
            }
            const double* mo = s.mon + g_k * r;
            for (int e = g_e0 + g_part; e < g_e1; e += LPR) g = fma(-s.coef[e], mo[s.lst[e]], g);
          }
#pragma unroll
          for (int o = LPR / 2; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
          if (g_on && g_part == 0) s.b[my_step] = (float)g;
        } else {
          for (int row = tid; row < dim; row += NT) {
            const int k = row / n, q = row - k * n;
            double g = D[k + 1][0] * z0[q];
            for (int j = 0; j < K; ++j) g = fma(D[k + 1][j + 1], Z[j * zl + q], g);
            for (int e = s.ptr[q]; e < s.ptr[q + 1]; ++e)
              g = fma(-s.coef[e], s.mon[k * r + s.lst[e]], g);
            s.b[s.step[row]] = (float)g;
          }
        }
        sweep_bar<NW>();
        // dZ = inverse x residual; Z -= dZ.  The maxima of |dZ| and |Z| go by
        // their bits, which order like the values (|Z| by its upper word; a Z
        // that is not finite counts as an infinite dZ).
        unsigned dmax = 0, zmax = 0;
        auto apply = [&](int at, float d) {
          const double v = Z[at] - (double)d;
          Z[at] = v;
          const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
          zmax = max(zmax, hi);
          dmax = max(dmax, hi >= 0x7ff00000u ? 0x7f800000u : __float_as_uint(d) & 0x7fffffffu);
        };
        if constexpr (CPL > 0) {
          constexpr int R2 = RPW <= 8 ? 8 : 16;
          float bv[CPL], y[R2];
#pragma unroll
          for (int c = 0; c < CPL; ++c) bv[c] = s.b[lane + 32 * c];
#pragma unroll
          for (int k = 0; k < R2; ++k) {
            y[k] = 0.f;
            if (k < RPW)
#pragma unroll
              for (int c = 0; c < CPL; ++c) y[k] = fmaf(m[k][c], bv[c], y[k]);
          }
          const float mine = warp_rows_sum<float, R2>(y);
          if (my_z >= 0) apply(my_z, mine);
        } else {
          for (int i2 = warp; i2 < dim; i2 += NW) {
            float y = 0.f;
            for (int j = lane; j < dim; j += 32) y = fmaf(mat[(size_t)i2 * dim + j], s.b[j], y);
            for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
            if (lane == 0) {
              const int v = s.step[i2], k = v / n;
              apply(k * zl + v - k * n, y);
            }
          }
        }
        dmax = __reduce_max_sync(0xffffffffu, dmax);
        zmax = __reduce_max_sync(0xffffffffu, zmax);
        if (lane == 0) {
          wmax[its & 1][0][warp] = dmax;
          wmax[its & 1][1][warp] = zmax;
        }
        sweep_bar<NW>();
        dmax = __reduce_max_sync(0xffffffffu, lane < NW ? wmax[its & 1][0][lane] : 0u);
        zmax = __reduce_max_sync(0xffffffffu, lane < NW ? wmax[its & 1][1][lane] : 0u);
        if (dmax >= 0x7f800000u) { have = false; break; }
        const float dz = __uint_as_float(dmax);
        const float sc = fmaxf(1.f, (float)__hiloint2double((int)zmax, 0));
        // the contraction, while the correction is above the residual's rounding
        if (attempt == 0 && prev < INFINITY && dz > 1e-14f * sc) rate = fmaxf(rate, dz / prev);
        if (dz <= 1e-12f * sc) {
          // converged to the tolerance; a linear contraction leaves an error of about
          // rate / (1 - rate) dz: the short way goes on until that is small too, or
          // the correction is at rounding level or no longer halves
          if (attempt == 1 || dz <= 2e-16f * sc || dz > 0.5f * prev ||
              (rate > 0.f && rate * dz <= SHORT_REST * sc * (1.f - rate))) {
            ok = true;
            break;
          }
        } else if (attempt == 0) {
          if (its == 0 && dz > EASY_STEP * sc) break;
          if (dz > CHORD_RATE * prev) {
            if (made) break;
            have = false;
          }
        } else if (CPL != 1 || dz > CHORD_RATE * prev) {
          have = false;
        }
        prev = dz;
      }
    }
    if (!ok) {
      ++nfail;
      have = false;
      sweep_bar<NW>();
      for (int t = tid; t < dim; t += NT) {
        const int k = t / n, q = t - k * n;
        Z[k * zl + q] = z0[q];
      }
      sweep_bar<NW>();
    }
    // An ageing inverse costs iterations.  Once those above the least that any
    // element took with it add up to an inversion's cost (about 8 + K n / 6
    // iterations), invert again.  27 species: 13.5 us per element when kept for
    // good, 7.6 / 7.1 / 7.3 us at 2 / 1 / 0.5 times this limit; 10 species: 5.5,
    // 4.3 / 4.3 / 4.3 us.
    least = min(least, its);
    excess += its - least;
    if (excess > excess_max) have = false;
    double* xi = x + (size_t)i * np * n;
    double* z0n = s.z0[cur ^ 1];
    double* Zn = s.Z[cur ^ 1];
    auto finish = [&](int t, int k, int q) {
      xi[t] = k == 0 ? z0[q] : Z[(k - 1) * zl + q];
      double v = ext[k][0] * z0[q];
      for (int j = 1; j < np; ++j) v = fma(ext[k][j], Z[(j - 1) * zl + q], v);
      if (k == 0) z0n[q] = v;
      else Zn[(k - 1) * zl + q] = v;
    };
    if (e_k < np) finish(tid, e_k, e_q);
    for (int t = tid + NT; t < np * n; t += NT) {
      const int k = t / n;
      finish(t, k, t - k * n);
    }
  }
  if (tid == 0) *fails = nfail;
}

// One block per problem; the block is as large as the batch's largest problem
// needs, the surplus warps of a smaller one leave at once.
__global__ void __launch_bounds__(SWEEP_MAX_THREADS, 1)
k_sweep_b(const DevInst* __restrict__ insts, const int* __restrict__ act) {
  extern __shared__ double sm[];
  const DevInst& I = insts[act[blockIdx.x]];
  const int dim = I.P.K * I.P.n;
  if ((int)threadIdx.x >= sweep_threads(dim)) return;
  if (dim <= 32) sweep_one<4, 8, 1, 4>(I.P, I.x, I.fails, nullptr, sm);
  else if (dim <= 64) sweep_one<8, 8, 2, 2>(I.P, I.x, I.fails, nullptr, sm);
  else if (dim <= 96) sweep_one<16, 6, 3, 1>(I.P, I.x, I.fails, nullptr, sm);
  else if (dim <= 128) sweep_one<16, 8, 4, 1>(I.P, I.x, I.fails, nullptr, sm);
  else if (dim <= 160) sweep_one<16, 10, 5, 1>(I.P, I.x, I.fails, nullptr, sm);
  else if (dim <= SWEEP_REG_DIM) sweep_one<16, 12, 6, 1>(I.P, I.x, I.fails, nullptr, sm);
  else sweep_one<16, 1, 0, 1>(I.P, I.x, I.fails, I.sweep_work, sm);
}

size_t sweep_work_floats(const DevProb& P) {
  const size_t dim = (size_t)P.K * P.n;
  return dim > SWEEP_REG_DIM && dim * dim * sizeof(float) > 150 * 1024 ? dim * dim : 0;
}

size_t sweep_smem_bytes(const DevProb& P) {
  return sweep_mem_bytes(P, sweep_work_floats(P) == 0);
}

int sweep_block_threads(const DevProb& P) { return sweep_threads(P.K * P.n); }

cudaError_t launch_sweep_b(const DevInst* insts, const int* act, int A, int threads, size_t smem,
                           cudaStream_t st) {
  if (A == 0) return cudaSuccess;
  const cudaError_t e = opt_in_smem(k_sweep_b, smem);
  if (e != cudaSuccess) return e;
  count_launch();
  k_sweep_b<<<A, threads, smem, st>>>(insts, act);
  return cudaGetLastError();
}

}  // namespace collo
