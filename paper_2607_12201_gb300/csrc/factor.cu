// Structured, pivot-free factorization and solve of the element-banded KKT
// system bordered by the parameter block.
//
// The paper attributes most of the GPU benefit to sparse linear algebra on a
// KKT system put in a "pivoting-free factorizable form", with parallelism at
// the level of the elimination tree (Abstract; Introduction).  Here the
// elimination tree is explicit:
//
//  1. Element condensation (one CUDA block per element, all elements in
//     parallel): the element's 8n unknowns are ordered as n (state,
//     multiplier) pairs per group -- (z1,c1), (z2,c2), (z0,c3) interior and
//     (z3,c0) interface -- and the 3n interior pairs are eliminated with
//     static 2x2 pivots [[w, j], [j, -delta_c]].  Their determinant is
//     -(w delta_c + j^2) < 0 for the collocation Jacobian entry j, so each pivot
//     is nonsingular whatever the sign of the Hessian entry w; the sequence is
//     Gaussian elimination without pivoting on the element's square
//     collocation Jacobian.  The parameter border rides along as extra rows.
//  2. Block cyclic reduction over the chain of 2n x 2n interface blocks
//     (ceil(log2 N) levels; at each level the odd blocks are eliminated in
//     parallel, each updating its two neighbours, creating the n x n fill
//     coupling between them, and contributing to the parameter Schur block).
//  3. The p x p parameter Schur complement, summed from all contributions in
//     a fixed order and factored in FP64 (LDL^T, 1x1 pivots).
//
// Inertia is counted from every pivot block (Sylvester's law of inertia).
// T = double (plain path) or float (mixed path; residuals and refinement
// are FP64 elsewhere).
#include <algorithm>
#include <climits>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "collo_internal.cuh"
#include "subst.cuh"

namespace collo {

constexpr int FBS = 256;   // threads per factor block

__device__ inline void pivot_inertia(double a, double b, double d, int& pos, int& neg, int& zero) {
  const double det = fma(a, d, -(b * b));
  if (!(det == det) || det == 0.0 || !isfinite(det)) { zero += 2; return; }
  if (det < 0) { pos += 1; neg += 1; return; }
  if (a + d > 0) pos += 2; else neg += 2;
}

// Packed lower triangle: entry (r, c), c <= r, at r (r + 1) / 2 + c.
__host__ __device__ inline int tri_at(int r, int c) { return r * (r + 1) / 2 + c; }

// Layouts of a block's lower triangle.  PackedTri (shared memory, where every
// byte counts): rows one after the other.  RowBlockTri (global slab): blocks
// of 32 rows, each row-major with its leading dimension cut to the block's last
// column, so that 32 x 32 tiles start on 128-byte lines (16 entries per row are
// above the diagonal on average and never used).
struct PackedTri {
  static __host__ __device__ int at(int r, int c) { return tri_at(r, c); }
  static __host__ __device__ size_t elems(int msz) {
    return ((size_t)msz * (msz + 1) / 2 + 3) & ~size_t(3);   // a multiple of 16 bytes
  }
};
struct RowBlockTri {
  static __host__ __device__ int at(int r, int c) {
    const int b = r >> 5;
    return 32 * (b + 1) * (16 * b + (r & 31)) + c;
  }
  static __host__ __device__ size_t elems(int msz) {
    const size_t b = (msz + 31) >> 5;
    return 512 * b * (b + 1);
  }
};
// The symmetric entry (a, b) of a triangle A.
template <class Lay, typename T>
__device__ inline T sym_at(const T* A, int a, int b) {
  return A[a >= b ? Lay::at(a, b) : Lay::at(b, a)];
}

// Tile t of a lower triangle of tiles, numbered row by row: (ti, tj), tj <= ti.
__device__ inline void tri_tile(int t, int& ti, int& tj) {
  int i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  ti = i;
  tj = t - i * (i + 1) / 2;
}

// Panel buffer leading dimension: at least PANEL_PAD rows past msz, so that every
// warp tile of trailing_update reads inside the buffer; a multiple of 4 (16-byte
// loads of consecutive rows in trailing_update, of a column's diagonal part in
// the panel eliminations) but not of 8, so that the column copies into it meet
// at most four ways in a bank.
constexpr int PANEL_PAD = 89;
__host__ __device__ inline int panel_ld(int msz) { return (((msz + 92) >> 3) << 3) + 4; }

// The tiles of a trailing update that a warp takes: lo .. hi - 1 in turn, or, with
// a counter in shared memory, lo and on, one after the other among the block's
// warps (its next one is asked for before a tile is computed).
struct TileTurns {
  int lo, hi;
  int* count;
  int t, next;
  __device__ int take() const {
    int v = 0;
    if ((threadIdx.x & 31) == 0) v = atomicAdd(count, 1);
    return lo + __shfl_sync(0xffffffffu, v, 0);
  }
  __device__ int first() { return t = count ? take() : lo < hi ? lo : INT_MAX; }
  __device__ void ahead() { next = count ? take() : t + 1 < hi ? t + 1 : INT_MAX; }
  __device__ int step() { return t = next; }
};
__device__ inline TileTurns tiles_in_turn(int lo, int hi) { return {lo, hi, nullptr, 0, 0}; }
__device__ inline TileTurns tiles_shared(int lo, int* count) { return {lo, 0, count, 0, 0}; }

// Trailing update of pair_eliminate_packed for kernels with a small register
// budget (the cyclic-reduction blocks inside the cooperative factorization
// kernel when it runs three blocks per SM): 4 x 4 tiles of the packed
// triangle, one per thread at a time; A[r][c] -= (sum_k Lp[k][r] W[k][c]), the
// sum in ascending k, subtracted once (the same arithmetic per entry as
// trailing_update, so the result does not depend on which of the two a
// launch uses).
// Tiles go to the warps in chunks of 32 (lane by lane), taken by TileTurns.
template <typename T, class Lay>
__device__ __noinline__ void trailing_update_tiles4(T* A, int msz, int cend, int K,
                                                    const T* __restrict__ Lp,
                                                    const T* __restrict__ W, int ldw,
                                                    TileTurns turns) {
  const int lane = threadIdx.x & 31;
  const int ntr = (msz - cend + 3) >> 2;
  const int ntiles = ntr * (ntr + 1) / 2, nch = (ntiles + 31) >> 5;
  for (int ch = turns.first(); ch < nch; ch = turns.step()) {
    turns.ahead();
    const int t = 32 * ch + lane;
    if (t < ntiles) {
      int ti, tj;
      tri_tile(t, ti, tj);
      const int r0 = cend + 4 * ti, cb = cend + 4 * tj;
      // the tile's entries are loaded first, so that their latency (the
      // triangle may be in global memory) overlaps the products below
      T cur[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int r = r0 + u, c = cb + v;
          cur[u][v] = (r < msz && c <= r) ? A[Lay::at(r, c)] : T(0);
        }
      T acc[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = T(0);
      for (int k = 0; k < K; ++k) {
        T lr[4], uc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          lr[u] = (r0 + u < msz) ? Lp[k * ldw + r0 + u] : T(0);
          uc[u] = (cb + u < msz) ? W[k * ldw + cb + u] : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = fma(lr[u], uc[v], acc[u][v]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + u;
        if (r >= msz) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int c = cb + v;
          if (c <= r) A[Lay::at(r, c)] = cur[u][v] - acc[u][v];
        }
      }
    }
  }
}
// Chunks that hold the tiles of the next 2 PB rows and columns.
__device__ inline int tiles4_head(int PB) {
  return (PB / 2 * (PB / 2 + 1) / 2 + 31) >> 5;
}

// Two FP32 values in one 64-bit register, and the packed multiply-add on them
// (each half rounded like fmaf): half the issue slots of two scalar ones.
__device__ inline unsigned long long pack2(float a, float b) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ inline void unpack2(unsigned long long d, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
}
__device__ inline unsigned long long fma2(unsigned long long a, unsigned long long b,
                                          unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Accumulators of a register tile of TR consecutive rows and TC columns:
// acc[u][v] += l[u] w[v].  FP32 rows go in packed pairs.
template <typename T, int TR, int TC>
struct TileAcc {
  T a[TR][TC];
  __device__ void clear() {
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) a[u][v] = T(0);
  }
  // l: TR consecutive entries (16-byte aligned), w: columns 8 entries apart
  __device__ void add(const T* __restrict__ l, const T* __restrict__ w) {
    T lr[TR], uc[TC];
#pragma unroll
    for (int u = 0; u < TR; u += 2) {
      const double2 q = *reinterpret_cast<const double2*>(l + u);
      lr[u] = q.x;
      lr[u + 1] = q.y;
    }
#pragma unroll
    for (int v = 0; v < TC; ++v) uc[v] = w[8 * v];
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) a[u][v] = fma(lr[u], uc[v], a[u][v]);
  }
  // the same with w in runs of two columns, the runs 16 apart
  __device__ void add_runs(const T* __restrict__ l, const T* __restrict__ w) {
    T lr[TR], uc[TC];
#pragma unroll
    for (int u = 0; u < TR; u += 2) {
      const double2 q = *reinterpret_cast<const double2*>(l + u);
      lr[u] = q.x;
      lr[u + 1] = q.y;
    }
#pragma unroll
    for (int v = 0; v < TC; v += 2) {
      const double2 q = *reinterpret_cast<const double2*>(w + 8 * v);
      uc[v] = q.x;
      uc[v + 1] = q.y;
    }
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) a[u][v] = fma(lr[u], uc[v], a[u][v]);
  }
  __device__ T get(int u, int v) const { return a[u][v]; }
};
template <int TR, int TC>
struct TileAcc<float, TR, TC> {
  unsigned long long a[TR / 2][TC];
  __device__ void clear() {
#pragma unroll
    for (int u = 0; u < TR / 2; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) a[u][v] = 0ull;
  }
  __device__ void add(const float* __restrict__ l, const float* __restrict__ w) {
    ulonglong2 lr[TR / 4];
    unsigned long long uc[TC];
#pragma unroll
    for (int u = 0; u < TR / 4; ++u) lr[u] = reinterpret_cast<const ulonglong2*>(l)[u];
#pragma unroll
    for (int v = 0; v < TC; ++v) uc[v] = pack2(w[8 * v], w[8 * v]);
#pragma unroll
    for (int u = 0; u < TR / 4; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) {
        a[2 * u][v] = fma2(lr[u].x, uc[v], a[2 * u][v]);
        a[2 * u + 1][v] = fma2(lr[u].y, uc[v], a[2 * u + 1][v]);
      }
  }
  // the same with w in runs of four columns, the runs 32 apart
  __device__ void add_runs(const float* __restrict__ l, const float* __restrict__ w) {
    ulonglong2 lr[TR / 4];
    unsigned long long uc[TC];
#pragma unroll
    for (int u = 0; u < TR / 4; ++u) lr[u] = reinterpret_cast<const ulonglong2*>(l)[u];
#pragma unroll
    for (int v = 0; v < TC; v += 4) {
      const float4 q = *reinterpret_cast<const float4*>(w + 8 * v);
      uc[v] = pack2(q.x, q.x);
      uc[v + 1] = pack2(q.y, q.y);
      uc[v + 2] = pack2(q.z, q.z);
      uc[v + 3] = pack2(q.w, q.w);
    }
#pragma unroll
    for (int u = 0; u < TR / 4; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) {
        a[2 * u][v] = fma2(lr[u].x, uc[v], a[2 * u][v]);
        a[2 * u + 1][v] = fma2(lr[u].y, uc[v], a[2 * u + 1][v]);
      }
  }
  __device__ float get(int u, int v) const {
    float x, y;
    unpack2(a[u >> 1][v], x, y);
    return (u & 1) ? y : x;
  }
};

// Trailing update of pair_eliminate_packed: A[r][c] -= sum_k Lp[k][r] W[k][c]
// for cend <= c <= r < msz (packed lower triangle, shared or global memory),
// the sum over k = 0..K-1 in ascending order, subtracted once.  Warp-blocked
// register tiles: a warp owns 4 TR rows x 8 TC columns of the trailing
// matrix, lane (ty, tx) = (lane / 8, lane % 8) the TR consecutive rows r0 + TR
// ty and the columns c0 + tx + 8v (v < TC): per k a thread's rows arrive in
// 16-byte loads (broadcast over its eight lanes) and its columns in runs of
// eight, and A is read and written in full 32-byte sectors.  Tiles start at a
// multiple of four rows for those loads.  TR x TC is set by
// the register budget of the calling kernel; out of line, so that the tile
// gets the kernel's whole register budget.  Rows and columns past msz are
// computed from the panel buffers' padding and never stored.
// Bound: FP32 multiply-adds against shared-memory loads and issue slots.  In
// isolation (K = 32, 16 warps) scalar multiply-adds with scalar loads reach 69 of
// the SM's 128 lanes per clock, packed ones with 16-byte loads 88.
template <typename T, int TR, int TC>
__device__ __noinline__ void trailing_update(T* A, int msz, int cend, int K,
                                             const T* __restrict__ Lp, const T* __restrict__ W,
                                             int ldw, TileTurns turns) {
  constexpr int WR = 4 * TR, WC = 8 * TC;
  static_assert(WR <= PANEL_PAD && WC <= PANEL_PAD, "panel buffers padded for the warp tile");
  const int lane = threadIdx.x & 31;
  const int ty = lane >> 3, tx = lane & 7;
  const int rbase = cend & ~3;
  const int nbr = (msz - rbase + WR - 1) / WR;
  int t = turns.first(), t0 = 0;
  for (int bi = 0; bi < nbr; ++bi) {
    // tiles t0 .. t0 + nbc - 1: those of tile row bi that meet the lower triangle
    const int nbc = (min(msz, rbase + (bi + 1) * WR) - cend + WC - 1) / WC;
    for (; t - t0 < nbc; t = turns.step()) {
      turns.ahead();
      const int bj = t - t0;
      const int r0 = rbase + bi * WR + TR * ty, c0 = cend + bj * WC + tx;
      const T* lb = Lp + r0;
      const T* wb = W + c0;
      // the tile's entries are loaded first, so that their latency (the
      // triangle may be in global memory) overlaps the products
      T cur[TR][TC];
#pragma unroll
      for (int u = 0; u < TR; ++u)
#pragma unroll
        for (int v = 0; v < TC; ++v) {
          const int r = r0 + u, c = c0 + 8 * v;
          cur[u][v] = (r < msz && c <= r) ? A[tri_at(r, c)] : T(0);
        }
      TileAcc<T, TR, TC> acc;
      acc.clear();
#pragma unroll 2
      for (int k = 0; k < K; ++k) acc.add(lb + k * ldw, wb + k * ldw);
#pragma unroll
      for (int u = 0; u < TR; ++u) {
        const int r = r0 + u;
        if (r >= msz) continue;
#pragma unroll
        for (int v = 0; v < TC; ++v) {
          const int c = c0 + 8 * v;
          if (c <= r) A[tri_at(r, c)] = cur[u][v] - acc.get(u, v);
        }
      }
    }
    t0 += nbc;
  }
}
// Tiles that hold the next 2 PB <= 4 TR rows and columns: the first tile row's.
template <int TR, int TC>
__device__ inline int packed_head(int msz, int cend) {
  return (min(msz, (cend & ~3) + 4 * TR) - cend + 8 * TC - 1) / (8 * TC);
}

// Four (FP32) or two (FP64) consecutive entries at a 16-byte boundary.
template <typename T>
struct alignas(16) Quad {
  T v[16 / sizeof(T)];
};

// The same update of a triangle in the slab (RowBlockTri), in tiles on its
// 128-byte lines: a warp owns a block's 32 rows x 8 TC columns (FP32: 64, or 32 at
// the end of a row block), lane (ty, tx) the rows 8 ty .. 8 ty + 7 and TC columns
// in 16-byte runs, 8 lanes side by side.
// Every access is 16 bytes per lane over whole lines and none is predicated:
// entries above the diagonal, past msz or before cend (in the tiles that
// straddle it) take part too and are never read again.
// Bound: the shared-memory loads of the products, which fill a warp's registers
// at 128 bytes per cycle whether lanes share an address or not: 12 wavefronts
// per 32 multiply-adds of a lane in an 8 x 4 tile, 8 in an 8 x 8 one; then L2 for
// the tile itself.  50 species, 2000 elements, cycles per element in all trailing
// updates (condensation and reduction): 756 000 with the packed triangle in the
// slab, whose rows start anywhere (4 to 8 lines per access, each predicated),
// 583 000 in 8 x 4 tiles on whole lines, 440 000 in 8 x 8 ones (both beside the
// next diagonal block, below).  FP64 keeps 8 x 2 tiles: its pipe is the bound.
template <typename T, int TC>
__device__ inline void slab_tile(T* a, int ld, const T* lb, const T* wb, int K, int ldw) {
  constexpr int TR = 8, Q = 16 / sizeof(T), NQ = TC / Q;
  // rows whose entries are loaded before the products (the rest after them, in
  // the registers of the operands): what the kernels' 128 registers hold
  constexpr int AHEAD = NQ == 1 ? TR : 0, PART = NQ == 1 ? TR : TR / 2;
  Quad<T> cur[PART][NQ];
  auto load = [&](int u0) {
#pragma unroll
    for (int u = 0; u < PART; ++u)
#pragma unroll
      for (int g = 0; g < NQ; ++g)
        cur[u][g] = *reinterpret_cast<const Quad<T>*>(a + (u0 + u) * ld + 8 * Q * g);
  };
  if (AHEAD) load(0);
  TileAcc<T, TR, TC> acc;
  acc.clear();
#pragma unroll 2
  for (int k = 0; k < K; ++k) acc.add_runs(lb + k * ldw, wb + k * ldw);
#pragma unroll
  for (int u0 = 0; u0 < TR; u0 += PART) {
    if (!AHEAD) load(u0);
#pragma unroll
    for (int u = 0; u < PART; ++u)
#pragma unroll
      for (int g = 0; g < NQ; ++g) {
#pragma unroll
        for (int i = 0; i < Q; ++i) cur[u][g].v[i] -= acc.get(u0 + u, Q * g + i);
        *reinterpret_cast<Quad<T>*>(a + (u0 + u) * ld + 8 * Q * g) = cur[u][g];
      }
  }
}
template <typename T, int TC>
__device__ __noinline__ void trailing_update_slab(T* A, int msz, int cend, int K,
                                                  const T* __restrict__ Lp,
                                                  const T* __restrict__ W, int ldw,
                                                  TileTurns turns) {
  constexpr int Q = 16 / sizeof(T), WC = 8 * TC, HC = 8 * Q;   // HC: columns of a narrow tile
  static_assert(32 <= PANEL_PAD, "tiles inside the panel buffers");
  const int lane = threadIdx.x & 31;
  const int ty = lane >> 3, tx = lane & 7;
  if (msz <= cend) return;
  const int nb = (msz + 31) >> 5, cb = cend & ~(HC - 1);
  int t = turns.first(), t0 = 0;
  for (int b = cend >> 5; b < nb; ++b) {
    // tiles t0 .. t0 + nbc - 1: those of row block b
    const int ld = 32 * (b + 1), nbc = (ld - cb + WC - 1) / WC;
    for (; t - t0 < nbc; t = turns.step()) {
      turns.ahead();
      const int c0 = cb + (t - t0) * WC;
      T* a = A + 512 * b * (b + 1) + 8 * ty * ld + c0 + Q * tx;
      const T* lb = Lp + 32 * b + 8 * ty;
      const T* wb = W + c0 + Q * tx;
      if (TC > Q && c0 + HC < ld) slab_tile<T, TC>(a, ld, lb, wb, K, ldw);
      else slab_tile<T, Q>(a, ld, lb, wb, K, ldw);
    }
    t0 += nbc;
  }
}
// columns per lane
template <typename T>
constexpr int SLAB_TC = sizeof(T) == 4 ? 8 : 2;
// Tiles that hold the next panel's diagonal block: those of the first row block
// (panels start at a multiple of 2 PB, so the block lies in it).
template <typename T, int TC>
__device__ inline int slab_head(int cend) {
  return (32 * ((cend >> 5) + 1) - (cend & ~(8 * 16 / (int)sizeof(T) - 1)) + 8 * TC - 1) / (8 * TC);
}

// One pair's update of a row's remaining panel columns: x[j] -= l0 U0[j] +
// l1 U1[j] for j = kk + 2 .. 2 PB - 1, each by two multiply-adds.  U0, U1: the
// pair's unscaled columns at the panel's own rows (the same for every row, read
// as shared-memory broadcasts).  Entries past the panel's last column are
// updated from whatever the buffer holds and not used.
template <typename T, int PB>
__device__ inline void pair_row_update(T (&x)[2 * PB], int kk, const T* __restrict__ U0,
                                       const T* __restrict__ U1, T l0, T l1) {
  constexpr int Q = 16 / sizeof(T);
#pragma unroll
  for (int g = 0; g < 2 * PB / Q; ++g) {
    if (Q * g + Q - 1 < kk + 2) continue;
    const Quad<T> u0 = reinterpret_cast<const Quad<T>*>(U0)[g];
    const Quad<T> u1 = reinterpret_cast<const Quad<T>*>(U1)[g];
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (Q * g + i >= kk + 2)
        x[Q * g + i] = fma(-l1, u1.v[i], fma(-l0, u0.v[i], x[Q * g + i]));
  }
}

// Pivot inverse (ia, ib, id) of the pair (a, b, d); zero where it has none.
template <typename T>
__device__ inline void pivot_inverse(T a, T b, T d, T& ia, T& ib, T& id) {
  const T det = fma(a, d, -(b * b));
  if (det != T(0) && isfinite(det)) {
    const T inv = T(1) / det;
    ia = d * inv; ib = -b * inv; id = a * inv;
  } else {
    ia = ib = id = T(0);
  }
}

// Entries cp .. cp + K - 1 of row r of the triangle (K even, the rest zero or
// unused).
template <class Lay, int N, typename T>
__device__ inline void load_row(const T* A, int r, int cp, int K, T (&x)[N]) {
  const T* row = A + Lay::at(r, cp);
  if constexpr (std::is_same<Lay, RowBlockTri>::value) {
    constexpr int Q = 16 / sizeof(T);
#pragma unroll
    for (int g = 0; g < N / Q; ++g) {
      Quad<T> q{};
      if (Q * g < K) q = reinterpret_cast<const Quad<T>*>(row)[g];
#pragma unroll
      for (int i = 0; i < Q; ++i) x[Q * g + i] = q.v[i];
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) x[j] = j < K ? row[j] : T(0);
  }
}

// Two passes eliminate a panel's pairs.  panel_diag: the panel's own rows (rows
// and columns cp .. cp + K - 1) by one warp, lane r holding row cp + r in
// registers; a pair's two columns, final once the earlier pairs are applied, go
// to ud (entry (r, c) at ud[c LU + r]), from where every lane reads them; L
// columns of these rows to Lout, pivots to piv.  panel_rows: the rows below
// (cp + K .. msz - 1), one thread per row, the row's panel entries in registers:
// final unscaled entries to W, multipliers to Lp and Lout.  pinv: the pairs'
// pivot inverses.
// Bound: panel_diag the chain of pivots (a shuffle and a reciprocal per pair;
// FP64: the FP64 pipe), panel_rows shared-memory loads and stores.
template <int PB>
constexpr int UD_LD = 2 * PB;
// window_update reads up to PB entries past the last column
template <int PB>
constexpr int UD_ELEMS = 2 * PB * UD_LD<PB> + PB;

template <class Lay, int PB>
__device__ __noinline__ void panel_diag(const double* A, int cp, int K, double* ud,
                                        double* __restrict__ Lout, int lds, double (*piv)[3]) {
  constexpr int LU = UD_LD<PB>;
  const int lane = threadIdx.x & 31;
  double x[2 * PB];
  load_row<Lay>(A, cp + (lane < K ? lane : 0), cp, K, x);
#pragma unroll
  for (int kk = 0; kk < 2 * PB; kk += 2) {
    if (kk >= K) break;
    double* U0 = ud + kk * LU;
    double* U1 = U0 + LU;
    if (lane >= kk && lane < K) {
      U0[lane] = x[kk];
      U1[lane] = x[kk + 1];
    }
    __syncwarp();
    const double a = U0[kk], b = U0[kk + 1], d = U1[kk + 1];
    double ia, ib, id;
    pivot_inverse(a, b, d, ia, ib, id);
    if (lane == 0) {
      piv[kk >> 1][0] = a; piv[kk >> 1][1] = b; piv[kk >> 1][2] = d;
    }
    const double l0 = fma(x[kk], ia, x[kk + 1] * ib);
    const double l1 = fma(x[kk], ib, x[kk + 1] * id);
    if (lane > kk + 1 && lane < K) {
      Lout[(size_t)(cp + kk) * lds + cp + lane] = l0;
      Lout[(size_t)(cp + kk + 1) * lds + cp + lane] = l1;
    }
    pair_row_update<double, PB>(x, kk, U0, U1, l0, l1);
  }
}

template <class Lay, int PB>
__device__ __noinline__ void panel_rows(const double* A, double* W, double* Lp, int ldw, int msz,
                                        int cp, int K, const double* ud,
                                        double* __restrict__ Lout, int lds,
                                        const double (*pinv)[3]) {
  constexpr int LU = UD_LD<PB>;
  for (int r = cp + K + threadIdx.x; r < msz; r += blockDim.x) {
    double x[2 * PB];
    load_row<Lay>(A, r, cp, K, x);
    double* lo = Lout + (size_t)cp * lds + r;
#pragma unroll
    for (int kk = 0; kk < 2 * PB; kk += 2) {
      if (kk >= K) break;
      const double ia = pinv[kk >> 1][0], ib = pinv[kk >> 1][1], id = pinv[kk >> 1][2];
      const double l0 = fma(x[kk], ia, x[kk + 1] * ib);
      const double l1 = fma(x[kk], ib, x[kk + 1] * id);
      W[kk * ldw + r] = x[kk];
      W[(kk + 1) * ldw + r] = x[kk + 1];
      Lp[kk * ldw + r] = l0;
      Lp[(kk + 1) * ldw + r] = l1;
      lo[(size_t)kk * lds] = l0;
      lo[(size_t)(kk + 1) * lds] = l1;
      pair_row_update<double, PB>(x, kk, ud + kk * LU, ud + (kk + 1) * LU, l0, l1);
    }
  }
}

// FP32: a window of the row moves along it, x[i] holding the row's entries of
// columns kk + 2i and kk + 2i + 1 (kk: the current pair's first column), so that
// the multiply-adds go in packed pairs and one loop body serves two pairs:
// panels of 16 pairs run a window of 16 over the first half and one of 8 over the
// rest; panels of 8 are unrolled (the loop's idle entries cost more than its
// shorter code gains).  Entries past the panel are computed from whatever lies
// there and not used.

// The pairs from column k0 on, at most PB / 2 of them and none from k1 on:
// publish(kk, x0, x1) the pair's columns of this row, multipliers(kk, x0, x1,
// l0, l1), then the update of the window's later entries from the pair's columns
// at the panel's own rows (in ud; loaded between the two, so that the loads
// overlap the multipliers' chain).
template <int PB, int NW, class Publish, class Multipliers>
__device__ inline void window_pairs(unsigned long long (&w)[NW], int k0, int k1, int K,
                                    const float* ud, Publish publish, Multipliers multipliers) {
  constexpr int LU = UD_LD<PB>;
  // G: the window's packed entries that are done
  auto one = [&](int kk, const float* U0, auto G) {
    constexpr int g0 = decltype(G)::value;
    float x0, x1, l0, l1;
    unpack2(w[g0 - 1], x0, x1);
    publish(kk, x0, x1);
    ulonglong2 u0[NW / 2], u1[NW / 2];
#pragma unroll
    for (int g = g0 / 2; g < NW / 2; ++g) {
      u0[g] = reinterpret_cast<const ulonglong2*>(U0)[g];
      u1[g] = reinterpret_cast<const ulonglong2*>(U0 + LU)[g];
    }
    multipliers(kk, x0, x1, l0, l1);
    const unsigned long long m0 = pack2(-l0, -l0), m1 = pack2(-l1, -l1);
#pragma unroll
    for (int g = g0 / 2; g < NW / 2; ++g) {
      if (2 * g >= g0) w[2 * g] = fma2(m1, u1[g].x, fma2(m0, u0[g].x, w[2 * g]));
      w[2 * g + 1] = fma2(m1, u1[g].y, fma2(m0, u0[g].y, w[2 * g + 1]));
    }
  };
#pragma unroll(PB == 8 ? PB / 4 : 1)
  for (int i = 0; i < PB / 4; ++i) {
    const int kk = k0 + 4 * i;
    if (kk >= k1) break;
    const float* U = ud + kk * LU + kk;   // 16-byte aligned
    one(kk, U, std::integral_constant<int, 1>());
    if (kk + 2 < K) one(kk + 2, U + 2 * LU, std::integral_constant<int, 2>());
#pragma unroll
    for (int j = 0; j < NW; ++j) w[j] = j + 2 < NW ? w[j + 2] : 0ull;   // two pairs on
  }
}
// All pairs of a panel on the row x.
template <int PB, class Publish, class Multipliers>
__device__ inline void panel_window(const float (&x)[2 * PB], int K, const float* ud,
                                    Publish publish, Multipliers multipliers) {
  unsigned long long w[PB], y[PB / 2];
#pragma unroll
  for (int i = 0; i < PB; ++i) w[i] = pack2(x[2 * i], x[2 * i + 1]);
  window_pairs<PB>(w, 0, min(K, PB), K, ud, publish, multipliers);
#pragma unroll
  for (int i = 0; i < PB / 2; ++i) y[i] = w[i];
  window_pairs<PB>(y, PB, K, K, ud, publish, multipliers);
}

template <class Lay, int PB>
__device__ __noinline__ void panel_diag(const float* A, int cp, int K, float* ud,
                                        float* __restrict__ Lout, int lds, float (*piv)[3]) {
  constexpr int LU = UD_LD<PB>;
  const int lane = threadIdx.x & 31;
  float x[2 * PB];
  load_row<Lay>(A, cp + (lane < K ? lane : 0), cp, K, x);
  auto publish = [&](int kk, float x0, float x1) {
    if (lane >= kk && lane < K) {
      ud[kk * LU + lane] = x0;
      ud[(kk + 1) * LU + lane] = x1;
    }
    __syncwarp();
  };
  panel_window<PB>(x, K, ud, publish, [&](int kk, float x0, float x1, float& l0, float& l1) {
    const float a = __shfl_sync(0xffffffffu, x0, kk);
    const float b = __shfl_sync(0xffffffffu, x0, kk + 1);
    const float d = __shfl_sync(0xffffffffu, x1, kk + 1);
    float ia, ib, id;
    pivot_inverse(a, b, d, ia, ib, id);
    if (lane == 0) {
      piv[kk >> 1][0] = a; piv[kk >> 1][1] = b; piv[kk >> 1][2] = d;
    }
    l0 = fma(x0, ia, x1 * ib);
    l1 = fma(x0, ib, x1 * id);
    if (lane > kk + 1 && lane < K) {
      Lout[(size_t)(cp + kk) * lds + cp + lane] = l0;
      Lout[(size_t)(cp + kk + 1) * lds + cp + lane] = l1;
    }
  });
}

template <class Lay, int PB>
__device__ __noinline__ void panel_rows(const float* A, float* W, float* Lp, int ldw, int msz,
                                        int cp, int K, const float* ud,
                                        float* __restrict__ Lout, int lds,
                                        const float (*pinv)[3]) {
  for (int r = cp + K + threadIdx.x; r < msz; r += blockDim.x) {
    float x[2 * PB];
    load_row<Lay>(A, r, cp, K, x);
    float* lo = Lout + (size_t)cp * lds + r;
    auto publish = [&](int kk, float x0, float x1) {
      W[kk * ldw + r] = x0;
      W[(kk + 1) * ldw + r] = x1;
    };
    panel_window<PB>(x, K, ud, publish, [&](int kk, float x0, float x1, float& l0, float& l1) {
      const float ia = pinv[kk >> 1][0], ib = pinv[kk >> 1][1], id = pinv[kk >> 1][2];
      l0 = fma(x0, ia, x1 * ib);
      l1 = fma(x0, ib, x1 * id);
      Lp[kk * ldw + r] = l0;
      Lp[(kk + 1) * ldw + r] = l1;
      lo[(size_t)kk * lds] = l0;
      lo[(size_t)(kk + 1) * lds] = l1;
    });
  }
}

// The panel's own columns between the two passes, one buffer per CUDA block.
template <typename T>
__device__ inline T* ud_buffer() {
  __shared__ __align__(16) T ud[UD_ELEMS<16>];
  return ud;
}

// Eliminate the first npairs (state, multiplier) pairs of the symmetric msz x
// msz matrix A, stored as a lower triangle (layout Lay), blocked right-looking:
// pairs are taken in panels of PB.  Warp 0 eliminates the pairs on the panel's
// own rows (panel_diag); every thread replays the same eliminations on its rows
// below (panel_rows; a row's multipliers depend only on the diagonal block);
// then the trailing matrix receives one rank-2PB update from the multipliers
// Lp[j][r] and the unscaled columns W[j][r] (leading dimension ldw =
// panel_ld(msz)), in register tiles of TR x TC (4 x 4 per thread at a time for
// TR = 0).  The next panel's diagonal block only needs the trailing tiles it
// lies in: warp 0 takes those first and runs panel_diag for it while the other
// warps go on with the rest (in sequence, this phase was 170 000 of the 1.05
// million cycles of an element at 50 species, 81 000 of 402 000 at 27).
// Every entry sees the arithmetic, in the order, of the pair-by-pair
// elimination: the pivot inverse ia = d / det, ib = -b / det, id = a / det;
// multipliers l0 = x0 ia + x1 ib, l1 = x0 ib + x1 id; the panel's remaining
// columns updated pair by pair; trailing entries by the sum over the panel's
// 2 PB columns in ascending order, subtracted once.
// L columns go to Lout[c * lds + r] (rows r > pair), pivots (a, b, d) to
// Dout[3 q]; inert[0..2] receives the pivots' inertia (counted off the
// elimination's path, by the last warp: its FP64 sign tests are slow).  The
// trailing block (rows and columns >= 2 npairs) is left in A.
// PB is 8 for blocks held in shared memory and 16 for blocks in the global
// slab (half the trailing passes over global memory, twice the arithmetic per
// entry read and written).
template <typename T, class Lay, int PB, int TR, int TC>
__device__ void pair_eliminate_packed(T* A, int msz, int npairs, T* __restrict__ Lout, int lds,
                                      T* __restrict__ Dout, T* Lp, T* W,
                                      int* __restrict__ inert) {
  const int tid = threadIdx.x, nt = blockDim.x, ldw = panel_ld(msz);
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  __shared__ T piv[PB][3], pinv[PB][3];   // pivots and their inverses of the panel's pairs
  __shared__ int turn;                    // trailing tiles taken so far
  T* ud = ud_buffer<T>();
  int pos = 0, neg = 0, zero = 0;
  auto diag = [&](int q0) {
    const int K = 2 * (min(q0 + PB, npairs) - q0);
    panel_diag<Lay, PB>(A, 2 * q0, K, ud, Lout, lds, piv);
    __syncwarp();
    if (lane < K / 2) {
      pivot_inverse(piv[lane][0], piv[lane][1], piv[lane][2], pinv[lane][0], pinv[lane][1],
                    pinv[lane][2]);
#pragma unroll
      for (int i = 0; i < 3; ++i) Dout[3 * (q0 + lane) + i] = piv[lane][i];
    }
  };
  if (warp == 0) diag(0);
  __syncthreads();
  for (int q0 = 0; q0 < npairs; q0 += PB) {
    const int pe = min(q0 + PB, npairs);
    const int cp = 2 * q0, cend = 2 * pe, K = cend - cp;
    panel_rows<Lay, PB>(A, W, Lp, ldw, msz, cp, K, ud, Lout, lds, pinv);
    if (tid == 0) turn = 0;
    if (warp == nw - 1 && lane < K / 2)
      pivot_inertia((double)piv[lane][0], (double)piv[lane][1], (double)piv[lane][2], pos, neg,
                    zero);
    __syncthreads();
    // trailing rank-K update of rows / columns >= cend (lower part)
    auto trailing = [&](TileTurns turns) {
      if constexpr (TR == 0)
        trailing_update_tiles4<T, Lay>(A, msz, cend, K, Lp, W, ldw, turns);
      else if constexpr (std::is_same<Lay, RowBlockTri>::value)
        trailing_update_slab<T, SLAB_TC<T>>(A, msz, cend, K, Lp, W, ldw, turns);
      else
        trailing_update<T, TR, TC>(A, msz, cend, K, Lp, W, ldw, turns);
    };
    int head = 0;
    if (pe < npairs) {
      if constexpr (TR == 0) head = tiles4_head(PB);
      else if constexpr (std::is_same<Lay, RowBlockTri>::value)
        head = slab_head<T, SLAB_TC<T>>(cend);
      else head = packed_head<TR, TC>(msz, cend);
      if (warp == 0) {
        trailing(tiles_in_turn(0, head));
        __syncwarp();
        diag(pe);
      }
    }
    trailing(tiles_shared(head, &turn));
    __syncthreads();
  }
  if (warp == nw - 1) {
    pos = __reduce_add_sync(0xffffffffu, pos);
    neg = __reduce_add_sync(0xffffffffu, neg);
    zero = __reduce_add_sync(0xffffffffu, zero);
    if (lane == 0) { inert[0] = pos; inert[1] = neg; inert[2] = zero; }
  }
}

// Storage of a block of msz rows factored by pair_eliminate_packed: the two
// panel buffers Lp, W (2 PB x panel_ld(msz) each) and the packed triangle
// (msz (msz + 1) / 2).  Everything in shared memory (PB = 8) when it fits the
// factorization limit; otherwise (PB = 16) the triangle in a per-CUDA-block
// global slab (L2-resident) and the panel buffers in shared memory, or, when
// even they do not fit, in the slab behind the triangle.
template <typename T>
__host__ __device__ inline int big_pb(int msz) {
  const size_t full8 = sizeof(T) * (2 * (size_t)16 * panel_ld(msz) + PackedTri::elems(msz));
  return full8 <= FACTOR_SMEM_LIMIT ? 8 : 16;
}
template <typename T>
__host__ __device__ inline size_t big_panel_elems(int msz) {
  return 2 * (size_t)(2 * big_pb<T>(msz)) * panel_ld(msz);
}
// pair_eliminate_packed with PB = 8 (triangle in shared memory) or pb (8 or 16,
// triangle in the global slab, whose panel buffers are sized for 16)
template <typename T, class Lay, int TR, int TC>
__device__ inline void pair_eliminate_big(T* A, int msz, int npairs, T* __restrict__ Lout,
                                          int lds, T* __restrict__ Dout, T* Lp, T* W,
                                          int* __restrict__ inert, int pb) {
  if (std::is_same<Lay, RowBlockTri>::value && pb == 16)
    pair_eliminate_packed<T, Lay, 16, TR, TC>(A, msz, npairs, Lout, lds, Dout, Lp, W, inert);
  else
    pair_eliminate_packed<T, Lay, 8, TR, TC>(A, msz, npairs, Lout, lds, Dout, Lp, W, inert);
}
template <typename T>
__host__ __device__ inline bool panel_in_global(int msz) {
  return sizeof(T) * big_panel_elems<T>(msz) > FACTOR_SMEM_LIMIT;
}
template <typename T>
__host__ __device__ inline size_t slab_elems(int msz) {
  return RowBlockTri::elems(msz) + (panel_in_global<T>(msz) ? big_panel_elems<T>(msz) : 0);
}
template <typename T>
struct BigPlace {
  T* A;
  T* Lp;
  T* W;
};
// Pointers of block storage for this CUDA block (full: all in shared memory).
template <typename T>
__device__ inline BigPlace<T> big_place(unsigned char* smraw, T* work, int msz, bool full) {
  const size_t pn = big_panel_elems<T>(msz) / 2;
  T* slab = work + (size_t)blockIdx.x * slab_elems<T>(msz);
  const bool pg = !full && panel_in_global<T>(msz);
  T* Lp = pg ? slab + RowBlockTri::elems(msz) : reinterpret_cast<T*>(smraw);
  T* A = full ? Lp + 2 * pn : slab;
  return {A, Lp, Lp + pn};
}

// use(load(i)) for i = 0 .. cnt - 1 over the threads of the block, B independent
// loads of a thread in flight before the first use (stores in use() would
// otherwise keep the compiler from moving the next load up).
template <int B, class Load, class Use>
__device__ inline void for_loaded(int cnt, Load load, Use use) {
  const int nt = blockDim.x;
  for (int i = threadIdx.x; i < cnt; i += B * nt) {
    decltype(load(0)) v[B];
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (i + b * nt < cnt) v[b] = load(i + b * nt);
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (i + b * nt < cnt) use(i + b * nt, v[b]);
  }
}

// Scatter assembly of element e's KKT block (packed lower triangle blk, zeroed)
// from its FP64 derivative blocks Wzz, JZ (K n^2), Wzt, JT (K n p), Wobj
// ((K+1)^2 n) and the barrier diagonal sig ((K+1) n, or NULL: zero), which may be in
// shared or global memory.  Out of line (it is not on the elimination's
// path).  Three passes separated by barriers over the nt
// threads of the block: disjoint entries (point Hessian blocks, the identity
// parts of the collocation rows D[k][j], continuity / initial rows, -delta_c,
// border), sums onto those (objective blocks, -h df/dz), then the diagonal.
template <typename T, class Lay>
__device__ __noinline__ void elem_scatter(const DevProb& P, int e, const double* Wzz,
                                          const double* JZ, const double* Wzt, const double* JT,
                                          const double* Wobj, const double* sig, double dw,
                                          double dc, T* blk);
template <typename T, class Tr>
__device__ __noinline__ void gauss_chain_out(const DevProb& P, const DevFactor<T>& F, int e,
                                             int i0, double dc, Tr tr);

// ---- 1. element condensation --------------------------------------------------
// One CUDA block condenses element e: assemble the bordered (2 (K+1) n + p)
// block, eliminate the K n interior pairs, write L, pivots, the 2n x 2n chain
// block, its border, the p x p Schur contribution and the coupling (Radau:
// -I; Gauss: gauss_chain_out).  For blocks above the register-tile limit
// (elem_factor_rt below).  TR x TC: the trailing update's register tile
// (trailing_update), set by the calling kernel's register budget.
template <typename T, class Lay, int TR, int TC>
__device__ void elem_factor_big(const DevProb& P, const DevEval& E,
                                const double* __restrict__ sigma, double dw, double dc,
                                const DevFactor<T>& F, int e, const BigPlace<T>& pl, int pb) {
  const int n = P.n, p = P.p, m = P.m, ext = P.ext, K = P.K, npt = P.np;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nint = K * n;          // interior pairs
  const int i0 = 2 * nint;         // first chain row (2Kn)
  const size_t nn = (size_t)n * n, np = (size_t)n * p;
  T* A = pl.A;
  const int nq = (int)(Lay::elems(ext) * sizeof(T) / 16);
  for (int i = tid; i < nq; i += nt) reinterpret_cast<int4*>(A)[i] = make_int4(0, 0, 0, 0);
  __syncthreads();
  elem_scatter<T, Lay>(P, e, E.Wzz + (size_t)e * K * nn, E.JZ + (size_t)e * K * nn,
                  E.Wzt + (size_t)e * K * np, E.JT + (size_t)e * K * np,
                  E.Wobj + (size_t)e * npt * npt * n,
                  sigma ? sigma + (size_t)e * npt * n : nullptr, dw, dc, A);
  const int ldl = factor_ld<T>(ext);
  pair_eliminate_big<T, Lay, TR, TC>(A, ext, nint, F.Lel + (size_t)e * (2 * nint) * ldl, ldl,
                                F.Del + (size_t)e * nint * 3, pl.Lp, pl.W,
                                F.inert + (size_t)e * 3, pb);
  const int n2 = 2 * n;
  auto tr = [&](int a, int b) { return sym_at<Lay>(A, a, b); };
  double* Sc = F.Scon + (size_t)e * p * p;
  for (int idx = tid; idx < p * p; idx += nt) {
    const int q = idx / p, q2 = idx - q * p;
    Sc[idx] = (double)tr(m + q, m + q2);
  }
  if (P.gauss) {
    gauss_chain_out<T>(P, F, e, i0, dc, tr);
    __syncthreads();
    return;
  }
  T* Aif = F.Aif + (size_t)e * n2 * n2;
  for (int idx = tid; idx < n2 * n2; idx += nt) {
    const int u = idx / n2, v = idx - u * n2;
    Aif[idx] = tr(i0 + u, i0 + v);
  }
  T* Bif = F.Bif + (size_t)e * n2 * p;
  if constexpr (std::is_same<Lay, RowBlockTri>::value) {
    // four rows q of a column per thread, so that the slab's rows are read along
    // their lines
    for (int idx = tid; idx < n2 * ((p + 3) >> 2); idx += nt) {
      const int q4 = idx / n2, u = idx - q4 * n2;
      T v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * q4 + i < p) v[i] = A[Lay::at(m + 4 * q4 + i, i0 + u)];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * q4 + i < p) Bif[u * p + 4 * q4 + i] = v[i];
    }
  } else {
    for (int idx = tid; idx < n2 * p; idx += nt) {
      const int u = idx / p, q = idx - u * p;
      Bif[idx] = A[Lay::at(m + q, i0 + u)];
    }
  }
  T* C = F.Cpl + (size_t)e * n * n;
  for (int idx = tid; idx < n * n; idx += nt) {
    const int s2 = idx / n, t = idx - s2 * n;
    C[idx] = (!chain_start(P, e) && s2 == t) ? T(-1) : T(0);
  }
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(FBS)
k_elem_factor(DevProb P, DevEval E, const double* __restrict__ sigma, double dw, double dc,
              DevFactor<T> F, int use_smem, int slab_pb) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BigPlace<T> pl = big_place<T>(smraw, F.work, P.ext, use_smem != 0);
  constexpr int TC = sizeof(T) == 4 ? 8 : 4;
  for (int e = blockIdx.x; e < P.N; e += gridDim.x)
    if (use_smem) elem_factor_big<T, PackedTri, 8, TC>(P, E, sigma, dw, dc, F, e, pl, 8);
    else elem_factor_big<T, RowBlockTri, 8, TC>(P, E, sigma, dw, dc, F, e, pl, slab_pb);
}

// ---- 1'. pair elimination with the block held in registers -------------------------
// The same elimination as pair_eliminate, organised for small blocks
// (ext <= RT_MAX_EXT): the lower triangle is cut into 4 x 4 tiles and each of
// the NT threads keeps up to TPT tiles in registers for the whole
// elimination.  For every pair the owners of the pair's tile column publish
// the two pivot columns (rows >= the pair) into a shared vector; after one
// barrier every thread forms the pivot inverse and the multipliers of its own
// rows and applies the rank-2 update to its tiles.  The shared vector
// alternates between two buffers, so one barrier per pair suffices: a buffer
// is rewritten only after the barrier that follows all reads of it.  Entries
// that are already eliminated, above the diagonal or past ext take harmless
// finite updates and are never read again.
//   entry(r, c), c <= r < ext: the block's lower triangle (assembly);
//   sink(r, c, v), 2 npairs <= c <= r < ext: the eliminated trailing block;
//   bar(): barrier over the NT threads; tid in [0, NT).
// L columns go to Lout[c * lds + r] (rows r > pair), pivots (a, b, d) to
// Dout[3 q] and pivs[q] (recorded by thread 0, in PAIRED mode by the owner of
// the diagonal tile); after the loop the threads count the pivots' inertia
// into cnt[0..2].  In PAIRED mode the loop's barrier is named barrier 1 over
// the warps that still have work (below); bar() is used outside the loop.
constexpr int RT_MAX_TR = 31;            // tile rows: ext <= 124
constexpr int RT_UB = 4 * RT_MAX_TR + 4;  // rows per pivot-column buffer

template <typename T>
struct alignas(2 * sizeof(T)) Pair {
  T x, y;
};
// Pivot-column buffers: two per elimination, 16-byte aligned for load4.
template <typename T>
struct alignas(16) PivotBuf {
  Pair<T> v[2 * RT_UB];
};

// Four consecutive entries of a pivot-column buffer (16-byte aligned).
__device__ inline void load4(const Pair<float>* p, float x[4], float y[4]) {
  const float4 u = reinterpret_cast<const float4*>(p)[0];
  const float4 v = reinterpret_cast<const float4*>(p)[1];
  x[0] = u.x; y[0] = u.y; x[1] = u.z; y[1] = u.w;
  x[2] = v.x; y[2] = v.y; x[3] = v.z; y[3] = v.w;
}
__device__ inline void load4(const Pair<double>* p, double x[4], double y[4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const double2 w = reinterpret_cast<const double2*>(p)[u];
    x[u] = w.x; y[u] = w.y;
  }
}

template <typename T>
struct Pivot {
  T a, b, d;
};
// Correctly rounded reciprocal (the same value as 1 / x).
__device__ inline float recip_rn(float x) { return __frcp_rn(x); }
__device__ inline double recip_rn(double x) { return __drcp_rn(x); }

constexpr int RT_MAX_PAIRS = 2 * RT_MAX_TR + 2;   // pairs of a block of <= 124 rows
constexpr int RT_MAX_THREADS = 512;               // threads of a register-tiled block

// Tiles are owned in pairs along a tile row: pair (ti, k) is tiles (ti, 2k) and
// (ti, 2k + 1) (the second absent when 2k + 1 > ti), so the multipliers of the
// row are formed once for both.  Pairs are numbered column pair by column pair
// (k ascending, then ti from 2k to R - 1; R - 2k pairs in column pair k), so
// that the threads of a warp hold neighbouring column pairs and finish
// together: a pair has no work left after pair step 4k + 1 (one tile) or
// 4k + 3 (two tiles), when its columns are eliminated and published.
__host__ __device__ inline int tile_pairs(int R) { return (R + 1) * (R + 1) / 4; }
__device__ inline void tile_pair(int t, int R, int& ti, int& k) {
  // first pair of column pair k: k (R + 1 - k)
  int c = (int)(0.5f * ((float)(R + 1) - sqrtf((float)((R + 1) * (R + 1) - 4 * t))));
  if (c < 0) c = 0;
  while (c > 0 && c * (R + 1 - c) > t) --c;
  while ((c + 1) * (R - c) <= t) ++c;
  k = c;
  ti = 2 * c + (t - c * (R + 1 - c));
}

// PAIRED: each thread owns TPP row pairs of tiles (above); otherwise TPP
// single tiles (for latency-bound small blocks, where every thread should
// hold a tile).
template <typename T, int TPP, bool PAIRED, class Entry, class Sink, class Bar>
__device__ void pair_eliminate_rt(int tid, int nt, int ext, int npairs, Entry entry,
                                  T* __restrict__ Lout, int lds, T* __restrict__ Dout, Sink sink,
                                  Bar bar, Pair<T>* ub, Pivot<T>* pivs, int* cnt) {
  constexpr int H = PAIRED ? 2 : 1;
  const int R = (ext + 3) >> 2, npr = PAIRED ? tile_pairs(R) : R * (R + 1) / 2;
  for (int r = tid; r < 2 * RT_UB; r += nt) ub[r] = Pair<T>{T(0), T(0)};
  int ti[TPP], tj0[TPP];
  bool two[TPP];
  T a[TPP][H][4][4];
#pragma unroll
  for (int j = 0; j < TPP; ++j) {
    const int t = tid + nt * j;
    int k = 0;
    ti[j] = -1;
    if (PAIRED) {
      if (t < npr) tile_pair(t, R, ti[j], k);
      tj0[j] = 2 * k;
      two[j] = tj0[j] + 1 <= ti[j];
    } else {
      tj0[j] = 0;
      if (t < npr) tri_tile(t, ti[j], tj0[j]);
      two[j] = false;
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int r = 4 * ti[j] + u, c = 4 * (tj0[j] + h) + v;
          a[j][h][u][v] = (ti[j] >= 0 && (h == 0 || two[j]) && r < ext && c <= r) ? entry(r, c)
                                                                                  : T(0);
        }
  }
  // PAIRED: a warp leaves the pair loop once none of its threads has work left
  // (exit pair = max over its threads of 4k + 2 or 4k + 4); the loop's barrier
  // (named barrier 1) of pair q counts the warps whose exit pair is >= q: those
  // still working wait on it, the one leaving at q only arrives, so its reads
  // of the previous pivot buffer are ordered before that buffer is rewritten.
  int* s_exit = nullptr;
  int* s_count = nullptr;
  int my_exit = npairs;
  if constexpr (PAIRED) {
    __shared__ int exit_of_warp[RT_MAX_THREADS / 32];
    __shared__ int count_of_pair[RT_MAX_PAIRS];
    s_exit = exit_of_warp;
    s_count = count_of_pair;
    int qd = 0;
#pragma unroll
    for (int j = 0; j < TPP; ++j)
      if (ti[j] >= 0) qd = max(qd, min(npairs, two[j] ? 2 * tj0[j] + 4 : 2 * tj0[j] + 2));
    qd = (int)__reduce_max_sync(0xffffffffu, (unsigned)qd);
    if ((tid & 31) == 0) s_exit[tid >> 5] = qd;
  }
  bar();
  if constexpr (PAIRED) {
    const int nw = nt >> 5;
    for (int q = tid; q < npairs; q += nt) {
      int c = 0;
      for (int w = 0; w < nw; ++w) c += s_exit[w] >= q ? 32 : 0;
      s_count[q] = c;
    }
    my_exit = s_exit[tid >> 5];
    bar();
  }
  for (int q = 0; q < npairs; ++q) {
    if constexpr (PAIRED) {
      if (q >= my_exit) {
        asm volatile("bar.arrive 1, %0;" ::"r"(s_count[q]) : "memory");
        break;
      }
    }
    const int c0 = 2 * q, c1 = c0 + 1, tq = c0 >> 2;
    const bool hi = (c0 & 2) != 0;
    Pair<T>* b = ub + (q & 1) * RT_UB;
#pragma unroll
    for (int j = 0; j < TPP; ++j)
#pragma unroll
      for (int h = 0; h < H; ++h)
        if (ti[j] >= 0 && tj0[j] + h == tq && (h == 0 || two[j]))
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = 4 * ti[j] + u;
            if (r >= c0 && r < ext)
              b[r] = Pair<T>{hi ? a[j][h][u][2] : a[j][h][u][0], hi ? a[j][h][u][3] : a[j][h][u][1]};
          }
    if constexpr (PAIRED) asm volatile("bar.sync 1, %0;" ::"r"(s_count[q]) : "memory");
    else bar();
    const T pa = b[c0].x, pb = b[c1].x, pd = b[c1].y;
    const T det = fma(pa, pd, -(pb * pb));
    T ia, ib, id;
    if (det != T(0) && isfinite(det)) {
      const T inv = recip_rn(det);
      ia = pd * inv; ib = -pb * inv; id = pa * inv;
    } else {
      ia = ib = id = T(0);
    }
    // the pivots are recorded by thread 0, or in PAIRED mode by the owner of the
    // diagonal tile (tq, tq), which works at this step
    bool writer = tid == 0;
    if constexpr (PAIRED) {
      writer = false;
#pragma unroll
      for (int j = 0; j < TPP; ++j)
        writer = writer || (ti[j] == tq && (tj0[j] == tq || (two[j] && tj0[j] + 1 == tq)));
    }
    if (writer) {
      Dout[3 * q + 0] = pa; Dout[3 * q + 1] = pb; Dout[3 * q + 2] = pd;
      pivs[q] = Pivot<T>{pa, pb, pd};
    }
#pragma unroll
    for (int j = 0; j < TPP; ++j) {
      if (ti[j] < 0 || 4 * ti[j] + 3 <= c1) continue;   // no live row
      T l0[4], l1[4], xr0[4], xr1[4];
      load4(b + 4 * ti[j], xr0, xr1);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        l0[u] = fma(xr0[u], ia, xr1[u] * ib);
        l1[u] = fma(xr0[u], ib, xr1[u] * id);
      }
      if (tj0[j] == tq || (two[j] && tj0[j] + 1 == tq))
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = 4 * ti[j] + u;
          if (r > c1 && r < ext) {
            Lout[(size_t)c0 * lds + r] = l0[u];
            Lout[(size_t)c1 * lds + r] = l1[u];
          }
        }
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int tj = tj0[j] + h;
        if ((h == 1 && !two[j]) || 4 * tj + 3 <= c1) continue;   // no live column
        T y0[4], y1[4];
        load4(b + 4 * tj, y0, y1);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v)
            a[j][h][u][v] = fma(-l1[u], y1[v], fma(-l0[u], y0[v], a[j][h][u][v]));
      }
    }
  }
  const int cs = 2 * npairs;
#pragma unroll
  for (int j = 0; j < TPP; ++j) {
    if (ti[j] < 0) continue;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      if (h == 1 && !two[j]) continue;
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int r = 4 * ti[j] + u, c = 4 * (tj0[j] + h) + v;
          if (r < ext && c <= r && c >= cs) sink(r, c, a[j][h][u][v]);
        }
    }
  }
  // inertia of the pivots (exact FP64 sign test), off the elimination's
  // critical path: cnt[0..2] = (pos, neg, zero) after the final barrier
  if (tid < 3) cnt[tid] = 0;
  bar();
  int pos = 0, neg = 0, zero = 0;
  for (int q = tid; q < npairs; q += nt)
    pivot_inertia((double)pivs[q].a, (double)pivs[q].b, (double)pivs[q].d, pos, neg, zero);
  if (pos) atomicAdd(&cnt[0], pos);
  if (neg) atomicAdd(&cnt[1], neg);
  if (zero) atomicAdd(&cnt[2], zero);
  bar();
}

struct CtaBar {
  __device__ void operator()() const { __syncthreads(); }
};
// Barrier over the 128 threads of one half of a 256-thread block (named
// barrier 1 + half; barrier 0 is __syncthreads).
struct HalfBar {
  int id;
  __device__ void operator()() const {
    if (id == 1) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
  }
};

// Element block of elem_factor_rt, assembled in shared memory as a packed
// lower triangle (entry (r, c), c <= r, at r (r + 1) / 2 + c) by structured
// scatter passes over the element's derivative blocks, then loaded into the
// threads' register tiles; after the elimination the trailing blocks go back
// through the same buffer and leave in coalesced stores.
template <typename T>
__host__ __device__ inline size_t elem_blk_bytes(const DevProb& P) {
  return (sizeof(T) * ((size_t)P.ext * (P.ext + 1) / 2) + 15) & ~size_t(15);
}
// The element's FP64 derivative blocks (Wzz, JZ: K n^2 each; Wzt, JT: K n p
// each; Wobj: (K+1)^2 n; sigma: (K+1) n), staged behind the triangle.
__host__ __device__ inline size_t elem_raw_doubles(const DevProb& P) {
  const size_t K = P.K, np = P.np;
  return 2 * K * P.n * P.n + 2 * K * P.n * P.p + (np * np + np) * P.n;
}
template <typename T>
__host__ __device__ inline size_t elem_stage_bytes(const DevProb& P) {
  return elem_blk_bytes<T>(P) + sizeof(double) * elem_raw_doubles(P);
}
// i / d and i % d for 0 <= i < 2^22 and 1 <= d <= 4096 through the float
// reciprocal inv = 1 / d: (i + 0.5) / d lies at least 0.5 / d from an integer,
// far more than the float rounding of the product, so the truncation is exact.
__device__ inline int quot(int i, int d, float inv) {
  return (int)(((float)i + 0.5f) * inv);
}
// local index of the state of point j / the multiplier of the element's
// constraint k (groups of grp_point / grp_con): Radau (z1,c1), (z2,c2),
// (z0,c3), (z3,c0); Gauss (z1,c1) .. (z4,c4), (z0, c0 of the next element),
// whose multiplier is k = 0 here
struct LocIndex {
  int n, K;
  bool gauss;
  __device__ int state(int j, int s) const {
    const int g = j == 0 ? (gauss ? K : K - 1) : ((!gauss && j == K) ? K : j - 1);
    return 2 * (g * n + s);
  }
  __device__ int dual(int k, int s) const { return 2 * ((k == 0 ? K : k - 1) * n + s) + 1; }
};

// Element condensation (same elimination as elem_factor_big) with
// pair_eliminate_rt over the nt threads of the block.
// Assembly of element e's KKT block (packed lower triangle in `blk`, shared
// memory) from its derivative blocks.  Kept out of line: inlined, it changes
// how the elimination that follows is compiled (about a quarter more
// instructions there).
template <typename T>
__device__ __noinline__ void elem_assemble_rt(const DevProb& P, const DevEval& E,
                                              const double* __restrict__ sigma, double dw,
                                              double dc, int e, T* blk) {
  const int n = P.n, p = P.p, ext = P.ext, K = P.K, npt = P.np;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nn = n * n, np = n * p, ntri = ext * (ext + 1) / 2;
  const int nob = npt * npt * n, nsg = npt * n;
  // the derivative blocks arrive by asynchronous copies issued all at once
  // (one memory latency per element) while the triangle is cleared
  double* Wzz = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(blk) +
                                          elem_blk_bytes<T>(P));
  double* JZ = Wzz + K * nn;
  double* Wzt = JZ + K * nn;
  double* JT = Wzt + K * np;
  double* Wobj = JT + K * np;
  double* sig = Wobj + nob;
  {
    auto stage = [&](double* dst, const double* src, int cnt) {
      for (int i = tid; i < cnt; i += nt) cp_async_elem(dst + i, src + i);
    };
    stage(Wzz, E.Wzz + (size_t)e * K * nn, K * nn);
    stage(JZ, E.JZ + (size_t)e * K * nn, K * nn);
    stage(Wzt, E.Wzt + (size_t)e * K * np, K * np);
    stage(JT, E.JT + (size_t)e * K * np, K * np);
    stage(Wobj, E.Wobj + (size_t)e * nob, nob);
    if (sigma) stage(sig, sigma + (size_t)e * nsg, nsg);
    else
      for (int i = tid; i < nsg; i += nt) sig[i] = 0.0;
    cp_async_commit();
  }
  for (int i = tid; i < ntri; i += nt) blk[i] = T(0);
  cp_async_wait_all();
  __syncthreads();
  elem_scatter<T, PackedTri>(P, e, Wzz, JZ, Wzt, JT, Wobj, sig, dw, dc, blk);
}

template <typename T, class Lay>
__device__ __noinline__ void elem_scatter(const DevProb& P, int e, const double* Wzz,
                                          const double* JZ, const double* Wzt, const double* JT,
                                          const double* Wobj, const double* sig, double dw,
                                          double dc, T* blk) {
  const int n = P.n, p = P.p, m = P.m, K = P.K, np = P.np;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nn = n * n, np_ = n * p;
  // by value: P may be in global memory, where each store to the triangle would
  // have its fields read again
  const LocIndex ix{n, K, P.gauss != 0};
  auto put = [&](int a, int b, T v) { blk[a >= b ? Lay::at(a, b) : Lay::at(b, a)] = v; };
  // an entry and what is added to it
  struct Sum {
    T* at;
    T old;
    double v;
  };
  auto sum = [&](int a, int b, double v) {
    T* t = blk + (a >= b ? Lay::at(a, b) : Lay::at(b, a));
    return Sum{t, *t, v};
  };
  auto store = [&](int, const Sum& q) { *q.at = q.old + (T)q.v; };
  // 1. disjoint entries: point Hessian blocks, the identity parts of the
  //    collocation rows (D[k][j]), continuity / initial rows, -delta_c, border
  const float inv_n = 1.f / (float)n, inv_p = p > 0 ? 1.f / (float)p : 0.f;
  const float inv_np = 1.f / (float)np;
  for_loaded<4>(K * nn, [&](int i) { return Wzz[i]; }, [&](int i, double v) {
    const int rs = quot(i, n, inv_n), sb = i - rs * n;   // rs = k n + sa
    const int k = quot(rs, n, inv_n), sa = rs - k * n;
    if (sa >= sb) put(ix.state(k + 1, sa), ix.state(k + 1, sb), (T)v);
  });
  for (int i = tid; i < K * np * n; i += nt) {
    const int kj = quot(i, n, inv_n), s2 = i - kj * n;
    const int k1 = quot(kj, np, inv_np), j = kj - k1 * np;
    put(ix.dual(k1 + 1, s2), ix.state(j, s2), (T)P.D[k1 + 1][j]);
  }
  if (!P.gauss) {
    // the element's own continuity / initial row c0 on z0
    for (int s2 = tid; s2 < n; s2 += nt) put(ix.dual(0, s2), ix.state(0, s2), T(1));
  } else if (chain_next(P, e)) {
    // the next element's continuity row: -b_j on every point of this element
    for (int i = tid; i < np * n; i += nt) {
      const int j = quot(i, n, inv_n), s2 = i - j * n;
      put(ix.dual(0, s2), ix.state(j, s2), (T)(-P.bw[j]));
    }
  }
  for (int i = tid; i < np * n; i += nt) {
    const int k = quot(i, n, inv_n), s2 = i - k * n;
    const int a = ix.dual(k, s2);
    put(a, a, (T)(-dc));
  }
  if constexpr (std::is_same<Lay, RowBlockTri>::value) {
    // a warp takes 8 (point, species) x 16 parameters, four of them per lane, so
    // that it meets few lines both in the derivatives' rows and in the slab's
    // (50 species, cycles per element: 100 000 with a warp's lanes along either
    // one, which then meet 32 lines in the other, 58 000 so)
    const int Kn = K * n, nks = (Kn + 7) >> 3, nq = (p + 15) >> 4, lane = tid & 31;
    for (int i = tid >> 5; i < nks * nq; i += nt >> 5) {
      const int q16 = i / nks, q4 = 4 * q16 + (lane & 3);
      const int ks = 8 * (i - q16 * nks) + (lane >> 2);   // ks = k n + s
      if (ks >= Kn) continue;
      const int k = quot(ks, n, inv_n), s2 = ks - k * n;
      const int cz = ix.state(k + 1, s2), cl = ix.dual(k + 1, s2);
      double w[4], j[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (4 * q4 + u < p) {
          w[u] = Wzt[ks * p + 4 * q4 + u];
          j[u] = JT[ks * p + 4 * q4 + u];
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (4 * q4 + u < p) {
          put(m + 4 * q4 + u, cz, (T)w[u]);
          put(m + 4 * q4 + u, cl, (T)j[u]);
        }
    }
  } else {
    for_loaded<4>(K * np_, [&](int i) { return make_double2(Wzt[i], JT[i]); },
                  [&](int i, double2 v) {
      const int ks = quot(i, p, inv_p), q = i - ks * p;     // ks = k n + s
      const int k = quot(ks, n, inv_n), s2 = ks - k * n;
      put(m + q, ix.state(k + 1, s2), (T)v.x);
      put(m + q, ix.dual(k + 1, s2), (T)v.y);
    });
  }
  __syncthreads();
  // 2. sums onto those: objective blocks (same species across points) and the
  //    -h df/dz part of the collocation rows
  const int np2 = np * np;
  const float inv_np2 = 1.f / (float)np2;
  for_loaded<4>(np2 * n, [&](int i) {
    const int s2 = quot(i, np2, inv_np2), jj = i - s2 * np2;
    const int ja = quot(jj, np, inv_np), jb = jj - ja * np;
    const int a = ix.state(ja, s2), b = ix.state(jb, s2);
    return a >= b ? sum(a, b, Wobj[i]) : Sum{nullptr, T(0), 0.0};
  }, [&](int i, const Sum& q) { if (q.at) store(i, q); });
  for_loaded<4>(K * nn, [&](int i) {
    const int rs = quot(i, n, inv_n), sp = i - rs * n;   // rs = k n + sd
    const int k = quot(rs, n, inv_n), sd = rs - k * n;
    return sum(ix.dual(k + 1, sd), ix.state(k + 1, sp), JZ[i]);
  }, store);
  __syncthreads();
  // 3. barrier diagonal and delta_w on the states
  for (int i = tid; i < np * n; i += nt) {
    const int j = quot(i, n, inv_n), s2 = i - j * n;
    const int a = ix.state(j, s2);
    store(i, sum(a, a, (sig ? sig[i] : 0.0) + dw));
  }
  __syncthreads();
}

// Gauss points: the trailing chain group of element e, (z_e0, c_(e+1)0)
// pairs at local rows i0 + 2s, i0 + 2s + 1, leaves in three parts: the z part
// of chain block e (its c part and the constant identity between them are
// written here only when e starts a chain, otherwise by element e - 1), the c
// part of chain block e + 1 with the coupling Cpl[e + 1] = K[c_(e+1)0, z_e0],
// and the borders of both.  tr(a, b): the trailing block's symmetric entry.
// Out of line, so that it does not add to the register demand of the
// elimination kernels it is called from.
template <typename T, class Tr>
__device__ __noinline__ void gauss_chain_out(const DevProb& P, const DevFactor<T>& F, int e,
                                             int i0, double dc, Tr tr) {
  const int n = P.n, p = P.p, m = P.m, n2 = 2 * n;
  const int tid = threadIdx.x, nt = blockDim.x;
  const bool start = chain_start(P, e), next = chain_next(P, e);
  T* Ae = F.Aif + (size_t)e * n2 * n2;
  for (int i = tid; i < n * n; i += nt) {
    const int s2 = i / n, t = i - s2 * n;
    Ae[(2 * s2) * n2 + 2 * t] = tr(i0 + 2 * s2, i0 + 2 * t);
    Ae[(2 * s2) * n2 + 2 * t + 1] = s2 == t ? T(1) : T(0);
    Ae[(2 * s2 + 1) * n2 + 2 * t] = s2 == t ? T(1) : T(0);
    if (start) Ae[(2 * s2 + 1) * n2 + 2 * t + 1] = s2 == t ? (T)(-dc) : T(0);
  }
  T* Be = F.Bif + (size_t)e * n2 * p;
  for (int i = tid; i < n * p; i += nt) {
    const int s2 = i / p, q = i - s2 * p;
    Be[(2 * s2) * p + q] = tr(m + q, i0 + 2 * s2);
    if (start) Be[(2 * s2 + 1) * p + q] = T(0);
  }
  if (start) {
    T* C = F.Cpl + (size_t)e * n * n;
    for (int i = tid; i < n * n; i += nt) C[i] = T(0);
  }
  if (next) {
    T* An = F.Aif + (size_t)(e + 1) * n2 * n2;
    T* Cn = F.Cpl + (size_t)(e + 1) * n * n;
    for (int i = tid; i < n * n; i += nt) {
      const int s2 = i / n, t = i - s2 * n;
      An[(2 * s2 + 1) * n2 + 2 * t + 1] = tr(i0 + 2 * s2 + 1, i0 + 2 * t + 1);
      Cn[i] = tr(i0 + 2 * s2 + 1, i0 + 2 * t);
    }
    T* Bn = F.Bif + (size_t)(e + 1) * n2 * p;
    for (int i = tid; i < n * p; i += nt) {
      const int s2 = i / p, q = i - s2 * p;
      Bn[(2 * s2 + 1) * p + q] = tr(m + q, i0 + 2 * s2 + 1);
    }
  }
}

template <typename T, int TPT>
__device__ void elem_factor_rt(const DevProb& P, const DevEval& E,
                               const double* __restrict__ sigma, double dw, double dc,
                               const DevFactor<T>& F, int e, Pair<T>* ub, T* blk) {
  const int n = P.n, p = P.p, m = P.m, ext = P.ext;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nint = P.K * n, i0 = 2 * nint, n2 = 2 * n;
  const float inv_n = 1.f / (float)n, inv_p = p > 0 ? 1.f / (float)p : 0.f;
  elem_assemble_rt<T>(P, E, sigma, dw, dc, e, blk);
  auto entry = [&](int r, int c) -> T { return blk[tri_at(r, c)]; };
  auto sink = [&](int r, int c, T val) { blk[tri_at(r, c)] = val; };
  __shared__ Pivot<T> pivs[RT_MAX_PAIRS];
  __shared__ int cnt[3];
  const int ldl = factor_ld<T>(ext);
  pair_eliminate_rt<T, TPT, true>(tid, nt, ext, nint, entry,
                            F.Lel + (size_t)e * (2 * nint) * ldl, ldl,
                            F.Del + (size_t)e * nint * 3, sink, CtaBar{}, ub, pivs, cnt);
  if (tid == 0) {
    F.inert[e * 3 + 0] = cnt[0]; F.inert[e * 3 + 1] = cnt[1]; F.inert[e * 3 + 2] = cnt[2];
  }
  // trailing block: chain block (2n x 2n, both triangles), its border (p x 2n),
  // parameter part (FP64)
  if (P.gauss) {
    __syncthreads();
    auto tr = [&](int a, int b) { return a >= b ? blk[tri_at(a, b)] : blk[tri_at(b, a)]; };
    gauss_chain_out<T>(P, F, e, i0, dc, tr);
    double* Sc = F.Scon + (size_t)e * p * p;
    for (int i = tid; i < p * p; i += nt) {
      const int q = quot(i, p, inv_p), q2 = i - q * p;
      Sc[i] = (double)(q >= q2 ? blk[tri_at(m + q, m + q2)] : blk[tri_at(m + q2, m + q)]);
    }
    return;
  }
  const float inv_n2 = 1.f / (float)n2;
  T* Aif = F.Aif + (size_t)e * n2 * n2;
  for (int i = tid; i < n2 * n2; i += nt) {
    const int u = quot(i, n2, inv_n2), v = i - u * n2;
    Aif[i] = u >= v ? blk[tri_at(i0 + u, i0 + v)] : blk[tri_at(i0 + v, i0 + u)];
  }
  T* Bif = F.Bif + (size_t)e * n2 * p;
  for (int i = tid; i < n2 * p; i += nt) {
    const int u = quot(i, p, inv_p), q = i - u * p;
    Bif[i] = blk[tri_at(m + q, i0 + u)];
  }
  double* Sc = F.Scon + (size_t)e * p * p;
  for (int i = tid; i < p * p; i += nt) {
    const int q = quot(i, p, inv_p), q2 = i - q * p;
    Sc[i] = (double)(q >= q2 ? blk[tri_at(m + q, m + q2)] : blk[tri_at(m + q2, m + q)]);
  }
  T* C = F.Cpl + (size_t)e * n * n;
  for (int idx = tid; idx < n * n; idx += nt) {
    const int s2 = quot(idx, n, inv_n), t = idx - s2 * n;
    C[idx] = (!chain_start(P, e) && s2 == t) ? T(-1) : T(0);
  }
}

// Tile pairs per thread of elem_factor_rt (1) and its block size for an element
// of size ext (a multiple of 32 threads covering every tile; 0 when the
// element is too large and elem_factor_big is used).
template <typename T>
__host__ __device__ constexpr int rt_tpt() { return 1; }   // tile pairs per thread
template <typename T>
__host__ __device__ inline int rt_block_threads(int ext) {
  const int R = (ext + 3) >> 2;
  if (R > RT_MAX_TR) return 0;
  const int per = (tile_pairs(R) + rt_tpt<T>() - 1) / rt_tpt<T>();
  const int nt = (per + 31) / 32 * 32;
  return nt < 64 ? 64 : nt;
}

// Register cap of the element kernels: enough for the tiles, few enough for
// four (float) or two (double) blocks of 192 threads per SM.
template <typename T>
constexpr int rt_maxnreg() { return sizeof(T) == 4 ? 80 : 128; }

template <typename T>
__global__ void __maxnreg__(rt_maxnreg<T>())
k_elem_factor_rt(DevProb P, DevEval E, const double* __restrict__ sigma, double dw, double dc,
                 DevFactor<T> F) {
  __shared__ PivotBuf<T> ub;
  extern __shared__ double stage_dyn[];
  elem_factor_rt<T, rt_tpt<T>()>(P, E, sigma, dw, dc, F, blockIdx.x, ub.v,
                                 reinterpret_cast<T*>(stage_dyn));
}

// ---- 2. one level of block cyclic reduction -------------------------------------
// Eliminates the blocks at odd multiples of `stride` (final = 1: block 0 alone).
// Local order of the extended block: [interface of block i (2n) | z3 of the
// left neighbour (n) | c0 of the right neighbour (n) | theta (p)].
// Kept out of line: inside the cooperative kernel (80 registers per thread for
// the latency-bound register-tiled reduction blocks) its register demand would
// otherwise shape the whole kernel.
template <typename T, class Lay, int TR, int TC>
__device__ __noinline__ void bcr_factor_big(const DevProb& P, const DevFactor<T>& F, int stride,
                                            int final_level, int bi, const BigPlace<T> pl,
                                            int pb) {
  const int n = P.n, p = P.p, N = P.N, bext = P.bext, n2 = 2 * n;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int i = final_level ? 0 : stride * (2 * bi + 1);
  const int L = final_level ? -1 : i - stride;
  const int R = (!final_level && i + stride < N) ? i + stride : -1;
  const T* Ai = F.Aif + (size_t)i * n2 * n2;
  const T* Ci = F.Cpl + (size_t)i * n * n;
  const T* CR = R >= 0 ? F.Cpl + (size_t)R * n * n : nullptr;
  const T* Bi = F.Bif + (size_t)i * n2 * p;
  T* A = pl.A;
  auto entry = [&](int a, int b) {
    T v = T(0);
    if (a < n2) {
      v = Ai[a * n2 + b];
    } else if (b < n2) {
      if (a < 3 * n) {                       // z3 of left neighbour, t = a - 2n
        if (L >= 0 && (b & 1)) v = Ci[(b >> 1) * n + (a - n2)];
      } else if (a < 4 * n) {                // c0 of right neighbour, s = a - 3n
        if (R >= 0 && !(b & 1)) v = CR[(a - 3 * n) * n + (b >> 1)];
      } else {                               // theta row q = a - 4n
        v = Bi[b * p + (a - 4 * n)];
      }
    }
    return v;
  };
  // a warp per row, four columns of a lane in flight
  for (int a = tid >> 5; a < bext; a += nt >> 5)
    for (int b0 = tid & 31; b0 <= a; b0 += 128) {
      T v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (b0 + 32 * i <= a) v[i] = entry(a, b0 + 32 * i);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (b0 + 32 * i <= a) A[Lay::at(a, b0 + 32 * i)] = v[i];
    }
  __syncthreads();
  const int ldl = factor_ld<T>(bext);
  pair_eliminate_big<T, Lay, TR, TC>(A, bext, n, F.Lb + (size_t)i * n2 * ldl, ldl,
                                F.Db + (size_t)i * n * 3, pl.Lp, pl.W,
                                F.inert + (size_t)(N + i) * 3, pb);
  // scatter the trailing (Schur) block into the neighbours
  auto tr = [&](int a, int b) { return sym_at<Lay>(A, a, b); };
  if (L >= 0) {
    T* AL = F.Aif + (size_t)L * n2 * n2;
    for (int idx = tid; idx < n * n; idx += nt) {
      const int t = idx / n, t2 = idx - t * n;
      AL[(2 * t) * n2 + 2 * t2] += tr(n2 + t, n2 + t2);
    }
    T* BL = F.Bif + (size_t)L * n2 * p;
    for (int idx = tid; idx < n * p; idx += nt) {
      const int t = idx / p, q = idx - t * p;
      BL[(2 * t) * p + q] += A[Lay::at(4 * n + q, n2 + t)];
    }
  }
  if (R >= 0) {
    T* AR = F.Aif + (size_t)R * n2 * n2;
    T* CRw = F.Cpl + (size_t)R * n * n;
    for (int idx = tid; idx < n * n; idx += nt) {
      const int s2 = idx / n, s3 = idx - s2 * n;
      AR[(2 * s2 + 1) * n2 + 2 * s3 + 1] += tr(3 * n + s2, 3 * n + s3);
      CRw[idx] = (L >= 0) ? A[Lay::at(3 * n + s2, n2 + s3)] : T(0);
    }
    T* BR = F.Bif + (size_t)R * n2 * p;
    for (int idx = tid; idx < n * p; idx += nt) {
      const int s2 = idx / p, q = idx - s2 * p;
      BR[(2 * s2 + 1) * p + q] += A[Lay::at(4 * n + q, 3 * n + s2)];
    }
  }
  double* Sc = F.Scon + (size_t)(N + i) * p * p;
  for (int idx = tid; idx < p * p; idx += nt) {
    const int q = idx / p, q2 = idx - q * p;
    Sc[idx] = (double)tr(4 * n + q, 4 * n + q2);
  }
  __syncthreads();
}

// Cyclic-reduction block (same result as bcr_factor_big) with
// pair_eliminate_rt on one half (128 threads) of the block: tid in [0, 128).
// Its inputs are first staged in `stage` (T elements, bcr_stage_elems):
// the block's interface block [2n][2n], its coupling [n][n], the right
// neighbour's coupling [n][n] and its border [2n][p].
// After the elimination the same buffer holds the trailing block (2n + p rows,
// packed lower triangle) on its way to the neighbours.
__host__ __device__ inline size_t bcr_stage_elems(int n, int p) {
  const size_t in = 6 * (size_t)n * n + 2 * (size_t)n * p, m2 = 2 * (size_t)n + p;
  const size_t out = m2 * (m2 + 1) / 2;
  return in > out ? in : out;
}
// Starts the staging of cyclic-reduction block bi's inputs into `stage` (one
// half, tid in [0, 128)); the copies are complete for this thread after
// cp_async_wait_all and for the half after a barrier that follows it.  A
// block's inputs are not written by any other block of its level, so they
// can be staged while the half still works on its previous block.
template <typename T>
__device__ void bcr_stage_issue(const DevProb& P, const DevFactor<T>& F, int stride,
                                int final_level, int bi, int tid, T* stage) {
  const int n = P.n, p = P.p, N = P.N, n2 = 2 * n;
  const int i = final_level ? 0 : stride * (2 * bi + 1);
  const int R = (!final_level && i + stride < N) ? i + stride : -1;
  T* Ai = stage;
  T* Ci = Ai + 4 * n * n;
  T* CR = Ci + n * n;
  T* Bi = CR + n * n;
  const T* gA = F.Aif + (size_t)i * n2 * n2;
  const T* gC = F.Cpl + (size_t)i * n * n;
  const T* gCR = R >= 0 ? F.Cpl + (size_t)R * n * n : nullptr;
  const T* gB = F.Bif + (size_t)i * n2 * p;
  for (int k = tid; k < 4 * n * n; k += 128) cp_async_elem(Ai + k, gA + k);
  for (int k = tid; k < n * n; k += 128) {
    cp_async_elem(Ci + k, gC + k);
    if (gCR) cp_async_elem(CR + k, gCR + k);
    else CR[k] = T(0);
  }
  for (int k = tid; k < n2 * p; k += 128) cp_async_elem(Bi + k, gB + k);
  cp_async_commit();
}

// Factorization of a block whose inputs are staged (complete and visible to
// the half).
template <typename T, int TPT>
__device__ void bcr_factor_staged(const DevProb& P, const DevFactor<T>& F, int stride,
                                  int final_level, int bi, int tid, HalfBar bar, Pair<T>* ub,
                                  T* stage, Pivot<T>* pivs, int* cnt) {
  const int n = P.n, p = P.p, N = P.N, bext = P.bext, n2 = 2 * n;
  const int i = final_level ? 0 : stride * (2 * bi + 1);
  const int L = final_level ? -1 : i - stride;
  const int R = (!final_level && i + stride < N) ? i + stride : -1;
  T* Ai = stage;
  T* Ci = Ai + 4 * n * n;
  T* CR = Ci + n * n;
  T* Bi = CR + n * n;
  auto entry = [&](int a, int b) -> T {
    if (a < n2) return Ai[a * n2 + b];
    if (b >= n2) return T(0);
    if (a < 3 * n)                 // z3 of left neighbour, t = a - 2n
      return (L >= 0 && (b & 1)) ? Ci[(b >> 1) * n + (a - n2)] : T(0);
    if (a < 4 * n)                 // c0 of right neighbour, s = a - 3n
      return (R >= 0 && !(b & 1)) ? CR[(a - 3 * n) * n + (b >> 1)] : T(0);
    return Bi[b * p + (a - 4 * n)];  // theta row q = a - 4n
  };
  // the trailing (Schur) block, local rows [z3 of L (n) | c0 of R (n) | theta (p)],
  // is collected in the staging buffer (the inputs are in registers by now) ...
  const int b2 = 2 * n;
  auto sink = [&](int r, int c, T val) { stage[tri_at(r - b2, c - b2)] = val; };
  const int ldl = factor_ld<T>(bext);
  pair_eliminate_rt<T, TPT, false>(tid, 128, bext, n, entry, F.Lb + (size_t)i * n2 * ldl, ldl,
                            F.Db + (size_t)i * n * 3, sink, bar, ub, pivs, cnt);
  if (tid == 0) {
    int* in = F.inert + (size_t)(N + i) * 3;
    in[0] = cnt[0]; in[1] = cnt[1]; in[2] = cnt[2];
  }
  // ... and added into the neighbours in coalesced passes of independent
  // read-modify-writes: z3 x z3 into the left neighbour's interface block and
  // border, c0 x c0 into the right one's, the new coupling c0(R) x z3(L), and
  // the p x p part into this block's parameter contribution
  auto tr = [&](int a, int b) { return a >= b ? stage[tri_at(a, b)] : stage[tri_at(b, a)]; };
  const float inv_n = 1.f / (float)n, inv_p = p > 0 ? 1.f / (float)p : 0.f;
  if (L >= 0) {
    T* AL = F.Aif + (size_t)L * n2 * n2;
    for (int k = tid; k < n * n; k += 128) {
      const int t = quot(k, n, inv_n), t2 = k - t * n;
      AL[(2 * t) * n2 + 2 * t2] += tr(t, t2);
    }
    T* BL = F.Bif + (size_t)L * n2 * p;
    for (int k = tid; k < n * p; k += 128) {
      const int t = quot(k, p, inv_p), q = k - t * p;
      BL[(2 * t) * p + q] += tr(2 * n + q, t);
    }
  }
  if (R >= 0) {
    T* AR = F.Aif + (size_t)R * n2 * n2;
    T* CRw = F.Cpl + (size_t)R * n * n;
    for (int k = tid; k < n * n; k += 128) {
      const int s2 = quot(k, n, inv_n), t = k - s2 * n;
      AR[(2 * s2 + 1) * n2 + 2 * t + 1] += tr(n + s2, n + t);
      CRw[k] = L >= 0 ? tr(n + s2, t) : T(0);
    }
    T* BR = F.Bif + (size_t)R * n2 * p;
    for (int k = tid; k < n * p; k += 128) {
      const int s2 = quot(k, p, inv_p), q = k - s2 * p;
      BR[(2 * s2 + 1) * p + q] += tr(2 * n + q, n + s2);
    }
  }
  double* Sc = F.Scon + (size_t)(N + i) * p * p;
  for (int k = tid; k < p * p; k += 128) {
    const int q = quot(k, p, inv_p), q2 = k - q * p;
    Sc[k] = (double)tr(2 * n + q, 2 * n + q2);
  }
  bar();   // the buffer is restaged by this half's next block
}

// bcr_factor_staged with its staging waited for (no overlap).
template <typename T, int TPT>
__device__ void bcr_factor_rt(const DevProb& P, const DevFactor<T>& F, int stride,
                              int final_level, int bi, int tid, HalfBar bar, Pair<T>* ub,
                              T* stage, Pivot<T>* pivs, int* cnt) {
  bcr_stage_issue<T>(P, F, stride, final_level, bi, tid, stage);
  cp_async_wait_all();
  bar();
  bcr_factor_staged<T, TPT>(P, F, stride, final_level, bi, tid, bar, ub, stage, pivs, cnt);
}

// Tiles per thread of bcr_factor_rt for P (single tiles; 0: use bcr_factor_big).
__host__ __device__ inline int bcr_rt_tiles(int bext) {
  const int R = (bext + 3) >> 2;
  if (R > RT_MAX_TR) return 0;
  const int tpt = (R * (R + 1) / 2 + 127) / 128;
  return tpt <= 2 ? tpt : 0;
}

__host__ __device__ inline int bcr_level_blocks(int N, int stride) {
  return (N - stride + 2 * stride - 1) / (2 * stride);
}

template <typename T, int BT>
__global__ void __launch_bounds__(FBS)
k_bcr_factor(DevProb P, DevFactor<T> F, int stride, int final_level, int use_smem, int slab_pb) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nblk = final_level ? 1 : bcr_level_blocks(P.N, stride);
  if constexpr (BT > 0) {
    // two blocks of the level per CUDA block, one per half
    __shared__ PivotBuf<T> ub[2];
    __shared__ Pivot<T> pivs[2][RT_MAX_PAIRS];
    __shared__ int cnt[2][3];
    const int half = threadIdx.x >> 7;
    T* stage = reinterpret_cast<T*>(smraw) + half * bcr_stage_elems(P.n, P.p);
    for (int bi = 2 * blockIdx.x + half; bi < nblk; bi += 2 * gridDim.x)
      bcr_factor_rt<T, BT>(P, F, stride, final_level, bi, threadIdx.x & 127, HalfBar{1 + half},
                           ub[half].v, stage, pivs[half], cnt[half]);
  } else {
    const BigPlace<T> pl = big_place<T>(smraw, F.work, P.bext, use_smem != 0);
    constexpr int TC = sizeof(T) == 4 ? 8 : 4;
    for (int bi = blockIdx.x; bi < nblk; bi += gridDim.x)
      if (use_smem)
        bcr_factor_big<T, PackedTri, 8, TC>(P, F, stride, final_level, bi, pl, 8);
      else
        bcr_factor_big<T, RowBlockTri, 8, TC>(P, F, stride, final_level, bi, pl, slab_pb);
  }
}

// ---- 3. parameter Schur complement (FP64) ------------------------------------------
// part[g][l] = sum of X[c][l] over the g-th of G contiguous chunks of c.
constexpr int CS_BS = 256;
__device__ inline double chunk_sum_item(const double* __restrict__ X, int C, int L, int G, int g,
                                        int l) {
  const int c0 = (int)((long long)C * g / G), c1 = (int)((long long)C * (g + 1) / G);
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int c = c0;
  for (; c + 3 < c1; c += 4) {
    a0 += X[(size_t)c * L + l];
    a1 += X[(size_t)(c + 1) * L + l];
    a2 += X[(size_t)(c + 2) * L + l];
    a3 += X[(size_t)(c + 3) * L + l];
  }
  for (; c < c1; ++c) a0 += X[(size_t)c * L + l];
  return (a0 + a1) + (a2 + a3);
}

__global__ void __launch_bounds__(CS_BS)
k_chunk_sums(const double* __restrict__ X, int C, int L, int G, double* __restrict__ part) {
  const int l = blockIdx.x * CS_BS + threadIdx.x;
  const int g = blockIdx.y;
  if (l >= L) return;
  part[(size_t)g * L + l] = chunk_sum_item(X, C, L, G, g, l);
}

cudaError_t launch_chunk_sums(const double* X, int C, int L, double* part, cudaStream_t st) {
  if (L <= 0) return cudaSuccess;
  dim3 grid(ceil_div(L, CS_BS), n_chunks(C));
  count_launch();
  k_chunk_sums<<<grid, CS_BS, 0, st>>>(X, C, L, n_chunks(C), part);
  return cudaGetLastError();
}

// Sum of the chunk sums of entry l, by one thread: four interleaved partial sums,
// sixteen loads in flight.
__device__ inline double sum_chunks(const double* __restrict__ part, int G, int L, int l) {
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  const int G4 = G & ~3;
  for (int g0 = 0; g0 < G4; g0 += 16) {
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = g0 + i < G4 ? part[(size_t)(g0 + i) * L + l] : 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (g0 + i < G4) a[i & 3] += v[i];
  }
  for (int g = G4; g < G; ++g) a[0] += part[(size_t)g * L + l];
  return (a[0] + a[1]) + (a[2] + a[3]);
}

// Total of entry idx of the p x p contributions, left in its first chunk's place
// (by the one thread that handles the entry); only the lower triangle is used.
__device__ inline void schur_total(double* chunkS, int N, int p, int idx) {
  const int q = idx / p, q2 = idx - q * p;
  if (q2 <= q) chunkS[idx] = sum_chunks(chunkS, n_chunks(2 * N), p * p, idx);
}
__global__ void __launch_bounds__(CS_BS) k_schur_total(double* chunkS, int N, int p) {
  const int idx = blockIdx.x * CS_BS + threadIdx.x;
  if (idx < p * p) schur_total(chunkS, N, p, idx);
}

// The same sum by the four lanes of a quad (quarter 0 .. 3), which call together,
// whatever the warp's other lanes do: the four partial sums of sum_chunks, each
// with its loads in flight at once, added in its order; every lane of the quad
// returns it.
__device__ inline double sum_chunks4(const double* __restrict__ part, int G, int L, int l,
                                     int quarter) {
  const int G4 = G & ~3;
  double a = 0.0;
  for (int g0 = quarter; g0 < G4; g0 += 32) {
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = g0 + 4 * i < G4 ? part[(size_t)(g0 + 4 * i) * L + l] : 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (g0 + 4 * i < G4) a += v[i];
  }
  if (quarter == 0)
    for (int g = G4; g < G; ++g) a += part[(size_t)g * L + l];
  const unsigned quad = 0xfu << (threadIdx.x & 28);
  a += __shfl_xor_sync(quad, a, 1);
  return a + __shfl_xor_sync(quad, a, 2);
}

constexpr int SBS = 256;
// Whether the block that factors the Schur complement also totals its entries
// (schur_total): one entry of the lower triangle per thread at most.  The totals are
// then one pass over the chunk sums; from two passes on, all blocks share them and a
// grid barrier follows.  A factorization of two species, 50 elements 123.0 us with the
// barrier, 122.1 without, 11 species (253 entries), 100 elements 220.1 and 216.7, 10
// species, 400 elements equal.
__host__ __device__ inline bool schur_totals_inside(int p) { return p * (p + 1) / 2 <= SBS; }
// One block: S = (total of all contributions) + diag(W_thth + sigma + dw), FP64
// LDL^T with 1x1 pivots, total inertia.  sums: the chunk sums (summed: their
// totals, schur_total, in the first chunk's place).  work: schur_doubles(p) doubles
// in dynamic shared memory, or S.S itself when that does not fit: the matrix,
// lower triangle column-major (entry (r, c) at c ld + r, the layout of the
// factor left in S.S), and three columns of multipliers.
// Bound: the chain of pivots, each a reciprocal (some 400 cycles in FP64) behind
// the update of its column.  Warp 0 updates column k + 1 first and inverts its
// pivot while the other warps apply column k to the columns beyond: one barrier
// per column, and the reciprocal is off the other warps' path.
__device__ void schur_block(const DevProb& P, const int* __restrict__ inert,
                            const double* __restrict__ sums, bool summed,
                            const double* __restrict__ wtt, const double* __restrict__ sigma,
                            double dw, const DevSchur& S, double* work) {
  __shared__ long long cnt[3];
  __shared__ long long red[3][SBS];
  const int p = P.p, N = P.N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ld = schur_ld(p);
  const size_t nz = (size_t)N * P.np * P.n;
  double* A = work;
  double* lbuf = A + (size_t)p * ld;
  for (int t = tid; t < p * (p + 1) / 2; t += SBS) {
    int q, q2;
    tri_tile(t, q, q2);
    const int idx = q * p + q2;
    double v = summed ? sums[idx] : sum_chunks(sums, n_chunks(2 * N), p * p, idx);
    if (q == q2) v += wtt[q] + (sigma ? sigma[nz + q] : 0.0) + dw;
    A[(size_t)q2 * ld + q] = v;
  }
  {
    long long a = 0, b = 0, c = 0;
    for (int k = tid; k < 2 * N; k += SBS) { a += inert[3 * k]; b += inert[3 * k + 1]; c += inert[3 * k + 2]; }
    red[0][tid] = a; red[1][tid] = b; red[2][tid] = c;
    __syncthreads();
    for (int s = SBS / 2; s > 0; s >>= 1) {
      if (tid < s) { red[0][tid] += red[0][tid + s]; red[1][tid] += red[1][tid + s]; red[2][tid] += red[2][tid + s]; }
      __syncthreads();
    }
    if (tid == 0) { cnt[0] = red[0][0]; cnt[1] = red[1][0]; cnt[2] = red[2][0]; }
  }
  __syncthreads();
  // multipliers of column k (final) into buffer k % 3, its pivot counted; warp 0
  auto finish = [&](int k) {
    const double d = A[(size_t)k * ld + k];
    const bool ok = (d != 0.0) && isfinite(d);
    const double inv = ok ? 1.0 / d : 0.0;
    double* l = lbuf + (size_t)(k % 3) * p;
    for (int r = k + 1 + lane; r < p; r += 32) l[r] = A[(size_t)k * ld + r] * inv;
    if (lane == 0) {
      if (!ok) cnt[2] += 1; else if (d > 0) cnt[0] += 1; else cnt[1] += 1;
      S.Sd[k] = d;
    }
  };
  // column c -= l u[c], rows c .. p - 1
  auto apply = [&](int c, const double* l, const double* u) {
    const double uc = u[c];
    double* col = A + (size_t)c * ld;
    for (int r = c + lane; r < p; r += 32) col[r] = fma(-l[r], uc, col[r]);
  };
  if (warp == 0 && p > 0) finish(0);
  __syncthreads();
  for (int k = 0; k < p; ++k) {
    const double* l = lbuf + (size_t)(k % 3) * p;
    const double* u = A + (size_t)k * ld;
    if (warp == 0) {
      if (k + 1 < p) {
        apply(k + 1, l, u);
        __syncwarp();
        finish(k + 1);
      }
    } else {
      // the multipliers of the column before leave for S.S (where they may
      // replace the column itself, which nobody reads any more)
      if (warp == 1 && k > 0) {
        const double* lp = lbuf + (size_t)((k - 1) % 3) * p;
        for (int r = k + lane; r < p; r += 32) S.S[(size_t)(k - 1) * ld + r] = lp[r];
      }
      for (int c = k + 1 + warp; c < p; c += SBS / 32 - 1) apply(c, l, u);
    }
    __syncthreads();
  }
  if (tid == 0) { S.inertia[0] = cnt[0]; S.inertia[1] = cnt[1]; S.inertia[2] = cnt[2]; }
  __syncthreads();
}

__global__ void __launch_bounds__(SBS)
k_schur(DevProb P, const int* __restrict__ inert, const double* __restrict__ chunkS,
        const double* __restrict__ wtt, const double* __restrict__ sigma, double dw,
        DevSchur S, int in_global) {
  extern __shared__ double sS[];
  schur_block(P, inert, chunkS, true, wtt, sigma, dw, S, in_global ? S.S : sS);
}

// ---- solves: one warp or a group of them per block -----------------------------------
// Blocks of at most SOLVE_NARROW rows are solved by one warp each, eight at a
// time in a CUDA block; larger ones by the whole CUDA block, or, many of them at
// once, by groups of its warps (subst.cuh, launch_solve_b).  One solve against one warp per block throughout, two columns loaded per step: 10
// species, 400 elements 148 -> 133 us; 27 species, 415 elements 394 -> 166 us; 50
// species, 2000 elements 1692 -> 671 us.
constexpr int SOLVE_NARROW = 128;
constexpr int SOLVE_G = SUB_WARPS;
// Rows up to which groups of four warps beat one of eight when there are many wide
// blocks (launch_solve_b).
constexpr int SOLVE_G4_ROWS = 320;
static_assert(SUB_WARPS == FBS / 32, "one block's warps");
__host__ __device__ inline bool elem_solve_wide(const DevProb& P) { return P.ext > SOLVE_NARROW; }
__host__ __device__ inline bool bcr_solve_wide(const DevProb& P) { return P.bext > SOLVE_NARROW; }
// Dynamic shared memory of a solve kernel: narrow blocks of at most pn rows, wide
// ones of at most pw, a parameter block of max_p (each 0: none).  Three panels in
// flight per group (two, one), if two CUDA blocks then still fit an SM; else as
// many as one block has room for.
constexpr size_t SOLVE_HALF_SM = 110 * 1024;
template <typename T, int G>
static size_t group_smem(int msz, int groups, int most = SUB_STAGES, bool half = false) {
  const size_t v = sizeof(T) * sub_vec_elems(msz), pn = sub_slot_bytes<T, G>(msz);
  auto bytes = [&](int st) { return groups * ((v + st * pn + 15) & ~size_t(15)); };
  for (size_t cap : {SOLVE_HALF_SM, size_t(200 * 1024)})
    for (int st = most; st > 1 && !(half && cap > SOLVE_HALF_SM); --st)
      if (bytes(st) <= cap) return bytes(st);
  return bytes(1);
}
// many[0], many[1]: many narrow / wide blocks (more than two for each warp / CUDA
// block the device holds).  Then two CUDA blocks per SM hide the chains better than
// more panels in flight, if one panel of each kind leaves room for them, and many
// narrow blocks do with one panel each.  A solve of the first 64, 32 and 16 problems of 5
// to 50 species (100 to 2000 elements): 7.2, 4.2 and 2.0 ms with one CUDA block per SM,
// 4.6, 2.8 and 1.44 with two; one warp per block throughout 5.0, 3.3 and 2.1.  50
// species alone, 2000 elements: 773 against 671 us.
template <typename T>
size_t solve_smem(int pn, int pw, int max_p, const bool (&many)[2]) {
  auto need = [&](bool half) {
    size_t b = max_p > 0 ? group_smem<double, SOLVE_G>(max_p, 1, SUB_STAGES, half) : 0;
    if (pn > 0) b = std::max(b, group_smem<T, 1>(pn, SOLVE_G, many[0] ? 1 : SUB_STAGES, half));
    if (pw > 0) b = std::max(b, group_smem<T, SOLVE_G>(pw, 1, SUB_STAGES, half));
    return b;
  };
  const size_t b = many[0] || many[1] ? need(true) : 0;
  if (b > 0 && b <= SOLVE_HALF_SM) return pw > 0 ? SOLVE_HALF_SM : b;
  return need(false);
}
// The part of the `bytes` of dynamic shared memory of this thread's group, for
// blocks of up to msz rows.
template <typename T, int G>
__device__ inline SubMem<T, G> sub_mem(unsigned char* sm, size_t bytes, int msz,
                                       unsigned long long* bars, int* err) {
  const int g = group_index<G>();
  const size_t share = (bytes / (SOLVE_G / G)) & ~size_t(15);
  return sub_carve<T, G>(sm + g * share, share, msz, bars + g * SUB_STAGES, err);
}
constexpr int SOLVE_BARS = SOLVE_G * SUB_STAGES;   // barriers of a kernel's narrow groups

// The L columns of element e and of reduction block i.
template <typename T>
__device__ inline FactorCols<T> elem_cols(const DevProb& P, const DevFactor<T>& F, int e) {
  const int ld = factor_ld<T>(P.ext), nc = 2 * P.K * P.n;
  return {F.Lel + (size_t)e * nc * ld, ld, P.ext, nc};
}
template <typename T>
__device__ inline FactorCols<T> bcr_cols(const DevProb& P, const DevFactor<T>& F, int i) {
  const int ld = factor_ld<T>(P.bext), nc = 2 * P.n;
  return {F.Lb + (size_t)i * nc * ld, ld, P.bext, nc};
}
// Block bi of the level with this stride (final_level: the last block).
__device__ inline int bcr_block(int stride, int final_level, int bi) {
  return final_level ? 0 : stride * (2 * bi + 1);
}

template <typename T>
__device__ inline void pair_solve_d(T a, T b, T d, T w0, T w1, T& v0, T& v1) {
  const T det = fma(a, d, -(b * b));
  if (det != T(0) && isfinite(det)) {
    const T inv = recip_rn(det);
    v0 = fma(d, w0, -(b * w1)) * inv;
    v1 = fma(a, w1, -(b * w0)) * inv;
  } else {
    v0 = T(0); v1 = T(0);
  }
}

// local index a < m -> position in the API-layout KKT vector of element e.
// Radau: every local row is an unknown of the element.
__device__ inline size_t elem_global(const DevProb& P, int e, int a) {
  const int n = P.n;
  const size_t nx = (size_t)P.N * 4 * n + P.p;
  const int pr = a >> 1, g = (pr >= n) + (pr >= 2 * n) + (pr >= 3 * n), s = pr - g * n;
  if (a & 1) return nx + ((size_t)e * 4 + grp_con(0, 3, g)) * n + s;
  return ((size_t)e * 4 + grp_point(0, 3, g)) * n + s;
}
// Gauss: the chain group's multipliers are the next element's c0, absent
// (-1) after a chain's last element, whose block has zero rows there apart
// from -delta_c.
__device__ inline long long elem_global_gauss(const DevProb& P, int e, int a) {
  const int n = P.n, np = P.np;
  const size_t nx = (size_t)P.N * np * n + P.p;
  const int pr = a >> 1, g = pr / n, s = pr - g * n;
  if (a & 1) {
    if (g == P.K) return chain_next(P, e) ? (long long)(nx + (size_t)(e + 1) * np * n + s) : -1;
    return (long long)(nx + ((size_t)e * np + g + 1) * n + s);
  }
  return (long long)(((size_t)e * np + (g < P.K ? g + 1 : 0)) * n + s);
}
// w[a] = v[global index of a] (0 where there is none) for a in [lo, hi), or
// the reverse when store (Gauss elements, by thread tid of nt; out of line).
template <typename T>
__device__ __noinline__ void gauss_elem_gather(const DevProb& P, int e, const double* v, T* w,
                                               int lo, int hi, int tid, int nt) {
  for (int a = lo + tid; a < hi; a += nt) {
    const long long gi = elem_global_gauss(P, e, a);
    w[a] = gi >= 0 ? (T)v[gi] : T(0);
  }
}
template <typename T>
__device__ __noinline__ void gauss_elem_scatter(const DevProb& P, int e, const T* w, double* v,
                                                int lo, int hi, int tid, int nt) {
  for (int a = lo + tid; a < hi; a += nt) {
    const long long gi = elem_global_gauss(P, e, a);
    if (gi >= 0) v[gi] = (double)w[a];
  }
}

// Gauss points: chain right-hand sides after element e's forward
// elimination (wt: the trailing rows (z_e0, c_(e+1)0) interleaved): the z part
// of chain block e and the c part of chain block e + 1 (the rhs of c_(e+1)0
// updated by this element's elimination); a chain's first element also sets
// its own c part, the rhs of its initial condition.  Thread tid of nt.
template <typename T>
__device__ __noinline__ void gauss_chain_rhs(const DevProb& P, const DevFactor<T>& F,
                                             const double* __restrict__ b, int e, const T* wt,
                                             int tid, int nt) {
  const int n = P.n;
  const size_t nx = (size_t)P.N * P.np * n + P.p;
  T* Rif = F.Rif + (size_t)e * 2 * n;
  const bool start = chain_start(P, e), next = chain_next(P, e);
  for (int s2 = tid; s2 < n; s2 += nt) {
    Rif[2 * s2] = wt[2 * s2];
    if (start) Rif[2 * s2 + 1] = (T)b[nx + (size_t)e * P.np * n + s2];
    if (next) F.Rif[(size_t)(e + 1) * 2 * n + 2 * s2 + 1] = wt[2 * s2 + 1];
  }
}

// Forward substitution of element e by a group of G warps: V, the chain rows'
// right-hand side and the parameter rows' contribution.  Here and below, the
// block's first panels have been asked for (sub_start), and next() asks for
// those of the group's next block once this one's substitution is done.
template <typename T, int G, class Next>
__device__ void elem_fwd_one(const DevProb& P, const DevFactor<T>& F, const double* __restrict__ b,
                             int e, SubMem<T, G>& sm, Next next) {
  constexpr int NT = 32 * G;
  const int tid = group_tid<G>();
  const int n = P.n, ext = P.ext, m = P.m, p = P.p, nint = P.K * n;
  T* w = sm.w;
  if (!P.gauss) {
    for (int a = tid; a < ext; a += NT) w[a] = a < m ? (T)b[elem_global(P, e, a)] : T(0);
  } else {
    gauss_elem_gather<T>(P, e, b, w, 0, m, tid, NT);
    for (int a = m + tid; a < ext; a += NT) w[a] = T(0);
  }
  group_sync<G>();
  const T* D = F.Del + (size_t)e * nint * 3;   // asked for before the substitution
  T d0 = T(0), d1 = T(0), d2 = T(0);
  if (tid < nint) { d0 = D[3 * tid]; d1 = D[3 * tid + 1]; d2 = D[3 * tid + 2]; }
  sm.ring.phases = group_forward<G, true>(w, sm.ring, elem_cols(P, F, e));
  next();
  T* V = F.Vint + (size_t)e * 2 * nint;
  for (int q = tid; q < nint; q += NT) {
    if (q >= NT) { d0 = D[3 * q]; d1 = D[3 * q + 1]; d2 = D[3 * q + 2]; }
    T v0, v1;
    pair_solve_d<T>(d0, d1, d2, w[2 * q], w[2 * q + 1], v0, v1);
    V[2 * q] = v0; V[2 * q + 1] = v1;
  }
  T* Rif = F.Rif + (size_t)e * 2 * n;
  if (!P.gauss) {
    for (int u = tid; u < 2 * n; u += NT) Rif[u] = w[2 * nint + u];
  } else {
    gauss_chain_rhs<T>(P, F, b, e, w + 2 * nint, tid, NT);
  }
  double* Rth = F.Rth + (size_t)e * p;
  for (int q = tid; q < p; q += NT) Rth[q] = (double)w[m + q];
  group_sync<G>();
}

template <typename T, int G, class Next>
__device__ void bcr_fwd_one(const DevProb& P, const DevFactor<T>& F, int stride, int final_level,
                            int bi, SubMem<T, G>& sm, Next next) {
  constexpr int NT = 32 * G;
  const int tid = group_tid<G>();
  const int n = P.n, p = P.p, N = P.N, bext = P.bext, n2 = 2 * n;
  const int i = bcr_block(stride, final_level, bi);
  const int L = final_level ? -1 : i - stride;
  const int R = (!final_level && i + stride < N) ? i + stride : -1;
  const T* Rii = F.Rif + (size_t)i * n2;
  T* w = sm.w;
  for (int a = tid; a < bext; a += NT) w[a] = a < n2 ? Rii[a] : T(0);
  // what the end needs from memory, asked for before the substitution: pivots
  // and the neighbours' right-hand sides (this block alone adds to these entries)
  const T* D = F.Db + (size_t)i * n * 3;
  T* RL = F.Rif + (size_t)(L >= 0 ? L : 0) * n2;
  T* RR = F.Rif + (size_t)(R >= 0 ? R : 0) * n2;
  T d0 = T(0), d1 = T(0), d2 = T(0), rl = T(0), rr = T(0);
  if (tid < n) {
    d0 = D[3 * tid]; d1 = D[3 * tid + 1]; d2 = D[3 * tid + 2];
    if (L >= 0) rl = RL[2 * tid];
    if (R >= 0) rr = RR[2 * tid + 1];
  }
  group_sync<G>();
  sm.ring.phases = group_forward<G, true>(w, sm.ring, bcr_cols(P, F, i));
  next();
  T* V = F.Vb + (size_t)i * n2;
  for (int q = tid; q < n; q += NT) {
    if (q >= NT) {
      d0 = D[3 * q]; d1 = D[3 * q + 1]; d2 = D[3 * q + 2];
      if (L >= 0) rl = RL[2 * q];
      if (R >= 0) rr = RR[2 * q + 1];
    }
    T v0, v1;
    pair_solve_d<T>(d0, d1, d2, w[2 * q], w[2 * q + 1], v0, v1);
    V[2 * q] = v0; V[2 * q + 1] = v1;
    if (L >= 0) RL[2 * q] = rl + w[n2 + q];
    if (R >= 0) RR[2 * q + 1] = rr + w[3 * n + q];
  }
  double* Rth = F.Rth + (size_t)(N + i) * p;
  for (int q = tid; q < p; q += NT) Rth[q] = (double)w[4 * n + q];
  group_sync<G>();
}

// Parameter solve by one block of FBS threads: rhs = b_theta + chunk sums of the
// contributions, then the FP64 LDL^T of the Schur complement.  Up to 32 parameters
// (one panel) every thread fetches its share of the factor while the right-hand
// side is summed, and one warp solves with it forward and back, in the arithmetic of
// the panels; those would fetch it twice, each time behind the solve (two species, 200
// elements 99.7 -> 95.0 us a solve, 8 species, 60 elements 69.8 -> 68.2).
__device__ void theta_solve_block(const DevProb& P, const double* __restrict__ chunkR,
                                  const double* __restrict__ b, const DevSchur& S,
                                  double* __restrict__ sol, SubMem<double, SOLVE_G>& sm) {
  const int p = P.p, N = P.N, tid = threadIdx.x;
  const size_t nz = (size_t)N * P.np * P.n;
  double* sv = sm.w;
  const FactorCols<double> L{S.S, factor_ld<double>(p), p, p};
  const bool one_panel = p <= 32;
  const int ld = sub_ld(p);
  double* l = reinterpret_cast<double*>(sm.ring.slots);   // one panel: entry (r, c) at c ld + r
  double d = 0.0;
  if (one_panel) {
    if (tid < p) d = S.Sd[tid];
    for (int i = tid; i < p * p; i += FBS) {
      const int c = i / p, r = i - c * p;
      if (r > c) l[c * ld + r] = S.S[(size_t)c * L.ld + r];
    }
  } else {
    sub_start<SOLVE_G>(sm.ring, L, true);
  }
  for (int q = tid >> 2; q < p; q += FBS / 4) {
    const double v = sum_chunks4(chunkR, n_chunks(2 * N), p, q, tid & 3);
    if ((tid & 3) == 0) sv[q] = b[nz + q] + v;
  }
  __syncthreads();
  if (one_panel) {
    if (tid < 32) {
      const int lane = tid, row = min(lane, p - 1);
      double v = lane < p ? sv[lane] : 0.0;
#pragma unroll 4
      for (int k = 0; k < p; ++k) {
        const double u = fma(-l[k * ld + row], __shfl_sync(0xffffffffu, v, k), v);
        v = lane > k ? u : v;
      }
      v = (d != 0.0 && isfinite(d)) ? v / d : 0.0;
#pragma unroll 4
      for (int j = p - 1; j > 0; --j) {
        const double u = fma(-l[row * ld + j], __shfl_sync(0xffffffffu, v, j), v);
        v = lane < j ? u : v;
      }
      if (lane < p) { sol[nz + lane] = v; S.xth[lane] = v; }
    }
  } else {
    sm.ring.phases = group_forward<SOLVE_G, false>(sv, sm.ring, L);
    sub_start<SOLVE_G>(sm.ring, L, false);
    for (int k = tid; k < p; k += FBS) {
      d = S.Sd[k];
      sv[k] = (d != 0.0 && isfinite(d)) ? sv[k] / d : 0.0;
    }
    __syncthreads();
    sm.ring.phases = group_backward<SOLVE_G, false>(sv, sm.sums, sm.ring, L);
    for (int q = tid; q < p; q += FBS) { sol[nz + q] = sv[q]; S.xth[q] = sv[q]; }
  }
  sub_release();
  __syncthreads();
}

__global__ void __launch_bounds__(FBS)
k_theta_solve(DevProb P, const double* __restrict__ chunkR, const double* __restrict__ b,
              DevSchur S, double* __restrict__ sol, int* err, size_t smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bars[SUB_STAGES];
  sub_init<SOLVE_G>(bars, 1);
  sub_ready();
  SubMem<double, SOLVE_G> sm = sub_mem<double, SOLVE_G>(smraw, smem, P.p, bars, err);
  theta_solve_block(P, chunkR, b, S, sol, sm);
}

template <typename T, int G, class Next>
__device__ void bcr_bwd_one(const DevProb& P, const DevFactor<T>& F, const DevSchur& S,
                            double* __restrict__ sol, int stride, int final_level, int bi,
                            SubMem<T, G>& sm, Next next) {
  constexpr int NT = 32 * G;
  const int tid = group_tid<G>();
  const int n = P.n, p = P.p, N = P.N, bext = P.bext, n2 = 2 * n, np = P.np, cpt = P.cpt;
  const int i = bcr_block(stride, final_level, bi);
  const int L = final_level ? -1 : i - stride;
  const int R = (!final_level && i + stride < N) ? i + stride : -1;
  const size_t nx = (size_t)N * np * n + p;
  const T* V = F.Vb + (size_t)i * n2;
  T* x = sm.w;
  for (int a = tid; a < bext; a += NT) {
    T v = T(0);
    if (a < n2) {
      v = V[a];
    } else if (a < 3 * n) {
      if (L >= 0) v = (T)sol[((size_t)L * np + cpt) * n + (a - n2)];
    } else if (a < 4 * n) {
      if (R >= 0) v = (T)sol[nx + (size_t)R * np * n + (a - 3 * n)];
    } else {
      v = (T)S.xth[a - 4 * n];
    }
    x[a] = v;
  }
  group_sync<G>();
  sm.ring.phases = group_backward<G, true>(x, sm.sums, sm.ring, bcr_cols(P, F, i));
  next();
  for (int s = tid; s < n; s += NT) {
    sol[((size_t)i * np + cpt) * n + s] = (double)x[2 * s];
    sol[nx + (size_t)i * np * n + s] = (double)x[2 * s + 1];
  }
  group_sync<G>();
}

template <typename T, int G, class Next>
__device__ void elem_bwd_one(const DevProb& P, const DevFactor<T>& F, const DevSchur& S,
                             double* __restrict__ sol, int e, SubMem<T, G>& sm, Next next) {
  constexpr int NT = 32 * G;
  const int tid = group_tid<G>();
  const int n = P.n, ext = P.ext, m = P.m;
  const int nint = P.K * n;
  const T* V = F.Vint + (size_t)e * 2 * nint;
  T* x = sm.w;
  for (int a = tid; a < 2 * nint; a += NT) x[a] = V[a];
  if (!P.gauss) {
    for (int a = 2 * nint + tid; a < m; a += NT) x[a] = (T)sol[elem_global(P, e, a)];
  } else {
    gauss_elem_gather<T>(P, e, sol, x, 2 * nint, m, tid, NT);
  }
  for (int a = m + tid; a < ext; a += NT) x[a] = (T)S.xth[a - m];
  group_sync<G>();
  sm.ring.phases = group_backward<G, true>(x, sm.sums, sm.ring, elem_cols(P, F, e));
  next();
  if (!P.gauss)
    for (int a = tid; a < 2 * nint; a += NT) sol[elem_global(P, e, a)] = (double)x[a];
  else
    gauss_elem_scatter<T>(P, e, x, sol, 0, 2 * nint, tid, NT);
  group_sync<G>();
}

// One launch per phase: a narrow block per warp or a wide one per CUDA block
// (G = SOLVE_G).
template <typename T, int G>
__global__ void __launch_bounds__(FBS)
k_elem_solve(DevProb P, DevFactor<T> F, DevSchur S, const double* __restrict__ b,
             double* __restrict__ sol, int fwd, size_t smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bars[SOLVE_BARS];
  sub_init<G>(bars, SOLVE_G / G);
  sub_ready();
  SubMem<T, G> sm = sub_mem<T, G>(smraw, smem, P.ext, bars, &F.gbar->err);
  const int e = G > 1 ? blockIdx.x : blockIdx.x * SOLVE_G + (threadIdx.x >> 5);
  if (e >= P.N) return;
  sub_start<G>(sm.ring, elem_cols(P, F, e), fwd != 0);
  if (fwd) elem_fwd_one<T, G>(P, F, b, e, sm, [] {});
  else elem_bwd_one<T, G>(P, F, S, sol, e, sm, [] {});
}

template <typename T, int G>
__global__ void __launch_bounds__(FBS)
k_bcr_solve(DevProb P, DevFactor<T> F, DevSchur S, double* __restrict__ sol, int fwd, int stride,
            int final_level, size_t smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bars[SOLVE_BARS];
  sub_init<G>(bars, SOLVE_G / G);
  sub_ready();
  SubMem<T, G> sm = sub_mem<T, G>(smraw, smem, P.bext, bars, &F.gbar->err);
  const int nblk = final_level ? 1 : bcr_level_blocks(P.N, stride);
  const int bi = G > 1 ? blockIdx.x : blockIdx.x * SOLVE_G + (threadIdx.x >> 5);
  if (bi >= nblk) return;
  sub_start<G>(sm.ring, bcr_cols(P, F, bcr_block(stride, final_level, bi)), fwd != 0);
  if (fwd) bcr_fwd_one<T, G>(P, F, stride, final_level, bi, sm, [] {});
  else bcr_bwd_one<T, G>(P, F, S, sol, stride, final_level, bi, sm, [] {});
}

// ---- persistent cooperative kernels ------------------------------------------------
// A whole factorization or a whole solve in one cooperative launch: the phases
// of the elimination tree (elements, each cyclic-reduction level, the
// parameter block) are separated by a grid barrier instead of kernel
// boundaries.  Barrier e of a launch completes when the arrival counter
// reaches (e + 1) * gridDim.x: a block arrives with one release reduction
// and waits by polling the counter (no returning atomic on the way, nothing
// to reset between barriers).  The last block to leave the kernel zeroes the
// counter for the next launch.  The wait is bounded: after GridBar::spin_limit
// polls (GRID_SPIN_LIMIT when 0) it records an error in GridBar::err and
// continues, so a fault shows up as a status on the host instead of a hang.
constexpr long long GRID_SPIN_LIMIT = 20000000;   // ~1-2 s of polling

__device__ inline unsigned int ld_acquire_gpu(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// `epoch` counts the barriers this block has passed in the launch.
__device__ void grid_barrier(GridBar* gb, unsigned int& epoch) {
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    // extra and spin_limit are set by the host before the launch
    const unsigned int target = epoch * gridDim.x + gb->extra;
    const long long limit = gb->spin_limit > 0 ? gb->spin_limit : GRID_SPIN_LIMIT;
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->count) : "memory");
    long long spins = 0;
    while (ld_acquire_gpu(&gb->count) < target) {
      __nanosleep(32);
      if (++spins > limit) { atomicExch(&gb->err, 1); break; }
    }
  }
  __syncthreads();
}

// Called by every block as its last statement: every block has passed every
// barrier once the exit count reaches gridDim.x, so the counters can be zeroed.
__device__ void grid_exit(GridBar* gb) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int left = atomicAdd(&gb->exits, 1u) + 1u;
    if (left == gridDim.x) {
      atomicExch(&gb->count, 0u);
      atomicExch(&gb->exits, 0u);
    }
  }
}

// Descriptor of a lone instance in shared memory.  The acquire of a grid barrier
// empties the L1 cache, after which every read through the descriptor in global
// memory waits for the L2 again; with one instance its copy here is used instead.
struct LoneInst {
  alignas(16) unsigned char b[sizeof(DevInst)];
};
__device__ inline void lone_load(LoneInst& s, const DevInst* insts, const int* act, int A) {
  static_assert(sizeof(DevInst) % 8 == 0, "copied by 8-byte words");
  if (A == 1) {
    const double* src = reinterpret_cast<const double*>(insts + act[0]);
    double* dst = reinterpret_cast<double*>(s.b);
    for (int i = threadIdx.x; i < (int)(sizeof(DevInst) / 8); i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
}

// ---- batched persistent kernels -------------------------------------------------------
// Work of all active instances of a batch in one cooperative launch.  Plan
// arrays (device memory, written by the host):
//   pre_elem[A+1]       prefix of element counts
//   pre_lv[l][A+1]      prefix of cyclic-reduction blocks eliminated at level l
//   pre_cs[A+1]         prefix of chunk-sum items (chunks x p^2 for the factor,
//                       chunks x p for the solve)
// Per-instance flags (InstFlags) say whether that instance's blocks fit the
// kernel's shared memory or use its global slabs.
template <typename T>
__device__ inline const DevFactor<T>& inst_factor(const DevInst& I);
template <>
__device__ inline const DevFactor<float>& inst_factor<float>(const DevInst& I) { return I.F32; }
template <>
__device__ inline const DevFactor<double>& inst_factor<double>(const DevInst& I) { return I.F64; }

// Element condensation of a batch with elem_factor_rt: one block per element of
// the work list; instances without flag 4 are condensed inside k_factor_b.
template <typename T>
__global__ void __maxnreg__(rt_maxnreg<T>())
k_elem_factor_rt_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int A,
                   const int* __restrict__ pre_elem, const InstParams* __restrict__ prm,
                   const int* __restrict__ flags) {
  __shared__ PivotBuf<T> ub;
  extern __shared__ double stage_dyn[];
  const int t = blockIdx.x;
  const int k = find_item(pre_elem, A, t);
  if (!(flags[k] & 4)) return;
  const DevInst& I = insts[act[k]];
  elem_factor_rt<T, rt_tpt<T>()>(I.P, I.E, I.sigma, prm[k].dw, prm[k].dc, inst_factor<T>(I),
                                 t - pre_elem[k], ub.v, reinterpret_cast<T*>(stage_dyn));
}

// Element condensation of a batch for the instances whose element blocks are
// above the register-tile limit (without flag 4): elements of the work list
// taken in turn by the CUDA blocks of the grid (at most one global slab per
// CUDA block), block storage in shared memory (flag 1) or in the slab.
// BS threads per block (Schedule::big_threads): 512 with one block per SM, or
// 256 compiled for two blocks per SM (128 registers per thread), so that where
// the shared memory allows, two elements are condensed on an SM at once and
// one block's panel phases overlap the other's trailing update.
template <typename T, int BS>
__global__ void __launch_bounds__(BS, BS == 256 ? 2 : 1)
k_elem_factor_big_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int A,
                    const int* __restrict__ pre_elem, const InstParams* __restrict__ prm,
                    const int* __restrict__ flags, int slab_pb) {
  extern __shared__ __align__(16) unsigned char smraw[];
  for (int t = blockIdx.x; t < pre_elem[A]; t += gridDim.x) {
    const int k = find_item(pre_elem, A, t);
    if (flags[k] & 4) continue;   // condensed by k_elem_factor_rt_b
    const DevInst& I = insts[act[k]];
    const DevFactor<T>& F = inst_factor<T>(I);
    const bool full = (flags[k] & 1) != 0;
    const BigPlace<T> pl = big_place<T>(smraw, F.work, I.P.ext, full);
    // trailing tiles: 8 x 4 (FP32) or 8 x 2 (FP64) within 128 registers per thread
    constexpr int TC = sizeof(T) == 4 ? 4 : 2;
    const int e = t - pre_elem[k];
    const double dw = prm[k].dw, dc = prm[k].dc;
    if (full) elem_factor_big<T, PackedTri, 8, TC>(I.P, I.E, I.sigma, dw, dc, F, e, pl, 8);
    else elem_factor_big<T, RowBlockTri, 8, TC>(I.P, I.E, I.sigma, dw, dc, F, e, pl, slab_pb);
  }
}

// FP32: three blocks per SM (more reduction blocks in flight; the levels are
// latency bound), unless WIDE: when the reduction blocks of the batch need so
// much shared memory that one block per SM is all that fits, the kernel is
// compiled for one block per SM and its large blocks get warp-blocked register
// tiles (same arithmetic per entry).
template <typename T, int BT, int WIDE>
__global__ void __launch_bounds__(FBS, (sizeof(T) == 4 && !WIDE) ? 3 : 1)
k_factor_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int A,
           const int* __restrict__ pre_elem, const int* __restrict__ pre_lv, int maxL,
           const int* __restrict__ pre_cs, const InstParams* __restrict__ prm,
           const int* __restrict__ flags, GridBar* gb, size_t smem_bytes, int bcr_full,
           int slab_pb, int totals) {
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned int ep = 0;
  // 1. element condensation: done by k_elem_factor_rt_b / k_elem_factor_big_b
  // before this launch
  // 2. cyclic-reduction levels, then each instance's final block
  for (int lv = 0; lv <= maxL; ++lv) {
    const int* pre = pre_lv + (size_t)lv * (A + 1);
    const bool fin = lv == maxL;
    const int tot = fin ? A : pre[A];
    if constexpr (BT > 0) {
      // instances with flag 8: two blocks of the level per CUDA block
      __shared__ PivotBuf<T> ubh[2];
      __shared__ Pivot<T> pivh[2][RT_MAX_PAIRS];
      __shared__ int cnth[2][3];
      const int half = threadIdx.x >> 7, htid = threadIdx.x & 127;
      const HalfBar hbar{1 + half};
      // each half owns a fixed half of the dynamic shared memory (instances of
      // different sizes may share the block), split into two stage buffers:
      // the next block's inputs are copied into one while the current block
      // is factored from the other
      const size_t hb = (smem_bytes / 2) & ~size_t(15), bb = (hb / 2) & ~size_t(15);
      unsigned char* hbase = smraw + half * hb;
      auto stage_of = [&](int j) { return reinterpret_cast<T*>(hbase + (j & 1) * bb); };
      auto next_rt = [&](int t) {
        for (; t < tot; t += 2 * gridDim.x)
          if (flags[fin ? t : find_item(pre, A, t)] & 8) break;
        return t;
      };
      auto issue = [&](int t, int j) {
        const int k = fin ? t : find_item(pre, A, t);
        const DevInst& I = insts[act[k]];
        bcr_stage_issue<T>(I.P, inst_factor<T>(I), fin ? 1 : 1 << lv, fin ? 1 : 0,
                           fin ? 0 : t - pre[k], htid, stage_of(j));
      };
      int t = next_rt(2 * blockIdx.x + half), j = 0;
      if (t < tot) issue(t, 0);
      while (t < tot) {
        const int tn = next_rt(t + 2 * gridDim.x);
        cp_async_wait_all();
        hbar();
        // the other buffer's last block ended with a half barrier
        if (tn < tot) issue(tn, j + 1);
        const int k = fin ? t : find_item(pre, A, t);
        const DevInst& I = insts[act[k]];
        bcr_factor_staged<T, BT>(I.P, inst_factor<T>(I), fin ? 1 : 1 << lv, fin ? 1 : 0,
                                 fin ? 0 : t - pre[k], htid, hbar, ubh[half].v, stage_of(j),
                                 pivh[half], cnth[half]);
        t = tn;
        ++j;
      }
    }
    // the whole-block pass reuses the shared memory the halves staged in
    if (BT > 0 && bcr_full) __syncthreads();
    for (int t = blockIdx.x; bcr_full && t < tot; t += gridDim.x) {
      const int k = fin ? t : find_item(pre, A, t);
      if (BT > 0 && (flags[k] & 8)) continue;
      const DevInst& I = insts[act[k]];
      const DevFactor<T>& F = inst_factor<T>(I);
      const bool full = (flags[k] & 2) != 0;
      const BigPlace<T> pl = big_place<T>(smraw, F.work, I.P.bext, full);
      // trailing tiles: warp-blocked 8 x 4 when the kernel runs one block per
      // SM (WIDE), else the 4 x 4 tiles that fit 80 registers per thread
      constexpr int TR = WIDE ? 8 : 0, TC = WIDE ? 4 : 0;
      const int stride = fin ? 1 : 1 << lv, bi = fin ? 0 : t - pre[k];
      if (full) bcr_factor_big<T, PackedTri, TR, TC>(I.P, F, stride, fin, bi, pl, 8);
      else bcr_factor_big<T, RowBlockTri, TR, TC>(I.P, F, stride, fin, bi, pl, slab_pb);
    }
    grid_barrier(gb, ep);
  }
  // 3. chunk sums of the parameter contributions
  for (int t = blockIdx.x * FBS + threadIdx.x; t < pre_cs[A]; t += gridDim.x * FBS) {
    const int k = find_item(pre_cs, A, t);
    const DevInst& I = insts[act[k]];
    const DevFactor<T>& F = inst_factor<T>(I);
    const int L = I.P.p * I.P.p, G = n_chunks(2 * I.P.N);
    const int it = t - pre_cs[k];
    F.chunkS[it] = chunk_sum_item(F.Scon, 2 * I.P.N, L, G, it / L, it % L);
  }
  grid_barrier(gb, ep);
  // ... their totals
  if (totals) {
    for (int t = blockIdx.x * FBS + threadIdx.x; t < pre_cs[A]; t += gridDim.x * FBS) {
      const int k = find_item(pre_cs, A, t);
      const DevInst& I = insts[act[k]];
      if (t - pre_cs[k] < I.P.p * I.P.p && !schur_totals_inside(I.P.p))
        schur_total(inst_factor<T>(I).chunkS, I.P.N, I.P.p, t - pre_cs[k]);
    }
    grid_barrier(gb, ep);
  }
  // 4. parameter Schur complement, one block per instance
  for (int k = blockIdx.x; k < A; k += gridDim.x) {
    const DevInst& I = insts[act[k]];
    const DevFactor<T>& F = inst_factor<T>(I);
    const size_t need = sizeof(double) * schur_doubles(I.P.p);
    double* sS = need <= smem_bytes ? reinterpret_cast<double*>(smraw) : I.S.S;
    schur_block(I.P, F.inert, F.chunkS, !schur_totals_inside(I.P.p), I.E.wtt, I.sigma, prm[k].dw, I.S,
                sS);
    if (threadIdx.x == 0) {
      long long* o = reinterpret_cast<long long*>(I.out + O_INERT);
      o[0] = I.S.inertia[0]; o[1] = I.S.inertia[1]; o[2] = I.S.inertia[2];
    }
  }
  grid_exit(gb);
}

// Work lists of the batched solve: prefix arrays over the active instances of
// the elements and of the reduction blocks of each level, separately for the
// instances whose blocks are narrow (one warp each) and wide (one CUDA block).
struct SolvePlan {
  const int* elem[2];   // [wide][A + 1]
  const int* lv[2];     // [wide][level][A + 1]
};

// Batched solve.  Levels below `lsplit` run over the whole grid, a grid
// barrier after each; from level `lsplit` up (few blocks per instance) one
// block owns an instance and separates its levels by block barriers, and the
// same block then solves the parameter system and substitutes back down to
// level `lsplit`.  Every block solve is the same code as in the
// single-instance launches, so the result does not depend on the split.
template <typename T, int WG>
__global__ void __launch_bounds__(FBS, sizeof(T) == 4 ? 2 : 1)
k_solve_b(const DevInst* __restrict__ insts, const int* __restrict__ act, int A, SolvePlan sp,
          const int* __restrict__ pre_lv, int maxL, int lsplit,
          const int* __restrict__ pre_cs, int ir, int pn, int pw, int max_p, size_t smem,
          GridBar* gb) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int WIDE = SOLVE_G / WG;   // groups for wide blocks
  __shared__ unsigned long long bars[SOLVE_BARS + (WIDE + 1) * SUB_STAGES];
  __shared__ LoneInst lone;
  lone_load(lone, insts, act, A);
  unsigned long long* wide_bars = bars + SOLVE_BARS;
  unsigned long long* theta_bars = wide_bars + WIDE * SUB_STAGES;
  sub_init<1>(bars, SOLVE_G);
  sub_init<WG>(wide_bars, WIDE);
  sub_init<SOLVE_G>(theta_bars, 1);
  sub_ready();
  auto inst = [&](int k) -> const DevInst& {
    return A == 1 ? *reinterpret_cast<const DevInst*>(lone.b) : insts[act[k]];
  };
  unsigned int ep = 0;
  const int warp = threadIdx.x >> 5, wpb = FBS / 32;
  const int gw = blockIdx.x * wpb + warp, nw = gridDim.x * wpb;
  const int wg = blockIdx.x * WIDE + group_index<WG>(), nwg = gridDim.x * WIDE;
  // the three groups use the same shared memory, one at a time
  SubMem<T, 1> narrow = sub_mem<T, 1>(smraw, smem, max(pn, 1), bars, &gb->err);
  SubMem<T, WG> wide = sub_mem<T, WG>(smraw, smem, max(pw, 1), wide_bars, &gb->err);
  SubMem<double, SOLVE_G> theta =
      sub_mem<double, SOLVE_G>(smraw, smem, max(max_p, 1), theta_bars, &gb->err);
  auto phase_end = [&]() { sub_release(); grid_barrier(gb, ep); };
  // Items t0, t0 + step, ... of a list for one group: cols(I, i) are an item's L
  // columns, run(I, i, next) its substitution.
  auto list = [&](const int* pre, int t0, int step, auto& sm, bool fwd, auto&& cols, auto&& run) {
    constexpr int G = std::is_same_v<std::decay_t<decltype(sm)>, SubMem<T, 1>> ? 1 : WG;
    const int tot = pre[A];
    auto find = [&](int t) { return A == 1 ? 0 : find_item(pre, A, t); };
    int k = t0 < tot ? find(t0) : 0;
    if (t0 < tot) sub_start<G>(sm.ring, cols(inst(k), t0 - pre[k]), fwd);
    for (int t = t0; t < tot; t += step) {
      const int tn = t + step, kn = tn < tot ? find(tn) : 0;
      run(inst(k), t - pre[k],
          [&] { if (tn < tot) sub_start<G>(sm.ring, cols(inst(kn), tn - pre[kn]), fwd); });
      k = kn;
    }
  };
  // a phase's wide and narrow blocks; a kind that no instance has is not looked for
  // (a list's length is a read of the L2 on every level's path)
  auto both = [&](const int* narrows, const int* wides, bool fwd, auto&& cols, auto&& one) {
    if (pw > 0) {
      list(wides, wg, nwg, wide, fwd, cols, one(wide));
      sub_release();
      __syncthreads();
    }
    if (pn > 0) list(narrows, gw, nw, narrow, fwd, cols, one(narrow));
  };
  auto elems = [&](bool fwd) {
    auto cols = [&](const DevInst& I, int e) { return elem_cols(I.P, inst_factor<T>(I), e); };
    auto one = [&](auto& sm) {
      return [&, fwd](const DevInst& I, int e, auto next) {
        if (fwd) elem_fwd_one(I.P, inst_factor<T>(I), ir ? I.kr : I.ka, e, sm, next);
        else elem_bwd_one(I.P, inst_factor<T>(I), I.S, ir ? I.kc : I.kb, e, sm, next);
      };
    };
    both(sp.elem[0], sp.elem[1], fwd, cols, one);
  };
  auto level = [&](int lv, bool fwd) {
    const size_t o = (size_t)lv * (A + 1);
    auto cols = [&](const DevInst& I, int bi) {
      return bcr_cols(I.P, inst_factor<T>(I), bcr_block(1 << lv, 0, bi));
    };
    auto one = [&](auto& sm) {
      return [&, fwd](const DevInst& I, int bi, auto next) {
        if (fwd) bcr_fwd_one(I.P, inst_factor<T>(I), 1 << lv, 0, bi, sm, next);
        else bcr_bwd_one(I.P, inst_factor<T>(I), I.S, ir ? I.kc : I.kb, 1 << lv, 0, bi, sm, next);
      };
    };
    both(sp.lv[0] + o, sp.lv[1] + o, fwd, cols, one);
  };
  // the levels from lsplit up of instance k, by this block
  auto top = [&](const DevInst& I, int k, int lv, bool fwd) {
    const int fin = lv == maxL, stride = fin ? 1 : 1 << lv;
    const int* pre = pre_lv + (size_t)lv * (A + 1);
    const int nb = fin ? 1 : pre[k + 1] - pre[k];
    auto run = [&](int bi, auto& sm, auto g) {
      constexpr int G = decltype(g)::value;
      sub_start<G>(sm.ring, bcr_cols(I.P, inst_factor<T>(I), bcr_block(stride, fin, bi)), fwd);
      if (fwd) bcr_fwd_one(I.P, inst_factor<T>(I), stride, fin, bi, sm, [] {});
      else bcr_bwd_one(I.P, inst_factor<T>(I), I.S, ir ? I.kc : I.kb, stride, fin, bi, sm, [] {});
    };
    if (bcr_solve_wide(I.P))
      for (int bi = group_index<WG>(); bi < nb; bi += WIDE)
        run(bi, wide, std::integral_constant<int, WG>{});
    else
      for (int bi = warp; bi < nb; bi += wpb) run(bi, narrow, std::integral_constant<int, 1>{});
    sub_release();
    __syncthreads();
  };
  elems(true);
  phase_end();
  for (int lv = 0; lv < lsplit; ++lv) {
    level(lv, true);
    phase_end();
  }
  for (int k = blockIdx.x; k < A; k += gridDim.x)
    for (int lv = lsplit; lv <= maxL; ++lv) top(inst(k), k, lv, true);
  phase_end();
  for (int t = blockIdx.x * FBS + threadIdx.x; t < pre_cs[A]; t += gridDim.x * FBS) {
    const int k = find_item(pre_cs, A, t);
    const DevInst& I = inst(k);
    const DevFactor<T>& F = inst_factor<T>(I);
    const int L = I.P.p, G = n_chunks(2 * I.P.N);
    const int it = t - pre_cs[k];
    F.chunkR[it] = chunk_sum_item(F.Rth, 2 * I.P.N, L, G, it / L, it % L);
  }
  phase_end();
  for (int k = blockIdx.x; k < A; k += gridDim.x) {
    const DevInst& I = inst(k);
    theta_solve_block(I.P, inst_factor<T>(I).chunkR, ir ? I.kr : I.ka, I.S, ir ? I.kc : I.kb,
                      theta);
    for (int lv = maxL; lv >= lsplit; --lv) top(I, k, lv, false);
  }
  phase_end();
  for (int lv = lsplit - 1; lv >= 0; --lv) {
    level(lv, false);
    phase_end();
  }
  elems(false);
  grid_exit(gb);
}

// ---- host launchers ------------------------------------------------------------------
int bcr_levels(int N) {
  int lv = 0;
  for (int s = 1; s < N; s *= 2) ++lv;
  return lv;
}

// Dynamic shared memory of a panel-eliminated block: everything (full), or
// the panel buffers only when the block is in a global slab (none when they
// are in the slab too).
template <typename T>
static size_t panel_smem(int msz, bool full) {
  const size_t panel = sizeof(T) * big_panel_elems<T>(msz);
  if (full) return panel + sizeof(T) * PackedTri::elems(msz);
  return panel_in_global<T>(msz) ? 0 : panel;
}
template <typename T>
size_t elem_factor_smem(const DevProb& P, bool full) { return panel_smem<T>(P.ext, full); }
template <typename T>
size_t bcr_factor_smem(const DevProb& P, bool full) { return panel_smem<T>(P.bext, full); }

// Largest dynamic shared memory of a factorization block.  One limit decides
// both whether a block is factored in shared memory (here and in the batched
// plans) and whether its global slab is allocated; it leaves room for the
// static shared memory of the persistent kernels (< 27 KB) under 227 KB.
constexpr size_t SMEM_LIMIT = FACTOR_SMEM_LIMIT;

template <typename T>
bool elem_uses_smem(const DevProb& P) { return elem_factor_smem<T>(P, true) <= SMEM_LIMIT; }
template <typename T>
bool bcr_uses_smem(const DevProb& P) { return bcr_factor_smem<T>(P, true) <= SMEM_LIMIT; }

// Global workspace (in T elements) needed when a block does not fit in shared memory.
template <typename T>
size_t factor_work_elems(const DevProb& P, int n_slabs) {
  size_t w = 0;
  if (!elem_uses_smem<T>(P)) w = std::max(w, slab_elems<T>(P.ext) * n_slabs);
  if (!bcr_uses_smem<T>(P)) w = std::max(w, slab_elems<T>(P.bext) * n_slabs);
  return w;
}

template <typename T>
cudaError_t launch_elem_factor(const DevProb& P, const DevEval& E, const double* sigma, double dw,
                               double dc, const DevFactor<T>& F, cudaStream_t st) {
  const int rtn = rt_block_threads<T>(P.ext);
  if (rtn > 0) {
    const size_t sm = elem_stage_bytes<T>(P);
    opt_in_smem(k_elem_factor_rt<T>, sm, true);
    count_launch();
    k_elem_factor_rt<T><<<P.N, rtn, sm, st>>>(P, E, sigma, dw, dc, F);
    return cudaGetLastError();
  }
  bool es = elem_uses_smem<T>(P);
  size_t sm = elem_factor_smem<T>(P, es);
  opt_in_smem(k_elem_factor<T>, sm);
  int grid = es ? P.N : std::min(P.N, F.n_slabs);
  count_launch();
  k_elem_factor<T><<<grid, FBS, sm, st>>>(P, E, sigma, dw, dc, F, es ? 1 : 0,
                                           schedule().slab_pairs);
  return cudaGetLastError();
}

template <typename KernelT>
static int coop_grid(KernelT kern, int threads, size_t smem, int want, int reserve = 0) {
  // co-resident blocks per SM per (device, kernel, threads, shared memory),
  // cached: the query costs more host time than a launch.  `reserve` SMs are
  // left out (kernels of another stream hold them), so that the whole grid
  // fits on the others.
  struct Key {
    int dev;
    const void* k;
    int threads;
    size_t smem;
    bool operator<(const Key& o) const {
      return std::tie(dev, k, threads, smem) < std::tie(o.dev, o.k, o.threads, o.smem);
    }
  };
  static std::mutex mu;
  static std::map<Key, std::pair<int, int>> cache;   // (blocks per SM, SMs)
  int dev = 0;
  cudaGetDevice(&dev);
  const Key key{dev, (const void*)kern, threads, smem};
  int per = -1, sms = 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) { per = it->second.first; sms = it->second.second; }
  }
  if (per < 0) {
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = {per, sms};
  }
  const int usable = std::max(1, sms - std::max(0, reserve));
  return std::max(0, std::min(want, per * usable));
}

template <typename T>
cudaError_t launch_factor(const DevProb& P, const DevEval& E, const double* sigma, double dw,
                          double dc, const DevFactor<T>& F, const DevSchur& S, cudaStream_t st) {
  const bool es = elem_uses_smem<T>(P), bs = bcr_uses_smem<T>(P);
  const size_t sme = elem_factor_smem<T>(P, es), smb = bcr_factor_smem<T>(P, bs);
  const size_t sms = sizeof(double) * schur_doubles(P.p);
  cudaError_t e;
  if ((e = launch_elem_factor<T>(P, E, sigma, dw, dc, F, st)) != cudaSuccess) return e;
  const int bt = bcr_rt_tiles(P.bext);
  auto bcr_level = [&](int s, int fin) -> cudaError_t {
    const int nblk = fin ? 1 : bcr_level_blocks(P.N, s);
    const size_t smr = 2 * sizeof(T) * bcr_stage_elems(P.n, P.p);
    count_launch();
    if (bt == 1 || bt == 2) {
      auto kern = bt == 1 ? k_bcr_factor<T, 1> : k_bcr_factor<T, 2>;
      opt_in_smem(kern, smr);
      kern<<<(nblk + 1) / 2, FBS, smr, st>>>(P, F, s, fin, 1, schedule().slab_pairs);
    } else {
      opt_in_smem(k_bcr_factor<T, 0>, smb);
      const int g = bs ? nblk : std::min(nblk, F.n_slabs);
      k_bcr_factor<T, 0><<<g, FBS, smb, st>>>(P, F, s, fin, bs ? 1 : 0, schedule().slab_pairs);
    }
    return cudaGetLastError();
  };
  for (int s = 1; s < P.N; s *= 2)
    if ((e = bcr_level(s, 0)) != cudaSuccess) return e;
  if ((e = bcr_level(1, 1)) != cudaSuccess) return e;
  // the Schur block works in shared memory up to the factorization limit,
  // otherwise in S.S itself
  const bool sg = sms > SMEM_LIMIT;
  if (!sg) opt_in_smem(k_schur, sms);
  if ((e = launch_chunk_sums(F.Scon, 2 * P.N, P.p * P.p, F.chunkS, st)) != cudaSuccess) return e;
  if (P.p > 0) {
    count_launch();
    k_schur_total<<<ceil_div((long long)P.p * P.p, CS_BS), CS_BS, 0, st>>>(F.chunkS, P.N, P.p);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  count_launch();
  k_schur<<<1, SBS, sg ? 0 : sms, st>>>(P, F.inert, F.chunkS, E.wtt, sigma, dw, S, sg ? 1 : 0);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_solve(const DevProb& P, const DevFactor<T>& F, const DevSchur& S,
                         const double* b, double* sol, cudaStream_t st) {
  const bool ew = elem_solve_wide(P), bw = bcr_solve_wide(P);
  const bool few[2] = {false, false};
  const size_t sme = solve_smem<T>(ew ? 0 : P.ext, ew ? P.ext : 0, 0, few);
  const size_t smb = solve_smem<T>(bw ? 0 : P.bext, bw ? P.bext : 0, 0, few);
  const size_t smt = solve_smem<T>(0, 0, std::max(P.p, 1), few);
  cudaError_t e;
  auto grid = [](bool wide, int items) { return wide ? items : ceil_div(items, SOLVE_G); };
  auto run = [&](auto kern, int g, size_t sm, auto... args) -> cudaError_t {
    opt_in_smem(kern, sm, true);
    count_launch();
    kern<<<g, FBS, sm, st>>>(args..., sm);
    return cudaGetLastError();
  };
  auto elems = [&](int fwd) {
    return run(ew ? k_elem_solve<T, SOLVE_G> : k_elem_solve<T, 1>, grid(ew, P.N), sme, P, F, S, b,
               sol, fwd);
  };
  auto level = [&](int fwd, int s, int fin) {
    const int g = grid(bw, fin ? 1 : bcr_level_blocks(P.N, s));
    return run(bw ? k_bcr_solve<T, SOLVE_G> : k_bcr_solve<T, 1>, g, smb, P, F, S, sol, fwd, s, fin);
  };
  if ((e = elems(1)) != cudaSuccess) return e;
  std::vector<int> strides;
  for (int s = 1; s < P.N; s *= 2) strides.push_back(s);
  for (int s : strides)
    if ((e = level(1, s, 0)) != cudaSuccess) return e;
  if ((e = level(1, 1, 1)) != cudaSuccess) return e;
  if ((e = launch_chunk_sums(F.Rth, 2 * P.N, P.p, F.chunkR, st)) != cudaSuccess) return e;
  if ((e = run(k_theta_solve, 1, smt, P, (const double*)F.chunkR, b, S, sol, &F.gbar->err)) !=
      cudaSuccess)
    return e;
  if ((e = level(0, 1, 1)) != cudaSuccess) return e;
  for (int k = (int)strides.size() - 1; k >= 0; --k)
    if ((e = level(0, strides[k], 0)) != cudaSuccess) return e;
  return elems(0);
}

// Batched launchers.  `grid_cap` limits the grid when some instance uses its
// global slabs (at most n_slabs blocks may run).  Factorization parts: 1 the
// register-tiled element kernel, 4 the large-element kernel, 2 the rest (cyclic
// reduction and parameter Schur complement in the cooperative kernel).
template <typename T>
cudaError_t launch_factor_b(const DevInst* insts, const int* act, int A, const int* pre_elem,
                            const int* pre_lv, int maxL, const int* pre_cs,
                            const InstParams* prm, const int* flags, GridBar* gb, size_t smem,
                            int grid_cap, int rt_threads, size_t rt_smem, int tot_elem,
                            int big_grid, size_t big_smem, int bcr_tpt, int bcr_full, int max_p, int parts,
                            cudaStream_t st, int reserve) {
  if (A == 0) return cudaSuccess;
  if ((parts & 1) && rt_threads > 0 && tot_elem > 0) {
    if (rt_threads > RT_MAX_THREADS) return cudaErrorInvalidValue;
    opt_in_smem(k_elem_factor_rt_b<T>, rt_smem, true);
    count_launch();
    k_elem_factor_rt_b<T><<<tot_elem, rt_threads, rt_smem, st>>>(insts, act, A, pre_elem, prm,
                                                                 flags);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const Schedule sch = schedule();
  if ((parts & 4) && big_grid > 0) {
    count_launch();
    if (sch.big_threads == 256) {
      opt_in_smem(k_elem_factor_big_b<T, 256>, big_smem, true);
      k_elem_factor_big_b<T, 256><<<big_grid, 256, big_smem, st>>>(insts, act, A, pre_elem, prm,
                                                                   flags, sch.slab_pairs);
    } else {
      opt_in_smem(k_elem_factor_big_b<T, 512>, big_smem, true);
      k_elem_factor_big_b<T, 512><<<big_grid, 512, big_smem, st>>>(insts, act, A, pre_elem, prm,
                                                                   flags, sch.slab_pairs);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (!(parts & 2)) return cudaSuccess;
  // one block per SM is all that fits when smem exceeds a third of an SM's
  // shared memory: then the kernel variant compiled for one block per SM
  int dev = 0, smem_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  const bool wide = sizeof(T) == 4 && bcr_full && 3 * (smem + 1024) > (size_t)smem_sm;
  auto kern = bcr_tpt == 1 ? k_factor_b<T, 1, 0>
              : bcr_tpt == 2 ? k_factor_b<T, 2, 0> : k_factor_b<T, 0, 0>;
  if constexpr (sizeof(T) == 4)
    if (wide)
      kern = bcr_tpt == 1 ? k_factor_b<T, 1, 1>
             : bcr_tpt == 2 ? k_factor_b<T, 2, 1> : k_factor_b<T, 0, 1>;
  opt_in_smem(kern, smem, true);
  int grid = coop_grid(kern, FBS, smem, grid_cap, reserve);
  if (grid < 1) return cudaErrorInvalidConfiguration;
  int slab_pb = sch.slab_pairs;
  int totals = schur_totals_inside(max_p) ? 0 : 1;
  void* args[] = {(void*)&insts, (void*)&act, &A, (void*)&pre_elem, (void*)&pre_lv, &maxL,
                  (void*)&pre_cs, (void*)&prm, (void*)&flags, &gb, &smem, &bcr_full, &slab_pb, &totals};
  count_launch();
  return cudaLaunchCooperativeKernel((void*)kern, dim3(grid), dim3(FBS), args, smem, st);
}

template <typename T>
cudaError_t launch_solve_b(const DevInst* insts, const int* act, int A,
                           const int* const elem[2], const int* const lv[2], const int* pre_lv,
                           int maxL, int lsplit, const int* pre_cs, int ir, int pn, int pw,
                           const bool (&many)[2], bool most, GridBar* gb, int max_p,
                           int grid_want, cudaStream_t st, int reserve) {
  if (A == 0) return cudaSuccess;
  size_t smem = solve_smem<T>(pn, pw, std::max(max_p, 1), many);
  // Wide blocks: a group's chain costs the same whatever its size, and only the rows
  // below it gain from more warps.  With several blocks for each CUDA block the device
  // holds, more and smaller groups cover one another's chains: two warps each
  // as long as four such groups have a panel each in the memory (about 200 rows in
  // FP32), four warps from twice as many blocks on up to SOLVE_G4_ROWS.  One solve of A problems of
  // 400 elements by groups of 8 / 4 / 2 warps, us: 16 species, A = 2 182 / 177 / 172, A = 32
  // 754 / 560 / 518; 20 species, A = 32 978 / 773 / 736; 27 species (one panel of 35 KB), A =
  // 2 233 / 245, A = 4 312 / 302, A = 32 1395 / 1189; 33 species, A = 4 372 / 371; 36, A = 8
  // 590 / 615.
  auto kern = k_solve_b<T, SOLVE_G>;
  if (many[1] && SOLVE_G / 2 * group_smem<T, 2>(pw, 1, 1) <= smem)
    kern = k_solve_b<T, 2>;
  else if (most && pw <= SOLVE_G4_ROWS && SOLVE_G / 4 * group_smem<T, 4>(pw, 1, 1) <= smem)
    kern = k_solve_b<T, 4>;
  opt_in_smem(kern, smem, true);
  int grid = coop_grid(kern, FBS, smem, grid_want, reserve);
  if (grid < 1) return cudaErrorInvalidConfiguration;
  SolvePlan sp{{elem[0], elem[1]}, {lv[0], lv[1]}};
  void* args[] = {(void*)&insts, (void*)&act, &A, &sp, (void*)&pre_lv, &maxL,
                  &lsplit, (void*)&pre_cs, &ir, &pn, &pw, &max_p, &smem, &gb};
  count_launch();
  return cudaLaunchCooperativeKernel((void*)kern, dim3(grid), dim3(FBS), args, smem, st);
}

template cudaError_t launch_factor_b<float>(const DevInst*, const int*, int, const int*,
                                            const int*, int, const int*, const InstParams*,
                                            const int*, GridBar*, size_t, int, int, size_t, int,
                                            int, size_t, int, int, int, int, cudaStream_t, int);
template cudaError_t launch_factor_b<double>(const DevInst*, const int*, int, const int*,
                                             const int*, int, const int*, const InstParams*,
                                             const int*, GridBar*, size_t, int, int, size_t, int,
                                             int, size_t, int, int, int, int, cudaStream_t, int);
int bcr_rt_tiles_of(const DevProb& P) { return bcr_rt_tiles(P.bext); }
size_t elem_rt_stage_bytes(const DevProb& P, bool f32) {
  return f32 ? elem_stage_bytes<float>(P) : elem_stage_bytes<double>(P);
}
size_t bcr_rt_stage_bytes(const DevProb& P, bool f32) {
  const size_t one = (f32 ? sizeof(float) : sizeof(double)) * bcr_stage_elems(P.n, P.p);
  return 4 * ((one + 15) & ~size_t(15));   // two halves, two stage buffers each
}
int elem_rt_threads(const DevProb& P, bool f32) {
  return f32 ? rt_block_threads<float>(P.ext) : rt_block_threads<double>(P.ext);
}
bool solve_wide(const DevProb& P, bool elem) { return elem ? elem_solve_wide(P) : bcr_solve_wide(P); }
template cudaError_t launch_solve_b<float>(const DevInst*, const int*, int, const int* const[2],
                                           const int* const[2], const int*, int, int, const int*,
                                           int, int, int, const bool (&)[2], bool, GridBar*, int, int,
                                           cudaStream_t, int);
template cudaError_t launch_solve_b<double>(const DevInst*, const int*, int, const int* const[2],
                                            const int* const[2], const int*, int, int, const int*,
                                            int, int, int, const bool (&)[2], bool, GridBar*, int, int,
                                           cudaStream_t, int);
template size_t elem_factor_smem<float>(const DevProb&, bool);
template size_t elem_factor_smem<double>(const DevProb&, bool);
template size_t bcr_factor_smem<float>(const DevProb&, bool);
template size_t bcr_factor_smem<double>(const DevProb&, bool);

template cudaError_t launch_factor<double>(const DevProb&, const DevEval&, const double*, double,
                                           double, const DevFactor<double>&, const DevSchur&,
                                           cudaStream_t);
template cudaError_t launch_factor<float>(const DevProb&, const DevEval&, const double*, double,
                                          double, const DevFactor<float>&, const DevSchur&,
                                          cudaStream_t);
template cudaError_t launch_solve<double>(const DevProb&, const DevFactor<double>&,
                                          const DevSchur&, const double*, double*, cudaStream_t);
template cudaError_t launch_solve<float>(const DevProb&, const DevFactor<float>&,
                                         const DevSchur&, const double*, double*, cudaStream_t);
template cudaError_t launch_elem_factor<double>(const DevProb&, const DevEval&, const double*,
                                                double, double, const DevFactor<double>&,
                                                cudaStream_t);
template cudaError_t launch_elem_factor<float>(const DevProb&, const DevEval&, const double*,
                                               double, double, const DevFactor<float>&,
                                               cudaStream_t);
template size_t factor_work_elems<double>(const DevProb&, int);
template size_t factor_work_elems<float>(const DevProb&, int);

}  // namespace collo
