// Substitutions through the eliminated columns of a block, by a group of one, two,
// four or eight warps.
//
// Bound: the chain of dependent columns, and the memory latency of the factor's
// entries behind it (for many large blocks, their bandwidth).  Columns are taken
// in panels; a panel's factor entries, diagonal block and rows below, are copied
// to shared memory one or two panels ahead by bulk copies (one per column, a
// transaction barrier per panel), the first panels of the group's next block
// while the current one finishes, so the chain itself rarely waits for memory.
// The group's shared memory is divided for the block at hand, so that a smaller
// block than the launch's largest has more panels ahead.
// Per panel, the group's first warp solves the diagonal
// block, one right-hand-side entry per lane, passing each solved pair on by
// shuffles; then every thread applies the panel to its rows below (forward), or
// has summed its rows' part of the panel's columns before (backward).
#pragma once
#include "collo_internal.cuh"

namespace collo {

// Sums over the warp of y[0 .. R-1] per lane, R a power of two up to 32: halves
// are exchanged instead of adding every value across all lanes (R - 1 + 5 -
// log2 R shuffles instead of 5 R).  Lane l returns the sum of row
// l >> (5 - log2 R).
template <typename T, int R>
__device__ inline T warp_rows_sum(T (&y)[R]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = R / 2; h > 0; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const T keep = up ? y[k + h] : y[k], give = up ? y[k] : y[k + h];
      y[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  T v = y[0];
#pragma unroll
  for (; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Asynchronous copies (cp.async) of single elements from global to shared memory.
template <typename T>
__device__ inline void cp_async_elem(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// L columns of an eliminated block, unit lower, column-major: entry (row r,
// column c), r > c, at p[c ld + r]; p 16-byte aligned, ld = factor_ld(rows).
template <typename T>
struct FactorCols {
  const T* p;
  int ld, rows, cols;
};

// Leading dimension of a panel in shared memory: a multiple of 16 bytes, and 4
// modulo 8 entries so that the diagonal block is also read across its columns
// (backward) at no more than four ways in a bank.
__host__ __device__ inline int sub_ld(int msz) { return ((msz + 7) >> 3 << 3) + 4; }
// Columns of a panel: 32, or 16 for a single warp, halved until two panels fit
// SUB_STAGE_BYTES.  It depends on the block alone (the back substitution's sums
// are ordered by panel), not on the launch.
constexpr size_t SUB_STAGE_BYTES = 190 * 1024;
template <typename T, int G>
__host__ __device__ inline int sub_panel(int msz) {
  int pc = G > 1 ? 32 : 16;
  while (pc > 2 && 2 * sizeof(T) * (size_t)pc * sub_ld(msz) > SUB_STAGE_BYTES) pc >>= 1;
  return pc;
}
// Elements of a group's vector with its panel sums (32 behind it), and of one panel.
__host__ __device__ inline size_t sub_vec_elems(int msz) { return (size_t)((msz + 7) & ~7) + 32; }
template <typename T, int G>
__host__ __device__ inline size_t sub_panel_elems(int msz) {
  return (size_t)sub_panel<T, G>(msz) * sub_ld(msz);
}
// Bytes of a panel's slot for blocks of up to msz rows (a smaller block may take
// wider panels).
template <typename T, int G>
__host__ __device__ inline size_t sub_slot_bytes(int msz) {
  const size_t own = sizeof(T) * sub_panel_elems<T, G>(msz);
  const bool widest = sub_panel<T, G>(msz) == (G > 1 ? 32 : 16);
  return widest || own > SUB_STAGE_BYTES / 2 ? own : SUB_STAGE_BYTES / 2;
}

// ---- transaction barriers and bulk copies ---------------------------------------------
__device__ inline void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ inline void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// 16-byte aligned addresses, a multiple of 16 bytes.
__device__ inline void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst), "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ inline bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// A wait gives up after this many tries (each suspends the thread for a time set
// by the hardware) and records the error.
constexpr int SUB_WAIT_TRIES = 1 << 22;

constexpr int SUB_STAGES = 3;   // most panels in flight

// A group's ring of panels in shared memory (the same on every thread of the
// group): `bytes` of it, divided into slots by the block at hand (sub_start), as
// many as it has room for; slot: the next panel's; phases: each barrier's
// phase, a bit per slot.  Kept in registers and passed by value.
struct SubRing {
  unsigned char* slots;     // [stages][slot_bytes]
  unsigned bar;             // [SUB_STAGES] barriers, shared-space address
  int bytes, slot_bytes, stages;
  int slot;
  unsigned phases;
  int* err;                 // GridBar::err
};

// Groups of G of the block's eight warps.  A block's result does not depend on G > 1:
// panels are those of the block's rows, a row of the forward substitution takes the
// columns in their order, and a column's sum of the backward one is over the
// lanes' strided rows and then the same tree, whichever warp has it.
constexpr int SUB_WARPS = 8;
template <int G>
__device__ inline int group_index() { return (int)threadIdx.x / (32 * G); }
template <int G>
__device__ inline void group_sync() {
  if constexpr (G == 1) __syncwarp();
  else if constexpr (G == SUB_WARPS) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + group_index<G>()), "n"(32 * G) : "memory");
}

// Thread of the group.
template <int G>
__device__ inline int group_tid() { return (int)threadIdx.x % (32 * G); }

// A group's memory for blocks of up to msz rows in `bytes` at p (16-byte
// aligned): vector and sums, ring; bar: its SUB_STAGES barriers, initialised
// (sub_init).
template <typename T, int G>
struct SubMem {
  T* w;
  T* sums;
  SubRing ring;
};
template <typename T, int G>
__device__ inline SubMem<T, G> sub_carve(unsigned char* p, size_t bytes, int msz,
                                         unsigned long long* bar, int* err) {
  SubMem<T, G> m;
  const size_t v = sub_vec_elems(msz);
  m.w = reinterpret_cast<T*>(p);
  m.sums = m.w + (v - 32);
  m.ring.slots = reinterpret_cast<unsigned char*>(m.w + v);
  m.ring.bar = (unsigned)__cvta_generic_to_shared(bar);
  m.ring.bytes = (int)(bytes - sizeof(T) * v);
  m.ring.slot_bytes = m.ring.stages = m.ring.slot = 0;
  m.ring.phases = 0;
  m.ring.err = err;
  return m;
}
// Warps of a group that ask for panels (a barrier's arrivals): all but the one that
// carries the chain, where there are others.
template <int G>
constexpr int SUB_ASKING = G > 1 ? G - 1 : 1;
// Initialises the barriers of n groups of G (all of a kernel's, then sub_ready; the
// whole block calls).
template <int G>
__device__ inline void sub_init(unsigned long long* bar, int n) {
  if ((int)threadIdx.x < n * SUB_STAGES)
    mbar_init((unsigned)__cvta_generic_to_shared(bar + threadIdx.x), SUB_ASKING<G>);
}
__device__ inline void sub_ready() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
}
// Shared memory written by threads is given over to bulk copies: before the
// barrier that precedes the first such copy.
__device__ inline void sub_release() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Asks for the panel of L whose first column is cp (no panel outside 0 <= cp <
// cols), into a slot that every thread has left.  A copy takes its warp some 40
// cycles, so the columns are dealt out to the warps that do not carry the chain:
// one of them alone was still asking when the chain was done (27 to 50 species: 430 of
// 2300 cycles of a forward panel and 1000 of 2900 of a backward one).  With this and
// the ring divided per block, one solve at 27 species, 415 elements 197 -> 166 us, 50
// species, 2000 elements 842 -> 671 us.
template <int G, typename T>
__device__ inline void sub_ask(const SubRing& R, int slot, const FactorCols<T>& L, int cp, int pc,
                               int ld) {
  constexpr int Q = 16 / sizeof(T);
  constexpr int NW = SUB_ASKING<G>;
  const int w = G > 1 ? (group_tid<G>() >> 5) - 1 : 0, lane = threadIdx.x & 31;
  if (cp >= 0 && cp < L.cols && w >= 0) {
    const int K = min(pc, L.cols - cp), r0 = cp & ~(Q - 1);
    const int mine = w < K ? (K - w + NW - 1) / NW : 0;   // columns w, w + NW, ...
    const unsigned bytes = (unsigned)((L.rows - r0 + Q - 1) & ~(Q - 1)) * (unsigned)sizeof(T);
    const unsigned bar = R.bar + 8 * slot;
    if (lane == 0) mbar_expect(bar, bytes * (unsigned)mine);
    __syncwarp();
    const unsigned dst = (unsigned)__cvta_generic_to_shared(R.slots) + slot * R.slot_bytes;
    const int c = w + lane * NW;
    if (lane < mine)
      bulk_load(dst + (unsigned)(c * ld * (int)sizeof(T)), L.p + (size_t)(cp + c) * L.ld + r0,
                bytes, bar);
    __syncwarp();
  }
}

// Waits for the next panel; returns its slot.
__device__ inline int sub_next(SubRing& R) {
  const int slot = R.slot;
  const unsigned bar = R.bar + 8 * slot;
  const unsigned phase = (R.phases >> slot) & 1u;
  if (!mbar_try(bar, phase)) {
    int tries = 0;
    while (!mbar_try(bar, phase))
      if (++tries > SUB_WAIT_TRIES) { atomicExch(R.err, 1); break; }
  }
  R.phases ^= 1u << slot;
  if (++R.slot == R.stages) R.slot = 0;
  return slot;
}

// Divides the ring, which is empty, for a block and asks for the first panels of its
// forward (from the first column) or backward (from the last panel) substitution.
template <int G, typename T>
__device__ inline void sub_start(SubRing& R, const FactorCols<T>& L, bool forward) {
  const int pc = sub_panel<T, G>(L.rows), ld = sub_ld(L.rows);
  R.slot_bytes = pc * ld * (int)sizeof(T);
  R.stages = 1;
#pragma unroll
  for (int st = 2; st <= SUB_STAGES; ++st)
    if (st * R.slot_bytes <= R.bytes) R.stages = st;
  R.slot = 0;
  const int first = forward ? 0 : (L.cols - 1) & ~(pc - 1), step = forward ? pc : -pc;
  for (int q = 0, cp = first; q < max(1, R.stages - 1); ++q, cp += step)
    sub_ask<G>(R, q, L, cp, pc, ld);
}

// w = L^{-1} w (length L.rows, shared memory), w visible to the group, the
// block's panels started (sub_start); the
// result is visible to the group on return, the ring is empty.  Returns its phases.  PAIRS: columns come in pairs whose two
// rows are not coupled (entry (2q + 1, 2q) is absent).
template <int G, bool PAIRS, typename T>
__device__ __noinline__ unsigned group_forward(T* w, SubRing R, const FactorCols<T> L) {
  constexpr int NT = 32 * G, PC = G > 1 ? 32 : 16, Q = 16 / sizeof(T);
  constexpr unsigned FULL = 0xffffffffu;
  __builtin_assume(__isShared(w));
  const int tid = group_tid<G>(), lane = threadIdx.x & 31;
  const int msz = L.rows, ncol = L.cols, pc = sub_panel<T, G>(msz), ld = sub_ld(msz);
  const int ahead = (R.stages - 1) * pc;
  for (int cp = 0; cp < ncol; cp += pc) {
    const int K = min(pc, ncol - cp), cend = cp + K, r0 = cp & ~(Q - 1);
    // row r of column k of the panel: st[k ld + r - r0]
    const int slot = sub_next(R);
    const T* st = reinterpret_cast<const T*>(R.slots + (size_t)slot * R.slot_bytes);
    __builtin_assume(__isShared(st));
    group_sync<G>();    // every thread has left the panel before
    if (R.stages > 1) sub_ask<G>(R, slot == 0 ? R.stages - 1 : slot - 1, L, cp + ahead, pc, ld);
    if (tid < 32) {
      // this lane's row of the diagonal block; nothing on and above the
      // diagonal (PAIRS: nor inside a pair).  Short loops: a few blocks per
      // launch run this code, so fetching instructions counts.
      const T* d = st + (cp - r0) + min(lane, K - 1);
      T v = lane < K ? w[cp + lane] : T(0);
      if constexpr (PAIRS) {
#pragma unroll 4
        for (int k = 0; k < K; k += 2) {
          const bool on = lane > k + 1;
          const T l0 = d[k * ld], l1 = d[(k + 1) * ld];
          const T w0 = __shfl_sync(FULL, v, k), w1 = __shfl_sync(FULL, v, k + 1);
          const T u = fma(-l1, w1, fma(-l0, w0, v));
          v = on ? u : v;
        }
      } else {
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
          const T l0 = d[k * ld];
          const T u = fma(-l0, __shfl_sync(FULL, v, k), v);
          v = lane > k ? u : v;
        }
      }
      if (lane < K) w[cp + lane] = v;
    }
    group_sync<G>();
    for (int r = cend + tid; r < msz; r += NT) {
      const T* s = st + (r - r0);
      T acc = w[r];
      if (K == PC) {
#pragma unroll 8
        for (int k = 0; k < PC; ++k) acc = fma(-s[k * ld], w[cp + k], acc);
      } else {
#pragma unroll 2
        for (int k = 0; k < K; ++k) acc = fma(-s[k * ld], w[cp + k], acc);
      }
      w[r] = acc;
    }
    if (R.stages == 1) {
      group_sync<G>();
      sub_ask<G>(R, 0, L, cp + pc, pc, ld);
    }
  }
  group_sync<G>();
  return R.phases;
}

// Back substitution, the block's panels started: x (length L.rows) holds the right-hand side in
// its first L.cols entries and the known tail behind them; the first L.cols entries
// become x_c - sum_{r > c} L[r][c] x_r from the last column to the first.  The
// panel sums are over the lanes' strided rows, then a fixed shuffle tree.
// sums: 32 entries of shared memory.
template <int G, bool PAIRS, typename T>
__device__ __noinline__ unsigned group_backward(T* x, T* sums, SubRing R, const FactorCols<T> L) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int PC = G > 1 ? 32 : 16, CW = PC / G;   // columns a warp sums at once
  constexpr int Q = 16 / sizeof(T);
  __builtin_assume(__isShared(x));
  __builtin_assume(__isShared(sums));
  const int tid = group_tid<G>(), lane = threadIdx.x & 31, warp = tid >> 5;
  const int msz = L.rows, ncol = L.cols, pc = sub_panel<T, G>(msz), ld = sub_ld(msz);
  const int ahead = (R.stages - 1) * pc;
  for (int cp = ncol > 0 ? (ncol - 1) & ~(pc - 1) : -1; cp >= 0; cp -= pc) {
    const int K = min(pc, ncol - cp), cend = cp + K, r0 = cp & ~(Q - 1);
    const int slot = sub_next(R);
    const T* st = reinterpret_cast<const T*>(R.slots + (size_t)slot * R.slot_bytes);
    __builtin_assume(__isShared(st));
    group_sync<G>();    // the panel above is solved, and left by every thread
    if (R.stages > 1) sub_ask<G>(R, slot == 0 ? R.stages - 1 : slot - 1, L, cp - ahead, pc, ld);
    const int k0 = warp * CW;
    if (k0 < K) {
      T acc[CW];
#pragma unroll
      for (int c = 0; c < CW; ++c) acc[c] = T(0);
#pragma unroll 2
      for (int r = cend + lane; r < msz; r += 32) {
        const T xr = x[r];
        const T* s = st + (r - r0) + k0 * ld;
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = fma(k0 + c < K ? s[c * ld] : T(0), xr, acc[c]);
      }
      const T s = warp_rows_sum<T, CW>(acc);
      constexpr int SH = CW == 16 ? 1 : CW == 8 ? 2 : 3;   // lane l has column l >> SH
      if ((lane & ((1 << SH) - 1)) == 0) sums[k0 + (lane >> SH)] = s;
    }
    group_sync<G>();
    if (tid < 32) {
      // this lane's column of the diagonal block
      const T* d = st + min(lane, K - 1) * ld + (cp - r0);
      T t = lane < K ? x[cp + lane] - sums[lane] : T(0);
      if constexpr (PAIRS) {
#pragma unroll 4
        for (int j = K - 2; j > 0; j -= 2) {
          const T l0 = d[j], l1 = d[j + 1];
          const T x0 = __shfl_sync(FULL, t, j), x1 = __shfl_sync(FULL, t, j + 1);
          const T u = fma(-l1, x1, fma(-l0, x0, t));
          t = lane < j ? u : t;
        }
      } else {
#pragma unroll 4
        for (int j = K - 1; j > 0; --j) {
          const T l0 = d[j];
          const T u = fma(-l0, __shfl_sync(FULL, t, j), t);
          t = lane < j ? u : t;
        }
      }
      if (lane < K) x[cp + lane] = t;
    }
    if (R.stages == 1) {
      group_sync<G>();
      sub_ask<G>(R, 0, L, cp - pc, pc, ld);
    }
  }
  group_sync<G>();
  return R.phases;
}

}  // namespace collo
