// The two kernels of one PDHG step attempt (Sec. II.E iteration, PDLP form):
//
//   k_dual    : K x' (sliced ELL, warp per 32-row slice) fused with the
//               projected dual step y' = max(y_lo, y + sigma (q - 2 K x' + K x));
//               FP32 recomputes K x in the same matrix pass (gathering x and
//               x'), FP64 reads the stored K x and writes K x' (StoresKx),
//               the lazy y-average update, and the FP64 partial sums ||dy||^2 and
//               dy^T K dx.  The block that finishes last reduces the partials in
//               fixed order and takes the adaptive step decision (accept/reject,
//               next eta) on the device.
//   k_adjoint : K^T y' for an accepted step (else the cached K^T y), the
//               x-average update, and -- fused -- the primal step of the NEXT
//               attempt x'' = proj_[l,u](x - tau (c - K^T y)) with ||dx||^2.
//
// Buffers are double-buffered by a parity bit in the device state: the
// current iterate is buf[par], the candidate buf[1-par]; accepting flips par.
#include "internal.cuh"

namespace ucpdhg {

// Row dot products of U consecutive slices (U = 1, or 2 or 4 slices of one group:
// one width w unless kRunsOwn) with x1 and, if TWO, with x2 in the same matrix pass;
// lane = row within each slice.  The columns of a slice come from its runs (8 B per 32
// entries: the gather is then one or two contiguous pieces and needs no index
// load of its own) or, where it has none, from the explicit indices.
//
// What bounds these sweeps is not DRAM but the instructions and dependent round
// trips per 32 rows (the time per row is the same for a matrix that stays in L2),
// so a warp takes U slices whose entries and operand rows lie at fixed distances:
// loads without predicates or address arithmetic of their own, U E entries, their
// gathers and 4 U (5 U) operands in flight together.  Warps in flight count as much:
// chunks of E = 4 at U = 2 spill at 64 registers (44.5 us for K x' of the 6717-bus
// day) and lose a quarter of the warps at 80 (44.9).  With column runs and the order
// of build_layout, FP32, 6717-bus 96-period day: K x' 49.3 -> 36.9 us, K^T y' 36.5 ->
// 22.8 us; FP64 107 -> 83 and 61 -> 51 us, where the FP64 pipe is the bound.
//
// soff[s0] and soff[s0 + U] (clamped past the end, giving empty slices).  The
// per-attempt kernels load the NEXT group's offsets one iteration ahead, so this
// L2 round trip is off the critical path.
struct SliceSpan {
  int o, w, mode;  // first slot, entries per row, kRuns*
};
template <class T, int U>
__device__ __forceinline__ int2 slice_offsets(const SellView<T>& A, int s0) {
  return make_int2(__ldg(A.soff + min(s0, A.nslices)), __ldg(A.soff + min(s0 + U, A.nslices)));
}
template <int U>
__device__ __forceinline__ SliceSpan slice_span(int2 ob) {
  return {ob.x & ~(kSlice - 1), ((ob.y >> 5) - (ob.x >> 5)) / U, ob.x & (kSlice - 1)};
}

// Run words of the next 32 / U k-columns of each of the U slices: lane t holds the
// one of slice t U / 32.  One coalesced load (issued an iteration ahead by the
// per-attempt kernels) instead of a dependent one before every gather: entries and
// gathers then leave together.  The 4 registers of the two iterations are there at
// two slices per warp (6717-bus day, FP32, K x' 39.2 -> 36.9 us, K^T y' 25.0 ->
// 22.8); at one slice and 40 registers they spill (45 -> 52 us), so U = 1 reads each
// word where it is used.
template <class T, int U>
__device__ __forceinline__ int2 run_words(const SellView<T>& A, const SliceSpan& g, int k0, int lane) {
  constexpr int W = 32 / U;
  if (U == 1) return int2{};
  const int k = k0 + lane % W;
  return (g.mode != kRunsNone && k < g.w) ? __ldg(A.runs + (g.o >> 5) + (lane / W) * g.w + k)
                                          : make_int2(0, (int)((unsigned)kSlice << kRunBits));
}

// E entries of each slice from k0 on; rw: the run words from k-column kw on.
template <class T, int U, int E, int MODE, bool TWO, bool TAIL>
__device__ __forceinline__ void dot_chunk(const SellView<T>& A, const SliceSpan& g, int2 rw, int kw, int k0,
                                          int lane, const T* __restrict__ x1, const T* __restrict__ x2,
                                          T (&acc1)[U], T (&acc2)[U]) {
  int c[U][E];
  T v[U][E];
  [[maybe_unused]] bool indices = false;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const bool ok = !TAIL || k0 + e < g.w;
      const int slot = g.o + (u * g.w + k0 + e) * kSlice;
      if (MODE == kRunsNone) {
        c[u][e] = ok ? __ldg(A.col + slot + lane) : 0;
      } else {
        int2 r = make_int2(0, (int)((unsigned)kSlice << kRunBits));
        if constexpr (U == 1) {
          if (ok) r = __ldg(A.runs + (slot >> 5));
        } else {
          const int t = u * (32 / U) + k0 + e - kw;
          r.x = __shfl_sync(0xffffffffu, rw.x, t);
          if (MODE != kRunsOne) r.y = __shfl_sync(0xffffffffu, rw.y, t);
        }
        if (MODE == kRunsOne) {
          c[u][e] = r.x + lane;
        } else {
          c[u][e] = run_col(r, lane);
          if (MODE == kRunsMixed) indices |= run_split(r) == 0;
        }
      }
      v[u][e] = ok ? __ldg(A.val + slot + lane) : (T)0;
    }
  // one branch for the chunk: a branch per k-column keeps the later loads behind it
  if (MODE == kRunsMixed && indices) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (!TAIL || k0 + e < g.w) c[u][e] = __ldg(A.col + g.o + (u * g.w + k0 + e) * kSlice + lane);
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (!TAIL || k0 + e < g.w) {
        acc1[u] += v[u][e] * __ldg(x1 + c[u][e]);
        if (TWO) acc2[u] += v[u][e] * __ldg(x2 + c[u][e]);
      }
}

template <class T, int U, int MODE, bool TWO>
__device__ __forceinline__ void sell_dot_mode(const SellView<T>& A, const SliceSpan& g, int2 rw, int lane,
                                              const T* __restrict__ x1, const T* __restrict__ x2,
                                              T (&acc1)[U], T (&acc2)[U]) {
  if constexpr (U == 1) {
    if (g.w <= 2)
      dot_chunk<T, U, 2, MODE, TWO, true>(A, g, rw, 0, 0, lane, x1, x2, acc1, acc2);
    else if (MODE == kRunsNone) {
      // rows without runs may be long: eight unpredicated entries in flight (100000
      // rows of 40 random entries, FP32: K^T y' 22.4 -> 19.3 us, K x' 37.1 -> 35.7)
      int k0 = 0;
      for (; k0 + 8 <= g.w; k0 += 8)
        dot_chunk<T, U, 8, MODE, TWO, false>(A, g, rw, 0, k0, lane, x1, x2, acc1, acc2);
      for (; k0 < g.w; k0 += 4) dot_chunk<T, U, 4, MODE, TWO, true>(A, g, rw, 0, k0, lane, x1, x2, acc1, acc2);
    } else
      for (int k0 = 0; k0 < g.w; k0 += 4)
        dot_chunk<T, U, 4, MODE, TWO, true>(A, g, rw, 0, k0, lane, x1, x2, acc1, acc2);
  } else {
    constexpr int W = 32 / U;  // a multiple of the chunks
    for (int kw = 0;;) {
      const int end = min(g.w, kw + W);
      int k0 = kw;
      for (; k0 + 2 <= end; k0 += 2)
        dot_chunk<T, U, 2, MODE, TWO, false>(A, g, rw, kw, k0, lane, x1, x2, acc1, acc2);
      if (k0 < end) dot_chunk<T, U, 1, MODE, TWO, false>(A, g, rw, kw, k0, lane, x1, x2, acc1, acc2);
      kw += W;
      if (kw >= g.w) break;
      rw = run_words<T, U>(A, g, kw, lane);
    }
  }
}

// Slices of their own widths (groups with a row far longer than the rest), one after
// the other, eight unpredicated entries in flight: such a row is a serial chain of its
// warp (K x of the 4224-bus, 18-period day with a row of 20000 entries: 1.74 ms; 2.5 ms
// with predicated chunks of four, 6.4 ms where the row widens its whole group).  Only
// compiled into the kernels for matrices with such groups (OWN): in the others it
// would cost 1 % (FP32 K x' of the 6717-bus day 36.9 -> 37.2 us, its FP64 solve 73.6 ->
// 74.4 ms).
template <class T, int U, bool TWO>
__device__ __forceinline__ void sell_dot_own(const SellView<T>& A, int s0, int lane, const T* __restrict__ x1,
                                             const T* __restrict__ x2, T (&acc1)[U], T (&acc2)[U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const SliceSpan g = slice_span<1>(slice_offsets<T, 1>(A, s0 + u));
    T a1[1] = {0}, a2[1] = {0};
    int k0 = 0;
    for (; k0 + 8 <= g.w; k0 += 8)
      dot_chunk<T, 1, 8, kRunsNone, TWO, false>(A, g, int2{}, 0, k0, lane, x1, x2, a1, a2);
    for (; k0 < g.w; ++k0)
      dot_chunk<T, 1, 1, kRunsNone, TWO, false>(A, g, int2{}, 0, k0, lane, x1, x2, a1, a2);
    acc1[u] = a1[0];
    acc2[u] = a2[0];
  }
}

// s0: the first of the U slices, g: their span.
template <class T, int U, bool TWO, bool OWN>
__device__ __forceinline__ void sell_dot_pre(const SellView<T>& A, int s0, const SliceSpan& g, int2 rw, int lane,
                                             const T* __restrict__ x1, const T* __restrict__ x2,
                                             T (&acc1)[U], T (&acc2)[U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) acc1[u] = acc2[u] = 0;
  if (g.mode == kRunsOne)
    sell_dot_mode<T, U, kRunsOne, TWO>(A, g, rw, lane, x1, x2, acc1, acc2);
  else if (g.mode == kRunsTwo)
    sell_dot_mode<T, U, kRunsTwo, TWO>(A, g, rw, lane, x1, x2, acc1, acc2);
  else if (g.mode == kRunsMixed)
    sell_dot_mode<T, U, kRunsMixed, TWO>(A, g, rw, lane, x1, x2, acc1, acc2);
  else if (OWN && g.mode == kRunsOwn)
    sell_dot_own<T, U, TWO>(A, s0, lane, x1, x2, acc1, acc2);
  else
    sell_dot_mode<T, U, kRunsNone, TWO>(A, g, rw, lane, x1, x2, acc1, acc2);
}

template <class T, int U, int MINB, bool OWN = false>
__global__ void __launch_bounds__(kBlock, MINB) k_dual(IterArgs<T> a) {
  grid_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  // matrix only: before the previous kernel ends
  int2 ob = slice_offsets<T, U>(a.K, gw * U), nb = U == 1 ? ob : slice_offsets<T, U>(a.K, (gw + nw) * U);
  int2 rw = run_words<T, U>(a.K, slice_span<U>(ob), 0, lane);
  grid_wait_prior();
  DevState* st = a.st;
  __shared__ DualScalars<T> sc;
  if (threadIdx.x == 0) dual_scalars<T>(st, sc);
  __syncthreads();
  if (sc.done) return;
  const int p = sc.p;
  const bool has_pw = sc.has_pw;
  const T pwT = sc.pw;
  const T sigma = sc.sigma;
  const T* __restrict__ xn = a.x[1 - p];
  const T* __restrict__ xc = a.x[p];
  const T* __restrict__ yc = a.y[p];
  T* __restrict__ yn = a.y[1 - p];
  // partials in the iterate precision up to the block totals (FP64
  // throughput on this GPU is ~1/60 of FP32); the step rule is a heuristic
  T acc_dy2 = 0, acc_int = 0;
  for (int s0 = gw * U; s0 < a.K.nslices; s0 += nw * U) {
    // next group's run words, the offsets of the one after it
    const int2 nrw = run_words<T, U>(a.K, slice_span<U>(nb), 0, lane);
    const int2 nnb = slice_offsets<T, U>(a.K, s0 + (U == 1 ? 1 : 2) * nw * U);
    const int i0 = s0 * kSlice + lane;
    // row operands do not depend on the product: load them first so their
    // latency overlaps the matrix stream (vectors are allocated in whole groups)
    T yo[U], qi[U], lo[U], yb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * kSlice;
      yo[u] = yc[i];
      qi[u] = a.q[i];
      lo[u] = a.ylo ? a.ylo[i] : (T)0;
      yb[u] = has_pw ? a.ybar[i] : (T)0;
    }
    // FP32: K x' and K x in one pass (K x recomputed: an L2 gather instead of
    // a stream read and write of m values).  FP64: K x' only, K x read.
    T kx[U], ko[U];
    if constexpr (StoresKx<T>::value) {
#pragma unroll
      for (int u = 0; u < U; ++u) ko[u] = a.Kx[p][i0 + u * kSlice];
      T unused[U];
      sell_dot_pre<T, U, false, OWN>(a.K, s0, slice_span<U>(ob), rw, lane, xn, xn, kx, unused);
    } else {
      sell_dot_pre<T, U, true, OWN>(a.K, s0, slice_span<U>(ob), rw, lane, xn, xc, kx, ko);
    }
    ob = U == 1 ? nnb : nb;
    nb = nnb;
    rw = nrw;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * kSlice;
      T t = qi[u] - (T)2 * kx[u];
      t = t + ko[u];
      T v = yo[u] + sigma * t;
      if (i >= a.m_eq) v = max_of(v, lo[u]);
      // FP64: rows whose multiplier is zero and stays zero (most inequalities) add
      // exact zeros below.  A warp of them leaves out 5 of its 9 FP64 instructions
      // (16 clocks each on the pipe that bounds this kernel) and the store of ybar:
      // 6717-bus day 94 -> 83 us.  (K^T y' gains nothing from the like: 51 -> 55 us.)
      bool idle = false;
      if constexpr (sizeof(T) == 8)
        idle = __all_sync(0xffffffffu, i >= a.m || (!non_zero(v) && !non_zero(yo[u]) && finite_bits(kx[u]) &&
                                                    finite_bits(ko[u])));
      if (i < a.m) {
        yn[i] = v;
        if constexpr (StoresKx<T>::value) a.Kx[1 - p][i] = kx[u];
        if (idle) continue;
        if (has_pw) a.ybar[i] = yb[u] + pwT * yo[u];
        const T dy = v - yo[u];
        const T dk = kx[u] - ko[u];
        acc_dy2 += dy * dy;
        acc_int += dy * dk;
      }
    }
  }
  T acc[2] = {acc_dy2, acc_int};
  if (publish_partials_t<2, T>(acc, a.partials, &st->counter)) {
    double tot[2];
    final_sum_t<2, T>(a.partials, gridDim.x, tot);
    if (threadIdx.x == 0) {
      decide_step(st, a, tot[0], tot[1]);
      st->counter = 0;
    }
  }
}

template <class T, int U, int MINB, bool OWN = false>
__global__ void __launch_bounds__(kBlock, MINB) k_adjoint(IterArgs<T> a) {
  grid_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  // matrix only: before the previous kernel ends
  int2 ob = slice_offsets<T, U>(a.KT, gw * U), nb = U == 1 ? ob : slice_offsets<T, U>(a.KT, (gw + nw) * U);
  int2 rw = run_words<T, U>(a.KT, slice_span<U>(ob), 0, lane);
  grid_wait_prior();
  DevState* st = a.st;
  __shared__ AdjScalars<T> sc;
  if (threadIdx.x == 0) adj_scalars<T>(st, sc);
  __syncthreads();
  if (sc.done) return;
  const int p = sc.p;
  const int acc_last = sc.acc_last;
  const bool upd_avg = sc.upd_avg;
  const T wlT = sc.wl;
  const T tau = sc.tau;
  const T* __restrict__ yc = a.y[p];
  const T* __restrict__ xc = a.x[p];
  T* __restrict__ kty = a.KTy[p];
  T* __restrict__ xn = a.x[1 - p];
  T acc_dx2 = 0;
  for (int s0 = gw * U; s0 < a.KT.nslices; s0 += nw * U) {
    const int2 nrw = run_words<T, U>(a.KT, slice_span<U>(nb), 0, lane);
    const int2 nnb = slice_offsets<T, U>(a.KT, s0 + (U == 1 ? 1 : 2) * nw * U);
    const int j0 = s0 * kSlice + lane;
    T x0[U], cj[U], lj[U], uj[U], xb[U], g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * kSlice;
      x0[u] = xc[j];
      cj[u] = a.c[j];
      lj[u] = a.l[j];
      uj[u] = a.u[j];
      xb[u] = upd_avg ? a.xbar[j] : (T)0;
    }
    if (acc_last) {
      T unused[U];
      sell_dot_pre<T, U, false, OWN>(a.KT, s0, slice_span<U>(ob), rw, lane, yc, yc, g, unused);
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) g[u] = kty[j0 + u * kSlice];
    }
    ob = U == 1 ? nnb : nb;
    nb = nnb;
    rw = nrw;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * kSlice;
      if (j < a.n) {
        if (acc_last) kty[j] = g[u];
        if (upd_avg) a.xbar[j] = xb[u] + wlT * x0[u];
        T v = x0[u] - tau * (cj[u] - g[u]);
        v = min(max(v, lj[u]), uj[u]);
        xn[j] = v;
        const T d = v - x0[u];
        acc_dx2 += d * d;
      }
    }
  }
  T acc[1] = {acc_dx2};
  if (publish_partials_t<1, T>(acc, a.partials, &st->counter)) {
    double tot[1];
    final_sum_t<1, T>(a.partials, gridDim.x, tot);
    if (threadIdx.x == 0) {
      st->dx2 = tot[0];
      st->counter = 0;
    }
  }
}

// ---- software-pipelined variants (one slice per warp) -------------------------
//
// A warp sweeps its slices s, s + nw, s + 2 nw, ...  While the gathers of slice
// s are in flight, the first kStage entries (columns and values) and the row
// operands of slice s + nw are already loading, and the offsets of s + 2 nw
// before them: two dependent round trips per slice (matrix from HBM, gathered
// vector from L2) overlap instead of following each other.  Entries beyond
// kStage (the long minimum-up/down rows) are read after the gathers.

constexpr int kStage = 4;

// Explicit column indices here: the runs' second word would take four more
// registers of the two stages (spills at 48 registers: 75 against 50 us for K x').
template <class T>
struct SliceStage {
  SliceSpan g;
  int c[kStage];
  T v[kStage];
};

template <class T>
__device__ __forceinline__ void stage_slice(const SellView<T>& A, int2 ob, int lane, SliceStage<T>& st) {
  st.g = slice_span<1>(ob);
  const int o = st.g.o + lane, w = st.g.w;
#pragma unroll
  for (int e = 0; e < kStage; ++e) {
    const bool ok = e < w;
    st.c[e] = ok ? __ldg(A.col + o + e * kSlice) : 0;
    st.v[e] = ok ? __ldg(A.val + o + e * kSlice) : (T)0;
  }
}

// Row products of a staged slice with x1 and (if TWO) x2.
template <class T, bool TWO>
__device__ __forceinline__ void staged_dot(const SellView<T>& A, const SliceStage<T>& st, int lane,
                                           const T* __restrict__ x1, const T* __restrict__ x2,
                                           T& acc1, T& acc2) {
  T a1[1] = {0}, a2[1] = {0};
#pragma unroll
  for (int e = 0; e < kStage; ++e)
    if (e < st.g.w) {
      a1[0] += st.v[e] * __ldg(x1 + st.c[e]);
      if (TWO) a2[0] += st.v[e] * __ldg(x2 + st.c[e]);
    }
  int k0 = kStage;
  for (; k0 + 8 <= st.g.w; k0 += 8)
    dot_chunk<T, 1, 8, kRunsNone, TWO, false>(A, st.g, int2{}, 0, k0, lane, x1, x2, a1, a2);
  for (; k0 < st.g.w; k0 += 4)
    dot_chunk<T, 1, 4, kRunsNone, TWO, true>(A, st.g, int2{}, 0, k0, lane, x1, x2, a1, a2);
  acc1 = a1[0];
  acc2 = a2[0];
}

template <class T, int MINB>
__global__ void __launch_bounds__(kBlock, MINB) k_dual_pipe(IterArgs<T> a) {
  grid_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  const int ns = a.K.nslices;
  // matrix only before the previous kernel ends: the warp's first slice
  // (entries) and the offsets of its second
  SliceStage<T> cur;
  stage_slice<T>(a.K, slice_offsets<T, 1>(a.K, gw), lane, cur);
  int2 nb = slice_offsets<T, 1>(a.K, gw + nw);
  grid_wait_prior();
  DevState* st = a.st;
  __shared__ DualScalars<T> sc;
  if (threadIdx.x == 0) dual_scalars<T>(st, sc);
  __syncthreads();
  if (sc.done) return;
  const int p = sc.p;
  const bool has_pw = sc.has_pw;
  const T pwT = sc.pw;
  const T sigma = sc.sigma;
  const T* __restrict__ xn = a.x[1 - p];
  const T* __restrict__ xc = a.x[p];
  const T* __restrict__ yc = a.y[p];
  T* __restrict__ yn = a.y[1 - p];
  T acc_dy2 = 0, acc_int = 0;
  constexpr bool kStored = StoresKx<T>::value;
  T yo, qi, lo, yb, kxo;
  auto row_ops = [&](int s, T& y0, T& q0, T& l0, T& b0, T& k0) {
    const int i = s * kSlice + lane;
    y0 = q0 = l0 = b0 = k0 = 0;
    if (s < ns && i < a.m) {
      y0 = yc[i];
      q0 = a.q[i];
      if (i >= a.m_eq) l0 = dual_floor(a.ylo, i, a.m_eq);
      if (has_pw) b0 = a.ybar[i];
      if (kStored) k0 = a.Kx[p][i];
    }
  };
  row_ops(gw, yo, qi, lo, yb, kxo);
  for (int s = gw; s < ns; s += nw) {
    // next slice: entries and row operands; offsets two slices ahead
    SliceStage<T> nxt;
    T yo2, qi2, lo2, yb2, kxo2;
    stage_slice<T>(a.K, nb, lane, nxt);
    row_ops(s + nw, yo2, qi2, lo2, yb2, kxo2);
    nb = slice_offsets<T, 1>(a.K, s + 2 * nw);
    T kx, ko;
    if constexpr (kStored) {
      T unused;
      staged_dot<T, false>(a.K, cur, lane, xn, xn, kx, unused);
      ko = kxo;
    } else {
      staged_dot<T, true>(a.K, cur, lane, xn, xc, kx, ko);
    }
    const int i = s * kSlice + lane;
    if (i < a.m) {
      T t = qi - (T)2 * kx;
      t = t + ko;
      T v = yo + sigma * t;
      if (i >= a.m_eq) v = max(v, lo);
      yn[i] = v;
      if (kStored) a.Kx[1 - p][i] = kx;
      if (has_pw) a.ybar[i] = yb + pwT * yo;
      const T dy = v - yo;
      acc_dy2 += dy * dy;
      acc_int += dy * (kx - ko);
    }
    cur = nxt;
    yo = yo2;
    qi = qi2;
    lo = lo2;
    yb = yb2;
    kxo = kxo2;
  }
  T acc[2] = {acc_dy2, acc_int};
  if (publish_partials_t<2, T>(acc, a.partials, &st->counter)) {
    double tot[2];
    final_sum_t<2, T>(a.partials, gridDim.x, tot);
    if (threadIdx.x == 0) {
      decide_step(st, a, tot[0], tot[1]);
      st->counter = 0;
    }
  }
}

template <class T, int MINB>
__global__ void __launch_bounds__(kBlock, MINB) k_adjoint_pipe(IterArgs<T> a) {
  grid_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  const int ns = a.KT.nslices;
  // matrix only before the previous kernel ends (used only if the step it
  // decides is accepted)
  SliceStage<T> cur;
  stage_slice<T>(a.KT, slice_offsets<T, 1>(a.KT, gw), lane, cur);
  int2 nb = slice_offsets<T, 1>(a.KT, gw + nw);
  grid_wait_prior();
  DevState* st = a.st;
  __shared__ AdjScalars<T> sc;
  if (threadIdx.x == 0) adj_scalars<T>(st, sc);
  __syncthreads();
  if (sc.done) return;
  const int p = sc.p;
  const int acc_last = sc.acc_last;
  const bool upd_avg = sc.upd_avg;
  const T wlT = sc.wl;
  const T tau = sc.tau;
  const T* __restrict__ yc = a.y[p];
  const T* __restrict__ xc = a.x[p];
  T* __restrict__ kty = a.KTy[p];
  T* __restrict__ xn = a.x[1 - p];
  T acc_dx2 = 0;
  auto col_ops = [&](int s, T& x0, T& c0, T& l0, T& u0, T& b0, T& g0) {
    const int j = s * kSlice + lane;
    x0 = c0 = l0 = u0 = b0 = g0 = 0;
    if (s < ns && j < a.n) {
      x0 = xc[j];
      c0 = a.c[j];
      l0 = a.l[j];
      u0 = a.u[j];
      if (upd_avg) b0 = a.xbar[j];
      if (!acc_last) g0 = kty[j];
    }
  };
  T x0, cj, lj, uj, xb, g;
  col_ops(gw, x0, cj, lj, uj, xb, g);
  for (int s = gw; s < ns; s += nw) {
    SliceStage<T> nxt;
    nxt.g.w = 0;
    T x2, c2, l2, u2, b2, g2;
    if (acc_last) {
      stage_slice<T>(a.KT, nb, lane, nxt);
      nb = slice_offsets<T, 1>(a.KT, s + 2 * nw);
    }
    col_ops(s + nw, x2, c2, l2, u2, b2, g2);
    if (acc_last) {
      T unused;
      staged_dot<T, false>(a.KT, cur, lane, yc, yc, g, unused);
    }
    const int j = s * kSlice + lane;
    if (j < a.n) {
      if (acc_last) kty[j] = g;
      if (upd_avg) a.xbar[j] = xb + wlT * x0;
      T v = x0 - tau * (cj - g);
      v = min(max(v, lj), uj);
      xn[j] = v;
      const T d = v - x0;
      acc_dx2 += d * d;
    }
    cur = nxt;
    x0 = x2;
    cj = c2;
    lj = l2;
    uj = u2;
    xb = b2;
    g = g2;
  }
  T acc[1] = {acc_dx2};
  if (publish_partials_t<1, T>(acc, a.partials, &st->counter)) {
    double tot[1];
    final_sum_t<1, T>(a.partials, gridDim.x, tot);
    if (threadIdx.x == 0) {
      st->dx2 = tot[0];
      st->counter = 0;
    }
  }
}

// x = proj_[l,u](0), y = proj(0), averages and anchors reset; K^T y.
template <class T>
__global__ void k_init_vectors(IterArgs<T> a) {
  const int64_t N = a.n > a.m ? a.n : a.m;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N;
       t += (int64_t)gridDim.x * blockDim.x) {
    if (t < a.n) {
      T v = min(max((T)0, a.l[t]), a.u[t]);
      a.x[0][t] = v;
      a.x[1][t] = v;
      a.xa[t] = v;
      a.xbar[t] = 0;
      if (a.xbar64) a.xbar64[t] = 0.0;
    }
    if (t < a.m) {
      T v = 0;
      if ((int)t >= a.m_eq) v = max(v, dual_floor(a.ylo, (int)t, a.m_eq));
      a.y[0][t] = v;
      a.y[1][t] = v;
      a.ya[t] = v;
      a.ybar[t] = 0;
      if (a.ybar64) a.ybar64[t] = 0.0;
    }
  }
}

// Product of one row without its padding slots.  They gather what their neighbours'
// run leads to: times their zero that adds nothing to a sum unless it is infinite or a
// NaN, as entries of a caller's vector may be.
template <class T>
__device__ __noinline__ T dot_entries(const T* val, const int32_t* col, int w, const T* x) {
  T acc = 0;
  for (int k = 0; k < w; ++k)
    if (!is_padding(val[k * kSlice])) acc += val[k * kSlice] * x[col[k * kSlice]];
  return acc;
}

// y = A x, or with perm the FP64 result in another order, out[perm[r]] = (A x)_r
// (pdhg_apply_K: the unscrambling, and for FP32 the widening, in the same pass).  U
// slices per warp, one pass over the matrix without a loop: a sweep this short is all
// latency.  LONG (U = 1): sixteen unpredicated entries in flight from the explicit
// indices, and the registers for them (three blocks per SM instead of five or more).
template <class T, int U, bool LONG>
__global__ void __launch_bounds__(kBlock, LONG ? 3 : U == 1 ? 8 : sizeof(T) == 4 ? 6 : 5)
    k_spmv_into(SellView<T> A, const T* __restrict__ x, T* __restrict__ y, const int32_t* __restrict__ perm,
                double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int s0 = ((blockIdx.x * kBlock + threadIdx.x) >> 5) * U;
  if (s0 >= A.nslices) return;
  T acc[U], unused[U];
  int to[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = (s0 + u) * kSlice + lane;
    to[u] = perm && r < A.rows ? __ldg(perm + r) : r;
  }
  const SliceSpan g = slice_span<U>(slice_offsets<T, U>(A, s0));
  if constexpr (LONG) {
    acc[0] = 0;
    int k0 = 0;
    for (; k0 + 16 <= g.w; k0 += 16)
      dot_chunk<T, 1, 16, kRunsNone, false, false>(A, g, int2{}, 0, k0, lane, x, x, acc, unused);
    for (; k0 < g.w; k0 += 4)
      dot_chunk<T, 1, 4, kRunsNone, false, true>(A, g, int2{}, 0, k0, lane, x, x, acc, unused);
  } else {
    sell_dot_pre<T, U, false, false>(A, s0, g, run_words<T, U>(A, g, 0, lane), lane, x, x, acc, unused);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = (s0 + u) * kSlice + lane;
    if (r < A.rows) {
      const int o = g.o + u * g.w * kSlice + lane;
      const T v = finite_bits(acc[u]) ? acc[u] : dot_entries<T>(A.val + o, A.col + o, g.w, x);
      if (perm)
        out[to[u]] = (double)v;
      else
        y[r] = v;
    }
  }
}

__global__ void k_state_init(DevState* st, RoundInit r, const double* scalars) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (r.reset_steps) {
    st->eta = r.eta > 0.0 ? r.eta : scalars[0];
    st->omega = r.omega > 0.0 ? r.omega : scalars[1];
  }
  st->dx2 = 0.0;
  st->w_last = 0.0;
  st->pending_w = 0.0;
  st->wsum = 0.0;
  st->avg_div = 0.0;
  st->par = 0;
  st->accepted_last = 0;
  st->k = 0;
  st->since_restart = 0;
  st->accepted = 0;
  st->restarts = 0;
  st->checks = 0;
  st->kkt0 = 0.0;
  st->kkt_prev = 0.0;
  st->restart_now = 0;
  st->restart_to_avg = 0;
  st->done = 0;
  st->status = 0;
  st->best_is_avg = 0;
  st->numeric = 0;
  st->tol = r.tol;
  st->ir_red = r.ir_red;
  st->fold = 0;
  st->round_target = r.tol;
  st->max_k = r.max_k;
  st->max_checks = r.max_checks;
  st->k_offset = r.k_offset;
  st->t_limit_ns = r.t_limit_ns;
  if (r.first_round) {
    st->t_start = globaltimer_ns();
    for (int i = 0; i < 3; ++i) {
      st->t_tol[i] = -1.0;
      st->k_tol[i] = -1;
    }
    st->n_trace_a = 0;
    st->n_trace_c = 0;
  }
  st->beta_suff = r.beta_suff;
  st->beta_nec = r.beta_nec;
  st->beta_art = r.beta_art;
  st->omega_smooth = r.omega_smooth;
  st->red_exp = r.red_exp;
  st->grow_exp = r.grow_exp;
  st->infeas_eps = r.infeas_eps;
  st->fold_every = r.fold_every;
  st->wait_timeout = 0;
  st->fixed = r.fixed;
  st->art_total = r.art_total;
  st->trace_on = r.trace_on;
  st->trace_cap_a = r.trace_cap_a;
  st->trace_cap_c = r.trace_cap_c;
  st->qnorm = scalars[2];
  st->cnorm = scalars[3];
  st->inv_dp = r.inv_dp;
  st->inv_dd = r.inv_dd;
  st->gap_w = r.gap_w > 0.0 ? r.gap_w : 1.0;
  st->const_p = scalars[6];
  st->const_d = scalars[7];
  st->refine = r.refine;
  st->counter = 0;
}

// ---------------------------------------------------------------------------

static int vgrid(int64_t n) {
  int64_t g = (n + kBlock - 1) / kBlock;
  if (g > 152 * 8) g = 152 * 8;
  return (int)(g < 1 ? 1 : g);
}

template <class T, int U, bool LONG>
static void spmv_slices(const SellView<T>& A, const T* x, T* y, const int32_t* perm, double* out, cudaStream_t s) {
  const int64_t warps = (A.nslices + U - 1) / U;
  const unsigned grid = (unsigned)((warps + kWarps - 1) / kWarps);
  k_spmv_into<T, U, LONG><<<grid < 1 ? 1 : grid, kBlock, 0, s>>>(A, x, y, perm, out);
}

// A slice is a serial chain of its warp, 0.27 us per entry of its rows in steps of two
// at two slices a warp.  That outlasts the rest where the widest slice has more than
// 1/65536 of the slots (LONG): K x of a transport LP (1600 rows of 700 and 900 entries)
// 276 -> 117 us, of 20000 x 20000 with 200 entries a row 84 -> 47 us.  Elsewhere LONG
// loses warps and the runs' short index reads: the 6717-bus day 68 -> 100 us.
template <class T>
static void spmv_any(const SellView<T>& A, const T* x, T* y, const int32_t* perm, double* out, cudaStream_t s) {
  if (A.widest >= 32 && (int64_t)A.widest * 65536 > (int64_t)A.slots)
    spmv_slices<T, 1, true>(A, x, y, perm, out, s);
  else if (A.own)
    spmv_slices<T, 1, false>(A, x, y, perm, out, s);
  else
    spmv_slices<T, 2, false>(A, x, y, perm, out, s);
}

template <class T>
void launch_spmv(const SellView<T>& A, const T* x, T* y, cudaStream_t s) {
  spmv_any<T>(A, x, y, nullptr, nullptr, s);
}

template <class T>
void launch_spmv_scatter(const SellView<T>& A, const T* x, const int32_t* perm, double* out, cudaStream_t s) {
  spmv_any<T>(A, x, nullptr, perm, out, s);
}

template <class T>
void launch_init_iterates(const IterArgs<T>& a, int grid, cudaStream_t s) {
  (void)grid;
  k_init_vectors<T><<<vgrid(a.n > a.m ? a.n : a.m), kBlock, 0, s>>>(a);
  launch_spmv<T>(a.KT, a.y[0], a.KTy[0], s);
  if (StoresKx<T>::value) launch_spmv<T>(a.K, a.x[0], a.Kx[0], s);
}

// Variants: 1, 2, 4 slices per warp; 0 software pipelined; 8 and 9 are the
// one-slice and the pipelined forms compiled for 8 resident blocks per SM
// (at most 32 registers, a few spilled to L1) -- more warps in flight against
// the HBM and L2 latency at the cost of the spills; 16 and 17 stage the matrix
// in shared memory with bulk copies (pdhg_staged.cu), one or two slices per
// warp at a time; 18 and 19 stage the row (column) operands with the matrix
// chunk (pdhg_rowstaged.cu); 20 and 21 keep two or three slices ahead in a
// per-warp shared-memory ring filled by cp.async (pdhg_ring.cu).
// Minimum resident blocks per SM that each variant is compiled for: the
// register budget that keeps the one-slice forms at 6 (FP32) or 5 (FP64)
// blocks per SM without spills (an unconstrained build takes ~58 registers and
// drops to 4 blocks per SM).
template <class T, int U>
struct MinBlocks {
  static constexpr int value = U == 1 ? (sizeof(T) == 4 ? 6 : 5) : (sizeof(T) == 4 ? 4 : 3);
};
template <class T>
struct MinBlocksPipe {
  static constexpr int value = sizeof(T) == 4 ? 5 : 3;
};

// One per-attempt kernel, with the programmatic-dependent-launch attribute when
// a.overlap is set (the kernel then overlaps its matrix prologue with the end
// of the previous kernel in the stream or graph).
template <class T>
static void launch_iter(void (*k)(IterArgs<T>), const IterArgs<T>& a, int grid, cudaStream_t s) {
  if (!a.overlap) {
    k<<<grid, kBlock, 0, s>>>(a);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, a);
}

template <class T>
void launch_dual(const IterArgs<T>& a, int grid, cudaStream_t s, int unroll) {
  constexpr int B = MinBlocks<T, 2>::value;
  static_assert(B == MinBlocks<T, 4>::value, "variants 2 and 4 share it");
  switch (unroll) {
    case 0: launch_iter<T>(k_dual_pipe<T, MinBlocksPipe<T>::value>, a, grid, s); break;
    case 2: launch_iter<T>(a.K.own ? k_dual<T, 2, B, true> : k_dual<T, 2, B>, a, grid, s); break;
    case 4: launch_iter<T>(a.K.own ? k_dual<T, 4, B, true> : k_dual<T, 4, B>, a, grid, s); break;
    case 8: launch_iter<T>(k_dual<T, 1, 8>, a, grid, s); break;
    case 9: launch_iter<T>(k_dual_pipe<T, 8>, a, grid, s); break;
    case 16: launch_dual_staged<T>(a, grid, s, 1); break;
    case 17: launch_dual_staged<T>(a, grid, s, 2); break;
    case 18: launch_dual_rowstaged<T>(a, grid, s, 1); break;
    case 19: launch_dual_rowstaged<T>(a, grid, s, 2); break;
    case 20: launch_dual_ring<T>(a, grid, s, 3); break;
    case 21: launch_dual_ring<T>(a, grid, s, 4); break;
    default: launch_iter<T>(k_dual<T, 1, MinBlocks<T, 1>::value>, a, grid, s); break;
  }
}

template <class T>
void launch_adjoint(const IterArgs<T>& a, int grid, cudaStream_t s, int unroll) {
  constexpr int B = MinBlocks<T, 2>::value;
  switch (unroll) {
    case 0: launch_iter<T>(k_adjoint_pipe<T, MinBlocksPipe<T>::value>, a, grid, s); break;
    case 2: launch_iter<T>(a.KT.own ? k_adjoint<T, 2, B, true> : k_adjoint<T, 2, B>, a, grid, s); break;
    case 4: launch_iter<T>(a.KT.own ? k_adjoint<T, 4, B, true> : k_adjoint<T, 4, B>, a, grid, s); break;
    case 8: launch_iter<T>(k_adjoint<T, 1, 8>, a, grid, s); break;
    case 9: launch_iter<T>(k_adjoint_pipe<T, 8>, a, grid, s); break;
    case 16: launch_adjoint_staged<T>(a, grid, s, 1); break;
    case 17: launch_adjoint_staged<T>(a, grid, s, 2); break;
    case 18: launch_adjoint_rowstaged<T>(a, grid, s, 1); break;
    case 19: launch_adjoint_rowstaged<T>(a, grid, s, 2); break;
    case 20: launch_adjoint_ring<T>(a, grid, s, 3); break;
    case 21: launch_adjoint_ring<T>(a, grid, s, 4); break;
    default: launch_iter<T>(k_adjoint<T, 1, MinBlocks<T, 1>::value>, a, grid, s); break;
  }
}

void launch_state_init(DevState* st, const RoundInit& r, const double* scalars, cudaStream_t s) {
  k_state_init<<<1, 32, 0, s>>>(st, r, scalars);
}

int blocks_per_sm_iter() {
  int best = 1 << 30;
  const void* fns[4] = {(const void*)&k_dual<double, 1, MinBlocks<double, 1>::value>,
                        (const void*)&k_adjoint<double, 1, MinBlocks<double, 1>::value>,
                        (const void*)&k_dual<float, 1, MinBlocks<float, 1>::value>,
                        (const void*)&k_adjoint<float, 1, MinBlocks<float, 1>::value>};
  for (const void* f : fns) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, kBlock, 0) != cudaSuccess) b = 4;
    best = b < best ? b : best;
  }
  return best < 1 ? 1 : best;
}

template void launch_spmv<double>(const SellView<double>&, const double*, double*, cudaStream_t);
template void launch_spmv<float>(const SellView<float>&, const float*, float*, cudaStream_t);
template void launch_spmv_scatter<double>(const SellView<double>&, const double*, const int32_t*, double*,
                                          cudaStream_t);
template void launch_spmv_scatter<float>(const SellView<float>&, const float*, const int32_t*, double*,
                                         cudaStream_t);
template void launch_init_iterates<double>(const IterArgs<double>&, int, cudaStream_t);
template void launch_init_iterates<float>(const IterArgs<float>&, int, cudaStream_t);
template void launch_dual<double>(const IterArgs<double>&, int, cudaStream_t, int);
template void launch_dual<float>(const IterArgs<float>&, int, cudaStream_t, int);
template void launch_adjoint<double>(const IterArgs<double>&, int, cudaStream_t, int);
template void launch_adjoint<float>(const IterArgs<float>&, int, cudaStream_t, int);

}  // namespace ucpdhg
