// Batched node LPs that share K, c and q and differ in their bounds (the
// branch-and-bound relaxations whose bounds the paper's PDHG provides,
// Sec. III.B), solved together: FP32 iterations, FP64 KKT checks and FP64
// iterative refinement, with per-instance step size, primal weight, restarts,
// refinement rounds and termination.
//
// Layout: every per-instance vector is interleaved, v[i * BP + b] (BP = 32 or
// 64 instance slots), so one sweep over K serves all instances: a warp owns a
// row, its lanes own instances, the row's column/value loads are broadcasts
// and the gather x[col * BP + b] is one contiguous 128/256 B access.
//
// Refinement rounds run inside the graph: when an instance's current iterate
// (x^, y^) halves the round's starting rel-KKT at a check without a restart,
// the next correction LP follows elementwise from the FP64 products the check
// already computed (K x^ and K^T y^):
//   q^' = f (q^ - K x^),  c^' = f (c^ - K^T y^),  [l^',u^'] = f ([l^,u^] - x^),
//   y_lo^' = f (y_lo^ - y^),  f = Delta'/Delta,  x* += x^/Delta,  y* += y^/Delta
// and the iteration state moves to the new coordinates v' = f (v - x^): the
// iterate becomes 0 (K x^ = K^T y^ = 0), anchors and averages shift with it,
// step size, primal weight and restart window carry over.  The whole batch is
// one CUDA graph whose while loop runs until every instance is done.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "internal.cuh"

namespace ucpdhg {
namespace {

constexpr int kBWarps = 8;            // warps per block of the row/column sweeps
constexpr int kBThreads = kBWarps * 32;
constexpr int kKktWarps = 4;          // smaller blocks for the FP64 check sweeps
constexpr int kApplyRows = 4;         // rows per block of the elementwise kernels (x BP threads)
constexpr int kRowS = 7, kColS = 9;   // per-candidate sums (as in the single-instance check,
                                      // including the infeasibility-ray sums)
// Rows (columns) a warp sweeps together in kb_dual (kb_adjoint): R = 4, 2 or 1
// adjacent slots of a slice, read as int4/float4, int2/float2 or scalars; the
// batched autotuner picks R and the grid per matrix and batch width.
template <int R>
__device__ __forceinline__ void load_slots(const int32_t* __restrict__ c, const float* __restrict__ v,
                                           int (&cc)[R], float (&vv)[R]) {
  if constexpr (R == 4) {
    const int4 c4 = __ldg(reinterpret_cast<const int4*>(c));
    const float4 v4 = __ldg(reinterpret_cast<const float4*>(v));
    cc[0] = c4.x; cc[1] = c4.y; cc[2] = c4.z; cc[3] = c4.w;
    vv[0] = v4.x; vv[1] = v4.y; vv[2] = v4.z; vv[3] = v4.w;
  } else if constexpr (R == 2) {
    const int2 c2 = __ldg(reinterpret_cast<const int2*>(c));
    const float2 v2 = __ldg(reinterpret_cast<const float2*>(v));
    cc[0] = c2.x; cc[1] = c2.y;
    vv[0] = v2.x; vv[1] = v2.y;
  } else {
    cc[0] = __ldg(c);
    vv[0] = __ldg(v);
  }
}

// Per-instance state (array of B structs in device memory).
struct BInst {
  double eta, omega, dx2, w_last, pending_w, wsum, avg_div;
  int32_t par, accepted_last;
  int64_t k, k_total, since_restart, accepted, restarts, checks;
  double kkt0, kkt_prev;
  int32_t restart_now, restart_to_avg;
  int32_t done, status, rounds, act;  // act: takes part in the next attempts
  int32_t refine, finalize, cand_avg, round_checks;  // round_checks: checks this round
  double rel_p, rel_d, rel_gap, rel_kkt, pobj, dobj;
  double round_target;
  double round_rel0;      // rel_kkt of the current iterate at the round's start
  double dp, dd;          // Delta_P, Delta_D of the current round
  double next_scale;      // Delta' / Delta for the refinement step
  double const_p, const_d;
  double t_tol[3];
  int64_t k_tol[3];
  // what the sweeps read of the above, converted where it changes (a block that
  // multiplies or divides in FP64 at its start waits for it): eta omega, eta /
  // omega, pending_w, w_last; and 1 / omega for the step decision
  float sigma, tau, pend, last;
  double inv_omega;
};

__device__ __forceinline__ void set_steps(BInst& I) {
  I.inv_omega = 1.0 / I.omega;
  I.sigma = (float)(I.eta * I.omega);
  I.tau = (float)(I.eta * I.inv_omega);
  I.pend = (float)I.pending_w;
  I.last = (float)I.w_last;
}

struct BGlobal {
  double tol, red;
  double beta_suff, beta_nec, beta_art, omega_smooth, red_exp, grow_exp;
  int64_t max_k;
  uint64_t t_start, t_limit_ns;
  double qnorm, cnorm;
  double infeas_eps;  // certificate tolerance of the infeasibility test (0: off)
  int32_t fold_every;  // a refinement round also ends after this many checks (0: off)
  int32_t n_real, all_done;
};

template <int BP>
struct BArgs {
  SellView<float> K, KT;      // FP32 values (iterations)
  SellView<double> K64, KT64; // FP64 values (checks)
  int32_t n, m, m_eq, B;
  // FP32 iterate data [len * BP]
  float *x[2], *y[2], *Kx[2], *KTy[2];
  float *xbar, *ybar, *xa, *ya;  // xbar, ybar: step-weighted sums since the last check
  double *xbar64, *ybar64;        // the sums since the last restart (FP64; the window's
                                  // FP32 sums are added in and cleared at every check,
                                  // so refinement folds re-express exact sums)
  float *cf, *lf, *uf, *qf, *ylf;
  // FP64 data [len * BP]
  double *xst, *yst;          // accumulated x*, y* (scaled space)
  double *ch, *lh, *uh;       // correction c^, l^, u^
  double *qh, *ylh;           // correction q^, y_lo^
  double *lo, *uo;            // instance bounds l~, u~ (scaled)
  double *Kzc, *Kza;          // K x^ of current / average (FP64)
  double *KTzc, *KTza;        // K^T y^ of current / average
  double *Kxa, *KTya;         // K x^, K^T y^ of the restart anchors (infeasibility rays)
  const double *c_obj, *q_obj, *iDr, *iDc, *Dr, *Dc;  // shared [len]
  BInst* inst;
  BGlobal* g;
  double* part;               // per-block partials
  uint32_t* tier;             // arrivals of grid_inst_sum: the groups, each group's blocks (0 between kernels)
  volatile int32_t* cancel;
  unsigned long long cond;
  int32_t in_graph;
};

// A lane's H = BP / 32 instances are neighbours, b = H lane + h, so that their
// values are one 8-byte access where both take part; idx is the first one's.
template <int H>
__device__ __forceinline__ void load_inst(const float* __restrict__ v, size_t idx, float (&o)[H]) {
  if constexpr (H == 2) {
    const float2 t = *reinterpret_cast<const float2*>(v + idx);
    o[0] = t.x;
    o[1] = t.y;
  } else {
    o[0] = v[idx];
  }
}
template <int H>
__device__ __forceinline__ void gather_inst(const float* __restrict__ v, size_t idx, float (&o)[H]) {
  if constexpr (H == 2) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(v + idx));
    o[0] = t.x;
    o[1] = t.y;
  } else {
    o[0] = __ldg(v + idx);
  }
}
template <int H>
__device__ __forceinline__ void load_inst(const double* __restrict__ v, size_t idx, double (&o)[H]) {
  if constexpr (H == 2) {
    const double2 t = *reinterpret_cast<const double2*>(v + idx);
    o[0] = t.x;
    o[1] = t.y;
  } else {
    o[0] = v[idx];
  }
}
template <int H>
__device__ __forceinline__ void store_inst(float* __restrict__ v, size_t idx, const float (&o)[H]) {
  if constexpr (H == 2)
    *reinterpret_cast<float2*>(v + idx) = make_float2(o[0], o[1]);
  else
    v[idx] = o[0];
}
template <int H, class T>
__device__ __forceinline__ void store_inst(T* __restrict__ v, size_t idx, const T (&o)[H], const bool (&on)[H]) {
  if constexpr (H == 2) {
    if (on[0] && on[1]) {
      if constexpr (sizeof(T) == 4)
        *reinterpret_cast<float2*>(v + idx) = make_float2(o[0], o[1]);
      else
        *reinterpret_cast<double2*>(v + idx) = make_double2(o[0], o[1]);
      return;
    }
  }
#pragma unroll
  for (int h = 0; h < H; ++h)
    if (on[h]) v[idx + h] = o[h];
}
// The same from the buffers that each instance's parity selects.
template <int H>
__device__ __forceinline__ void load_par(float* const (&v)[2], const int (&par)[H], size_t idx, float (&o)[H]) {
  if (H == 1 || par[0] == par[H - 1]) {
    load_inst<H>(par[0] ? v[1] : v[0], idx, o);
    return;
  }
#pragma unroll
  for (int h = 0; h < H; ++h) o[h] = (par[h] ? v[1] : v[0])[idx + h];
}

__host__ __device__ __forceinline__ double* preg(double* p, int r) { return p + (size_t)r * 8192 * 64 * 20; }

// Per-instance block reduction of NV values held by each lane for its instances
// b = first + step h: put_inst leaves them in smem [warps][BP][NV], sum_inst writes
// the sums to part[block][b][k] by threads b < BP.
template <int BP, int NV>
__device__ __forceinline__ void put_inst(const double (&v)[BP / 32][NV], double* smem, int first, int step) {
#pragma unroll
  for (int h = 0; h < BP / 32; ++h)
#pragma unroll
    for (int k = 0; k < NV; ++k) smem[((threadIdx.x >> 5) * BP + first + step * h) * NV + k] = v[h][k];
}
template <int BP, int NV, int WARPS>
__device__ __forceinline__ void sum_inst(const double* smem, double* out) {
  __syncthreads();
  if (threadIdx.x < BP) {
    const int b = threadIdx.x;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
      for (int w = 0; w < WARPS; ++w) s += smem[(w * BP + b) * NV + k];
      out[((size_t)blockIdx.x * BP + b) * NV + k] = s;
    }
  }
  __syncthreads();
}

// Per-instance sums of NV partials over `nblocks` blocks (layout
// part[blk][BP][NV]) by ALL threads of the calling block: thread t sums the
// blocks t/BP, t/BP + C, ... (C = blockDim / BP chunks) for instance t % BP,
// then the chunks are combined in order.  Deterministic; result valid in
// threads t < BP.  smem: [C][BP][NV] doubles.
template <int BP, int NV>
__device__ __forceinline__ void inst_final_sum(const double* part, int nblocks, double* smem,
                                               double (&out)[NV]) {
  const int b = threadIdx.x % BP, c = threadIdx.x / BP, C = blockDim.x / BP;
  double v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = 0.0;
  if (c < C)
#pragma unroll 8  // loads in flight: one block sums what the whole grid wrote
    for (int blk = c; blk < nblocks; blk += C)
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] += __ldcg(part + ((size_t)blk * BP + b) * NV + k);
#pragma unroll
  for (int k = 0; k < NV; ++k) smem[(c * BP + b) * NV + k] = v[k];
  __syncthreads();
  if (threadIdx.x < BP) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
      for (int cc = 0; cc < C; ++cc) s += smem[(cc * BP + b) * NV + k];
      out[k] = s;
    }
  }
  __syncthreads();
}

// True in the last of `count` blocks to arrive at *counter.
__device__ __forceinline__ bool last_arrival(uint32_t* counter, unsigned count) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == count - 1;
    if (last) *counter = 0;  // everyone has arrived: ready for the next kernel
  }
  __syncthreads();
  return last != 0;
}

// Per-instance sums over the grid of what block_inst_sum left in part[block]: true
// in one block, whose threads t < BP then hold them.  One block adding up the whole
// grid is bound by its FP64 pipe (two lanes a clock: 34 ns per block of 64 x 2
// values, 5 us of the 33 us of K x' for 64 node LPs of 200 buses at 152 blocks, and
// it kept the sweeps from more blocks), so the last of every kTier blocks adds up
// those, on its own SM, and the last of these the groups'.  Fixed order.
// Now 20.0 us at 304 blocks, K^T y' 25.5 -> 16.6; 9 node LPs of 24 buses 17.5 -> 13.2 ms
// for 512 attempts.
constexpr int kTier = 16;
constexpr int kTierCount = 1 + (kMaxBlocks + kTier - 1) / kTier;
constexpr size_t kTierSums = (size_t)kMaxBlocks * 64 * 3;  // of `part`, behind the blocks' own
template <int BP, int NV>
__device__ __forceinline__ bool grid_inst_sum(double* part, uint32_t* tier, double* smem, double (&tot)[NV]) {
  static_assert(BP * NV <= 64 * 3, "fits before kTierSums");
  const unsigned grp = blockIdx.x / kTier, groups = (gridDim.x + kTier - 1) / kTier;
  const unsigned cnt = min((unsigned)kTier, gridDim.x - grp * kTier);
  if (!last_arrival(tier + 1 + grp, cnt)) return false;
  inst_final_sum<BP, NV>(part + (size_t)grp * kTier * BP * NV, cnt, smem, tot);
  if (groups == 1) return true;
  double* sums = part + kTierSums;
  if (threadIdx.x < BP)
#pragma unroll
    for (int k = 0; k < NV; ++k) sums[((size_t)grp * BP + threadIdx.x) * NV + k] = tot[k];
  if (!last_arrival(tier, groups)) return false;
  inst_final_sum<BP, NV>(sums, groups, smem, tot);
  return true;
}

// ---------------------------------------------------------------- attempt kernels

// K x' and the projected dual step for every active instance; the last block
// takes each instance's adaptive step decision.
template <int BP, int RW>
__global__ void __launch_bounds__(kBThreads) kb_dual(BArgs<BP> a) {
  BGlobal* g = a.g;
  constexpr int H = BP / 32;
  __shared__ float s_sigma[BP], s_pw[BP];
  __shared__ int s_par[BP], s_act[BP];
  const int all_done = g->all_done;  // read with the instances' state, not before it
  if (threadIdx.x < BP) {
    const BInst& I = a.inst[threadIdx.x];
    s_sigma[threadIdx.x] = I.sigma;
    s_pw[threadIdx.x] = I.pend;
    s_par[threadIdx.x] = I.par;
    s_act[threadIdx.x] = I.act;
  }
  __syncthreads();
  if (all_done) return;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBThreads + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBThreads) >> 5;
  struct Lane {  // of the instances b = first + step h
    float sigma[H], pw[H];
    int par[H];
    bool on[H], upd[H];
  };
  auto lane_state = [&](int first, int step) {
    Lane s;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int b = first + step * h;
      s.sigma[h] = s_sigma[b];
      s.pw[h] = s_pw[b];
      s.par[h] = s_par[b];
      s.on[h] = s_act[b];
      s.upd[h] = s.on[h] && s.pw[h] != 0.f;
    }
    return s;
  };
  __shared__ double smem[kBWarps * BP * 2];
  // Where all lanes' instances agree in pairs on what they do and on their buffers
  // (always with one instance per lane; with two until a step of one is rejected, one
  // ends, or B is odd) every access is one of a lane's pair (b = 2 lane + h); else
  // each instance's are its own, a warp's contiguous (b = lane + 32 h).  64 node LPs of
  // 6049 buses x 48 periods, K x' and K^T y': 545 and 448 us in pairs, 624 and 537 us one
  // by one (708 and 612 us one by one with b = 2 lane + h), of 455 us for the vectors
  // of K x' alone at the copy bandwidth.
  const int nq = (a.m + RW - 1) / RW;
  auto sweep = [&](auto paired, const Lane& me) {
    constexpr int S = decltype(paired)::value ? H : 1;  // instances per access
    constexpr int N = H / S;                            // accesses per lane
    const int at = S * lane;                            // access g: instances at + 32 g ...
    float a_dy2[H], a_int[H];
#pragma unroll
    for (int h = 0; h < H; ++h) a_dy2[h] = a_int[h] = 0.f;
    const float *xg[N], *kxr[N], *yr[N];
    float *kxw[N], *yw[N];
#pragma unroll
    for (int g = 0; g < N; ++g) {
      const int p = me.par[g * S];
      xg[g] = me.on[g * S] ? a.x[1 - p] + at + 32 * g : nullptr;
      kxr[g] = a.Kx[p];
      yr[g] = a.y[p];
      kxw[g] = a.Kx[1 - p];
      yw[g] = a.y[1 - p];
    }
    for (int qd = gw; qd < nq; qd += nw) {
      const int i0 = qd * RW;  // RW consecutive rows of one slice
      const int s = i0 >> 5;
      const int o_s = __ldg(a.K.off + s);
      const int base = o_s + (i0 & 31);
      const int w = (__ldg(a.K.off + s + 1) - o_s) >> 5;
      // row operands do not depend on the products: issue them first so their
      // latency overlaps the matrix stream and the gathers
      float ko[RW][N][S], yo[RW][N][S], qv[RW][N][S], lo[RW][N][S], yb[RW][N][S], acc[RW][N][S];
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int g = 0; g < N; ++g) {
          const int i = i0 + r;
#pragma unroll
          for (int t = 0; t < S; ++t)
            ko[r][g][t] = yo[r][g][t] = qv[r][g][t] = lo[r][g][t] = yb[r][g][t] = acc[r][g][t] = 0.f;
          if (i < a.m && xg[g]) {
            const size_t idx = (size_t)i * BP + at + 32 * g;
            load_inst<S>(kxr[g], idx, ko[r][g]);
            load_inst<S>(yr[g], idx, yo[r][g]);
            load_inst<S>(a.qf, idx, qv[r][g]);
            if (i >= a.m_eq) load_inst<S>(a.ylf, idx, lo[r][g]);
            if (me.upd[g * S]) load_inst<S>(a.ybar, idx, yb[r][g]);
          }
        }
      // entry k of the group's rows: RW adjacent slots (16 B aligned:
      // slice offsets are multiples of 32 and i0 of RW)
#pragma unroll 2
      for (int k = 0; k < w; ++k) {
        int c[RW];
        float v[RW];
        load_slots<RW>(a.K.col + base + k * kSlice, a.K.val + base + k * kSlice, c, v);
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
          for (int g = 0; g < N; ++g)
            if (xg[g]) {
              float x[S];
              gather_inst<S>(xg[g], (size_t)c[r] * BP, x);
#pragma unroll
              for (int t = 0; t < S; ++t) acc[r][g][t] += v[r] * x[t];
            }
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const int i = i0 + r;
        if (i >= a.m) continue;
#pragma unroll
        for (int g = 0; g < N; ++g) {
          if (!xg[g]) continue;
          const size_t idx = (size_t)i * BP + at + 32 * g;
          float vn[S], bn[S];
#pragma unroll
          for (int t = 0; t < S; ++t) {
            const int h = g * S + t;
            float z = qv[r][g][t] - 2.f * acc[r][g][t];
            z = z + ko[r][g][t];
            float v = yo[r][g][t] + me.sigma[h] * z;
            if (i >= a.m_eq) v = fmaxf(v, lo[r][g][t]);
            vn[t] = v;
            bn[t] = yb[r][g][t] + me.pw[h] * yo[r][g][t];
            const float dy = v - yo[r][g][t], dk = acc[r][g][t] - ko[r][g][t];
            a_dy2[h] += dy * dy;
            a_int[h] += dy * dk;
          }
          store_inst<S>(kxw[g], idx, acc[r][g]);
          store_inst<S>(yw[g], idx, vn);
          if (me.upd[g * S]) store_inst<S>(a.ybar, idx, bn);
        }
      }
    }
    double v[H][2];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      v[h][0] = (double)a_dy2[h];
      v[h][1] = (double)a_int[h];
    }
    put_inst<BP, 2>(v, smem, at, S == H ? 1 : 32);
  };
  const Lane me = lane_state(H * lane, 1);
  if (__all_sync(0xffffffffu,
                 H == 1 || (me.par[0] == me.par[H - 1] && me.on[0] == me.on[H - 1] && me.upd[0] == me.upd[H - 1])))
    sweep(std::true_type{}, me);
  else
    sweep(std::false_type{}, lane_state(lane, 32));
  sum_inst<BP, 2, kBWarps>(smem, a.part);
  double tot[2];
  if (grid_inst_sum<BP, 2>(a.part, a.tier, smem, tot)) {
    double down = 0.0, up = 0.0;
    if (threadIdx.x < BP) {  // does not depend on the sums
      const int64_t k = a.inst[threadIdx.x].k_total + 2;
      down = 1.0 - step_power(k, g->red_exp);
      up = 1.0 + step_power(k, g->grow_exp);
    }
    if (threadIdx.x < BP) {
      const int b = threadIdx.x;
      BInst& I = a.inst[b];
      if (I.act) {
        // attempts of all rounds (a refinement round is a change of coordinates)
        const double dy2 = tot[0], inter = tot[1];
        const double eta = I.eta, omega = I.omega;
        const double movement = omega * I.dx2 + dy2 * I.inv_omega;
        const double interaction = 2.0 * fabs(inter);
        const double eta_max = interaction > 0.0 ? movement / interaction : INFINITY;
        const double eta_next = fmin(down * eta_max, up * eta);
        const int accept = eta <= eta_max;
        const double w = accept ? eta : 0.0;
        I.k += 1;
        I.k_total += 1;
        if (accept) {
          I.par = 1 - I.par;
          I.wsum += eta;
          I.accepted += 1;
        }
        I.w_last = I.pending_w = w;
        I.last = I.pend = (float)w;
        I.accepted_last = accept;
        I.since_restart += 1;
        I.eta = eta_next;
        I.tau = (float)(eta_next * I.inv_omega);
        I.sigma = (float)(eta_next * omega);
      }
    }
  }
}

// K^T y' for instances whose step was accepted, the x-average update and the
// next primal step x'' = proj(x - tau (c - K^T y)).
template <int BP, int RW>
__global__ void __launch_bounds__(kBThreads) kb_adjoint(BArgs<BP> a) {
  BGlobal* g = a.g;
  constexpr int H = BP / 32;
  __shared__ float s_tau[BP], s_wl[BP];
  __shared__ int s_par[BP], s_act[BP], s_acc[BP];
  const int all_done = g->all_done;
  if (threadIdx.x < BP) {
    const BInst& I = a.inst[threadIdx.x];
    s_tau[threadIdx.x] = I.tau;
    s_wl[threadIdx.x] = I.last;
    s_par[threadIdx.x] = I.par;
    s_act[threadIdx.x] = I.act;
    s_acc[threadIdx.x] = I.act && I.accepted_last;
  }
  __syncthreads();
  if (all_done) return;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBThreads + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBThreads) >> 5;
  struct Lane {  // as in kb_dual
    float tau[H], wl[H];
    int par[H];
    bool on[H], got[H], upd[H];  // active; new K^T y this attempt; the x-average moves
  };
  auto lane_state = [&](int first, int step) {
    Lane s;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int b = first + step * h;
      s.tau[h] = s_tau[b];
      s.wl[h] = s_wl[b];
      s.par[h] = s_par[b];
      s.on[h] = s_act[b];
      s.got[h] = s_acc[b];
      s.upd[h] = s.got[h] && s.wl[h] != 0.f;
    }
    return s;
  };
  __shared__ double smem[kBWarps * BP];
  const int nq = (a.n + RW - 1) / RW;
  auto sweep = [&](auto paired, const Lane& me) {  // as in kb_dual
    constexpr int S = decltype(paired)::value ? H : 1;
    constexpr int N = H / S;
    const int at = S * lane;
    float a_dx2[H];
#pragma unroll
    for (int h = 0; h < H; ++h) a_dx2[h] = 0.f;
    const float *yg[N], *xr[N];
    float *kty[N], *xw[N];
#pragma unroll
    for (int g = 0; g < N; ++g) {
      const int p = me.par[g * S];
      yg[g] = me.got[g * S] ? a.y[p] + at + 32 * g : nullptr;
      xr[g] = a.x[p];
      xw[g] = a.x[1 - p];
      kty[g] = a.KTy[p];
    }
    for (int qd = gw; qd < nq; qd += nw) {
      const int j0 = qd * RW;  // RW consecutive columns of one slice
      const int s = j0 >> 5;
      const int o_s = __ldg(a.KT.off + s);
      const int base = o_s + (j0 & 31);
      const int w = (__ldg(a.KT.off + s + 1) - o_s) >> 5;
      float x0[RW][N][S], cv[RW][N][S], lv[RW][N][S], uv[RW][N][S], xb[RW][N][S], acc[RW][N][S];
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int g = 0; g < N; ++g) {
          const int j = j0 + r;
#pragma unroll
          for (int t = 0; t < S; ++t)
            x0[r][g][t] = cv[r][g][t] = lv[r][g][t] = uv[r][g][t] = xb[r][g][t] = acc[r][g][t] = 0.f;
          if (j < a.n && me.on[g * S]) {
            const size_t idx = (size_t)j * BP + at + 32 * g;
            load_inst<S>(xr[g], idx, x0[r][g]);
            load_inst<S>(a.cf, idx, cv[r][g]);
            load_inst<S>(a.lf, idx, lv[r][g]);
            load_inst<S>(a.uf, idx, uv[r][g]);
            if (!yg[g]) load_inst<S>(kty[g], idx, acc[r][g]);  // the old K^T y
            if (me.upd[g * S]) load_inst<S>(a.xbar, idx, xb[r][g]);
          }
        }
#pragma unroll 2
      for (int k = 0; k < w; ++k) {
        int c[RW];
        float v[RW];
        load_slots<RW>(a.KT.col + base + k * kSlice, a.KT.val + base + k * kSlice, c, v);
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
          for (int g = 0; g < N; ++g)
            if (yg[g]) {
              float y[S];
              gather_inst<S>(yg[g], (size_t)c[r] * BP, y);
#pragma unroll
              for (int t = 0; t < S; ++t) acc[r][g][t] += v[r] * y[t];
            }
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const int j = j0 + r;
        if (j >= a.n) continue;
#pragma unroll
        for (int g = 0; g < N; ++g) {
          if (!me.on[g * S]) continue;
          const size_t idx = (size_t)j * BP + at + 32 * g;
          float vn[S], bn[S];
#pragma unroll
          for (int t = 0; t < S; ++t) {
            const int h = g * S + t;
            bn[t] = xb[r][g][t] + me.wl[h] * x0[r][g][t];
            float v = x0[r][g][t] - me.tau[h] * (cv[r][g][t] - acc[r][g][t]);
            v = fminf(fmaxf(v, lv[r][g][t]), uv[r][g][t]);
            vn[t] = v;
            const float d = v - x0[r][g][t];
            a_dx2[h] += d * d;
          }
          if (yg[g]) store_inst<S>(kty[g], idx, acc[r][g]);
          if (me.upd[g * S]) store_inst<S>(a.xbar, idx, bn);
          store_inst<S>(xw[g], idx, vn);
        }
      }
    }
    double v[H][1];
#pragma unroll
    for (int h = 0; h < H; ++h) v[h][0] = (double)a_dx2[h];
    put_inst<BP, 1>(v, smem, at, S == H ? 1 : 32);
  };
  const Lane me = lane_state(H * lane, 1);
  if (H == 1 || __all_sync(0xffffffffu, me.par[0] == me.par[H - 1] && me.on[0] == me.on[H - 1] &&
                                            me.got[0] == me.got[H - 1] && me.upd[0] == me.upd[H - 1]))
    sweep(std::true_type{}, me);
  else
    sweep(std::false_type{}, lane_state(lane, 32));
  sum_inst<BP, 1, kBWarps>(smem, a.part);
  double tot[1];
  if (grid_inst_sum<BP, 1>(a.part, a.tier, smem, tot)) {
    if (threadIdx.x < BP) {
      const int b = threadIdx.x;
      if (a.inst[b].act) a.inst[b].dx2 = tot[0];
    }
  }
}

// ---------------------------------------------------------------- checks (FP64)

// xbar64 += xbar: the window's sums join the FP64 sums before a check, so that the
// row side gathers one of them.
template <int BP>
__global__ void kb_flush_x(BArgs<BP> a) {
  if (a.g->all_done) return;
  const size_t N = (size_t)a.n * BP / 4;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < N; t += (size_t)gridDim.x * blockDim.x) {
    const float4 w = reinterpret_cast<const float4*>(a.xbar)[t];
    if (!(non_zero(w.x) || non_zero(w.y) || non_zero(w.z) || non_zero(w.w))) continue;
    double2* d = reinterpret_cast<double2*>(a.xbar64) + 2 * t;
    double2 p = d[0], q = d[1];
    p.x += to_f64(w.x);
    p.y += to_f64(w.y);
    q.x += to_f64(w.z);
    q.y += to_f64(w.w);
    d[0] = p;
    d[1] = q;
    reinterpret_cast<float4*>(a.xbar)[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Products of row i with two vectors of every instance, FP64 throughout; o, w: the
// first slot and the entries of its slice (loaded a row ahead).  E entries are in
// flight: four on the row side, so that most rows cost one round trip for the
// entries and one for the gathers; two on the column side, whose sums leave no
// registers for more (5.4 against 6.1 ms).
template <int BP, int E>
__device__ __forceinline__ void kb_dots(const SellView<double>& A, int o, int w, int i, int lane,
                                        float* const (&x)[2], const int (&par)[BP / 32],
                                        const double* __restrict__ xs, bool some, double (&d0)[BP / 32],
                                        double (&d1)[BP / 32]) {
  constexpr int H = BP / 32;
#pragma unroll
  for (int h = 0; h < H; ++h) d0[h] = d1[h] = 0.0;
  if (!some) return;
  for (int k0 = 0; k0 < w; k0 += E) {
    float g[E][H];
    double t[E][H], v[E];
    int c[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const bool ok = k0 + e < w;
      const int slot = o + (k0 + (ok ? e : 0)) * kSlice + (i & 31);
      c[e] = __ldg(A.col + slot);
      v[e] = __ldg(A.val + slot);
    }
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (k0 + e < w) {
        const size_t ci = (size_t)c[e] * BP + H * lane;
        load_par<H>(x, par, ci, g[e]);
        load_inst<H>(xs, ci, t[e]);
      }
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (k0 + e < w)
#pragma unroll
        for (int h = 0; h < H; ++h) {
          d0[h] += v[e] * to_f64(g[e][h]);
          d1[h] += v[e] * t[e][h];
        }
  }
}

// The infeasibility rays of each instance are the differences of its current
// and average iterates from its last restart anchor, tested as in the
// single-instance check (pdhg_kkt.cu): the anchors' FP64 products Kxa, KTya are
// seeded at the first check and moved at restarts and refinement folds.
// FP64-pipe bound like that check, and written like it; here a warp holds one
// row (column) of all instances, so what is left out as zero is a row inactive
// in every node LP.  64 node LPs of 6049 buses x 48 periods: row side 10.3 ms
// before, 5.6 ms now; column side 10.9 ms before, 5.4 ms now
// (row side at 80% of the FP64 pipe).
template <int BP>
__global__ void __launch_bounds__(kKktWarps * 32) kb_kkt_row(BArgs<BP> a, int init) {
  BGlobal* g = a.g;
  if (g->all_done) return;
  constexpr int H = BP / 32;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double acc[H][2 * kRowS], iw[H], idp2[H];
  float pw[H];
  int par[H];
  bool on[H], has_avg[H];
  bool some = false;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const BInst& I = a.inst[H * lane + h];
    has_avg[h] = I.wsum > 0.0;
    iw[h] = has_avg[h] ? 1.0 / I.wsum : 0.0;
    idp2[h] = 1.0 / (I.dp * I.dp);
    pw[h] = (float)I.pending_w;
    par[h] = I.par;
    on[h] = I.act;
    some = some || on[h];
#pragma unroll
    for (int k = 0; k < 2 * kRowS; ++k) acc[h][k] = 0.0;
  }
  int o_next = 0, e_next = 0;  // the next row's slice
  if (gw < a.m) {
    o_next = __ldg(a.K64.off + (gw >> 5));
    e_next = __ldg(a.K64.off + (gw >> 5) + 1);
  }
  for (int i = gw; i < a.m; i += nw) {
    const size_t idx = (size_t)i * BP + H * lane;
    const int o = o_next, w = (e_next - o_next) >> 5;
    if (i + nw < a.m) {
      o_next = __ldg(a.K64.off + ((i + nw) >> 5));
      e_next = __ldg(a.K64.off + ((i + nw) >> 5) + 1);
    }
    float yo[H], yb[H], ya[H];
    double yb64[H], qr[H], kanc[H], d0[H], d1[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      yo[h] = yb[h] = ya[h] = 0.f;
      yb64[h] = qr[h] = kanc[h] = 0.0;
    }
    if (some) {
      load_par<H>(a.y, par, idx, yo);
      load_inst<H>(a.ybar, idx, yb);
      load_inst<H>(a.ya, idx, ya);
      load_inst<H>(a.ybar64, idx, yb64);
      load_inst<H>(a.qh, idx, qr);
      if (!init) load_inst<H>(a.Kxa, idx, kanc);
    }
    const double qo = a.q_obj[i], idr = a.iDr[i], dr = a.Dr[i];
    kb_dots<BP, 4>(a.K64, o, w, i, lane, a.x, par, a.xbar64, some, d0, d1);
    const bool ineq = i >= a.m_eq;
    const double idr2 = idr * idr;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      d1[h] = has_avg[h] ? d1[h] * iw[h] : d0[h];
      if (init) kanc[h] = d0[h];
    }
    store_inst<H, double>(a.Kzc, idx, d0, on);
    store_inst<H, double>(a.Kza, idx, d1, on);
    if (init) store_inst<H, double>(a.Kxa, idx, d0, on);
    bool live = !finite_bits(qo);  // seen in q y alone (as in the single-instance check)
#pragma unroll
    for (int h = 0; h < H; ++h) {
      double r0 = on[h] ? qr[h] - d0[h] : 0.0, r1 = on[h] ? qr[h] - d1[h] : 0.0;
      double v0 = on[h] ? d0[h] - kanc[h] : 0.0, v1 = on[h] ? d1[h] - kanc[h] : 0.0;
      if (ineq) {
        r0 = pos_part(r0);
        r1 = pos_part(r1);
        v0 = neg_part(v0);
        v1 = neg_part(v1);
      }
      if (__any_sync(0xffffffffu, non_zero(r0) || non_zero(r1))) {
        const double q0 = r0 * r0, q1 = r1 * r1;
        acc[h][0] += q0;
        acc[h][1] += q0 * idr2;
        acc[h][kRowS + 0] += q1;
        acc[h][kRowS + 1] += q1 * idr2;
      }
      if (__any_sync(0xffffffffu, non_zero(v0) || non_zero(v1))) {
        acc[h][4] += (v0 * v0) * idr2;
        acc[h][kRowS + 4] += (v1 * v1) * idr2;
      }
      live = live || (on[h] && (non_zero(yo[h]) || non_zero(yb[h]) || non_zero(yb64[h]) || non_zero(ya[h])));
    }
    if (!__any_sync(0xffffffffu, live)) continue;
    double ybs[H];
    float zero[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      if (pw[h] != 0.f) yb[h] = yb[h] + pw[h] * yo[h];
      ybs[h] = to_f64(yb[h]) + yb64[h];
      zero[h] = 0.f;
    }
    store_inst<H, double>(a.ybar64, idx, ybs, on);
    store_inst<H, float>(a.ybar, idx, zero, on);
    const double dr2 = dr * dr;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const double y0 = on[h] ? to_f64(yo[h]) : 0.0, yan = on[h] ? to_f64(ya[h]) : 0.0;
      const double y1 = on[h] ? (has_avg[h] ? ybs[h] * iw[h] : y0) : 0.0;
      const double dd0 = y0 - yan, dd1 = y1 - yan, s0 = dd0 * dd0, s1 = dd1 * dd1;
      acc[h][2] += qo * y0;
      acc[h][3] += s0;
      acc[h][6] += qo * dd0;
      acc[h][kRowS + 2] += qo * y1;
      acc[h][kRowS + 3] += s1;
      acc[h][kRowS + 6] += qo * dd1;
      const bool n0 = ineq && is_neg(dd0), n1 = ineq && is_neg(dd1);
      if (__any_sync(0xffffffffu, n0 || n1)) {
        acc[h][5] += (n0 ? s0 : 0.0) * dr2;
        acc[h][kRowS + 5] += (n1 ? s1 : 0.0) * dr2;
      }
    }
  }
#pragma unroll
  for (int h = 0; h < H; ++h) {  // the unscaled LP's residual
    acc[h][1] *= idp2[h];
    acc[h][kRowS + 1] *= idp2[h];
  }
  __shared__ double smem[kKktWarps * BP * 2 * kRowS];
  put_inst<BP, 2 * kRowS>(acc, smem, H * lane, 1);
  sum_inst<BP, 2 * kRowS, kKktWarps>(smem, preg(a.part, 1));
}

template <int BP>
__global__ void __launch_bounds__(kKktWarps * 32) kb_kkt_col(BArgs<BP> a, int init) {
  BGlobal* g = a.g;
  if (g->all_done) return;
  constexpr int H = BP / 32;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double acc[H][2 * kColS], iw[H], idd[H];
  int par[H];
  bool on[H], has_avg[H];
  bool some = false;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const BInst& I = a.inst[H * lane + h];
    has_avg[h] = I.wsum > 0.0;
    iw[h] = has_avg[h] ? 1.0 / I.wsum : 0.0;
    idd[h] = 1.0 / I.dd;
    par[h] = I.par;
    on[h] = I.act;
    some = some || on[h];
#pragma unroll
    for (int k = 0; k < 2 * kColS; ++k) acc[h][k] = 0.0;
  }
  int o_next = 0, e_next = 0;  // the next row's slice
  if (gw < a.n) {
    o_next = __ldg(a.KT64.off + (gw >> 5));
    e_next = __ldg(a.KT64.off + (gw >> 5) + 1);
  }
  for (int j = gw; j < a.n; j += nw) {
    const size_t idx = (size_t)j * BP + H * lane;
    const int o = o_next, w = (e_next - o_next) >> 5;
    if (j + nw < a.n) {
      o_next = __ldg(a.KT64.off + ((j + nw) >> 5));
      e_next = __ldg(a.KT64.off + ((j + nw) >> 5) + 1);
    }
    float x0t[H], xat[H];
    double xs[H], lo[H], up[H], cr[H], kanc[H], e0[H], e1[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      x0t[h] = xat[h] = 0.f;
      xs[h] = lo[h] = up[h] = cr[h] = kanc[h] = 0.0;
    }
    if (some) {
      load_par<H>(a.x, par, idx, x0t);
      load_inst<H>(a.xa, idx, xat);
      load_inst<H>(a.xbar64, idx, xs);
      load_inst<H>(a.lo, idx, lo);
      load_inst<H>(a.uo, idx, up);
      load_inst<H>(a.ch, idx, cr);
      if (!init) load_inst<H>(a.KTya, idx, kanc);
    }
    const double co = a.c_obj[j], idc = a.iDc[j], dc = a.Dc[j];
    // kb_kkt_row has flushed the y window into ybar64
    kb_dots<BP, 2>(a.KT64, o, w, j, lane, a.y, par, a.ybar64, some, e0, e1);
    const double idc2 = idc * idc, dc2 = dc * dc;
    const bool cost = non_zero(co);
#pragma unroll
    for (int h = 0; h < H; ++h) {
      e1[h] = has_avg[h] ? e1[h] * iw[h] : e0[h];
      if (init) kanc[h] = e0[h];
    }
    store_inst<H, double>(a.KTzc, idx, e0, on);
    store_inst<H, double>(a.KTza, idx, e1, on);
    if (init) store_inst<H, double>(a.KTya, idx, e0, on);
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const bool lf = finite_bits(lo[h]), uf = finite_bits(up[h]);
      const double x0 = on[h] ? to_f64(x0t[h]) : 0.0, xan = on[h] ? to_f64(xat[h]) : 0.0;
      const double x1 = on[h] ? (has_avg[h] ? xs[h] * iw[h] : x0) : 0.0;
#pragma unroll
      for (int cnd = 0; cnd < 2; ++cnd) {
        double* ac = acc[h] + cnd * kColS;
        const double kty = cnd ? e1[h] : e0[h];
        const double xv = cnd ? x1 : x0;
        const double lam = on[h] ? cr[h] - kty : 0.0;
        const bool ln = is_neg(lam), la = ln ? uf : lf;
        const double rd = la ? 0.0 : lam;
        ac[3] += (la ? (ln ? up[h] : lo[h]) : 0.0) * lam;
        const double lr = on[h] ? kanc[h] - kty : 0.0;
        const bool rn = is_neg(lr), ra = rn ? uf : lf;
        const double vl = ra ? 0.0 : lr;
        ac[6] += (ra ? (rn ? up[h] : lo[h]) : 0.0) * lr;
        if (__any_sync(0xffffffffu, non_zero(rd))) {
          const double q = rd * rd;
          ac[0] += q;
          ac[1] += q * idc2;
        }
        if (__any_sync(0xffffffffu, non_zero(vl))) ac[5] += (vl * vl) * idc2;
        if (cost) ac[2] += co * xv;
        const double dx = xv - xan;
        if (__any_sync(0xffffffffu, non_zero(dx))) {
          const double q = dx * dx;
          ac[4] += q;
          if (cost) ac[8] += co * dx;
          const bool bad = non_zero(dx) && (is_neg(dx) ? lf : uf);
          if (__any_sync(0xffffffffu, bad)) ac[7] += (bad ? q : 0.0) * dc2;
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int c = 0; c < 2; ++c) {  // the unscaled LP's measures
      acc[h][c * kColS + 1] *= idd[h] * idd[h];
      acc[h][c * kColS + 3] *= idd[h];
    }
  __shared__ double smem[kKktWarps * BP * 2 * kColS];
  put_inst<BP, 2 * kColS>(acc, smem, H * lane, 1);
  sum_inst<BP, 2 * kColS, kKktWarps>(smem, preg(a.part, 2));
}

// Fixed-order totals of the check's partials, one block per instance (one block
// for all of them took 0.7 to 1.2 ms, these 12 to 29 us): tot[b][0..14) of the rows,
// tot[b][14..32) of the columns.
constexpr int kCheckS = 2 * (kRowS + kColS);
template <int BP>
__global__ void __launch_bounds__(kBlock) kb_check_sums(const BGlobal* g, const double* row, int nb_row,
                                                        const double* col, int nb_col, double* tot) {
  if (g->all_done) return;
  const int b = blockIdx.x;
  __shared__ double smem[kWarps * 2 * kColS];
  double r[2 * kRowS], c[2 * kColS];
#pragma unroll
  for (int k = 0; k < 2 * kRowS; ++k) r[k] = 0.0;
#pragma unroll
  for (int k = 0; k < 2 * kColS; ++k) c[k] = 0.0;
  for (int t = threadIdx.x; t < nb_row; t += kBlock)
#pragma unroll
    for (int k = 0; k < 2 * kRowS; ++k) r[k] += __ldcg(row + ((size_t)t * BP + b) * 2 * kRowS + k);
  block_sum<2 * kRowS>(r, smem);
  for (int t = threadIdx.x; t < nb_col; t += kBlock)
#pragma unroll
    for (int k = 0; k < 2 * kColS; ++k) c[k] += __ldcg(col + ((size_t)t * BP + b) * 2 * kColS + k);
  block_sum<2 * kColS>(c, smem);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 2 * kRowS; ++k) tot[b * kCheckS + k] = r[k];
#pragma unroll
    for (int k = 0; k < 2 * kColS; ++k) tot[b * kCheckS + 2 * kRowS + k] = c[k];
  }
}

// One thread per instance: termination, restart, primal weight, end of a
// refinement round; the while condition clears when every instance is done.
template <int BP>
__global__ void __launch_bounds__(64) kb_control(BArgs<BP> a, const double* tot, int init) {
  BGlobal* g = a.g;
  __shared__ int s_running;
  if (threadIdx.x == 0) s_running = 0;
  __syncthreads();
  const int b = threadIdx.x;
  if (b < BP && !g->all_done) {
    double rs[2 * kRowS], cs[2 * kColS];
#pragma unroll
    for (int k = 0; k < 2 * kRowS; ++k) rs[k] = tot[b * kCheckS + k];
#pragma unroll
    for (int k = 0; k < 2 * kColS; ++k) cs[k] = tot[b * kCheckS + 2 * kRowS + k];
    BInst& I = a.inst[b];
    I.restart_now = 0;
    I.refine = 0;
    I.finalize = 0;
    if (I.act) {
      const double omega = I.omega, idp = 1.0 / I.dp, idd = 1.0 / I.dd;
      double rel[2], relp[2], reld[2], relg[2], P[2], D[2], kw[2], rp2s[2], rd2s[2], gh[2], dxa[2],
          dya[2];
      bool finite = true;
      for (int c = 0; c < 2; ++c) {
        rp2s[c] = rs[c * kRowS + 0];
        const double rp2u = rs[c * kRowS + 1], qy = rs[c * kRowS + 2];
        dya[c] = rs[c * kRowS + 3];
        rd2s[c] = cs[c * kColS + 0];
        const double rd2u = cs[c * kColS + 1], cx = cs[c * kColS + 2], bnd = cs[c * kColS + 3];
        dxa[c] = cs[c * kColS + 4];
        for (int k = 0; k < kRowS; ++k) finite = finite && isfinite(rs[c * kRowS + k]);
        for (int k = 0; k < kColS; ++k) finite = finite && isfinite(cs[c * kColS + k]);
        P[c] = cx * idp + I.const_p;
        D[c] = qy * idd + I.const_d + bnd;
        relp[c] = sqrt(rp2u) / (1.0 + g->qnorm);
        reld[c] = sqrt(rd2u) / (1.0 + g->cnorm);
        relg[c] = fabs(P[c] - D[c]) / (1.0 + fabs(P[c]) + fabs(D[c]));
        rel[c] = fmax(relp[c], fmax(reld[c], relg[c]));
        // the correction LP's gap is Delta^2 times the LP's, its residuals
        // Delta times: weighting the gap by 1/Delta keeps the restart test
        // what it is for the same point in round 0 (up to a common factor)
        gh[c] = (P[c] - D[c]) * I.dp;
        kw[c] = sqrt(omega * rp2s[c] + rd2s[c] / omega + gh[c] * gh[c]);
      }
      const bool has_avg = I.wsum > 0.0;
      if (init) {
        I.kkt0 = I.kkt_prev = kw[0];
        I.round_target = fmax(g->tol, g->red * rel[0]);
        I.round_rel0 = rel[0];
      } else {
        I.checks += 1;
        I.round_checks += 1;
        I.pending_w = 0.0;
        const int best = (has_avg && rel[1] < rel[0]) ? 1 : 0;
        const uint64_t now = globaltimer_ns();
        const double thr[3] = {1e-4, 1e-6, 1e-8};
        for (int t = 0; t < 3; ++t)
          if (I.t_tol[t] < 0.0 && rel[best] <= thr[t]) {
            I.t_tol[t] = (double)(now - g->t_start) * 1e-9;
            I.k_tol[t] = I.k_total;
          }
        I.rel_p = relp[best];
        I.rel_d = reld[best];
        I.rel_gap = relg[best];
        I.rel_kkt = rel[best];
        I.pobj = P[best];
        I.dobj = D[best];
        int stop = 0;
        if (!finite) {
          stop = PDHG_STATUS_NUMERIC;
        } else if (rel[best] <= g->tol) {
          stop = PDHG_STATUS_OPTIMAL;
        } else if (I.k_total >= g->max_k) {
          stop = PDHG_STATUS_ITER_LIMIT;
        } else if (now - g->t_start >= g->t_limit_ns) {
          stop = PDHG_STATUS_TIME_LIMIT;
        } else if (a.cancel && *a.cancel) {
          stop = PDHG_STATUS_CANCELLED;
        } else if (g->infeas_eps > 0.0) {
          for (int c = 0; c < 2 && !stop; ++c) {
            const double d_obj = rs[c * kRowS + 6] + cs[c * kColS + 6];
            const double d_viol = sqrt(rs[c * kRowS + 5] + cs[c * kColS + 5]);
            const double p_obj = cs[c * kColS + 8];
            const double p_viol = sqrt(rs[c * kRowS + 4] + cs[c * kColS + 7]);
            if (d_obj > 0.0 && d_viol <= g->infeas_eps * d_obj)
              stop = PDHG_STATUS_PRIMAL_INFEASIBLE;
            else if (p_obj < 0.0 && p_viol <= g->infeas_eps * (-p_obj))
              stop = PDHG_STATUS_DUAL_INFEASIBLE;
          }
        }
        if (stop) {
          I.done = 1;
          I.act = 0;
          I.status = stop;
          I.finalize = 1;
          I.cand_avg = best;
        } else {
          int to_avg = (has_avg && kw[1] < kw[0]) ? 1 : 0;
          const double kc = kw[to_avg];
          int restart = (kc <= g->beta_suff * I.kkt0) ||
                        (kc <= g->beta_nec * I.kkt0 && kc > I.kkt_prev) ||
                        ((double)I.since_restart >= g->beta_art * (double)I.k_total);
          I.kkt_prev = kc;
          if (restart) {
            // distances in round-0 units (the correction coordinates are Delta
            // times larger): the "too small to update omega" test stays fixed
            const double Dx = sqrt(dxa[to_avg]) / I.dp, Dy = sqrt(dya[to_avg]) / I.dd;
            double om = omega;
            if (Dx > 1e-10 && Dy > 1e-10)
              om = exp(g->omega_smooth * log(Dy / Dx) + (1.0 - g->omega_smooth) * log(omega));
            I.omega = om;
            const double k0 = sqrt(om * rp2s[to_avg] + rd2s[to_avg] / om + gh[to_avg] * gh[to_avg]);
            I.restarts += 1;
            I.kkt0 = k0;
            I.kkt_prev = k0;
            I.avg_div = I.wsum;
            I.wsum = 0.0;
            I.since_restart = 0;
            I.restart_now = 1;
            I.restart_to_avg = to_avg;
          } else if (rel[0] <= I.round_target ||
                     (g->fold_every > 0 && I.round_checks >= g->fold_every &&
                      rel[0] <= I.round_rel0)) {
            // refinement fold (as pdhg_solve): the current iterate joins x*, y*
            // and kb_apply re-expresses the iteration state in the new
            // coordinates; step size, primal weight, averages and restart
            // window carry over
            const double relb = fmax(rel[0], 1e-300);
            const double scale = fmin(1.0 / relb, 1e12);
            const double f = scale / I.dp;  // Delta_P = Delta_D here
            I.refine = 1;
            I.round_checks = 0;
            I.cand_avg = 0;
            I.next_scale = f;
            I.round_target = fmax(g->tol, g->red * relb);
            I.round_rel0 = relb;
            I.rounds += 1;
            // KKT_w with the gap weighted back to round-0 units scales by f
            I.kkt0 *= f;
            I.kkt_prev *= f;
            I.rel_p = relp[0];
            I.rel_d = reld[0];
            I.rel_gap = relg[0];
            I.rel_kkt = rel[0];
            I.pobj = P[0];
            I.dobj = D[0];
          }
        }
      }
    }
    if (I.act) {
      I.eta = fmin(I.eta, fp32_step_cap(I.omega));  // FP32 range (see fp32_step_cap)
      set_steps(I);
    }
    if (!I.done) atomicAdd(&s_running, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0 && !init) {
    const int all = (s_running == 0) || g->all_done;
    g->all_done = all;
    if (a.in_graph) cudaGraphSetConditional(a.cond, all ? 0u : 1u);
  }
}

// Elementwise, thread (r, b) = (threadIdx.x / BP, threadIdx.x % BP): restart
// moves, refinement steps and final accumulation per instance, plus the new
// pending primal step; per-instance sums of ||dx||^2, c~^T x*, q~^T y*.
template <int BP>
__global__ void __launch_bounds__(kApplyRows * BP) kb_apply(BArgs<BP> a) {
  BGlobal* g = a.g;
  const int b = threadIdx.x % BP, r0 = threadIdx.x / BP;
  const BInst& I = a.inst[b];
  const int restart = I.restart_now, refine = I.refine, fin = I.finalize;
  const int any = restart || refine || fin;
  const int p = I.par;
  const double f = I.next_scale;
  const double idp = 1.0 / I.dp, idd = 1.0 / I.dd;
  const double iw = I.wsum > 0.0 ? 1.0 / I.wsum : 0.0;
  const double wsum = I.wsum;
  const double div = I.avg_div;
  const int cand_avg = I.cand_avg;
  const float tau = I.tau;
  double sdx = 0.0, scp = 0.0, scd = 0.0;
  if (any) {
    // rows
    for (int i = blockIdx.x * kApplyRows + r0; i < a.m; i += gridDim.x * kApplyRows) {
      const size_t idx = (size_t)i * BP + b;
      if (restart) {
        if (I.restart_to_avg) {
          a.y[p][idx] = (float)(((double)a.ybar[idx] + a.ybar64[idx]) / div);
          a.Kx[p][idx] = (float)a.Kza[idx];
        }
        a.ya[idx] = a.y[p][idx];
        a.ybar[idx] = 0.f;
        a.ybar64[idx] = 0.0;
        a.Kxa[idx] = I.restart_to_avg ? a.Kza[idx] : a.Kzc[idx];
      } else {
        const double yh = cand_avg ? ((double)a.ybar[idx] + a.ybar64[idx]) * iw : (double)a.y[p][idx];
        const double kz = cand_avg ? a.Kza[idx] : a.Kzc[idx];
        const double ys = a.yst[idx] + yh * idd;
        a.yst[idx] = ys;
        if (refine) {
          // fold at the current iterate (cand_avg = 0): new correction data,
          // then the state in the new coordinates v' = f (v - y^c)
          const double qn = f * (a.qh[idx] - kz);
          a.qh[idx] = qn;
          a.qf[idx] = (float)qn;
          if (i >= a.m_eq) {
            const double yl = f * (a.ylh[idx] - yh);
            a.ylh[idx] = yl;
            a.ylf[idx] = (float)yl;
          }
          a.ya[idx] = (float)(f * ((double)a.ya[idx] - yh));
          a.ybar64[idx] = f * ((double)a.ybar[idx] + a.ybar64[idx] - wsum * yh);
          a.ybar[idx] = 0.f;
          a.y[p][idx] = 0.f;
          a.Kx[p][idx] = 0.f;
          a.Kxa[idx] = f * (a.Kxa[idx] - kz);
        }
        scd += a.q_obj[i] * ys;
      }
    }
    // columns
    for (int j = blockIdx.x * kApplyRows + r0; j < a.n; j += gridDim.x * kApplyRows) {
      const size_t idx = (size_t)j * BP + b;
      if (restart) {
        a.KTya[idx] = I.restart_to_avg ? a.KTza[idx] : a.KTzc[idx];
        if (I.restart_to_avg) {
          a.x[p][idx] = (float)(((double)a.xbar[idx] + a.xbar64[idx]) / div);
          a.KTy[p][idx] = (float)a.KTza[idx];
        }
        const float x0 = a.x[p][idx];
        a.xa[idx] = x0;
        a.xbar[idx] = 0.f;
        a.xbar64[idx] = 0.0;
        float v = x0 - tau * (a.cf[idx] - a.KTy[p][idx]);
        v = fminf(fmaxf(v, a.lf[idx]), a.uf[idx]);
        a.x[1 - p][idx] = v;
        const double d = (double)(v - x0);
        sdx += d * d;
      } else {
        const double xh = cand_avg ? ((double)a.xbar[idx] + a.xbar64[idx]) * iw : (double)a.x[p][idx];
        const double kz = cand_avg ? a.KTza[idx] : a.KTzc[idx];
        const double xs = a.xst[idx] + xh * idp;
        a.xst[idx] = xs;
        if (refine) {
          const double cn = f * (a.ch[idx] - kz);
          // exact in FP64: the candidate may sit a rounding outside its bounds
          // (the FP32 iterate was projected onto FP32-rounded bounds, e.g. a
          // fixed variable); the new round corrects that, so no clamping here.
          // The round starts at x^ = y^ = 0 even if that is a rounding
          // outside [l^, u^]: the first projected step restores feasibility.
          const double ln = f * (a.lh[idx] - xh);
          const double un = f * (a.uh[idx] - xh);
          a.ch[idx] = cn;
          a.lh[idx] = ln;
          a.uh[idx] = un;
          a.cf[idx] = (float)cn;
          a.lf[idx] = (float)ln;
          a.uf[idx] = (float)un;
          a.xa[idx] = (float)(f * ((double)a.xa[idx] - xh));
          a.xbar64[idx] = f * ((double)a.xbar[idx] + a.xbar64[idx] - wsum * xh);
          a.xbar[idx] = 0.f;
          a.KTya[idx] = f * (a.KTya[idx] - kz);
          a.KTy[p][idx] = 0.f;
          a.x[p][idx] = 0.f;
          // the pending primal step from the new data (the same step in exact
          // arithmetic)
          float v = fminf(fmaxf(-tau * a.cf[idx], a.lf[idx]), a.uf[idx]);
          a.x[1 - p][idx] = v;
          sdx += (double)v * (double)v;
        }
        scp += a.c_obj[j] * xs;
      }
    }
  }
  __shared__ double smem[kApplyRows * BP * 3];
  smem[(r0 * BP + b) * 3 + 0] = sdx;
  smem[(r0 * BP + b) * 3 + 1] = scp;
  smem[(r0 * BP + b) * 3 + 2] = scd;
  __syncthreads();
  if (r0 == 0) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int rr = 0; rr < kApplyRows; ++rr) {
      s0 += smem[(rr * BP + b) * 3 + 0];
      s1 += smem[(rr * BP + b) * 3 + 1];
      s2 += smem[(rr * BP + b) * 3 + 2];
    }
    double* out = a.part + ((size_t)blockIdx.x * BP + b) * 3;
    out[0] = s0;
    out[1] = s1;
    out[2] = s2;
  }
  double tot[3];
  if (grid_inst_sum<BP, 3>(a.part, a.tier, smem, tot)) {
    if (threadIdx.x < BP) {
      BInst& J = a.inst[threadIdx.x];
      if (J.restart_now || J.refine || J.finalize) {
        const double s0 = tot[0], s1 = tot[1], s2 = tot[2];
        if (J.restart_now) {
          J.dx2 = s0;
        } else {
          J.const_p = s1;
          J.const_d = s2;
        }
        if (J.refine) {
          // the same iteration in the new coordinates: only the scale and the
          // pending step's length change
          J.dx2 = s0;
          J.dp *= J.next_scale;
          J.dd = J.dp;
        }
      }
      J.restart_now = 0;
      J.refine = 0;
      J.finalize = 0;
    }
  }
}

// ---------------------------------------------------------------- setup kernels

__global__ void kb_invert(const int32_t* __restrict__ perm, int32_t* __restrict__ inv, int n) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) inv[perm[t]] = t;
}

// Round-0 data of every instance.  The callers' bounds lie instance after instance
// in the original order, the solver's vectors column after column in the internal
// one: tiles of kTile original columns go through shared memory, so that both
// sides are read and written in whole sectors.  A bound equal to the shared LP's
// takes that one's scaled value (a division saved in all but the fixed columns).
// The first pending primal step x' = proj(x - tau c) (K^T y = 0) and its
// ||dx||^2 per block are formed on the way.
constexpr int kTile = 32;
template <int BP>
__global__ void __launch_bounds__(kBThreads) kb_setup_cols(
    BArgs<BP> a, const double* __restrict__ lb, const double* __restrict__ ub, const double* __restrict__ l0,
    const double* __restrict__ u0, const int32_t* __restrict__ inv_col, const double* __restrict__ Dc,
    const double* __restrict__ c_s, const double* __restrict__ l_s, const double* __restrict__ u_s) {
  __shared__ double tl[kTile][BP + 1], tu[kTile][BP + 1];
  const int b = threadIdx.x % BP;
  const float tau = a.inst[b].tau;
  double dx2 = 0.0;
  for (int64_t o0 = (int64_t)blockIdx.x * kTile; o0 < a.n; o0 += (int64_t)gridDim.x * kTile) {
    for (int t = threadIdx.x; t < kTile * BP; t += kBThreads) {
      const int oo = t % kTile, bb = t / kTile;
      if (o0 + oo < a.n && bb < a.B) {
        tl[oo][bb] = lb[(size_t)bb * a.n + o0 + oo];
        tu[oo][bb] = ub[(size_t)bb * a.n + o0 + oo];
      }
    }
    __syncthreads();
    for (int oo = threadIdx.x / BP; oo < kTile && o0 + oo < a.n; oo += kBThreads / BP) {
      const int64_t o = o0 + oo;
      const int j = inv_col[o];
      double lo = l_s[j], up = u_s[j];
      if (b < a.B) {
        const double l = tl[oo][b], u = tu[oo][b];
        if (__double_as_longlong(l) != __double_as_longlong(l0[o])) lo = l / Dc[j];
        if (__double_as_longlong(u) != __double_as_longlong(u0[o])) up = u / Dc[j];
      }
      const size_t t = (size_t)j * BP + b;
      const double c = c_s[j];
      const float cf = (float)c, lf = (float)lo, uf = (float)up;
      a.lo[t] = lo;
      a.uo[t] = up;
      a.lh[t] = lo;
      a.uh[t] = up;
      a.lf[t] = lf;
      a.uf[t] = uf;
      a.ch[t] = c;
      a.cf[t] = cf;
      a.xst[t] = 0.0;
      const float x0 = fminf(fmaxf(0.f, lf), uf);
      const float x1 = fminf(fmaxf(x0 - tau * cf, lf), uf);
      a.x[0][t] = x0;
      a.x[1][t] = x1;
      a.xa[t] = x0;
      a.xbar[t] = 0.f;
      a.xbar64[t] = 0.0;
      a.KTy[0][t] = a.KTy[1][t] = 0.f;
      if (__float_as_uint(x1) != __float_as_uint(x0)) {
        const double d = to_f64(x1) - to_f64(x0);
        dx2 += d * d;
      }
    }
    __syncthreads();
  }
  __shared__ double sm[kBThreads];
  sm[threadIdx.x] = dx2;
  __syncthreads();
  if (threadIdx.x < BP) {
    for (int k = 1; k < kBThreads / BP; ++k) dx2 += sm[threadIdx.x + k * BP];
    a.part[(size_t)blockIdx.x * BP + threadIdx.x] = dx2;
  }
}

template <int BP>
__global__ void kb_setup_rows(BArgs<BP> a, const double* __restrict__ q_s) {
  const int64_t N = (int64_t)a.m * BP;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / BP);
    const double q = q_s[i], yl = (i < a.m_eq) ? -INFINITY : 0.0;
    a.qh[t] = q;
    a.qf[t] = (float)q;
    a.ylh[t] = yl;
    a.ylf[t] = (float)yl;
    a.yst[t] = 0.0;
    a.y[0][t] = a.y[1][t] = 0.f;
    a.ya[t] = a.ybar[t] = 0.f;
    a.ybar64[t] = 0.0;
  }
}

// ||x' - x||^2 of each instance from the blocks of kb_setup_cols.
template <int BP>
__global__ void __launch_bounds__(kBlock) kb_first_dx2(BArgs<BP> a, int nb) {
  __shared__ double sm[kWarps];
  double v[1] = {0.0};
  for (int t = threadIdx.x; t < nb; t += kBlock) v[0] += __ldcg(a.part + (size_t)t * BP + blockIdx.x);
  block_sum<1>(v, sm);
  if (threadIdx.x == 0) a.inst[blockIdx.x].dx2 = v[0];
}

// K x for every slot (initial point of round 0).
template <int BP>
__global__ void __launch_bounds__(kBThreads) kb_spmm(BArgs<BP> a) {
  constexpr int H = BP / 32;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBThreads + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBThreads) >> 5;
  for (int i = gw; i < a.m; i += nw) {
    const int s = i >> 5, r = i & 31;
    const int o0 = __ldg(a.K.off + s) + r;
    const int w = (__ldg(a.K.off + s + 1) - __ldg(a.K.off + s)) >> 5;
    float acc[H];
#pragma unroll
    for (int h = 0; h < H; ++h) acc[h] = 0.f;
    for (int k = 0; k < w; ++k) {
      const int c = __ldg(a.K.col + o0 + k * kSlice);
      const float v = __ldg(a.K.val + o0 + k * kSlice);
#pragma unroll
      for (int h = 0; h < H; ++h) acc[h] += v * __ldg(a.x[0] + (size_t)c * BP + lane + 32 * h);
    }
#pragma unroll
    for (int h = 0; h < H; ++h) a.Kx[0][(size_t)i * BP + lane + 32 * h] = acc[h];
  }
}

// out[b][o] = D v[b] of internal element inv[o], through tiles as kb_setup_cols.
template <int BP>
__global__ void __launch_bounds__(kBThreads) kb_output(const double* __restrict__ v, const double* __restrict__ D,
                                                       const int32_t* __restrict__ inv, int64_t len, int B,
                                                       double* __restrict__ out) {
  __shared__ double tile[kTile][BP + 1];
  const int b = threadIdx.x % BP;
  for (int64_t o0 = (int64_t)blockIdx.x * kTile; o0 < len; o0 += (int64_t)gridDim.x * kTile) {
    for (int oo = threadIdx.x / BP; oo < kTile && o0 + oo < len; oo += kBThreads / BP) {
      const int j = inv[o0 + oo];
      tile[oo][b] = D[j] * v[(size_t)j * BP + b];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kTile * B; t += kBThreads) {
      const int oo = t % kTile, bb = t / kTile;
      if (o0 + oo < len) out[(size_t)bb * len + o0 + oo] = tile[oo][bb];
    }
    __syncthreads();
  }
}

__global__ void kb_init_state(BInst* inst, BGlobal* g, uint32_t* tier, int B, int BP, const double* scalars,
                              BGlobal gin) {
  const int b = threadIdx.x;
  for (int t = b; t < kTierCount; t += blockDim.x) tier[t] = 0;
  if (b == 0) {
    *g = gin;
    g->t_start = globaltimer_ns();
    g->qnorm = scalars[2];
    g->cnorm = scalars[3];
    g->all_done = 0;
  }
  if (b < BP) {
    BInst I;
    memset(&I, 0, sizeof(I));
    I.eta = scalars[0];
    I.omega = scalars[1];
    set_steps(I);
    I.act = b < B;
    I.done = b >= B;
    I.dp = I.dd = 1.0;
    I.next_scale = 1.0;
    I.rel_kkt = INFINITY;
    for (int t = 0; t < 3; ++t) {
      I.t_tol[t] = -1.0;
      I.k_tol[t] = -1;
    }
    inst[b] = I;
  }
}

struct Batched {
  int BP = 0, cap = 0;
  std::vector<void*> allocs;
  void* args = nullptr;  // BArgs<BP> host copy
  BInst* inst = nullptr;
  BInst* inst_host = nullptr;
  int32_t* done_host = nullptr;  // pinned copy of g->all_done (host-loop mode)
  BGlobal* g = nullptr;
  double* part = nullptr;
  uint32_t* tier = nullptr;
  int32_t *inv_row = nullptr, *inv_col = nullptr;  // original -> internal
  cudaGraphExec_t exec = nullptr;
  cudaGraph_t graph = nullptr;
  int grid_rows = 0, grid_cols = 0, grid_kr = 0, grid_kc = 0, grid_apply = 0;
  int rw_dual = 4, rw_adj = 4;  // rows (columns) per warp of the sweeps
  bool tuned = false, inverted = false;
};

template <int BP>
void launch_sweep_dual(const BArgs<BP>& a, int rw, int grid, cudaStream_t s) {
  if (rw == 1)
    kb_dual<BP, 1><<<grid, kBThreads, 0, s>>>(a);
  else if (rw == 2)
    kb_dual<BP, 2><<<grid, kBThreads, 0, s>>>(a);
  else
    kb_dual<BP, 4><<<grid, kBThreads, 0, s>>>(a);
}

template <int BP>
void launch_sweep_adjoint(const BArgs<BP>& a, int rw, int grid, cudaStream_t s) {
  if (rw == 1)
    kb_adjoint<BP, 1><<<grid, kBThreads, 0, s>>>(a);
  else if (rw == 2)
    kb_adjoint<BP, 2><<<grid, kBThreads, 0, s>>>(a);
  else
    kb_adjoint<BP, 4><<<grid, kBThreads, 0, s>>>(a);
}

template <class P>
cudaError_t balloc(Batched* bt, P** p, size_t count) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, count * sizeof(P) + 16);
  if (e == cudaSuccess) {
    bt->allocs.push_back(q);
    *p = (P*)q;
  }
  return e;
}

template <int BP>
int setup_batched(Workspace* w, Batched* bt, BArgs<BP>* out) {
  BArgs<BP> a{};
  const size_t n = (size_t)w->n * BP, m = (size_t)w->m * BP;
  cudaError_t e = cudaSuccess;
  auto F = [&](float** p, size_t c) { if (e == cudaSuccess) e = balloc(bt, p, c); };
  auto D = [&](double** p, size_t c) { if (e == cudaSuccess) e = balloc(bt, p, c); };
  for (int i = 0; i < 2; ++i) {
    F(&a.x[i], n);
    F(&a.y[i], m);
    F(&a.Kx[i], m);
    F(&a.KTy[i], n);
  }
  F(&a.xbar, n); F(&a.ybar, m); F(&a.xa, n); F(&a.ya, m);
  F(&a.cf, n); F(&a.lf, n); F(&a.uf, n); F(&a.qf, m); F(&a.ylf, m);
  D(&a.xst, n); D(&a.yst, m); D(&a.ch, n); D(&a.lh, n); D(&a.uh, n); D(&a.qh, m); D(&a.ylh, m);
  D(&a.lo, n); D(&a.uo, n); D(&a.Kzc, m); D(&a.Kza, m); D(&a.KTzc, n); D(&a.KTza, n);
  D(&a.Kxa, m); D(&a.KTya, n); D(&a.xbar64, n); D(&a.ybar64, m);
  if (e == cudaSuccess) e = balloc(bt, &bt->inst, BP);
  if (e == cudaSuccess) e = balloc(bt, &bt->g, 1);
  if (e == cudaSuccess) e = balloc(bt, &bt->part, (size_t)3 * 8192 * 64 * 20);
  if (e == cudaSuccess) e = balloc(bt, &bt->tier, kTierCount);
  if (e == cudaSuccess) e = balloc(bt, &bt->inv_row, w->m);
  if (e == cudaSuccess) e = balloc(bt, &bt->inv_col, w->n);
  if (e != cudaSuccess) {
    g_err = std::string("batched allocation: ") + cudaGetErrorString(e);
    return PDHG_ERR_NOMEM;
  }
  if (cudaMallocHost(&bt->inst_host, sizeof(BInst) * BP) != cudaSuccess ||
      cudaMallocHost(&bt->done_host, sizeof(int32_t)) != cudaSuccess) {
    g_err = "batched pinned allocation failed";
    return PDHG_ERR_NOMEM;
  }
  a.K = w->K.v32();
  a.KT = w->KT.v32();
  a.K64 = w->K.v64();
  a.KT64 = w->KT.v64();
  a.n = (int32_t)w->n;
  a.m = (int32_t)w->m;
  a.m_eq = (int32_t)w->m_eq;
  a.c_obj = w->c_s;
  a.q_obj = w->q_s;
  a.iDr = w->iDr;
  a.iDc = w->iDc;
  a.Dr = w->Dr;
  a.Dc = w->Dc;
  a.inst = bt->inst;
  a.g = bt->g;
  a.part = bt->part;
  a.tier = bt->tier;
  a.cancel = w->opts.cancel_flag;
  *out = a;
  const int sms = w->num_sms;
  // at least ~8 rows per warp, so the per-instance partials of small problems
  // stay few (their final sums sit on the critical path of every attempt)
  // the sweeps are grid-stride loops: one wave of resident blocks
  int occ_d = 0, occ_a = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_d, kb_dual<BP, 4>, kBThreads, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_a, kb_adjoint<BP, 4>, kBThreads, 0);
  occ_d = std::max(occ_d, 1);
  occ_a = std::max(occ_a, 1);
  bt->grid_rows = std::max(1, std::min(sms * occ_d, (int)((w->m + 8 * kBWarps - 1) / (8 * kBWarps))));
  bt->grid_cols = std::max(1, std::min(sms * occ_a, (int)((w->n + 8 * kBWarps - 1) / (8 * kBWarps))));
  bt->grid_kr = std::max(1, std::min(sms * 8, (int)((w->m + 8 * kKktWarps - 1) / (8 * kKktWarps))));
  bt->grid_kc = std::max(1, std::min(sms * 8, (int)((w->n + 8 * kKktWarps - 1) / (8 * kKktWarps))));
  bt->grid_apply = std::max(
      1, std::min(sms * 8, (int)((std::max(w->n, w->m) + 16 * kApplyRows - 1) / (16 * kApplyRows))));
  bt->grid_rows = std::min(bt->grid_rows, 8192);
  bt->grid_cols = std::min(bt->grid_cols, 8192);
  bt->grid_kr = std::min(bt->grid_kr, 8192);
  bt->grid_kc = std::min(bt->grid_kc, 8192);
  bt->grid_apply = std::min(bt->grid_apply, 8192);
  return PDHG_OK;
}

template <int BP>
void launch_body(const BArgs<BP>& a, Batched* bt, cudaStream_t s, int init) {
  if (!init) {
    for (int k = 0; k < kCheckEvery; ++k) {
      launch_sweep_dual<BP>(a, bt->rw_dual, bt->grid_rows, s);
      launch_sweep_adjoint<BP>(a, bt->rw_adj, bt->grid_cols, s);
    }
  }
  if (!init) kb_flush_x<BP><<<bt->grid_apply, 256, 0, s>>>(a);
  kb_kkt_row<BP><<<bt->grid_kr, kKktWarps * 32, 0, s>>>(a, init);
  kb_kkt_col<BP><<<bt->grid_kc, kKktWarps * 32, 0, s>>>(a, init);
  // the attempts' region of the partials is free here
  kb_check_sums<BP><<<BP, kBlock, 0, s>>>(a.g, preg(a.part, 1), bt->grid_kr, preg(a.part, 2), bt->grid_kc,
                                          a.part);
  kb_control<BP><<<1, 64, 0, s>>>(a, a.part, init);
  if (!init) kb_apply<BP><<<bt->grid_apply, kApplyRows * BP, 0, s>>>(a);
}

template <int BP>
int build_batched_graph(Workspace* w, Batched* bt, BArgs<BP> a) {
  if (bt->exec) return PDHG_OK;
  cudaGraph_t gph = nullptr;
  if (cudaGraphCreate(&gph, 0) != cudaSuccess) return PDHG_ERR_CUDA;
  cudaGraphConditionalHandle h;
  if (cudaGraphConditionalHandleCreate(&h, gph, 1, cudaGraphCondAssignDefault) != cudaSuccess)
    return PDHG_ERR_CUDA;
  alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)];
  std::memset(raw, 0, sizeof(raw));
  cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(raw);
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  if (cudaGraphAddNode(&node, gph, nullptr, nullptr, 0, &cp) != cudaSuccess) return PDHG_ERR_CUDA;
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  if (cudaStreamBeginCaptureToGraph(w->cap_stream, body, nullptr, nullptr, 0,
                                    cudaStreamCaptureModeThreadLocal) != cudaSuccess)
    return PDHG_ERR_CUDA;
  a.in_graph = 1;
  a.cond = (unsigned long long)h;
  launch_body<BP>(a, bt, w->cap_stream, 0);
  cudaGraph_t captured = nullptr;
  cudaError_t e = cudaStreamEndCapture(w->cap_stream, &captured);
  if (e != cudaSuccess) {
    g_err = std::string("batched graph capture: ") + cudaGetErrorString(e);
    return PDHG_ERR_CUDA;
  }
  e = cudaGraphInstantiate(&bt->exec, gph, 0);
  if (e != cudaSuccess) {
    g_err = std::string("batched graph instantiate: ") + cudaGetErrorString(e);
    return PDHG_ERR_CUDA;
  }
  bt->graph = gph;
  return PDHG_OK;
}

// Device state, round-0 data, first primal step and initial KKT_w of every
// instance.
template <int BP>
void batched_start(Workspace* w, Batched* bt, const BArgs<BP>& a, int B, const double* l_b,
                   const double* u_b, cudaStream_t s) {
  const pdhg_opts& o = w->opts;
  BGlobal gin{};
  gin.tol = o.tol;
  gin.red = o.ir_reduction;
  gin.beta_suff = o.beta_sufficient;
  gin.beta_nec = o.beta_necessary;
  gin.beta_art = o.beta_artificial;
  gin.omega_smooth = o.omega_smoothing;
  gin.red_exp = o.step_reduction_exp;
  gin.grow_exp = o.step_growth_exp;
  gin.max_k = o.max_iters;
  gin.t_limit_ns = (uint64_t)(o.time_limit_s * 1e9);
  gin.infeas_eps = o.infeas_tol > 0.0 ? std::max(o.infeas_tol, kFp32RayTol) : 0.0;  // FP32 iterates
  gin.fold_every = o.ir_fold_checks;
  gin.n_real = B;
  kb_init_state<<<1, BP < 32 ? 32 : BP, 0, s>>>(bt->inst, bt->g, bt->tier, B, BP, w->scalars, gin);
  const int gv = std::min(w->num_sms * 8, 8192);
  const int gt = (int)std::min<int64_t>((w->n + kTile - 1) / kTile, gv);
  kb_setup_cols<BP><<<gt, kBThreads, 0, s>>>(a, l_b, u_b, w->prob.l, w->prob.u, bt->inv_col, w->Dc, w->c_s, w->l_s,
                                             w->u_s);
  kb_setup_rows<BP><<<gv, 256, 0, s>>>(a, w->q_s);
  kb_first_dx2<BP><<<BP, kBlock, 0, s>>>(a, gt);
  kb_spmm<BP><<<bt->grid_rows, kBThreads, 0, s>>>(a);
  launch_body<BP>(a, bt, s, 1);  // initial KKT_w of every instance
}

// The batched autotuner: rows (columns) per warp R in {1, 2, 4} and the grid
// (1 to 8 blocks per SM, capped by occupancy and by one row group per warp) of each
// sweep, timed with CUDA events on this matrix and batch width.  UCPDHG_TUNE_LOG=1
// prints the table to stderr.
template <int BP>
int autotune_batched(Workspace* w, Batched* bt, const BArgs<BP>& a, int B, const double* l_b,
                     const double* u_b, cudaStream_t s) {
  bt->tuned = true;
  if (!w->opts.autotune) {
    // fixed shape: kernel_variant 1, 2 or 4 sets R of both sweeps, kernel_grid
    // their blocks (both grid-stride loops; partials hold kMaxBlocks blocks)
    const int kv = w->opts.kernel_variant;
    if (kv == 1 || kv == 2 || kv == 4) bt->rw_dual = bt->rw_adj = kv;
    if (w->opts.kernel_grid > 0) bt->grid_rows = bt->grid_cols = std::min(w->opts.kernel_grid, kMaxBlocks);
    return PDHG_OK;
  }
  const char* log_env = std::getenv("UCPDHG_TUNE_LOG");
  const bool log = log_env && log_env[0] == '1';
  batched_start<BP>(w, bt, a, B, l_b, u_b, s);
  const int sms = w->num_sms;
  for (int which = 0; which < 2; ++which) {
    const int64_t len = which == 0 ? w->m : w->n;
    float best = 1e30f;
    int best_rw = 4, best_grid = which == 0 ? bt->grid_rows : bt->grid_cols;
    for (int rw : {4, 2, 1}) {
      int occ = 0;
      if (which == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ, rw == 4 ? (const void*)kb_dual<BP, 4> : rw == 2 ? (const void*)kb_dual<BP, 2> : (const void*)kb_dual<BP, 1>,
            kBThreads, 0);
      else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ, rw == 4 ? (const void*)kb_adjoint<BP, 4> : rw == 2 ? (const void*)kb_adjoint<BP, 2> : (const void*)kb_adjoint<BP, 1>,
            kBThreads, 0);
      occ = std::max(occ, 1);
      // at most one row group per warp
      const int need = (int)std::max<int64_t>(1, (len + rw * kBWarps - 1) / (rw * kBWarps));
      for (int bps = 1; bps <= std::min(occ, 8); ++bps) {
        const int g = std::min(std::min(sms * bps, need), 8192);
        auto run = [&]() {
          if (which == 0)
            launch_sweep_dual<BP>(a, rw, g, s);
          else
            launch_sweep_adjoint<BP>(a, rw, g, s);
        };
        run();
        cudaEventRecord(w->ev[2], s);
        for (int r = 0; r < 3; ++r) run();
        cudaEventRecord(w->ev[3], s);
        if (cudaEventSynchronize(w->ev[3]) != cudaSuccess) {
          g_err = std::string("batched autotune: ") + cudaGetErrorString(cudaGetLastError());
          return PDHG_ERR_CUDA;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, w->ev[2], w->ev[3]);
        if (log)
          std::fprintf(stderr, "autotune batched B=%d %s rows/warp %d grid %d: %.2f us\n", B,
                       which == 0 ? "dual" : "adjoint", rw, g, ms * 1000.f / 3.f);
        if (ms < best * 0.98f) {
          best = ms;
          best_rw = rw;
          best_grid = g;
        }
        if (g == need) break;
      }
    }
    if (which == 0) {
      bt->rw_dual = best_rw;
      bt->grid_rows = best_grid;
    } else {
      bt->rw_adj = best_rw;
      bt->grid_cols = best_grid;
    }
  }
  return cudaGetLastError() == cudaSuccess ? PDHG_OK : PDHG_ERR_CUDA;
}

template <int BP>
int solve_batched_impl(Workspace* w, int B, const double* l_b, const double* u_b, double* x_out,
                       double* y_out, pdhg_result* res, cudaStream_t s) {
  Batched* bt = (Batched*)w->batched;
  if (bt && bt->BP != BP) return -99;  // caller rebuilds
  if (!bt) {
    bt = new Batched();
    bt->BP = BP;
    w->batched = bt;
    BArgs<BP> a;
    int rc = setup_batched<BP>(w, bt, &a);
    if (rc != PDHG_OK) return rc;
    bt->args = new BArgs<BP>(a);
  }
  if (!bt->inverted) {
    kb_invert<<<w->num_sms, 256, 0, s>>>(w->perm_row, bt->inv_row, (int)w->m);
    kb_invert<<<w->num_sms, 256, 0, s>>>(w->perm_col, bt->inv_col, (int)w->n);
    // a later call may use another stream
    if (cudaStreamSynchronize(s) != cudaSuccess) {
      g_err = std::string("batched setup: ") + cudaGetErrorString(cudaGetLastError());
      return PDHG_ERR_CUDA;
    }
    bt->inverted = true;
  }
  BArgs<BP> a = *(BArgs<BP>*)bt->args;
  a.B = B;
  a.in_graph = 0;
  const pdhg_opts& o = w->opts;
  if (!bt->tuned) {
    // time the sweeps' launch shapes on this batch (real attempts on scratch
    // state, re-initialised below), before the graph captures them
    launch_prepare(w, true, s);
    int rc = autotune_batched<BP>(w, bt, a, B, l_b, u_b, s);
    if (rc != PDHG_OK) return rc;
  }
  if (!o.host_loop) {
    int rc = build_batched_graph<BP>(w, bt, a);
    if (rc != PDHG_OK) return rc;
  }
  cudaEventRecord(w->ev[0], s);
  launch_prepare(w, true, s);
  batched_start<BP>(w, bt, a, B, l_b, u_b, s);
  if (o.host_loop) {
    // the graph body's kernels launched from the host (profilers cannot see
    // kernels inside a graph with conditional nodes); one wait per check
    for (;;) {
      launch_body<BP>(a, bt, s, 0);
      if (cudaMemcpyAsync(bt->done_host, &bt->g->all_done, sizeof(int32_t), cudaMemcpyDeviceToHost,
                          s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess) {
        g_err = std::string("batched host loop: ") + cudaGetErrorString(cudaGetLastError());
        return PDHG_ERR_CUDA;
      }
      if (*bt->done_host) break;
    }
  } else {
    cudaError_t e = cudaGraphLaunch(bt->exec, s);
    if (e != cudaSuccess) {
      g_err = std::string("batched graph launch: ") + cudaGetErrorString(e);
      return PDHG_ERR_CUDA;
    }
  }
  const int64_t gmax = std::min(w->num_sms * 8, 8192);
  if (x_out)
    kb_output<BP><<<(int)std::min<int64_t>((w->n + kTile - 1) / kTile, gmax), kBThreads, 0, s>>>(
        a.xst, w->Dc, bt->inv_col, w->n, B, x_out);
  if (y_out)
    kb_output<BP><<<(int)std::min<int64_t>((w->m + kTile - 1) / kTile, gmax), kBThreads, 0, s>>>(
        a.yst, w->Dr, bt->inv_row, w->m, B, y_out);
  cudaEventRecord(w->ev[1], s);
  if (cudaMemcpyAsync(bt->inst_host, bt->inst, sizeof(BInst) * BP, cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    g_err = std::string("batched solve: ") + cudaGetErrorString(cudaGetLastError());
    return PDHG_ERR_CUDA;
  }
  float ms = 0.f;
  cudaEventElapsedTime(&ms, w->ev[0], w->ev[1]);
  int64_t checks_max = 0;
  for (int b = 0; b < B; ++b) checks_max = std::max(checks_max, bt->inst_host[b].checks);
  const int passes = o.ruiz_iters + (o.pock_chambolle ? 1 : 0);
  const int64_t launches = 5 + passes + 5 + 4 + checks_max * (2 * kCheckEvery + 6) + 2;
  bool numeric = false;
  for (int b = 0; b < B; ++b) {
    const BInst& I = bt->inst_host[b];
    pdhg_result& r = res[b];
    std::memset(&r, 0, sizeof(r));
    r.status = I.status ? I.status : PDHG_STATUS_ITER_LIMIT;
    r.ir_rounds = I.rounds;
    r.iterations = I.k_total;
    r.accepted = I.accepted;
    r.restarts = I.restarts;
    r.checks = I.checks;
    r.rel_p = I.rel_p;
    r.rel_d = I.rel_d;
    r.rel_gap = I.rel_gap;
    r.rel_kkt = I.rel_kkt;
    r.primal_obj = I.pobj;
    r.dual_obj = I.dobj;
    r.solve_seconds = ms * 1e-3;
    for (int t = 0; t < 3; ++t) {
      r.time_to_tol[t] = I.t_tol[t];
      r.iters_to_tol[t] = I.k_tol[t];
    }
    r.eta = I.eta;
    r.omega = I.omega;
    r.kernel_launches = launches;
    numeric = numeric || I.status == PDHG_STATUS_NUMERIC;
  }
  if (numeric) {
    g_err = "NaN/Inf met in a batched KKT evaluation";
    return PDHG_ERR_NUMERIC;
  }
  return PDHG_OK;
}

}  // namespace

void batched_tuning(Workspace* w, int32_t* out) {
  const Batched* bt = (const Batched*)w->batched;
  const bool t = bt && bt->tuned;
  out[0] = t ? bt->rw_dual : -1;
  out[1] = t ? bt->grid_rows : 0;
  out[2] = t ? bt->rw_adj : -1;
  out[3] = t ? bt->grid_cols : 0;
}

void release_batched(Workspace* w) {
  Batched* bt = (Batched*)w->batched;
  if (!bt) return;
  if (bt->exec) cudaGraphExecDestroy(bt->exec);
  if (bt->graph) cudaGraphDestroy(bt->graph);
  if (bt->inst_host) cudaFreeHost(bt->inst_host);
  if (bt->done_host) cudaFreeHost(bt->done_host);
  for (void* p : bt->allocs) cudaFree(p);
  if (bt->args) {
    if (bt->BP == 64)
      delete (BArgs<64>*)bt->args;
    else
      delete (BArgs<32>*)bt->args;
  }
  delete bt;
  w->batched = nullptr;
}

}  // namespace ucpdhg

using namespace ucpdhg;

extern "C" int pdhg_solve_batched(void* ws, int32_t B, const double* l_b, const double* u_b,
                                  double* x_out, double* y_out, pdhg_result* res_b, void* stream) {
  g_err.clear();
  if (!ws || !l_b || !u_b || !res_b) {
    g_err = "pdhg_solve_batched: NULL argument";
    return PDHG_ERR_INVALID_ARG;
  }
  if (B < 1 || B > 64) {
    g_err = "pdhg_solve_batched: B must be in 1..64";
    return PDHG_ERR_INVALID_ARG;
  }
  Workspace* w = (Workspace*)ws;
  cudaStream_t s = (cudaStream_t)stream;
  const int BP = B <= 32 ? 32 : 64;
  if (w->batched && ((Batched*)w->batched)->BP != BP) release_batched(w);
  int rc = BP == 32 ? solve_batched_impl<32>(w, B, l_b, u_b, x_out, y_out, res_b, s)
                    : solve_batched_impl<64>(w, B, l_b, u_b, x_out, y_out, res_b, s);
  return rc;
}
