// 64 step attempts of a small LP in one launch (Sec. II.E iteration, PDLP form).
//
// On a small LP the two kernels of an attempt (pdhg_kernels.cu) spend their time
// on what surrounds the sweeps: the launch, the state read, the round trip for
// the matrix and the row operands, the last-block reduction.  Here one launch runs
// the 64 attempts between two checks.  Every block owns the slices s = block,
// block + gridDim, ... of K and of K^T, keeps their entries and the rows' and
// columns' operands in shared memory for the whole launch, and only the vectors
// that others gather (x', y') go through global memory, with a barrier over all
// blocks after each sweep.  K x is kept instead of recomputed (same sums in the same
// order, so the iterates are those of the separate kernels; the step-size sums
// are reduced in another fixed order).
//
// Up to 16 blocks run as one cluster (the barrier is the cluster's, the partial
// sums travel through distributed shared memory); larger grids are cooperative
// launches with a counter in global memory.  Every wait on it is bounded: a
// block that gives up sets DevState::wait_timeout and done and returns, and so do
// the blocks that wait for it.
#include <algorithm>

#include "internal.cuh"

namespace ucpdhg {
namespace {

constexpr int kResCluster = 16;
constexpr int kResBlocks = 160;  // most blocks of a cooperative launch (GB300: 152 SMs)
constexpr int kResStates = 7;                  // vectors kept per row and per column
constexpr size_t kResSmem = 223 * 1024;  // dynamic shared memory a block may take (227 KB less the static)

struct ResArgs {
  const int32_t* kloc;  // entry offset of each slice of K in its block's shared memory
  const int32_t* tloc;
  int32_t kcap, tcap;  // entries per block
  int32_t rcap, ccap;  // rows and columns per block
  int32_t polls;       // of grid_barrier before a block gives up
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Barrier over the blocks of a cooperative launch (one thread per block, after a
// barrier of its block): counts the block in and waits, bounded, until `target`
// arrivals.  False if it gave up.  A counter that all poll beats words with a tag
// per block that all collect (17.2 against 20.0 us per attempt at 152 blocks:
// 152 x 152 polled words cost more than the second round trip for the sums).
__device__ __forceinline__ bool grid_barrier(uint32_t* counter, unsigned target, int polls) {
  __threadfence();
  atomicAdd(counter, 1u);
  for (int it = 0; it < polls; ++it) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (v >= target) {
      __threadfence();
      return true;
    }
  }
  return false;
}

// Fixed-order totals of every block's NV values (one warp, after the barrier;
// valid in every lane).
template <int NV, class T>
__device__ __forceinline__ void sum_parts(const T* parts, int G, int lane, T (&tot)[NV]) {
  constexpr int N = (kResBlocks + 31) / 32;
  T v[N][NV];
#pragma unroll
  for (int n = 0; n < N; ++n)
#pragma unroll
    for (int e = 0; e < NV; ++e) v[n][e] = lane + 32 * n < G ? __ldcg(parts + (lane + 32 * n) * 4 + e) : (T)0;
#pragma unroll
  for (int e = 0; e < NV; ++e) {
    tot[e] = v[0][e];
#pragma unroll
    for (int n = 1; n < N; ++n) tot[e] += v[n][e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot[e] += __shfl_xor_sync(0xffffffffu, tot[e], o);
  }
}

// Block totals of NV values of T, valid in every lane of warp 0.
template <int NV, int WARPS, class T>
__device__ __forceinline__ void res_block_sum(T (&v)[NV], T* smem /* [WARPS * NV] */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = warp_sum_t<T>(v[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) smem[wid * NV + k] = v[k];
  __syncthreads();
  if (wid == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      v[k] = lane < WARPS ? smem[lane * NV + k] : (T)0;
#pragma unroll
      for (int o = WARPS / 2; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
}

// Scalars of the step decision, in the registers of thread 0 for the whole
// launch.  decide() is decide_step (common.cuh) with what does not depend on the
// sums taken out of the wait for them: the factors of the next step, and 1/omega
// in place of the divisions by omega (GB300's FP64 pipe makes each of them
// hundreds of cycles on the chain that every block waits for).
struct ResStep {
  double eta, omega, inv_omega, wsum, up, down;
  int64_t k, kg, accepted, since;
  int par, fixed;
};
__device__ __forceinline__ void step_factors(ResStep& r, const DevState& st) {
  r.down = 1.0 - step_power(r.kg + 2, st.red_exp);
  r.up = 1.0 + step_power(r.kg + 2, st.grow_exp);
}

// Products of one slice held in shared memory, gathered from vec: eight gathers
// (L2: the barrier has emptied L1) in flight per lane.
template <class T, int E>
__device__ __forceinline__ T res_chunk(const int32_t* col, const T* val, int k0, int w, int lane, const T* vec, T acc) {
  T v[E], x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool ok = k0 + e < w;
    v[e] = ok ? val[(k0 + e) * kSlice + lane] : (T)0;
    x[e] = ok ? vec[col[(k0 + e) * kSlice + lane]] : (T)0;
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (k0 + e < w) acc += v[e] * x[e];
  return acc;
}
template <class T>
__device__ __forceinline__ T res_dot(const int32_t* col, const T* val, int w, int lane, const T* vec) {
  if (w <= 4) return res_chunk<T, 4>(col, val, 0, w, lane, vec, (T)0);
  T acc = 0;
  for (int k0 = 0; k0 < w; k0 += 8) acc = res_chunk<T, 8>(col, val, k0, w, lane, vec, acc);
  return acc;
}

template <class T, bool CLUSTER, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) k_resident(IterArgs<T> a, ResArgs r) {
  extern __shared__ __align__(16) unsigned char res_raw[];
  __shared__ DevState st;
  __shared__ T red[WARPS * 2];
  __shared__ T parts[kResCluster * 4];  // cluster: every block's {||dy||^2, dy^T K dx, ||dx||^2}
  __shared__ int abort_s;
  __shared__ DualScalars<T> ds;
  __shared__ AdjScalars<T> as;
  const int b = blockIdx.x, G = gridDim.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < (int)(sizeof(DevState) / 4); t += WARPS * 32)
    reinterpret_cast<int*>(&st)[t] = reinterpret_cast<const int*>(a.st)[t];
  if (threadIdx.x == 0) abort_s = 0;
  __syncthreads();
  if (st.done) return;  // the same in every block
  ResStep rs_{};
  if (threadIdx.x == 0) {
    dual_scalars<T>(&st, ds);
    rs_.eta = st.eta;
    rs_.omega = st.omega;
    rs_.inv_omega = 1.0 / st.omega;
    rs_.wsum = st.wsum;
    rs_.k = st.k;
    rs_.kg = st.k_offset + st.k;
    rs_.accepted = st.accepted;
    rs_.since = st.since_restart;
    rs_.par = st.par;
    rs_.fixed = st.fixed;
  }

  T* kval = reinterpret_cast<T*>(res_raw);
  T* tval = kval + r.kcap;
  T* rs = tval + r.tcap;                // row state: y[2], K x[2], y sum, q, y_lo
  T* cs = rs + kResStates * r.rcap;     // column state: x[2], K^T y, x sum, c, l, u
  int32_t* kcol = reinterpret_cast<int32_t*>(cs + kResStates * r.ccap);
  int32_t* tcol = kcol + r.kcap;
  int2* ktab = reinterpret_cast<int2*>(tcol + r.tcap);  // {first entry, entries per row} of each slice
  int2* ttab = ktab + r.rcap / kSlice;
  T* sy[2] = {rs, rs + r.rcap};
  T* skx[2] = {rs + 2 * r.rcap, rs + 3 * r.rcap};
  T *sybar = rs + 4 * r.rcap, *sq = rs + 5 * r.rcap, *slo = rs + 6 * r.rcap;
  T* sx[2] = {cs, cs + r.ccap};
  T *skty = cs + 2 * r.ccap, *sxbar = cs + 3 * r.ccap, *sc = cs + 4 * r.ccap, *sl = cs + 5 * r.ccap,
    *su = cs + 6 * r.ccap;
  const int nk = a.K.nslices > b ? (a.K.nslices - 1 - b) / G + 1 : 0;
  const int nt = a.KT.nslices > b ? (a.KT.nslices - 1 - b) / G + 1 : 0;
  const int p0 = st.par;

  // each warp loads what it will use itself
  for (int l = wid; l < nk; l += WARPS) {
    const int s = b + l * G, o = a.K.off[s], n = a.K.off[s + 1] - o, q = r.kloc[s];
    for (int t = lane; t < n; t += 32) {
      kval[q + t] = a.K.val[o + t];
      kcol[q + t] = a.K.col[o + t];
    }
    if (lane == 0) ktab[l] = make_int2(q, n >> 5);
    __syncwarp();  // the entries are read across the warp below
    const int i = s * kSlice + lane, d = l * kSlice + lane;
    sy[p0][d] = a.y[p0][i];
    sybar[d] = a.ybar[i];
    sq[d] = a.q[i];
    slo[d] = a.ylo ? a.ylo[i] : (T)0;
    skx[p0][d] = StoresKx<T>::value ? a.Kx[p0][i] : res_dot<T>(kcol + q, kval + q, n >> 5, lane, a.x[p0]);
  }
  for (int l = wid; l < nt; l += WARPS) {
    const int s = b + l * G, o = a.KT.off[s], n = a.KT.off[s + 1] - o, q = r.tloc[s];
    for (int t = lane; t < n; t += 32) {
      tval[q + t] = a.KT.val[o + t];
      tcol[q + t] = a.KT.col[o + t];
    }
    if (lane == 0) ttab[l] = make_int2(q, n >> 5);
    const int j = s * kSlice + lane, d = l * kSlice + lane;
    sx[p0][d] = a.x[p0][j];
    sx[1 - p0][d] = a.x[1 - p0][j];
    skty[d] = a.KTy[p0][j];
    sxbar[d] = a.xbar[j];
    sc[d] = a.c[j];
    sl[d] = a.l[j];
    su[d] = a.u[j];
  }
  __syncthreads();
  if (CLUSTER) cluster_barrier();  // every block has started: its shared memory may be written

  double dx2 = st.dx2;   // ||x' - x||^2 of the pending candidate (warp 0)
  T part_dx2 = 0;        // this block's part of it (warp 0)
  unsigned target = 0;   // arrivals at the barrier (thread 0)
  // {||dy||^2, dy^T K dx, ||dx||^2} of each block
  T* gpart = reinterpret_cast<T*>(a.partials);

  for (int k = 0; k < kCheckEvery; ++k) {
    // ---- K x' and the dual step
    {
      const int p = ds.p;
      const bool has_pw = ds.has_pw;
      const T pw = ds.pw, sigma = ds.sigma;
      const T* xn = a.x[1 - p];
      T* yn = a.y[1 - p];
      T acc[2] = {0, 0};
      for (int l = wid; l < nk; l += WARPS) {
        const int2 e = ktab[l];
        const int i = (b + l * G) * kSlice + lane, d = l * kSlice + lane;
        const T kx = res_dot<T>(kcol + e.x, kval + e.x, e.y, lane, xn);
        if (i < a.m) {
          const T yo = sy[p][d], ko = skx[p][d];
          T t = sq[d] - (T)2 * kx;
          t = t + ko;
          T v = yo + sigma * t;
          if (i >= a.m_eq) v = max(v, slo[d]);
          yn[i] = v;
          sy[1 - p][d] = v;
          skx[1 - p][d] = kx;
          if (has_pw) sybar[d] = sybar[d] + pw * yo;
          const T dy = v - yo;
          acc[0] += dy * dy;
          acc[1] += dy * (kx - ko);
        }
      }
      res_block_sum<2, WARPS, T>(acc, red);
      double w_now = 0.0, max_now = 0.0, next_now = 0.0;  // thread 0
      int acc_now = 0;
      if (wid == 0) {
        // totals of all blocks in fixed order, then the step decision (every
        // block takes the same one)
        bool ok = true;
        T tot[2], dxt = 0;
        if constexpr (CLUSTER) {
          if (lane < G) {
            const unsigned dst = static_cast<uint32_t>(__cvta_generic_to_shared(parts + 4 * b));
            unsigned rem;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rem) : "r"(dst), "r"(lane));
            const T v3[3] = {acc[0], acc[1], part_dx2};
#pragma unroll
            for (int e = 0; e < 3; ++e) {
              if constexpr (sizeof(T) == 4)
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(rem + 4 * e), "f"(v3[e]) : "memory");
              else
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(rem + 8 * e), "d"(v3[e]) : "memory");
            }
          }
        } else {
          if (lane == 0) {
            __stcg(gpart + 4 * b, acc[0]);
            __stcg(gpart + 4 * b + 1, acc[1]);
            target += (unsigned)G;
          }
        }
        if (lane == 0) step_factors(rs_, st);
        if constexpr (!CLUSTER) {
          // the block's y' is ordered before by the barrier in the block sum
          if (lane == 0) ok = grid_barrier(&a.st->bar, target, r.polls);
          __syncwarp();
          sum_parts<2, T>(gpart, G, lane, tot);
        }
        if constexpr (CLUSTER) {
          __syncwarp();
          cluster_barrier();
          tot[0] = lane < G ? parts[4 * lane + 0] : (T)0;
          tot[1] = lane < G ? parts[4 * lane + 1] : (T)0;
          dxt = lane < G ? parts[4 * lane + 2] : (T)0;
#pragma unroll
          for (int o = kResCluster / 2; o > 0; o >>= 1) {
            tot[0] += __shfl_xor_sync(0xffffffffu, tot[0], o);
            tot[1] += __shfl_xor_sync(0xffffffffu, tot[1], o);
            dxt += __shfl_xor_sync(0xffffffffu, dxt, o);
          }
        }
        if (CLUSTER && k > 0) dx2 = (double)dxt;
        if (lane == 0) {
          const double movement = rs_.omega * dx2 + (double)tot[0] * rs_.inv_omega;
          const double interaction = 2.0 * fabs((double)tot[1]);
          const double eta = rs_.eta;
          const double eta_max = interaction > 0.0 ? movement / interaction : INFINITY;
          double eta_next = fmin(rs_.down * eta_max, rs_.up * eta);
          int accept = eta <= eta_max;
          if (rs_.fixed) {
            accept = 1;
            eta_next = eta;
          }
          w_now = accept ? eta : 0.0;
          acc_now = accept;
          max_now = eta_max;
          if (accept) rs_.par = 1 - rs_.par;
          as.p = ds.p = rs_.par;
          as.acc_last = accept;
          as.upd_avg = w_now != 0.0;
          as.wl = ds.pw = (T)w_now;
          ds.has_pw = w_now != 0.0;
          as.tau = (T)(eta_next * rs_.inv_omega);
          ds.sigma = (T)(eta_next * rs_.omega);
          next_now = eta_next;
          if (!ok) abort_s = 1;
        }
      } else if (CLUSTER) {
        cluster_barrier();
      }
      __syncthreads();
      if (!CLUSTER && abort_s) break;
      if (threadIdx.x == 0) {  // bookkeeping nobody waits for
        if (st.trace_on && a.trace_a) {  // every block writes the same record
          const int64_t t = st.n_trace_a;
          if (t < st.trace_cap_a) {
            double* rec = a.trace_a + t * 5;
            rec[0] = rs_.eta;
            rec[1] = rs_.omega;
            rec[2] = (double)acc_now;
            rec[3] = max_now;
            rec[4] = next_now;
          }
          st.n_trace_a = t + 1;
        }
        rs_.eta = next_now;
        rs_.wsum += w_now;
        rs_.accepted += acc_now;
        rs_.since += 1;
        rs_.k += 1;
        rs_.kg += 1;
        st.w_last = st.pending_w = w_now;
        st.accepted_last = acc_now;
      }
    }
    // ---- K^T y' of an accepted step, the x-average and the next primal step
    {
      const int p = as.p, acc_last = as.acc_last;
      const bool upd = as.upd_avg;
      const T wl = as.wl, tau = as.tau;
      const T* yc = a.y[p];
      T* xn = a.x[1 - p];
      T acc[1] = {0};
      for (int l = wid; l < nt; l += WARPS) {
        const int2 e = ttab[l];
        const int j = (b + l * G) * kSlice + lane, d = l * kSlice + lane;
        const T g = acc_last ? res_dot<T>(tcol + e.x, tval + e.x, e.y, lane, yc) : skty[d];
        if (j < a.n) {
          const T x0 = sx[p][d];
          skty[d] = g;
          if (upd) sxbar[d] = sxbar[d] + wl * x0;
          T v = x0 - tau * (sc[d] - g);
          v = min(max(v, sl[d]), su[d]);
          xn[j] = v;
          sx[1 - p][d] = v;
          const T dd = v - x0;
          acc[0] += dd * dd;
        }
      }
      res_block_sum<1, WARPS, T>(acc, red);
      part_dx2 = acc[0];
      if (k + 1 < kCheckEvery) {
        if constexpr (CLUSTER) {
          cluster_barrier();
        } else {
          if (wid == 0) {
            if (lane == 0) {
              __stcg(gpart + 4 * b + 2, acc[0]);
              target += (unsigned)G;
              if (!grid_barrier(&a.st->bar, target, r.polls)) abort_s = 1;
            }
          }
          __syncthreads();
          if (abort_s) break;
          if (wid == 0) {  // needed at the next decision only
            T tot[1];
            sum_parts<1, T>(gpart + 2, G, lane, tot);
            dx2 = (double)tot[0];
          }
        }
      }
    }
  }
  // the state the checks read, and the last ||dx||^2 over all blocks
  {
    const int p = as.p;
    for (int l = wid; l < nk; l += WARPS) {
      const int s = b + l * G, i = s * kSlice + lane, d = l * kSlice + lane;
      if (i < a.m) {
        a.ybar[i] = sybar[d];
        if (StoresKx<T>::value) a.Kx[p][i] = skx[p][d];
      }
    }
    for (int l = wid; l < nt; l += WARPS) {
      const int s = b + l * G, j = s * kSlice + lane, d = l * kSlice + lane;
      if (j < a.n) {
        a.KTy[p][j] = skty[d];
        if constexpr (sizeof(T) == 4) {  // the check reads the FP64 sums
          a.xbar64[j] += to_f64(sxbar[d]);
          a.xbar[j] = 0;
        } else {
          a.xbar[j] = sxbar[d];
        }
      }
    }
    if (threadIdx.x == 0) {
      volatile DevState* out = a.st;
      __stcg(gpart + 4 * b + 3, part_dx2);
      if (abort_s) out->wait_timeout = 1;
      __threadfence();
      const unsigned t = atomicAdd(&a.st->counter, 1u);
      if (t == (unsigned)G - 1) {  // last block out: the state of the attempts
        __threadfence();
        T d = 0;
        for (int g = 0; g < G; ++g) d += __ldcg(gpart + 4 * g + 3);
        st.dx2 = (double)d;
        st.eta = rs_.eta;
        st.wsum = rs_.wsum;
        st.k = rs_.k;
        st.accepted = rs_.accepted;
        st.since_restart = rs_.since;
        st.par = rs_.par;
        st.counter = st.bar = 0;
        if (out->wait_timeout) st.done = st.wait_timeout = 1;
        *a.st = st;
      }
    }
  }
}

template <class T>
size_t res_bytes(const ResArgs& r) {
  return sizeof(T) * ((size_t)r.kcap + r.tcap + (size_t)kResStates * (r.rcap + r.ccap)) +
         sizeof(int32_t) * ((size_t)r.kcap + r.tcap) + sizeof(int2) * ((size_t)(r.rcap + r.ccap) / kSlice);
}

// Entries of the slices s = b, b + G, ... of each block, one after the other.
int32_t deal_slices(const std::vector<int32_t>& off, int G, std::vector<int32_t>* loc) {
  const int ns = (int)off.size() - 1;
  std::vector<int32_t> fill(G, 0);
  loc->resize(ns);
  int32_t most = 0;
  for (int s = 0; s < ns; ++s) {
    (*loc)[s] = fill[s % G];
    fill[s % G] += off[s + 1] - off[s];
    most = std::max(most, fill[s % G]);
  }
  return most;
}

template <class T, bool CLUSTER, int WARPS>
cudaError_t res_launch(const IterArgs<T>& a, const ResidentPlan& pl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)pl.grid);
  cfg.blockDim = dim3(WARPS * 32);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (CLUSTER) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pl.grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const ResArgs r = {pl.kloc, pl.tloc, pl.kcap, pl.tcap, pl.rcap, pl.ccap, pl.polls};
  return cudaLaunchKernelEx(&cfg, k_resident<T, CLUSTER, WARPS>, a, r);
}

// Whether the device takes a launch of this plan.
template <class T, bool CLUSTER, int WARPS>
bool res_fits(const ResidentPlan& pl, int sms) {
  const void* fn = (const void*)&k_resident<T, CLUSTER, WARPS>;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem) != cudaSuccess)
    return false;
  if (CLUSTER) {
    if (pl.grid > 8 &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)pl.grid);
    cfg.blockDim = dim3(WARPS * 32);
    cfg.dynamicSmemBytes = pl.smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pl.grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n >= 1;
  }
  int per_sm = 0;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, WARPS * 32, pl.smem) == cudaSuccess &&
         per_sm >= 1 && pl.grid <= sms && pl.grid <= kResBlocks;
}

}  // namespace

template <class T>
bool plan_resident(const std::vector<int32_t>& koff, const std::vector<int32_t>& toff, int sms,
                   ResidentPlan* pl, std::vector<int32_t>* kloc, std::vector<int32_t>* tloc) {
  const int ks = (int)koff.size() - 1, ts = (int)toff.size() - 1;
  // one slice of K per warp where the cluster has that many, and as many blocks
  // as shared memory asks for
  for (int G = 1; G <= sms; G = G < kResCluster ? 2 * G : (G == kResCluster ? sms : sms + 1)) {
    if (G < kResCluster && G * 16 < ks) continue;
    // FP64 fills the FP64 pipe of 16 SMs at about 24 slices of K a block: above
    // that more SMs gain more than the cluster's cheaper barrier (29k rows, FP64:
    // 18.4 us per attempt on 16 blocks, 14.9 on 152)
    if (sizeof(T) == 8 && G <= kResCluster && ks > G * 24) continue;
    ResArgs r;
    r.kcap = deal_slices(koff, G, kloc);
    r.tcap = deal_slices(toff, G, tloc);
    r.rcap = (ks + G - 1) / G * kSlice;
    r.ccap = (ts + G - 1) / G * kSlice;
    const size_t bytes = res_bytes<T>(r);
    if (bytes > kResSmem) continue;
    pl->grid = G;
    pl->cluster = G <= kResCluster;
    pl->smem = bytes;
    pl->kcap = r.kcap;
    pl->tcap = r.tcap;
    pl->rcap = r.rcap;
    pl->ccap = r.ccap;
    pl->warps = (ks + G - 1) / G > 16 ? 32 : 16;
    const bool ok = pl->cluster ? (pl->warps == 32 ? res_fits<T, true, 32>(*pl, sms) : res_fits<T, true, 16>(*pl, sms))
                                : (pl->warps == 32 ? res_fits<T, false, 32>(*pl, sms) : res_fits<T, false, 16>(*pl, sms));
    cudaGetLastError();
    if (ok) return true;
  }
  return false;
}

template <class T>
cudaError_t launch_resident(const IterArgs<T>& a, const ResidentPlan& pl, cudaStream_t s) {
  if (pl.cluster) return pl.warps == 32 ? res_launch<T, true, 32>(a, pl, s) : res_launch<T, true, 16>(a, pl, s);
  return pl.warps == 32 ? res_launch<T, false, 32>(a, pl, s) : res_launch<T, false, 16>(a, pl, s);
}

template bool plan_resident<float>(const std::vector<int32_t>&, const std::vector<int32_t>&, int, ResidentPlan*,
                                   std::vector<int32_t>*, std::vector<int32_t>*);
template bool plan_resident<double>(const std::vector<int32_t>&, const std::vector<int32_t>&, int, ResidentPlan*,
                                    std::vector<int32_t>*, std::vector<int32_t>*);
template cudaError_t launch_resident<float>(const IterArgs<float>&, const ResidentPlan&, cudaStream_t);
template cudaError_t launch_resident<double>(const IterArgs<double>&, const ResidentPlan&, cudaStream_t);

}  // namespace ucpdhg
