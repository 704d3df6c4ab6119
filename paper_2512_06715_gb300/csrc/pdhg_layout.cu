// Internal layout (length-sorted orderings, sliced ELL) and the rescaling pass.
//
// Rows of K are reordered by decreasing length inside the equality block and
// inside the inequality block, columns by decreasing column count, so that each
// 32-row slice holds rows of (nearly) equal length and padding stays negligible
// on the UC sparsity (rows of 2 to ~25 entries); rows (columns) of one length are
// grouped so that a slice's gathers are contiguous (order_by_signature).  K and
// K^T are both kept in this layout; every vector the iterations touch lives in
// the internal order, so no permutation is applied inside the PDHG loop.
//
// Rescaling (the PDLP preconditioning of Applegate et al., cited in Sec. II.E):
// Ruiz l_inf passes r_i = 1/sqrt(max_j |K~_ij|), s_j = 1/sqrt(max_i |K~_ij|),
// then one Pock-Chambolle alpha = 1 pass with l_1 sums, both factors of a pass
// taken from the same K~.  The factors accumulate in Dr, Dc and the matrix is
// formed once at the end as K~_ij = K_ij (Dr_i Dc_j).
#include <algorithm>
#include <cstring>
#include <numeric>

#include "internal.cuh"

namespace ucpdhg {

namespace {

// Finalizer of a 64-bit hash (the multiply-xorshift of SplitMix64).
inline uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// Internal order of a set of rows (columns): by decreasing length, equal
// lengths grouped by signature in the order the signatures first occur, equal
// signatures in their original order.  perm receives `count` ids from `first`;
// members (optional) the size of each id's group.
void order_by_signature(int64_t first, int64_t count, const std::vector<int32_t>& len,
                        const std::vector<uint64_t>& sig, int32_t* perm, int32_t* members) {
  if (count == 0) return;
  // group ids by first occurrence (open addressing; lengths are part of the key)
  size_t cap = 16;
  while (cap < (size_t)count * 2) cap <<= 1;
  std::vector<int32_t> table(cap, -1), gid(count), glen;
  std::vector<int64_t> gsize;
  std::vector<int64_t> grep;  // a member of the group
  for (int64_t t = 0; t < count; ++t) {
    const int64_t i = first + t;
    size_t h = mix64(sig[i] + (uint64_t)len[i]) & (cap - 1);
    for (;; h = (h + 1) & (cap - 1)) {
      const int32_t g = table[h];
      if (g < 0) {
        table[h] = gid[t] = (int32_t)glen.size();
        glen.push_back(len[i]);
        gsize.push_back(1);
        grep.push_back(i);
        break;
      }
      if (glen[g] == len[i] && sig[grep[g]] == sig[i]) {
        gid[t] = g;
        ++gsize[g];
        break;
      }
    }
  }
  std::vector<int32_t> order(glen.size());
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return glen[a] > glen[b]; });
  std::vector<int64_t> pos(glen.size());
  int64_t at = 0;
  for (int32_t g : order) {
    pos[g] = at;
    at += gsize[g];
  }
  for (int64_t t = 0; t < count; ++t) {
    perm[pos[gid[t]]++] = (int32_t)(first + t);
    if (members) members[t] = (int32_t)gsize[gid[t]];
  }
}

// Offsets of the 32-row slices over the internal order.  Slices come in aligned
// groups of kGroup of one width, so that a warp sweeping a group (or half of one)
// finds its entries at fixed distances.  Returns the number of slices (a multiple
// of kGroup), -1 if the entries exceed 2^31.
int64_t slice_offsets_of(const std::vector<int32_t>& len, const std::vector<int32_t>& perm,
                         std::vector<int32_t>* off) {
  const int64_t rows = (int64_t)perm.size();
  const int64_t ng = (rows + kSlice * kGroup - 1) / (kSlice * kGroup);
  off->assign(ng * kGroup + 1, 0);
  int64_t tot = 0;
  for (int64_t g = 0; g < ng; ++g) {
    int32_t w = 0;
    const int64_t end = std::min(rows, (g + 1) * kSlice * kGroup);
    for (int64_t i = g * kSlice * kGroup; i < end; ++i) w = std::max(w, len[perm[i]]);
    for (int s = 0; s < kGroup; ++s) {
      tot += (int64_t)w * kSlice;
      if (tot >= (int64_t)1 << 31) return -1;
      (*off)[g * kGroup + s + 1] = (int32_t)tot;
    }
  }
  return ng * kGroup;
}

// Column runs of a sliced-ELL matrix (see SellView::runs).
void build_runs(const std::vector<int32_t>& off, const std::vector<int32_t>& col,
                const std::vector<int32_t>& src, int64_t ncols, std::vector<int32_t>* soff,
                std::vector<int32_t>* runs) {
  const int64_t ns = (int64_t)off.size() - 1;
  soff->assign(off.begin(), off.end());
  runs->assign((size_t)off[ns] / kSlice * 2, 0);
  for (int64_t g = 0; g < ns; g += kGroup) {
    const int64_t o0 = off[g], o1 = off[g + kGroup];
    int mode = ncols < ((int64_t)1 << kRunBits) ? kRunsOne : kRunsNone;
    for (int64_t o = o0; o < o1 && mode != kRunsNone; o += kSlice) {
      int32_t prev = -1, start[2] = {0, 0}, split = kSlice, pieces = 0;
      for (int lane = 0; lane < kSlice; ++lane) {
        // a padding slot (value 0) continues the run it follows, inside the vector
        int32_t c = col[o + lane];
        if (src[o + lane] < 0) c = (lane > 0 && prev + 1 < ncols) ? prev + 1 : 0;
        if (lane == 0 || c != prev + 1) {
          if (pieces == 2) {
            mode = kRunsNone;
            break;
          }
          if (pieces == 1) {
            split = lane;
            mode = kRunsTwo;
          }
          start[pieces++] = c;
        }
        prev = c;
      }
      (*runs)[o / kSlice * 2] = start[0];
      (*runs)[o / kSlice * 2 + 1] = (int32_t)(((uint32_t)split << kRunBits) | (uint32_t)start[1]);
    }
    for (int s = 0; s < kGroup; ++s) (*soff)[g + s] |= mode;
  }
}

}  // namespace

int build_layout(int64_t n, int64_t m, int64_t m_eq, const std::vector<int64_t>& rp,
                 const std::vector<int32_t>& col, const std::vector<double>& val, HostLayout* L,
                 std::string* err) {
  std::vector<int32_t> rlen(m), clen(n, 0);
  std::vector<uint64_t> rsig(m), csig(n, 0);
  for (size_t e = 0; e < col.size(); ++e) {
    if (col[e] < 0 || col[e] >= n) {
      *err = "column index out of range in CSR";
      return PDHG_ERR_INVALID_ARG;
    }
    clen[col[e]]++;
  }
  // Signatures that do not see a translation of the columns: a row's are its
  // values and its column distances from its first column, a column's are the
  // signatures of its rows and its place in them.  In a time-expanded model the
  // rows of one line (unit, bus) share a signature over all periods, and so do
  // its columns, so equal signatures kept in their original order run through
  // time and row r + 1 gathers column c + 1 where row r gathers column c.  Rows
  // that differ only in the unit they belong to (minimum up times: all values
  // +-1) are told apart by the signature of one of their columns, the one with
  // the most members: the others may be the few of the first or last periods.
  for (int64_t i = 0; i < m; ++i) {
    rlen[i] = (int32_t)(rp[i + 1] - rp[i]);
    uint64_t h = 0;
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
      uint64_t bits;
      std::memcpy(&bits, &val[e], sizeof(bits));
      h = mix64(h + (uint64_t)(col[e] - col[rp[i]]) + 0x9E3779B97F4A7C15ULL) + bits;
    }
    rsig[i] = mix64(h);
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e) csig[col[e]] += mix64(rsig[i] + (uint64_t)(e - rp[i]));
  }
  std::vector<int32_t> members(n);
  L->perm_col.resize(n);
  order_by_signature(0, n, clen, csig, L->perm_col.data(), members.data());
  for (int64_t i = 0; i < m; ++i) {
    int32_t best = -1;
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e)
      if (best < 0 || members[col[e]] > members[best]) best = col[e];
    if (best >= 0) rsig[i] = mix64(rsig[i] + csig[best]);
  }
  L->perm_row.resize(m);
  order_by_signature(0, m_eq, rlen, rsig, L->perm_row.data(), nullptr);
  order_by_signature(m_eq, m - m_eq, rlen, rsig, L->perm_row.data() + m_eq, nullptr);
  std::vector<int32_t> inv_row(m), inv_col(n);
  for (int64_t i = 0; i < m; ++i) inv_row[L->perm_row[i]] = (int32_t)i;
  for (int64_t j = 0; j < n; ++j) inv_col[L->perm_col[j]] = (int32_t)j;

  // ---- K in sliced ELL over internal rows ----
  const int64_t ks = slice_offsets_of(rlen, L->perm_row, &L->k_off);
  if (ks < 0) {
    *err = "padded nnz of K exceeds 2^31";
    return PDHG_ERR_UNSUPPORTED;
  }
  int64_t tot = L->k_off[ks];
  L->k_col.assign(tot, 0);
  L->k_src.assign(tot, -1);
  for (int64_t s = 0; s < ks; ++s) {
    for (int lane = 0; lane < kSlice; ++lane) {
      int64_t i = s * kSlice + lane;
      if (i >= m) continue;
      int32_t o = L->perm_row[i];
      for (int32_t k = 0; k < rlen[o]; ++k) {
        int64_t e = rp[o] + k;
        int64_t slot = L->k_off[s] + (int64_t)k * kSlice + lane;
        L->k_col[slot] = inv_col[col[e]];
        L->k_src[slot] = (int32_t)e;
      }
    }
  }

  // ---- K^T in sliced ELL over internal columns (entries by ascending row) ----
  std::vector<int64_t> cptr(n + 1, 0);
  for (int64_t j = 0; j < n; ++j) cptr[j + 1] = cptr[j] + clen[j];
  std::vector<int32_t> crow(col.size()), csrc(col.size());
  {
    std::vector<int64_t> fill(cptr.begin(), cptr.end() - 1);
    for (int64_t i = 0; i < m; ++i)
      for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
        int64_t pos = fill[col[e]]++;
        crow[pos] = (int32_t)i;
        csrc[pos] = (int32_t)e;
      }
  }
  const int64_t ts = slice_offsets_of(clen, L->perm_col, &L->t_off);
  if (ts < 0) {
    *err = "padded nnz of K^T exceeds 2^31";
    return PDHG_ERR_UNSUPPORTED;
  }
  tot = L->t_off[ts];
  L->t_col.assign(tot, 0);
  L->t_src.assign(tot, -1);
  for (int64_t s = 0; s < ts; ++s) {
    for (int lane = 0; lane < kSlice; ++lane) {
      int64_t j = s * kSlice + lane;
      if (j >= n) continue;
      int32_t o = L->perm_col[j];
      for (int64_t k = 0; k < clen[o]; ++k) {
        int64_t slot = L->t_off[s] + k * kSlice + lane;
        L->t_col[slot] = inv_row[crow[cptr[o] + k]];
        L->t_src[slot] = csrc[cptr[o] + k];
      }
    }
  }
  build_runs(L->k_off, L->k_col, L->k_src, n, &L->k_soff, &L->k_runs);
  build_runs(L->t_off, L->t_col, L->t_src, m, &L->t_soff, &L->t_runs);
  return PDHG_OK;
}

bool build_chunks(const std::vector<int32_t>& off, std::vector<int32_t>* chunks, int max_entries,
                  int max_slices) {
  chunks->clear();
  const int32_t ns = (int32_t)off.size() - 1;
  chunks->push_back(0);
  int32_t s0 = 0;
  for (int32_t s = 0; s < ns; ++s) {
    if (off[s + 1] - off[s] > max_entries) {
      chunks->clear();
      return false;
    }
    if (off[s + 1] - off[s0] > max_entries || s + 1 - s0 > max_slices) {
      chunks->push_back(s);
      s0 = s;
    }
  }
  if (ns > 0) chunks->push_back(ns);
  return true;
}

// ---------------------------------------------------------------------------
// kernels of the preparation pass

__global__ void k_load_vals(const int32_t* __restrict__ ksrc, const int32_t* __restrict__ tsrc,
                            const double* __restrict__ csr, double* __restrict__ kval,
                            double* __restrict__ tval, int64_t nk, int64_t nt) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nk + nt;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = t < nk ? ksrc[t] : tsrc[t - nk];
    (t < nk ? kval : tval - nk)[t] = (e >= 0) ? csr[e] : 0.0;
  }
}

__global__ void k_load_vecs(const int32_t* __restrict__ perm_col, const int32_t* __restrict__ perm_row,
                            const double* c, const double* l, const double* u, const double* q,
                            double* c_s, double* l_s, double* u_s, double* q_s, double* Dr,
                            double* Dc, int64_t n, int64_t m) {
  int64_t N = n > m ? n : m;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N;
       t += (int64_t)gridDim.x * blockDim.x) {
    if (t < n) {
      int32_t o = perm_col[t];
      c_s[t] = c[o];
      l_s[t] = l[o];
      u_s[t] = u[o];
      Dc[t] = 1.0;
    }
    if (t < m) {
      q_s[t] = q[perm_row[t]];
      Dr[t] = 1.0;
    }
  }
}

// One pass of the rescaling for both sides at once: per internal row of K and of
// K^T the max (Ruiz) or the sum (Pock-Chambolle) of |A_ij| drow_i dcol_j, and the
// row's new factor drow_i / sqrt(stat) (unchanged for an empty row), written to
// the other buffer so that both sides see the old factors.
// FP64-pipe bound (see common.cuh): one product per entry (the row's own factor
// is taken out of the max or sum), the max on the integer pipe, one reciprocal
// square root per row.  6717 buses, 96 periods, both sides: 314 us in four launches
// before, 134 us now.
template <bool SUM>
__global__ void __launch_bounds__(kBlock) k_scale_pass(SellView<double> K, SellView<double> KT,
                                                       const double* __restrict__ dr, const double* __restrict__ dc,
                                                       double* __restrict__ dr_new, double* __restrict__ dc_new) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  for (int t = gw; t < K.nslices + KT.nslices; t += nw) {
    const bool rows = t < K.nslices;
    const SellView<double>& A = rows ? K : KT;
    const double* __restrict__ dcol = rows ? dc : dr;
    const int s = rows ? t : t - K.nslices;
    const int o = A.off[s] + lane, w = (A.off[s + 1] - A.off[s]) >> 5;
    const int r = s * kSlice + lane;
    const double d = r < A.rows ? (rows ? dr : dc)[r] : 0.0;
    double sum = 0.0;
    unsigned long long top = 0;  // non-negative doubles compare as integers
    for (int k0 = 0; k0 < w; k0 += 4) {
      double v[4], c[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool ok = k0 + e < w;
        v[e] = ok ? __ldg(A.val + o + (k0 + e) * kSlice) : 0.0;
        c[e] = ok ? __ldg(dcol + __ldg(A.col + o + (k0 + e) * kSlice)) : 0.0;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (SUM) {
          sum += fabs(v[e]) * c[e];
        } else {
          const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v[e]) * c[e]);
          if (b > top && b <= 0x7ff0000000000000ull) top = b;  // a NaN is passed over, as by fmax
        }
      }
    }
    if (r < A.rows) {
      const double stat = (SUM ? sum : __longlong_as_double((long long)top)) * d;
      (rows ? dr_new : dc_new)[r] = stat > 0.0 ? d * rsqrt(stat) : d;
    }
  }
}

// K~ = K (drow_i dcol_j); the product of the two factors is formed first so that
// K and K^T get bit-identical values.  Both matrices in one launch, with the FP32
// copy (val32 not null) and max |K~| per block of the sweep over K.
__global__ void __launch_bounds__(kBlock) k_scale_vals(SellView<double> K, SellView<double> KT, double* kval,
                                                       double* tval, float* kval32, float* tval32,
                                                       const double* __restrict__ dr, const double* __restrict__ dc,
                                                       double* max_partials) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nw = (gridDim.x * kBlock) >> 5;
  unsigned long long top = 0;
  for (int t = gw; t < K.nslices + KT.nslices; t += nw) {
    const bool rows = t < K.nslices;
    const SellView<double>& A = rows ? K : KT;
    const double* __restrict__ dcol = rows ? dc : dr;
    double* val = rows ? kval : tval;
    float* val32 = rows ? kval32 : tval32;
    const int s = rows ? t : t - K.nslices;
    const int o = A.off[s] + lane, w = (A.off[s + 1] - A.off[s]) >> 5;
    const int r = s * kSlice + lane;
    const bool in = r < A.rows;  // padding rows hold zeros
    const double d = in ? (rows ? dr : dc)[r] : 0.0;
    for (int k0 = 0; k0 < w; k0 += 4) {
      double v[4], c[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool ok = k0 + e < w;
        v[e] = ok ? val[o + (k0 + e) * kSlice] : 0.0;
        c[e] = ok ? __ldg(dcol + __ldg(A.col + o + (k0 + e) * kSlice)) : 0.0;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (k0 + e < w) {
          const double x = in ? v[e] * (d * c[e]) : 0.0;
          val[o + (k0 + e) * kSlice] = x;
          if (val32) val32[o + (k0 + e) * kSlice] = (float)x;
          const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(x));
          if (rows && b > top && b <= 0x7ff0000000000000ull) top = b;
        }
    }
  }
#pragma unroll
  for (int q = 16; q > 0; q >>= 1) {
    const unsigned long long b = __shfl_down_sync(0xffffffffu, top, q);
    if (b > top) top = b;
  }
  __shared__ unsigned long long sm[kWarps];
  if (lane == 0) sm[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < kWarps; ++q)
      if (sm[q] > top) top = sm[q];
    max_partials[blockIdx.x] = __longlong_as_double((long long)top);
  }
}

// Scaled vectors plus the norms ||c||, ||q|| (unscaled) and ||c~||, ||q~||, and
// max |K~| as per-block partials (deterministic final pass in k_prepare_final).
__global__ void k_scale_vecs(double* c_s, double* l_s, double* u_s, double* q_s,
                             const double* __restrict__ Dr, const double* __restrict__ Dc, int64_t n,
                             int64_t m, double* partials, double* iDr, double* iDc) {
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t N = n > m ? n : m;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N;
       t += (int64_t)gridDim.x * blockDim.x) {
    if (t < n) {
      double c = c_s[t], d = Dc[t];
      v[0] += c * c;
      double cs = d * c;
      c_s[t] = cs;
      v[2] += cs * cs;
      iDc[t] = 1.0 / d;
      // most bounds are 0 or infinite and stay so: no division for those
      const double l = l_s[t], u = u_s[t];
      if (finite_bits(l) && non_zero(l)) l_s[t] = l / d;
      if (finite_bits(u) && non_zero(u)) u_s[t] = u / d;
    }
    if (t < m) {
      double q = q_s[t];
      v[1] += q * q;
      iDr[t] = 1.0 / Dr[t];
      double qs = Dr[t] * q;
      q_s[t] = qs;
      v[3] += qs * qs;
    }
  }
  __shared__ double smem[kWarps * 4];
  block_sum<4>(v, smem);
  if (threadIdx.x == 0)
    for (int k = 0; k < 4; ++k) partials[blockIdx.x * 4 + k] = v[k];
}

// scalars[0] = eta0 = 1/max|K~|, [1] = omega0, [2] = ||q||, [3] = ||c||,
// [4] = ||c~||, [5] = ||q~||.
__global__ void k_prepare_final(const double* vec_partials, int nb_vec, const double* max_partials,
                                int nb_max, double* scalars) {
  double v[4];
  final_sum<4>(vec_partials, nb_vec, v);
  __shared__ double mx_s[kWarps];
  double mx = 0.0;
  for (int b = threadIdx.x; b < nb_max; b += blockDim.x) mx = fmax(mx, max_partials[b]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) mx_s[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int t = 0; t < kWarps; ++t) r = fmax(r, mx_s[t]);
    double cn = sqrt(v[2]), qn = sqrt(v[3]);
    scalars[0] = r > 0.0 ? 1.0 / r : 1.0;
    scalars[1] = (cn > 1e-10 && qn > 1e-10) ? cn / qn : 1.0;
    scalars[2] = sqrt(v[1]);
    scalars[3] = sqrt(v[0]);
    scalars[4] = cn;
    scalars[5] = qn;
  }
}

template <class T>
__global__ void k_gather_perm(const int32_t* __restrict__ perm, const double* __restrict__ in,
                              T* __restrict__ out, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    out[t] = (T)in[perm[t]];
}

__global__ void k_scatter_perm(const int32_t* __restrict__ perm, const double* __restrict__ in,
                               double* __restrict__ out, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    out[perm[t]] = in[t];
}

// ---------------------------------------------------------------------------
// launchers

static int vec_grid(int64_t n, int sms) {
  int64_t g = (n + kBlock - 1) / kBlock;
  int64_t cap = (int64_t)sms * 8;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

template <class T>
void launch_gather_perm(const int32_t* perm, const double* in, T* out, int64_t n, cudaStream_t s) {
  k_gather_perm<T><<<vec_grid(n, 152), kBlock, 0, s>>>(perm, in, out, n);
}
template void launch_gather_perm<double>(const int32_t*, const double*, double*, int64_t, cudaStream_t);
template void launch_gather_perm<float>(const int32_t*, const double*, float*, int64_t, cudaStream_t);
void launch_scatter_perm(const int32_t* perm, const double* in, double* out, int64_t n,
                         cudaStream_t s) {
  k_scatter_perm<<<vec_grid(n, 152), kBlock, 0, s>>>(perm, in, out, n);
}

void launch_prepare(Workspace* w, bool f32, cudaStream_t s) {
  const int sms = w->num_sms;
  const int passes = w->opts.ruiz_iters + (w->opts.pock_chambolle ? 1 : 0);
  // sweeps over both matrices, one slice per warp (blocks retire at their own pace)
  const int64_t need = ((int64_t)w->K.nslices + w->KT.nslices + kWarps - 1) / kWarps;
  const int gs = (int)std::min<int64_t>(need, (int64_t)sms * 16);
  k_load_vals<<<vec_grid(w->K.nnz_pad + w->KT.nnz_pad, sms), kBlock, 0, s>>>(
      w->K.src, w->KT.src, w->prob.val, w->K.val64, w->KT.val64, w->K.nnz_pad, w->KT.nnz_pad);
  const int64_t N = w->n > w->m ? w->n : w->m;
  k_load_vecs<<<vec_grid(N, sms), kBlock, 0, s>>>(w->perm_col, w->perm_row, w->prob.c, w->prob.l,
                                                  w->prob.u, w->prob.q, w->c_s, w->l_s, w->u_s,
                                                  w->q_s, (passes & 1) ? w->fac_r : w->Dr,
                                                  (passes & 1) ? w->fac_c : w->Dc, w->n, w->m);
  // the factors change sides every pass and end in Dr, Dc
  for (int p = 0; p < passes; ++p) {
    const bool odd = (passes - p) & 1;
    const double *dr = odd ? w->fac_r : w->Dr, *dc = odd ? w->fac_c : w->Dc;
    double *dr_new = odd ? w->Dr : w->fac_r, *dc_new = odd ? w->Dc : w->fac_c;
    if (p >= w->opts.ruiz_iters)
      k_scale_pass<true><<<gs, kBlock, 0, s>>>(w->K.v64(), w->KT.v64(), dr, dc, dr_new, dc_new);
    else
      k_scale_pass<false><<<gs, kBlock, 0, s>>>(w->K.v64(), w->KT.v64(), dr, dc, dr_new, dc_new);
  }
  double* part_vec = w->partials;
  double* part_max = w->partials + (size_t)kMaxBlocks * kRegionStride;
  k_scale_vals<<<gs, kBlock, 0, s>>>(w->K.v64(), w->KT.v64(), w->K.val64, w->KT.val64, f32 ? w->K.val32 : nullptr,
                                     f32 ? w->KT.val32 : nullptr, w->Dr, w->Dc, part_max);
  const int gv = vec_grid(N, sms);
  k_scale_vecs<<<gv, kBlock, 0, s>>>(w->c_s, w->l_s, w->u_s, w->q_s, w->Dr, w->Dc, w->n, w->m,
                                     part_vec, w->iDr, w->iDc);
  k_prepare_final<<<1, kBlock, 0, s>>>(part_vec, gv, part_max, gs, w->scalars);
  w->values_f32 = f32;
}

}  // namespace ucpdhg
