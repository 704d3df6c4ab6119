// Internal layout (length-sorted orderings, sliced ELL) and the rescaling pass.
//
// Rows of K are reordered by (about) decreasing length inside the equality block
// and inside the inequality block, columns by decreasing column count, so that each
// 32-row slice holds rows of (nearly) equal length and padding stays small on the
// UC sparsity (rows of 2 to ~25 entries); rows (columns) of one kind stay together
// in time order so that a slice's gathers are contiguous (build_layout): 3 % padding
// on the 6717-bus day, 1 % with strictly equal lengths, but all k-columns of K and
// nearly all of K^T are then runs instead of 58 % of the entries, which took the
// FP32 sweeps from 39.7 + 29.5 to 36.9 + 22.8 us.  K and
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
#include <system_error>
#include <thread>

#include "internal.cuh"

namespace ucpdhg {

namespace {

// Finalizer of a 64-bit hash (the multiply-xorshift of SplitMix64).
inline uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// Groups of equal keys of the ids first, first + 1, ..., numbered by first
// occurrence (open addressing).
struct Groups {
  std::vector<int32_t> of;          // group of each id
  std::vector<int32_t> rep;         // a member
  std::vector<int32_t> size, most;  // members, longest length
  std::vector<int64_t> total;       // entries
};
Groups group_by(int64_t first, int64_t count, const std::vector<int32_t>& len, const std::vector<uint64_t>& key) {
  Groups g;
  size_t cap = 16;
  while (cap < (size_t)count * 2) cap <<= 1;
  std::vector<int32_t> table(cap, -1);
  g.of.resize(count);
  for (int64_t t = 0; t < count; ++t) {
    const int64_t i = first + t;
    size_t h = mix64(key[i]) & (cap - 1);
    while (table[h] >= 0 && key[g.rep[table[h]]] != key[i]) h = (h + 1) & (cap - 1);
    if (table[h] < 0) {
      table[h] = (int32_t)g.rep.size();
      g.rep.push_back((int32_t)i);
      g.size.push_back(0);
      g.most.push_back(0);
      g.total.push_back(0);
    }
    const int32_t q = table[h];
    g.of[t] = q;
    ++g.size[q];
    g.most[q] = std::max(g.most[q], len[i]);
    g.total[q] += len[i];
  }
  return g;
}

// Internal order of a set of rows (columns): groups of equal keys by decreasing
// longest length, equal lengths as they first occur, members in their original
// order.  A group whose members differ so much in length that padding them to the
// longest would cost more than a quarter of its entries is split by length.
void order_by_key(int64_t first, int64_t count, const std::vector<int32_t>& len, std::vector<uint64_t>& key,
                  int32_t* perm) {
  if (count == 0) return;
  Groups g = group_by(first, count, len, key);
  bool split = false;
  for (int64_t t = 0; t < count; ++t) {
    const int32_t q = g.of[t];
    if ((int64_t)g.most[q] * g.size[q] * 4 > g.total[q] * 5) {
      key[first + t] = mix64(key[first + t] + (uint64_t)len[first + t] + 1);
      split = true;
    }
  }
  if (split) g = group_by(first, count, len, key);
  std::vector<int32_t> order(g.rep.size());
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return g.most[a] > g.most[b]; });
  std::vector<int64_t> pos(g.rep.size());
  int64_t at = 0;
  for (int32_t q : order) {
    pos[q] = at;
    at += g.size[q];
  }
  for (int64_t t = 0; t < count; ++t) perm[pos[g.of[t]]++] = (int32_t)(first + t);
}

// The distance between one column and the next of its group that more than half
// of such pairs have: the columns per period of a time-expanded model.  0: none.
int64_t period_of(const Groups& g, int64_t n) {
  std::vector<int32_t> last(g.rep.size(), -1);
  int64_t cand = 0, votes = 0, pairs = 0, hits = 0;
  for (int pass = 0; pass < 2; ++pass) {
    std::fill(last.begin(), last.end(), -1);
    for (int64_t j = 0; j < n; ++j) {
      const int32_t prev = last[g.of[j]];
      last[g.of[j]] = (int32_t)j;
      if (prev < 0) continue;
      const int64_t d = j - prev;
      if (pass == 0) {  // majority vote
        if (votes == 0) cand = d;
        votes += d == cand ? 1 : -1;
      } else {
        ++pairs;
        hits += d == cand;
      }
    }
  }
  return hits * 2 > pairs && pairs * 2 > n ? cand : 0;
}

// Offsets of the 32-row slices over the internal order.  Slices come in aligned
// groups of kGroup of one width, so that a warp sweeping a group (or half of one)
// finds its entries at fixed distances.  A group whose slices keep their own widths
// (own, or where the common one would add more than a quarter to its slots and more
// than kOwnPadding k-columns: a row far longer than its neighbours, such as a budget
// or reserve row, would pad 128 rows instead of 32) is swept slice by slice: 40000
// columns and one full row take 1.4 instead of 5.2 million slots.  The second
// condition leaves rows of up to 42 entries in groups of one width whatever their
// neighbours (all of the scheduling LPs here: 28 at most).  Returns the number of slices (a multiple of kGroup), -1 if the
// entries exceed 2^31.
constexpr int64_t kOwnPadding = 128;
int64_t slice_offsets_of(const std::vector<int32_t>& len, const std::vector<int32_t>& perm, bool own,
                         std::vector<int32_t>* off) {
  const int64_t rows = (int64_t)perm.size();
  const int64_t ng = (rows + kSlice * kGroup - 1) / (kSlice * kGroup);
  off->assign(ng * kGroup + 1, 0);
  int64_t tot = 0;
  for (int64_t g = 0; g < ng; ++g) {
    int32_t w[kGroup], most = 0;
    int64_t sum = 0;
    for (int s = 0; s < kGroup; ++s) {
      const int64_t first = (g * kGroup + s) * kSlice;
      w[s] = 0;
      for (int64_t i = first; i < std::min(rows, first + kSlice); ++i) w[s] = std::max(w[s], len[perm[i]]);
      most = std::max(most, w[s]);
      sum += w[s];
    }
    const int64_t pad = (int64_t)most * kGroup - sum;
    const bool one = !own && (pad * 4 <= sum || pad <= kOwnPadding);
    for (int s = 0; s < kGroup; ++s) {
      tot += (int64_t)(one ? most : w[s]) * kSlice;
      if (tot >= (int64_t)1 << 31) return -1;
      (*off)[g * kGroup + s + 1] = (int32_t)tot;
    }
  }
  return ng * kGroup;
}

// Returns whether some groups keep a width per slice.
bool size_slots(const std::vector<int32_t>& off, std::vector<int32_t>* col, std::vector<int32_t>* src,
                std::vector<int32_t>* soff, std::vector<int32_t>* runs) {
  col->assign(off.back(), 0);
  src->assign(off.back(), -1);
  runs->assign((size_t)off.back() / kSlice * 2, 0);
  soff->assign(off.begin(), off.end());
  bool any = false;
  for (size_t g = 0; g + kGroup < off.size(); g += kGroup) {
    bool own = false;
    for (int s = 1; s < kGroup; ++s) own = own || off[g + s + 1] - off[g + s] != off[g + 1] - off[g];
    for (int s = 0; own && s < kGroup; ++s) (*soff)[g + s] |= kRunsOwn;
    any = any || own;
  }
  return any;
}

// Entries of the rows into their slots.  A row shorter than its slice sits at the
// front or at the back of its slots, whichever continues more of the previous
// row's columns (the horizon cuts minimum up time rows at their front, the columns
// of the same variables at their back).
template <class Col, class Src>
void place_entries(int64_t rows, const std::vector<int32_t>& perm, const std::vector<int32_t>& len,
                   const std::vector<int32_t>& off, Col&& col_of, Src&& src_of, std::vector<int32_t>* col,
                   std::vector<int32_t>* src) {
  for (int64_t i = 0; i < rows; ++i) {
    const int64_t s = i / kSlice, lane = i % kSlice;
    const int32_t o = perm[i], n = len[o], w = (off[s + 1] - off[s]) / kSlice;
    int32_t front = 0;
    if (n < w && i > 0) {
      const int64_t q = (i - 1) / kSlice, p0 = off[q] + (i - 1) % kSlice;
      const int32_t pw = (off[q + 1] - off[q]) / kSlice;
      int hits[2] = {0, 0};
      for (int at = 0; at < 2; ++at)
        for (int32_t k = 0; k < n; ++k) {
          const int32_t t = k + (at ? w - n : 0);
          if (t < pw && (*src)[p0 + (int64_t)t * kSlice] >= 0 &&
              (*col)[p0 + (int64_t)t * kSlice] + 1 == col_of(o, k))
            ++hits[at];
        }
      if (hits[1] > hits[0]) front = w - n;
    }
    if (n < w && i + 1 < rows && front == 0) {
      // the first of a run has only its successor to go by: the row after it, if longer
      const int32_t on = perm[i + 1], nn = len[on];
      if (nn > n && nn <= w) {
        int hits[2] = {0, 0};
        for (int at = 0; at < 2; ++at)
          for (int32_t k = 0; k < n; ++k)
            if (col_of(o, k) + 1 == col_of(on, k + (at ? nn - n : 0))) ++hits[at];
        if (hits[1] > hits[0]) front = w - n;
      }
    }
    for (int32_t k = 0; k < n; ++k) {
      const int64_t slot = off[s] + (int64_t)(front + k) * kSlice + lane;
      (*col)[slot] = col_of(o, k);
      (*src)[slot] = src_of(o, k);
    }
  }
}

// Column runs of a sliced-ELL matrix (see SellView::runs).  Groups with more than a
// quarter of their k-columns in more than two runs keep to the indices.
void build_runs(const std::vector<int32_t>& off, const std::vector<int32_t>& col,
                const std::vector<int32_t>& src, int64_t ncols, std::vector<int32_t>* soff,
                std::vector<int32_t>* runs) {
  const int64_t ns = (int64_t)off.size() - 1;
  if (ncols >= ((int64_t)1 << kRunBits)) return;
  for (int64_t g = 0; g < ns; g += kGroup) {
    const int64_t o0 = off[g], o1 = off[g + kGroup];
    if (((*soff)[g] & (kSlice - 1)) == kRunsOwn) continue;
    int64_t two = 0, more = 0;
    for (int64_t o = o0; o < o1; o += kSlice) {
      int32_t prev = -1, start[2] = {0, 0}, split = kSlice, pieces = 0;
      for (int lane = 0; lane < kSlice; ++lane) {
        // a padding slot (value 0) continues the run it follows, inside the vector
        int32_t c = col[o + lane];
        if (src[o + lane] < 0) c = (lane > 0 && prev + 1 < ncols) ? prev + 1 : 0;
        if (lane == 0 || c != prev + 1) {
          if (pieces < 2) start[pieces] = c;
          if (++pieces == 2) split = lane;
        }
        prev = c;
      }
      if (pieces == 2) ++two;
      if (pieces > 2) {
        ++more;
        split = 0;  // the indices
      }
      (*runs)[o / kSlice * 2] = start[0];
      (*runs)[o / kSlice * 2 + 1] = (int32_t)(((uint32_t)split << kRunBits) | (uint32_t)start[1]);
    }
    const int mode = more * 4 > (o1 - o0) / kSlice ? kRunsNone
                     : more                        ? kRunsMixed
                     : two                         ? kRunsTwo
                                                   : kRunsOne;
    for (int s = 0; s < kGroup; ++s) (*soff)[g + s] |= mode;
  }
}

// The internal order of rows and columns and the slices' offsets; rlen and clen
// receive the lengths.
int order_layout(int64_t n, int64_t m, int64_t m_eq, const std::vector<int64_t>& rp,
                 const std::vector<int32_t>& col, const std::vector<double>& val, HostLayout* L,
                 std::vector<int32_t>* rlen_out, std::vector<int32_t>* clen_out, std::string* err) {
  std::vector<int32_t>&rlen = *rlen_out, &clen = *clen_out;
  rlen.assign(m, 0);
  clen.assign(n, 0);
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
  // time and row r + 1 gathers column c + 1 where row r gathers column c.
  for (int64_t i = 0; i < m; ++i) {
    rlen[i] = (int32_t)(rp[i + 1] - rp[i]);
    uint64_t h = (uint64_t)rlen[i];
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
      uint64_t bits;
      std::memcpy(&bits, &val[e], sizeof(bits));
      h = mix64(h + (uint64_t)(col[e] - col[rp[i]]) + 0x9E3779B97F4A7C15ULL) + bits;
    }
    rsig[i] = mix64(h);
    for (int64_t e = rp[i]; e < rp[i + 1]; ++e) csig[col[e]] += mix64(rsig[i] + (uint64_t)(e - rp[i]));
  }
  const Groups cg = group_by(0, n, clen, csig);
  const int64_t period = period_of(cg, n);
  if (period > 1) {
    // Columns of one place in the period, rows of one kind at one place: the
    // places of their first, last and last but one column and the end values.
    // These do not change where the horizon cuts a row short (minimum up and down
    // times), so such rows and the columns that lose them keep their places in
    // the run of their unit, padded, instead of scattering over the lengths.
    for (int64_t j = 0; j < n; ++j) csig[j] = (uint64_t)(j % period);
    for (int64_t i = 0; i < m; ++i) {
      const int64_t b = rp[i], e = rp[i + 1];
      uint64_t h = e > b ? 1 : 0;
      if (e > b) {
        uint64_t v0, v1;
        std::memcpy(&v0, &val[b], sizeof(v0));
        std::memcpy(&v1, &val[e - 1], sizeof(v1));
        h = mix64(h + (uint64_t)(col[b] % period)) + v0;
        h = mix64(h + (uint64_t)(col[e - 1] % period)) + v1;
        if (e - b > 1) h = mix64(h + (uint64_t)(col[e - 2] % period));
      }
      rsig[i] = mix64(h);
    }
  } else {
    // Rows that differ only in the unit they belong to are told apart by the
    // signature of the column with the most members
    for (int64_t i = 0; i < m; ++i) {
      int32_t best = -1;
      for (int64_t e = rp[i]; e < rp[i + 1]; ++e)
        if (best < 0 || cg.size[cg.of[col[e]]] > cg.size[cg.of[best]]) best = col[e];
      if (best >= 0) rsig[i] = mix64(rsig[i] + csig[best]);
    }
    for (int64_t j = 0; j < n; ++j) csig[j] = mix64(csig[j] + (uint64_t)clen[j]);
  }
  L->perm_row.resize(m);
  order_by_key(0, m_eq, rlen, rsig, L->perm_row.data());
  order_by_key(m_eq, m - m_eq, rlen, rsig, L->perm_row.data() + m_eq);
  L->perm_col.resize(n);
  order_by_key(0, n, clen, csig, L->perm_col.data());
  if (slice_offsets_of(rlen, L->perm_row, false, &L->k_off) >= 0 &&
      slice_offsets_of(clen, L->perm_col, false, &L->t_off) >= 0)
    return PDHG_OK;
  // The order above pads rows of one kind to one length and slices to groups.  What
  // only fits below 2^31 slots without that is ordered by length alone.
  const auto by_length = [](std::vector<int32_t>* perm, int64_t first, int64_t last, const std::vector<int32_t>& len) {
    std::iota(perm->begin() + first, perm->begin() + last, (int32_t)first);
    std::stable_sort(perm->begin() + first, perm->begin() + last,
                     [&](int32_t a, int32_t b) { return len[a] > len[b]; });
  };
  by_length(&L->perm_row, 0, m_eq, rlen);
  by_length(&L->perm_row, m_eq, m, rlen);
  by_length(&L->perm_col, 0, n, clen);
  const char* over = slice_offsets_of(rlen, L->perm_row, true, &L->k_off) < 0   ? "K"
                     : slice_offsets_of(clen, L->perm_col, true, &L->t_off) < 0 ? "K^T"
                                                                                : nullptr;
  if (!over) return PDHG_OK;
  *err = std::string("padded nnz of ") + over + " exceeds 2^31";
  return PDHG_ERR_UNSUPPORTED;
}

}  // namespace

int count_slots(int64_t n, int64_t m, int64_t m_eq, const std::vector<int64_t>& rp, const std::vector<int32_t>& col,
                const std::vector<double>& val, int64_t* slots_k, int64_t* slots_kt, std::string* err) {
  HostLayout L;
  std::vector<int32_t> rlen, clen;
  const int rc = order_layout(n, m, m_eq, rp, col, val, &L, &rlen, &clen, err);
  if (rc != PDHG_OK) return rc;
  *slots_k = L.k_off.back();
  *slots_kt = L.t_off.back();
  return PDHG_OK;
}

int build_layout(int64_t n, int64_t m, int64_t m_eq, const std::vector<int64_t>& rp,
                 const std::vector<int32_t>& col, const std::vector<double>& val, HostLayout* L,
                 std::string* err) {
  std::vector<int32_t> rlen, clen;
  const int rc = order_layout(n, m, m_eq, rp, col, val, L, &rlen, &clen, err);
  if (rc != PDHG_OK) return rc;
  std::vector<int32_t> inv_row(m), inv_col(n);
  for (int64_t i = 0; i < m; ++i) inv_row[L->perm_row[i]] = (int32_t)i;
  for (int64_t j = 0; j < n; ++j) inv_col[L->perm_col[j]] = (int32_t)j;

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
  const auto widest = [](const std::vector<int32_t>& off) {
    int32_t w = 0;
    for (size_t t = 0; t + 1 < off.size(); ++t) w = std::max(w, (off[t + 1] - off[t]) / kSlice);
    return w;
  };
  L->k_wide = widest(L->k_off);
  L->t_wide = widest(L->t_off);
  L->k_own = size_slots(L->k_off, &L->k_col, &L->k_src, &L->k_soff, &L->k_runs);
  L->t_own = size_slots(L->t_off, &L->t_col, &L->t_src, &L->t_soff, &L->t_runs);
  // the two matrices side by side; nothing here allocates or throws
  const auto fill_k = [&]() noexcept {
    place_entries(
        m, L->perm_row, rlen, L->k_off, [&](int64_t o, int32_t k) { return inv_col[col[rp[o] + k]]; },
        [&](int64_t o, int32_t k) { return (int32_t)(rp[o] + k); }, &L->k_col, &L->k_src);
    build_runs(L->k_off, L->k_col, L->k_src, n, &L->k_soff, &L->k_runs);
  };
  std::thread other;
  if (col.size() > (1u << 18)) {  // below, starting a thread costs what it saves
    try {
      other = std::thread(fill_k);
    } catch (const std::system_error&) {
    }
  }
  if (!other.joinable()) fill_k();
  place_entries(
      n, L->perm_col, clen, L->t_off, [&](int64_t o, int32_t k) { return inv_row[crow[cptr[o] + k]]; },
      [&](int64_t o, int32_t k) { return csrc[cptr[o] + k]; }, &L->t_col, &L->t_src);
  build_runs(L->t_off, L->t_col, L->t_src, m, &L->t_soff, &L->t_runs);
  if (other.joinable()) other.join();
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
    const double v = e >= 0 ? csr[e] : 0.0;
    (t < nk ? kval : tval - nk)[t] = e < 0 ? -0.0 : non_zero(v) ? v : 0.0;
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
