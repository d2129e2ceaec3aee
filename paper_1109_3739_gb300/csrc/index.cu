// index.cu -- device pieces of SpRef and SpAsgn (Section 3.1).
//
// The selection matrices of the SpRef and SpAsgn listings are built on the
// device in CSR form (the constructor sparse(i, j, 1, m, n) for their
// special shapes):
//   SpRef  R = sparse(1:len(I), I, 1, len(I), m)  -> row t holds column I[t]
//          Q = sparse(J, 1:len(J), 1, n, len(J))  -> row k holds every p with
//                                                    J[p] == k, increasing
//   SpAsgn R = sparse(I, 1:mb, 1, ma, mb)         -> row I[q] holds column q
//          Q = sparse(1:nb, J, 1, nb, na)         -> row q holds column J[q]
// and the final step of SpAsgn, the elementwise product of A with the
// structural negation of S*A*T plus R*B*Q: an entry (r, c) of A is in the
// structure of S*A*T exactly when r is in I and c is in J, so the negation is
// applied through I and the inverse index map cpos, and neither S*A*T nor its
// negation is ever materialised (Section 3.1).  Nor is R*B*Q, when B's rows
// keep their order under J: its entries are B's, moved to rows I and columns J.
#include "common.cuh"
#include "internal.h"

namespace hs {

static int grid1(int64_t n, int nt = 256) {
  int64_t g = (n + nt - 1) / nt;
  int64_t cap = (int64_t)sm_count() * 16;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

#define GRID_STRIDE(i, n) \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

__global__ void k_iota_i64(int64_t *p, int64_t n) { GRID_STRIDE(i, n) p[i] = i; }

__global__ void k_fill_i32(int32_t *a, int64_t n, int32_t v) { GRID_STRIDE(i, n) a[i] = v; }
void launch_fill_i32(int32_t *a, int64_t n, int32_t v, cudaStream_t st) {
  if (n > 0) {
    count_launch();
    k_fill_i32<<<grid1(n), 256, 0, st>>>(a, n, v);
  }
}

__global__ void k_iota_i32(int32_t *p, int64_t n) { GRID_STRIDE(i, n) p[i] = (int32_t)i; }
void launch_iota_i32(int32_t *p, int64_t n, cudaStream_t st) {
  if (n > 0) {
    count_launch();
    k_iota_i32<<<grid1(n), 256, 0, st>>>(p, n);
  }
}

// Q of SpRef: counts per row k go to Qp[k+1]; indices outside [0, bound)
// are skipped (the host reports them), so this may run before the range check
__global__ void k_count_idx(const int32_t *X, int64_t n, int64_t bound, int64_t *cnt) {
  GRID_STRIDE(i, n) {
    const int32_t x = X[i];
    if (x >= 0 && x < bound) atomicAdd(reinterpret_cast<unsigned long long *>(cnt + x + 1), 1ull);
  }
}
void launch_build_Q_count(const int32_t *J, int64_t nJ, int64_t bound, int64_t *Qp_counts, cudaStream_t st) {
  if (nJ > 0) {
    count_launch();
    k_count_idx<<<grid1(nJ), 256, 0, st>>>(J, nJ, bound, Qp_counts);
  }
}
// the largest of n counts, into *out (zeroed by the caller)
__global__ void k_max_count(const int64_t *cnt, int64_t n, unsigned long long *out) {
  unsigned long long mx = 0;
  GRID_STRIDE(i, n) mx = max(mx, (unsigned long long)cnt[i]);
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(out, mx);
}
void launch_max_count(const int64_t *cnt, int64_t n, unsigned long long *out, cudaStream_t st) {
  if (n <= 0) return;
  count_launch();
  k_max_count<<<grid1(n), 256, 0, st>>>(cnt, n, out);
}

// Q of SpRef: cur holds the row offsets on entry and is advanced by atomics;
// rows are then put in increasing order of p by an insertion sort, used only
// when no row holds more than 32 entries (one per repetition of k in J)
__global__ void k_fill_idx(const int32_t *X, int64_t n, int64_t *cur, int32_t *out) {
  GRID_STRIDE(i, n) {
    const unsigned long long at = atomicAdd(reinterpret_cast<unsigned long long *>(cur + X[i]), 1ull);
    out[at] = (int32_t)i;
  }
}
__global__ void k_sort_short_rows(const int64_t *ptr, int32_t *j, int64_t rows) {
  GRID_STRIDE(r, rows) {
    const int64_t b = ptr[r], e = ptr[r + 1];
    for (int64_t x = b + 1; x < e; ++x) {
      const int32_t v = j[x];
      int64_t y = x - 1;
      while (y >= b && j[y] > v) {
        j[y + 1] = j[y];
        --y;
      }
      j[y + 1] = v;
    }
  }
}
// Qcur: a copy of the finished offsets (length n+1); Qj is sorted per row
// using the offsets that precede Qcur in the caller's layout (Qcur - (n+1))
void launch_build_Q_fill(const int32_t *J, int64_t nJ, int64_t *Qcur, int32_t *Qj, cudaStream_t st) {
  if (nJ > 0) {
    count_launch();
    k_fill_idx<<<grid1(nJ), 256, 0, st>>>(J, nJ, Qcur, Qj);
  }
}
void launch_sort_short_rows(const int64_t *ptr, int32_t *j, int64_t rows, cudaStream_t st) {
  if (rows > 0) {
    count_launch();
    k_sort_short_rows<<<grid1(rows), 256, 0, st>>>(ptr, j, rows);
  }
}

// ----------------------------------------------------- SpRef by gathering
// B = A(I, J) without forming R*A: the rows I[t] of A are laid end to end
// (gathered entry g of output row t is entry A.p[I[t]] + g - G[t] of A,
// G the scanned row lengths), every gathered entry (t, c, v) becomes one
// tuple (t, p, v) for each p with J[p] == c (Q's row c), and the tuples are
// sorted by (t, p) -- or, when J is strictly increasing, written in place,
// already in order.

// G[t + 1] = length of row I[t] (G[0] is zero)
__global__ void k_gather_len(const int64_t *Ap, const int32_t *I, int64_t nI, int64_t *G) {
  GRID_STRIDE(t, nI) G[t + 1] = Ap[I[t] + 1] - Ap[I[t]];
}
// inc[G[t]] += 1 for every row starting inside [0, total): after an
// inclusive scan, inc[g] - 1 is the output row of gathered entry g
__global__ void k_row_starts(const int64_t *G, int64_t nI, int64_t total, int64_t *inc) {
  GRID_STRIDE(t, nI) {
    const int64_t g = G[t];
    if (g < total) atomicAdd(reinterpret_cast<unsigned long long *>(inc + g), 1ull);
  }
}
__device__ __forceinline__ void gather_entry(const GatherArgs &a, int64_t g, int64_t &t, int64_t &q, int &c) {
  t = a.row[g] - 1;
  q = a.Ap[a.I[t]] + (g - a.G[t]);
  c = a.Aj[q];
}
// W[g] = number of tuples entry g makes (|{p : J[p] == c}|)
__global__ void k_gather_w(GatherArgs a, int64_t *W) {
  GRID_STRIDE(g, a.total) {
    int64_t t, q;
    int c;
    gather_entry(a, g, t, q, c);
    W[g] = (c >= 0 && c < a.ncols) ? a.Qp[c + 1] - a.Qp[c] : 0;
  }
}
__device__ __forceinline__ void copy_val(void *dst, int64_t at, const void *src, int64_t q, int vb) {
  if (vb == 8) reinterpret_cast<uint64_t *>(dst)[at] = reinterpret_cast<const uint64_t *>(src)[q];
  else if (vb == 4) reinterpret_cast<uint32_t *>(dst)[at] = reinterpret_cast<const uint32_t *>(src)[q];
}
// the tuples, entry g's at [W[g-1], W[g]) of the scanned counts
__global__ void k_gather_fill(GatherArgs a, const int64_t *W, int32_t *ti, int32_t *pj, void *tv) {
  GRID_STRIDE(g, a.total) {
    int64_t t, q;
    int c;
    gather_entry(a, g, t, q, c);
    int64_t at = g > 0 ? W[g - 1] : 0;
    if (at == W[g]) continue;  // no tuple (and c may be any id)
    for (int64_t k = a.Qp[c]; k < a.Qp[c + 1]; ++k, ++at) {
      ti[at] = (int32_t)t;
      pj[at] = a.Qj[k];
      copy_val(tv, at, a.Av, q, a.vb);
    }
  }
}
// J strictly increasing: each entry makes at most one tuple and a row's
// tuples come out in increasing p, so they are B's entries as they stand
__global__ void k_gather_direct(GatherArgs a, const int64_t *W, int32_t *Bj, void *Bv) {
  GRID_STRIDE(g, a.total) {
    const int64_t before = g > 0 ? W[g - 1] : 0;
    if (W[g] == before) continue;
    int64_t t, q;
    int c;
    gather_entry(a, g, t, q, c);
    Bj[before] = a.Qj[a.Qp[c]];
    copy_val(Bv, before, a.Av, q, a.vb);
  }
}
// B's offsets from the scanned tuple counts: Bp[t] = W[G[t] - 1]
__global__ void k_gather_offsets(const int64_t *G, int64_t nI, const int64_t *W, int64_t *Bp) {
  GRID_STRIDE(t, nI + 1) {
    const int64_t g = G[t];
    Bp[t] = g > 0 ? W[g - 1] : 0;
  }
}
// flag bit 4: J not strictly increasing
__global__ void k_check_increasing(const int32_t *X, int64_t n, int *flag) {
  GRID_STRIDE(i, n - 1) if (X[i] >= X[i + 1]) atomicOr(flag, 4);
}

void launch_gather_len(const int64_t *Ap, const int32_t *I, int64_t nI, int64_t *G, cudaStream_t st) {
  if (nI <= 0) return;
  count_launch();
  k_gather_len<<<grid1(nI), 256, 0, st>>>(Ap, I, nI, G);
}
void launch_row_starts(const int64_t *G, int64_t nI, int64_t total, int64_t *inc, cudaStream_t st) {
  if (nI <= 0 || total <= 0) return;
  count_launch();
  k_row_starts<<<grid1(nI), 256, 0, st>>>(G, nI, total, inc);
}
void launch_gather_w(const GatherArgs &a, int64_t *W, cudaStream_t st) {
  if (a.total <= 0) return;
  count_launch();
  k_gather_w<<<grid1(a.total), 256, 0, st>>>(a, W);
}
void launch_gather_fill(const GatherArgs &a, const int64_t *W, int32_t *ti, int32_t *pj, void *tv, cudaStream_t st) {
  if (a.total <= 0) return;
  count_launch();
  k_gather_fill<<<grid1(a.total), 256, 0, st>>>(a, W, ti, pj, tv);
}
void launch_gather_direct(const GatherArgs &a, const int64_t *W, int32_t *Bj, void *Bv, cudaStream_t st) {
  if (a.total <= 0) return;
  count_launch();
  k_gather_direct<<<grid1(a.total), 256, 0, st>>>(a, W, Bj, Bv);
}
void launch_gather_offsets(const int64_t *G, int64_t nI, const int64_t *W, int64_t *Bp, cudaStream_t st) {
  count_launch();
  k_gather_offsets<<<grid1(nI + 1), 256, 0, st>>>(G, nI, W, Bp);
}
void launch_check_increasing(const int32_t *X, int64_t n, int *flag, cudaStream_t st) {
  if (n <= 1) return;
  count_launch();
  k_check_increasing<<<grid1(n - 1), 256, 0, st>>>(X, n, flag);
}

// flag bit 1: an index outside [0, bound)
__global__ void k_check_range(const int32_t *X, int64_t n, int64_t bound, int *flag) {
  GRID_STRIDE(i, n) {
    const int32_t v = X[i];
    if (v < 0 || v >= bound) atomicOr(flag, 1);
  }
}
void launch_check_range(const int32_t *X, int64_t n, int64_t bound, int *flag, cudaStream_t st) {
  if (n > 0) {
    count_launch();
    k_check_range<<<grid1(n), 256, 0, st>>>(X, n, bound, flag);
  }
}

// pos[X[i]] = i (pos pre-filled with -1) for indices inside [0, bound);
// flag bit 1: an index out of range (skipped), bit 2: a repeated index.
__global__ void k_mark_positions(const int32_t *X, int64_t n, int64_t bound, int32_t *pos, int *flag) {
  GRID_STRIDE(i, n) {
    const int32_t v = X[i];
    if (v < 0 || v >= bound) {
      atomicOr(flag, 1);
      continue;
    }
    const int32_t old = atomicExch(pos + v, (int32_t)i);
    if (old != -1) atomicOr(flag, 2);
  }
}
void launch_mark_positions(const int32_t *X, int64_t n, int64_t bound, int32_t *pos, int *flag, cudaStream_t st) {
  if (n > 0) {
    count_launch();
    k_mark_positions<<<grid1(n), 256, 0, st>>>(X, n, bound, pos, flag);
  }
}

// SpAsgn R = sparse(I, 1:mb, 1, ma, mb) from rpos: counts, then entries
__global__ void k_rows_from_pos(const int32_t *pos, int64_t m, int64_t *cnt) {
  GRID_STRIDE(r, m) cnt[r + 1] = pos[r] >= 0 ? 1 : 0;
}
__global__ void k_fill_from_pos(const int32_t *pos, int64_t m, const int64_t *ptr, int32_t *out) {
  GRID_STRIDE(r, m) if (pos[r] >= 0) out[ptr[r]] = pos[r];
}
void launch_rows_from_pos(const int32_t *pos, int64_t m, int64_t *cnt, cudaStream_t st) {
  if (m > 0) {
    count_launch();
    k_rows_from_pos<<<grid1(m), 256, 0, st>>>(pos, m, cnt);
  }
}
void launch_fill_from_pos(const int32_t *pos, int64_t m, const int64_t *ptr, int32_t *out, cudaStream_t st) {
  if (m > 0) {
    count_launch();
    k_fill_from_pos<<<grid1(m), 256, 0, st>>>(pos, m, ptr, out);
  }
}
__global__ void k_add_i64(int64_t *p, int64_t n, int64_t add) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] += add;
}

void launch_add_i64(int64_t *p, int64_t n, int64_t add, cudaStream_t st) {
  if (n <= 0) return;
  int64_t g = (n + 255) / 256;
  const int64_t cap = (int64_t)sm_count() * 8;
  if (g > cap) g = cap;
  count_launch();
  k_add_i64<<<(int)g, 256, 0, st>>>(p, n, add);
}

void launch_iota_i64(int64_t *p, int64_t n, cudaStream_t st) {
  if (n > 0) {
    count_launch();
    k_iota_i64<<<grid1(n), 256, 0, st>>>(p, n);
  }
}

// ------------------------------------------------------------ SpAsgn merge

// extend-add collision: x (from A) (+) y (from B) in the semiring's add
__device__ void combine_val(const AsgnArgs &a, int64_t di, int64_t ai, int64_t xi) {
  const bool mn = a.add_kind == MIN_PLUS;
  switch (a.dtype) {
    case 0: {
      const double x = ((const double *)a.Av)[ai], y = ((const double *)a.Xv)[xi];
      ((double *)a.Cv)[di] = mn ? (y < x ? y : x) : x + y;
      break;
    }
    case 1: {
      const float x = ((const float *)a.Av)[ai], y = ((const float *)a.Xv)[xi];
      ((float *)a.Cv)[di] = mn ? (y < x ? y : x) : __fadd_rn(x, y);
      break;
    }
    case 2: {
      const int32_t x = ((const int32_t *)a.Av)[ai], y = ((const int32_t *)a.Xv)[xi];
      ((int32_t *)a.Cv)[di] = mn ? (y < x ? y : x) : (int32_t)((uint32_t)x + (uint32_t)y);
      break;
    }
    case 3: {
      const int64_t x = ((const int64_t *)a.Av)[ai], y = ((const int64_t *)a.Xv)[xi];
      ((int64_t *)a.Cv)[di] = mn ? (y < x ? y : x) : (int64_t)((unsigned long long)x + (unsigned long long)y);
      break;
    }
    default: break;
  }
}

// The merge runs over entries, not rows, so a hub row costs what its entries
// cost (assigning 20,000 edges into a 16M-entry graph: 6.62 of 7.20 ms with one
// lane walking each touched row, 0.23 of 0.30 ms so; its 270 MB of A and C
// take 0.04 ms at the copy rate).  X = R*B*Q as the
// entries of B moved to row I[i] and column J[c], in (row, column) order:
// entry t of X goes in front of A's entry at[t] (the first of its row whose
// column is not smaller).  A bit per entry of A says whether it is kept: an
// assignment drops the entries of the I x J block, extend-add those that X
// repeats (X's entry then carries the sum).  With K(q) the kept entries
// before q, A's entry q goes to K(q) + |{t : at[t] <= q}| and X's entry t to
// K(at[t]) + t.

// lengths of X's rows into XB[row + 1], and whether X's entries, taken as they
// lie in B, are in increasing column order inside every row: viol[0] counts
// the entries whose column is not above that of the entry before, viol[1] how
// many of those begin a row.  Indices out of range are skipped (dbg, or flag
// set by the marking, reports them).
__global__ void k_asgn_rows(AsgnX x, int64_t m, int64_t n, int64_t *XB, unsigned long long *viol, long long *dbg) {
  unsigned long long all = 0, starts = 0;
  auto col = [&](int64_t e) -> int {
    const int c = x.j[e];
    if (!HS_G(dbg, c >= 0 && c < x.nJ, 51, c)) return -1;
    return x.J[c];
  };
  GRID_STRIDE(e, x.nnz) if (e > 0) all += col(e) <= col(e - 1);
  GRID_STRIDE(i, x.rows) {
    const int64_t b = x.p[i], e = x.p[i + 1];
    const int r = x.I[i];
    if (!HS_G(dbg, b >= 0 && b <= e && e <= x.nnz, 3, e)) continue;
    if (e > b && r >= 0 && r < m) atomicAdd(reinterpret_cast<unsigned long long *>(XB + r + 1), (unsigned long long)(e - b));
    if (e > b && b > 0) starts += col(b) <= col(b - 1);
  }
  all = warp_sum(all);
  starts = warp_sum(starts);
  if (lane_id() == 0) {
    if (all) atomicAdd(viol, all);
    if (starts) atomicAdd(viol + 1, starts);
  }
}

// at[t] and the source of each entry of X (src[t] = its place in X's arrays;
// ~place when A has an entry there too, whose keep bit extend-add clears).
// Thread per entry: the row by a search of X's offsets, the place by a search
// of A's row.
__global__ void k_asgn_place(AsgnX x, AsgnArgs a, const int64_t *XB, int64_t *at, int64_t *src, uint32_t *keep) {
  GRID_STRIDE(e, x.nnz) {
    int64_t lo = 0, hi = x.rows;  // last row that starts at or before e
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (x.p[mid] <= e) lo = mid;
      else hi = mid;
    }
    const int64_t r = x.I ? (int64_t)x.I[lo] : lo;
    int c = x.j[e];
    if (x.J) {
      if (!HS_G(a.dbg, c >= 0 && c < x.nJ, 51, c)) continue;
      c = x.J[c];
    }
    const int64_t t = r >= 0 && r < a.m ? XB[r] + (e - x.p[lo]) : -1;
    if (t < 0 || t >= x.nnz) continue;  // a bad or repeated index: reported before at[] is used
    const int64_t a0 = a.Ap[r], a1 = a.Ap[r + 1];
    if (!HS_G(a.dbg, a0 >= 0 && a0 <= a1 && a1 <= a.nnzA, 3, a1)) continue;
    const int64_t q = lower_bound_col(a.Aj, a0, a1, c);
    const bool both = a.accumulate && q < a1 && a.Aj[q] == c;
    at[t] = q;
    src[t] = both ? ~e : e;
    if (both) atomicAnd(keep + (q >> 5), ~(1u << (q & 31)));
  }
}

// assignment: the entries of A inside the I x J block lose their keep bit.  A
// warp per row of I; a row of more than ASGN_LONG entries by the whole block.
constexpr int ASGN_LONG = 1024;
__device__ __forceinline__ void asgn_drop(const AsgnArgs &a, int64_t a0, int64_t a1, int64_t step, int64_t first,
                                          uint32_t *keep) {
  constexpr int U = 4;
  // words are aligned to 32 entries, lane l on bit l: one atomic per word
  for (int64_t q0 = (a0 & ~(int64_t)31) + first; q0 - lane_id() < a1; q0 += U * step) {
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t q = q0 + u * step;
      c[u] = q >= a0 && q < a1 ? a.Aj[q] : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned gone = __ballot_sync(FULL, c[u] >= 0 && c[u] < a.n && a.cpos[c[u]] >= 0);
      if (gone && lane_id() == 0) atomicAnd(keep + ((q0 + u * step) >> 5), ~gone);
    }
  }
}
__global__ void __launch_bounds__(256) k_asgn_drop(AsgnArgs a, const int32_t *I, int64_t nI, uint32_t *keep) {
  __shared__ int s_long[8], s_n;
  const int w = threadIdx.x >> 5;
  for (int64_t i0 = (int64_t)blockIdx.x * 8; i0 < nI; i0 += (int64_t)gridDim.x * 8) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t i = i0 + w;
    const int r = i < nI ? I[i] : -1;
    if (r >= 0 && r < a.m) {
      const int64_t a0 = a.Ap[r], a1 = a.Ap[r + 1];
      if (HS_G(a.dbg, a0 >= 0 && a0 <= a1 && a1 <= a.nnzA, 3, a1)) {
        if (a1 - a0 <= ASGN_LONG) asgn_drop(a, a0, a1, 32, lane_id(), keep);
        else if (lane_id() == 0) s_long[atomicAdd(&s_n, 1)] = r;
      }
    }
    __syncthreads();
    for (int k = 0; k < s_n; ++k) asgn_drop(a, a.Ap[s_long[k]], a.Ap[s_long[k] + 1], 256, threadIdx.x, keep);
    __syncthreads();
  }
}

// kept entries per word of 32 (bits past A's last entry do not count)
__global__ void k_asgn_words(const uint32_t *keep, int64_t nnz, int64_t nw, int64_t *S) {
  GRID_STRIDE(w, nw) {
    const int64_t left = nnz - w * 32;
    S[w] = __popc(left >= 32 ? keep[w] : keep[w] & ((1u << left) - 1u));
  }
}
// K(q): kept entries of A before q (S: inclusive scan of the words' counts)
__device__ __forceinline__ int64_t kept_before(const int64_t *S, const uint32_t *keep, int64_t q) {
  const int64_t w = q >> 5;
  const int b = (int)(q & 31);
  return (w ? S[w - 1] : 0) + (b ? __popc(keep[w] & ((1u << b) - 1u)) : 0);
}
__global__ void k_asgn_offsets(AsgnArgs a, const int64_t *XB, const int64_t *S, const uint32_t *keep) {
  const int64_t k0 = kept_before(S, keep, min(a.Ap[0], a.nnzA));
  GRID_STRIDE(r, a.m + 1) {
    const int64_t q = a.Ap[r];
    a.Cp[r] = XB[r] + (HS_G(a.dbg, q >= 0 && q <= a.nnzA, 3, q) ? kept_before(S, keep, q) - k0 : 0);
  }
}

// A's kept entries into C, a tile of consecutive entries per block: the
// entries of X that fall inside the tile are found by two searches of at[]
constexpr int ASGN_NT = 256, ASGN_PER = 8, ASGN_TILE = ASGN_NT * ASGN_PER;
__global__ void __launch_bounds__(ASGN_NT) k_asgn_fill_a(AsgnArgs a, const int64_t *at, int64_t nx, const int64_t *S,
                                                         const uint32_t *keep) {
  __shared__ int64_t s_at[ASGN_TILE];
  __shared__ int64_t s_lo, s_hi;
  const int64_t first = a.Ap[0], last = min(a.Ap[a.m], a.nnzA);
  const int64_t k0 = kept_before(S, keep, min(first, a.nnzA));
  const int64_t q0 = (int64_t)blockIdx.x * ASGN_TILE;
  const int w = threadIdx.x >> 5;
  int c[ASGN_PER];
#pragma unroll
  for (int u = 0; u < ASGN_PER; ++u) {
    const int64_t q = q0 + u * ASGN_NT + threadIdx.x;
    c[u] = q >= first && q < last ? a.Aj[q] : 0;
  }
  if (w < 2) {  // entries of X at or before the tile's first and last entry
    const int64_t key = w == 0 ? q0 : q0 + ASGN_TILE - 1;
    const int64_t r = warp_upper_bound(at, nx, key);
    if (lane_id() == 0) (w == 0 ? s_lo : s_hi) = r;
  }
  __syncthreads();
  const int64_t lo = s_lo, hi = s_hi;
  const bool staged = hi - lo <= ASGN_TILE;
  if (staged)
    for (int64_t t = lo + threadIdx.x; t < hi; t += ASGN_NT) s_at[t - lo] = at[t];
  __syncthreads();
#pragma unroll
  for (int u = 0; u < ASGN_PER; ++u) {
    const int64_t q = q0 + u * ASGN_NT + threadIdx.x;
    if (q < first || q >= last) continue;
    const uint32_t kw = keep[q >> 5];
    if (!((kw >> (q & 31)) & 1u)) continue;
    int64_t l = lo, h = hi;  // |{t : at[t] <= q}|
    while (l < h) {
      const int64_t mid = (l + h) >> 1;
      if ((staged ? s_at[mid - lo] : at[mid]) <= q) l = mid + 1;
      else h = mid;
    }
    const int64_t kb = (q >> 5) ? S[(q >> 5) - 1] : 0;
    const int64_t d = kb + __popc(kw & ((1u << (q & 31)) - 1u)) - k0 + l;
    if (!HS_G(a.dbg, d >= 0 && d < a.nnzC, 86, d)) continue;
    a.Cj[d] = c[u];
    copy_val(a.Cv, d, a.Av, q, a.vbytes);
  }
}
__global__ void k_asgn_fill_x(AsgnX x, AsgnArgs a, const int64_t *at, const int64_t *src, const int64_t *S,
                              const uint32_t *keep) {
  const int64_t k0 = kept_before(S, keep, min(a.Ap[0], a.nnzA));
  GRID_STRIDE(t, x.nnz) {
    const int64_t s = src[t], q = at[t];
    const int64_t e = s < 0 ? ~s : s;
    if (!HS_G(a.dbg, q >= 0 && q <= a.nnzA && e < x.nnz, 87, q)) continue;
    const int64_t d = kept_before(S, keep, q) - k0 + t;
    if (!HS_G(a.dbg, d >= 0 && d < a.nnzC, 86, d)) continue;
    a.Cj[d] = x.J ? x.J[x.j[e]] : x.j[e];
    if (s < 0) combine_val(a, d, q, e);
    else copy_val(a.Cv, d, a.Xv, e, a.vbytes);
  }
}

void launch_asgn_rows(const AsgnX &x, int64_t m, int64_t n, int64_t *XB, unsigned long long *viol, long long *dbg,
                      cudaStream_t st) {
  const int64_t work = x.nnz > x.rows ? x.nnz : x.rows;
  if (work <= 0) return;
  count_launch();
  k_asgn_rows<<<grid1(work), 256, 0, st>>>(x, m, n, XB, viol, dbg);
}
void launch_asgn_keep(const AsgnX &x, const AsgnArgs &a, const int32_t *I, int64_t nI, const int64_t *XB, int64_t *at,
                      int64_t *src, uint32_t *keep, int64_t *S, int64_t nw, cudaStream_t st) {
  if (x.nnz > 0) {
    count_launch();
    k_asgn_place<<<grid1(x.nnz), 256, 0, st>>>(x, a, XB, at, src, keep);
  }
  if (!a.accumulate && nI > 0) {
    count_launch();
    k_asgn_drop<<<grid1(nI * 32), 256, 0, st>>>(a, I, nI, keep);
  }
  if (nw > 0) {
    count_launch();
    k_asgn_words<<<grid1(nw), 256, 0, st>>>(keep, a.nnzA, nw, S);
  }
}
void launch_asgn_offsets(const AsgnArgs &a, const int64_t *XB, const int64_t *S, const uint32_t *keep,
                         cudaStream_t st) {
  count_launch();
  k_asgn_offsets<<<grid1(a.m + 1), 256, 0, st>>>(a, XB, S, keep);
}
void launch_asgn_fill(const AsgnX &x, const AsgnArgs &a, const int64_t *at, const int64_t *src, const int64_t *S,
                      const uint32_t *keep, cudaStream_t st) {
  if (a.m > 0 && a.nnzA > 0) {
    count_launch();
    k_asgn_fill_a<<<(unsigned)((a.nnzA + ASGN_TILE - 1) / ASGN_TILE), ASGN_NT, 0, st>>>(a, at, x.nnz, S, keep);
  }
  if (x.nnz > 0) {
    count_launch();
    k_asgn_fill_x<<<grid1(x.nnz), 256, 0, st>>>(x, a, at, src, S, keep);
  }
}

}  // namespace hs
