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
#include <type_traits>

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

__device__ __forceinline__ void copy_val(void *dst, int64_t at, const void *src, int64_t q, int vb) {
  if (vb == 8) reinterpret_cast<uint64_t *>(dst)[at] = reinterpret_cast<const uint64_t *>(src)[q];
  else if (vb == 4) reinterpret_cast<uint32_t *>(dst)[at] = reinterpret_cast<const uint32_t *>(src)[q];
}

__global__ void k_iota_i64(int64_t *p, int64_t n) { GRID_STRIDE(i, n) p[i] = i; }

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
// tuple (t, p, v) for each p with J[p] == c (Q's row c).  When J repeats no
// index, that is at most one tuple: Q is J's inverse map, the tuples lie row
// by row, in order when J is increasing, else each row is sorted.  When J
// repeats indices the tuples are sorted by (t, p).

// First look at A, I and J: flag bit 1: an index out of range, bit 2: J
// repeats an index, bit 4: J not strictly increasing; pos[J[p]] = p (filled
// with -1 before); G[t + 1] = length of row I[t] (0 for a bad index), the
// longest in *lmax.
__global__ void k_spref_begin(const int64_t *Ap, int64_t m, int64_t n, const int32_t *I, int64_t nI, const int32_t *J,
                              int64_t nJ, int32_t *pos, int64_t *G, int *flag, unsigned long long *lmax) {
  int bad = 0;
  unsigned long long mx = 0;
  GRID_STRIDE(p, nJ) {
    const int32_t c = J[p];
    if (c < 0 || c >= n) bad |= 1;
    else if (atomicExch(pos + c, (int32_t)p) != -1) bad |= 2;
    if (p + 1 < nJ && c >= J[p + 1]) bad |= 4;
  }
  GRID_STRIDE(t, nI) {
    const int32_t r = I[t];
    int64_t len = 0;
    if (r < 0 || r >= m) bad |= 1;
    else len = max(Ap[r + 1] - Ap[r], (int64_t)0);
    G[t + 1] = len;
    if (t == 0) G[0] = 0;
    mx = max(mx, (unsigned long long)len);
  }
  bad = __reduce_or_sync(FULL, bad);
  mx = warp_max(mx);
  if (lane_id() == 0) {
    if (bad) atomicOr(flag, bad);
    if (mx) atomicMax(lmax, mx);
  }
}
void launch_spref_begin(const int64_t *Ap, int64_t m, int64_t n, const int32_t *I, int64_t nI, const int32_t *J,
                        int64_t nJ, int32_t *pos, int64_t *G, int *flag, unsigned long long *lmax, cudaStream_t st) {
  const int64_t work = nI > nJ ? nI : nJ;
  if (work <= 0) return;
  count_launch();
  k_spref_begin<<<grid1(work), 256, 0, st>>>(Ap, m, n, I, nI, J, nJ, pos, G, flag, lmax);
}

// ---- J without repetitions: an entry makes at most one tuple.  A block takes
// 2048 gathered entries, finds the output rows they lie in by a search of G
// and notes for each entry its column p in B (-1: none) and its value, a bit
// per entry and the kept entries per word of 32; after a scan of the words'
// counts, K(g) = kept entries before g is an entry's place among the kept.
constexpr int SG_NT = 256, SG_PER = 8, SG_TILE = SG_NT * SG_PER;
__global__ void __launch_bounds__(SG_NT) k_spref_gather(SprefArgs a) {
  __shared__ int64_t s_g[SG_TILE], s_row[2];
  const int64_t g0 = (int64_t)blockIdx.x * SG_TILE, g1 = min(g0 + SG_TILE, a.total);
  if (threadIdx.x < 64) {
    const int64_t r = warp_upper_bound(a.G, a.nI + 1, threadIdx.x < 32 ? g0 : g1 - 1) - 1;
    if (lane_id() == 0) s_row[threadIdx.x >> 5] = r;
  }
  __syncthreads();
  const int64_t r0 = s_row[0], r1 = s_row[1];
  const bool staged = r1 - r0 < SG_TILE;
  if (staged)
    for (int64_t r = r0 + threadIdx.x; r <= r1; r += SG_NT) s_g[r - r0] = a.G[r];
  __syncthreads();
  int64_t q[SG_PER];
  int c[SG_PER], p[SG_PER];
#pragma unroll
  for (int u = 0; u < SG_PER; ++u) {
    const int64_t g = g0 + u * SG_NT + threadIdx.x;
    q[u] = -1;
    if (g >= g1) continue;
    int64_t l = r0, h = r1 + 1;  // last row that starts at or before g
    while (h - l > 1) {
      const int64_t mid = (l + h) >> 1;
      if ((staged ? s_g[mid - r0] : a.G[mid]) <= g) l = mid;
      else h = mid;
    }
    q[u] = a.Ap[a.I[l]] + (g - (staged ? s_g[l - r0] : a.G[l]));
  }
#pragma unroll
  for (int u = 0; u < SG_PER; ++u) c[u] = q[u] >= 0 ? a.Aj[q[u]] : -1;
#pragma unroll
  for (int u = 0; u < SG_PER; ++u) p[u] = c[u] >= 0 && c[u] < a.n ? __ldg(a.pos + c[u]) : -1;
#pragma unroll
  for (int u = 0; u < SG_PER; ++u) {
    const int64_t g = g0 + u * SG_NT + threadIdx.x;
    const unsigned m = __ballot_sync(FULL, p[u] >= 0);
    if (g < g1) a.P[g] = p[u];
    if (p[u] >= 0) copy_val(a.V, g, a.Av, q[u], a.vb);
    if (lane_id() == 0 && g < g1) {
      a.keep[g >> 5] = m;
      a.S[g >> 5] = __popc(m);
    }
  }
}
// the kept entries in order: B's entries as they stand when J is increasing
__global__ void __launch_bounds__(256) k_spref_emit(SprefArgs a, int32_t *Bj, void *Bv) {
  GRID_STRIDE(g, a.total) {
    const uint32_t kw = a.keep[g >> 5];
    if (!((kw >> (g & 31)) & 1u)) continue;
    const int64_t d = ((g >> 5) ? a.S[(g >> 5) - 1] : 0) + __popc(kw & ((1u << (g & 31)) - 1u));
    Bj[d] = a.P[g];
    copy_val(Bv, d, a.V, g, a.vb);
  }
}
// B's row offsets, the number of kept entries (longs[2]), and the rows that
// the bitmap kernel below would take (longs[0]) with their entries (longs[1])
__device__ __forceinline__ int64_t spref_kept(const SprefArgs &a, int64_t g) {
  const int64_t w = g >> 5;
  const int b = (int)(g & 31);
  return (w ? a.S[w - 1] : 0) + (b ? __popc(a.keep[w] & ((1u << b) - 1u)) : 0);
}
__global__ void k_spref_offsets(SprefArgs a, int64_t *Bp, unsigned long long *longs) {
  GRID_STRIDE(t, a.nI + 1) {
    const int64_t g = a.G[t], b = spref_kept(a, g);
    Bp[t] = b;
    if (t == a.nI) {
      longs[2] = (unsigned long long)b;
    } else if (a.G[t + 1] - g > SR_CTA) {
      const int64_t c = spref_kept(a, a.G[t + 1]) - b;
      if (c > SR_CTA) {
        atomicAdd(longs, 1ull);
        atomicAdd(longs + 1, (unsigned long long)c);
      }
    }
  }
}
// ti[d] = the row of B that kept entry d lies in
__global__ void k_spref_row_ids(const int64_t *Bp, int64_t nI, int64_t ntup, int32_t *ti) {
  __shared__ int64_t s_row[2];
  const int64_t d0 = (int64_t)blockIdx.x * SG_TILE, d1 = min(d0 + SG_TILE, ntup);
  if (threadIdx.x < 64) {
    const int64_t r = warp_upper_bound(Bp, nI + 1, threadIdx.x < 32 ? d0 : d1 - 1) - 1;
    if (lane_id() == 0) s_row[threadIdx.x >> 5] = r;
  }
  __syncthreads();
  for (int64_t d = d0 + threadIdx.x; d < d1; d += SG_NT) {
    int64_t l = s_row[0], h = s_row[1] + 1;  // last row that starts at or before d
    while (h - l > 1) {
      const int64_t mid = (l + h) >> 1;
      if (Bp[mid] <= d) l = mid;
      else h = mid;
    }
    ti[d] = (int32_t)l;
  }
}

// ---- rows into increasing order of p, for a J in any order.  The tuples of a
// row lie together already, so only rows are sorted, by their length: eight
// lanes a row of at most 8, a warp up to SR_WARP (ranks counted directly), a
// block up to SR_CTA (buckets in shared memory), and longer ones through a
// bitmap of B's columns (rank = set bits before p).  Every tuple is read and
// written once; a radix sort of all (row, p) keys took five passes.  Only the
// bitmap's cost grows with B's width, a sweep and two reads of the row for
// every 2^20 columns: spref_by_radix (internal.h) says when the radix sort is
// taken after all.
constexpr int SR_WARP = 64;
template <typename T> struct SprefRowArgs {
  const int64_t *Bp;
  int64_t nI, nJ;
  const int32_t *P;  // kept tuples, row by row
  const T *V;
  int32_t *Bj;
  T *Bv;
  int *count;        // rows left to the block kernel, to the bitmap kernel; their work counters; error
  int32_t *list;     // 2 * nI
  long long *dbg;
};
template <typename T>
__global__ void __launch_bounds__(256) k_spref_rows(SprefRowArgs<T> a) {
  constexpr bool HAS_VAL = !std::is_same<T, NoVal>::value;
  const int lane = lane_id(), sub = lane >> 3, l = lane & 7;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; t0 < a.nI; t0 += nw * 4) {
    const int64_t t = t0 + sub;
    const int64_t b = t < a.nI ? a.Bp[t] : 0;
    const int64_t c = t < a.nI ? a.Bp[t + 1] - b : 0;
    {
      const bool mine = c <= 8 && l < c;
      const int32_t p = mine ? a.P[b + l] : 0x7fffffff;
      T v{};
      if constexpr (HAS_VAL)
        if (mine) v = a.V[b + l];
      int rank = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) rank += __shfl_sync(FULL, p, (sub << 3) + j) < p;
      if (mine) {
        a.Bj[b + rank] = p;
        if constexpr (HAS_VAL) a.Bv[b + rank] = v;
      }
    }
    // longer rows: the whole warp, one row after the other
    for (unsigned more = __ballot_sync(FULL, l == 0 && c > 8); more; more &= more - 1) {
      const int src = __ffs(more) - 1;
      const int64_t rb = __shfl_sync(FULL, b, src), rc = __shfl_sync(FULL, c, src);
      if (rc > SR_WARP) {
        if (lane == 0) {
          const int kind = rc > SR_CTA;
          a.list[kind * a.nI + atomicAdd(a.count + kind, 1)] = (int32_t)(t0 + (src >> 3));
        }
        continue;
      }
      const int n = (int)rc;
      for (int e0 = 0; e0 < n; e0 += 64) {  // two of the row's tuples per lane
        const int ea = e0 + lane, eb = ea + 32;
        const int32_t pa = ea < n ? a.P[rb + ea] : 0x7fffffff, pb = eb < n ? a.P[rb + eb] : 0x7fffffff;
        int ra = 0, rk = 0;
        for (int x0 = 0; x0 < n; x0 += 32) {
          const int32_t px = x0 + lane < n ? a.P[rb + x0 + lane] : 0x7fffffff;
          const int lim = min(32, n - x0);
          for (int j = 0; j < lim; ++j) {
            const int32_t y = __shfl_sync(FULL, px, j);
            ra += y < pa;
            rk += y < pb;
          }
        }
        if (ea < n) {
          a.Bj[rb + ra] = pa;
          if constexpr (HAS_VAL) a.Bv[rb + ra] = a.V[rb + ea];
        }
        if (eb < n) {
          a.Bj[rb + rk] = pb;
          if constexpr (HAS_VAL) a.Bv[rb + rk] = a.V[rb + eb];
        }
      }
    }
  }
}
template <typename T> struct SprefCtaSmem {
  static constexpr size_t vb = std::is_same<T, NoVal>::value ? 0 : sizeof(T);
  static constexpr size_t arr = (size_t)SR_CTA * (4 + vb);          // keys and values
  static constexpr size_t work = (size_t)SR_CTA * (12 + vb) + 16;   // group_sort_emit's work
  static constexpr size_t bytes = 2 * arr + work;
};
template <typename T>
__global__ void __launch_bounds__(256) k_spref_rows_cta(SprefRowArgs<T> a) {
  constexpr bool HAS_VAL = !std::is_same<T, NoVal>::value;
  using L = SprefCtaSmem<T>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ EmitScratch es;
  __shared__ int s_item, wtmp[33];
  T *v0 = reinterpret_cast<T *>(smem), *v1 = reinterpret_cast<T *>(smem + L::arr);
  int *k0 = reinterpret_cast<int *>(smem + SR_CTA * L::vb), *k1 = reinterpret_cast<int *>(smem + L::arr + SR_CTA * L::vb);
  const int count = a.count[0];
  while (true) {
    if (threadIdx.x == 0) s_item = atomicAdd(a.count + 2, 1);
    __syncthreads();
    const int i = s_item;
    if (i >= count) break;
    const int64_t t = a.list[i];
    const int64_t b = a.Bp[t];
    const int c = (int)(a.Bp[t + 1] - b);
    for (int e = threadIdx.x; e < c; e += 256) {
      k0[e] = a.P[b + e];
      if constexpr (HAS_VAL) v0[e] = a.V[b + e];
    }
    __syncthreads();
    group_sort_emit<CtaGroup, T, HAS_VAL>(k0, v0, c, c, k1, v1, smem + 2 * L::arr, wtmp, &es, a.Bj + b,
                                          HAS_VAL ? a.Bv + b : nullptr, a.count + 4, SR_CTA, a.dbg);
    __syncthreads();
  }
}
constexpr int SR_NT = 1024, SR_WORDS = BITMAP_COLS / 32, SR_GROUPS = SR_WORDS / 32;
struct SprefBitSmem {
  unsigned bits[SR_WORDS];  // B's columns of the chunk
  uint16_t pre[SR_WORDS];   // set bits before the word in its group of 32 words
  int base[SR_GROUPS];      // set bits before the group
  int wtmp[33];
  int item;
};
template <typename T>
__global__ void __launch_bounds__(SR_NT) k_spref_rows_bits(SprefRowArgs<T> a) {
  constexpr bool HAS_VAL = !std::is_same<T, NoVal>::value;
  extern __shared__ __align__(16) unsigned char smem[];
  SprefBitSmem &sm = *reinterpret_cast<SprefBitSmem *>(smem);
  const int count = a.count[1], tid = threadIdx.x;
  while (true) {
    if (tid == 0) sm.item = atomicAdd(a.count + 3, 1);
    __syncthreads();
    const int i = sm.item;
    if (i >= count) break;
    const int64_t t = a.list[a.nI + i];
    const int64_t b = a.Bp[t], c = a.Bp[t + 1] - b;
    int64_t done = 0;  // entries with smaller columns than the chunk's
    for (int64_t lo = 0; lo < a.nJ; lo += BITMAP_COLS) {
      const int groups = (int)((min(a.nJ - lo, (int64_t)BITMAP_COLS) + 1023) >> 10);
      for (int w = tid; w < groups * 32; w += SR_NT) sm.bits[w] = 0u;
      __syncthreads();
      for (int64_t e = tid; e < c; e += SR_NT) {
        const int64_t x = a.P[b + e] - lo;
        if (x >= 0 && x < BITMAP_COLS) atomicOr(sm.bits + (x >> 5), 1u << (x & 31));
      }
      __syncthreads();
      for (int g = tid >> 5; g < groups; g += SR_NT / 32) {  // a warp per group, a word per lane
        const int w = g * 32 + lane_id();
        const int n1 = __popc(sm.bits[w]);
        const int incl = warp_incl_scan(n1);
        sm.pre[w] = (uint16_t)(incl - n1);
        if (lane_id() == 31) sm.base[g] = incl;
      }
      __syncthreads();
      const int tot = group_excl_scan<CtaGroup>(sm.base, groups, sm.wtmp);
      for (int64_t e = tid; e < c; e += SR_NT) {
        const int32_t p = a.P[b + e];
        const int64_t x = p - lo;
        if (x < 0 || x >= BITMAP_COLS) continue;
        const int w = (int)(x >> 5);
        const int64_t r = done + sm.base[w >> 5] + sm.pre[w] + __popc(sm.bits[w] & ((1u << (x & 31)) - 1u));
        if (!HS_G(a.dbg, r < c, 88, r)) continue;
        a.Bj[b + r] = p;
        if constexpr (HAS_VAL) a.Bv[b + r] = a.V[b + e];
      }
      done += tot;
      __syncthreads();
    }
  }
}

void launch_spref_gather(const SprefArgs &a, cudaStream_t st) {
  if (a.total <= 0) return;
  count_launch();
  k_spref_gather<<<(unsigned)((a.total + SG_TILE - 1) / SG_TILE), SG_NT, 0, st>>>(a);
}
void launch_spref_offsets(const SprefArgs &a, int64_t *Bp, unsigned long long *longs, cudaStream_t st) {
  count_launch();
  k_spref_offsets<<<grid1(a.nI + 1), 256, 0, st>>>(a, Bp, longs);
}
void launch_spref_row_ids(const int64_t *Bp, int64_t nI, int64_t ntup, int32_t *ti, cudaStream_t st) {
  if (ntup <= 0) return;
  count_launch();
  k_spref_row_ids<<<(unsigned)((ntup + SG_TILE - 1) / SG_TILE), SG_NT, 0, st>>>(Bp, nI, ntup, ti);
}
void launch_spref_emit(const SprefArgs &a, int32_t *Bj, void *Bv, cudaStream_t st) {
  if (a.total <= 0) return;
  count_launch();
  k_spref_emit<<<grid1(a.total), 256, 0, st>>>(a, Bj, Bv);
}
template <typename T>
static void spref_rows(const int64_t *Bp, int64_t nI, int64_t nJ, const int32_t *P, const void *V, int32_t *Bj,
                       void *Bv, int64_t lmax, int *count, int32_t *list, long long *dbg, cudaStream_t st) {
  const SprefRowArgs<T> a{Bp, nI, nJ, P, reinterpret_cast<const T *>(V), Bj, reinterpret_cast<T *>(Bv), count, list, dbg};
  count_launch();
  k_spref_rows<T><<<grid1(nI * 8), 256, 0, st>>>(a);
  if (lmax > SR_WARP) {
    const int fit = fit_per_sm(k_spref_rows_cta<T>, 256, SprefCtaSmem<T>::bytes);
    count_launch();
    k_spref_rows_cta<T><<<sm_count() * fit, 256, SprefCtaSmem<T>::bytes, st>>>(a);
  }
  if (lmax > SR_CTA) {
    fit_per_sm(k_spref_rows_bits<T>, SR_NT, sizeof(SprefBitSmem));
    count_launch();
    k_spref_rows_bits<T><<<sm_count(), SR_NT, sizeof(SprefBitSmem), st>>>(a);
  }
}
void launch_spref_rows(int vb, const int64_t *Bp, int64_t nI, int64_t nJ, const int32_t *P, const void *V, int32_t *Bj,
                       void *Bv, int64_t lmax, int *count, int32_t *list, long long *dbg, cudaStream_t st) {
  if (nI <= 0) return;
  if (vb == 8) spref_rows<unsigned long long>(Bp, nI, nJ, P, V, Bj, Bv, lmax, count, list, dbg, st);
  else if (vb == 4) spref_rows<uint32_t>(Bp, nI, nJ, P, V, Bj, Bv, lmax, count, list, dbg, st);
  else spref_rows<NoVal>(Bp, nI, nJ, P, V, Bj, Bv, lmax, count, list, dbg, st);
}

// ---- J with repetitions: every tuple (t, p) of an entry is laid out and the
// tuples are sorted
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
// lane walking each touched row, 0.19 of 0.27 ms so; its 270 MB of A and C
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
// warp per row of I, whole blocks for a row of more than ASGN_LONG entries.
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
// A long row by ASGN_PARTS blocks (blockIdx.y): it would hold up one block
// long after the others are done (a row of 3.5e4 entries: 40 us).
constexpr int ASGN_PARTS = 8;
__global__ void __launch_bounds__(256) k_asgn_drop(AsgnArgs a, const int32_t *I, int64_t nI, uint32_t *keep) {
  __shared__ int s_long[8 * ASGN_PARTS], s_n;
  const int w = threadIdx.x >> 5, part = blockIdx.y;
  // this block's rows: 64 at a time; a part takes every eighth of the short
  // ones and its share of all long ones
  for (int64_t i0 = (int64_t)blockIdx.x * 64; i0 < nI; i0 += (int64_t)gridDim.x * 64) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    if (threadIdx.x < 64) {
      const int64_t i = i0 + threadIdx.x;
      const int r = i < nI ? I[i] : -1;
      if (r >= 0 && r < a.m && a.Ap[r + 1] - a.Ap[r] > ASGN_LONG) s_long[atomicAdd(&s_n, 1)] = r;
    }
    {
      const int64_t i = i0 + part * 8 + w;
      const int r = i < nI ? I[i] : -1;
      if (r >= 0 && r < a.m) {
        const int64_t a0 = a.Ap[r], a1 = a.Ap[r + 1];
        if (HS_G(a.dbg, a0 >= 0 && a0 <= a1 && a1 <= a.nnzA, 3, a1) && a1 - a0 <= ASGN_LONG)
          asgn_drop(a, a0, a1, 32, lane_id(), keep);
      }
    }
    __syncthreads();
    for (int k = 0; k < s_n; ++k) {
      const int64_t a0 = a.Ap[s_long[k]], a1 = a.Ap[s_long[k] + 1];
      if (!HS_G(a.dbg, a0 >= 0 && a0 <= a1 && a1 <= a.nnzA, 3, a1)) continue;
      const int64_t share = ((a1 - a0 + ASGN_PARTS - 1) / ASGN_PARTS + 31) & ~(int64_t)31;
      const int64_t b0 = a0 + part * share, b1 = min(a1, b0 + share);
      if (b0 < b1) asgn_drop(a, b0, b1, 256, threadIdx.x, keep);
    }
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
template <typename V>  // the values' bits by width (NoVal: none); they are asked for with the columns
__global__ void __launch_bounds__(ASGN_NT) k_asgn_fill_a(AsgnArgs a, const int64_t *at, int64_t nx, const int64_t *S,
                                                         const uint32_t *keep) {
  __shared__ int64_t s_at[ASGN_TILE];
  __shared__ int64_t s_lo, s_hi;
  const int64_t first = a.Ap[0], last = min(a.Ap[a.m], a.nnzA);
  const int64_t k0 = kept_before(S, keep, min(first, a.nnzA));
  const int64_t q0 = (int64_t)blockIdx.x * ASGN_TILE;
  const int w = threadIdx.x >> 5;
  constexpr bool HAS_VAL = !std::is_same<V, NoVal>::value;
  int c[ASGN_PER];
  V v[ASGN_PER];
#pragma unroll
  for (int u = 0; u < ASGN_PER; ++u) {
    const int64_t q = q0 + u * ASGN_NT + threadIdx.x;
    const bool in = q >= first && q < last;
    c[u] = in ? __ldcs(a.Aj + q) : 0;
    if constexpr (HAS_VAL) v[u] = in ? __ldcs(reinterpret_cast<const V *>(a.Av) + q) : V{};
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
    if constexpr (HAS_VAL) reinterpret_cast<V *>(a.Cv)[d] = v[u];
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
    const int64_t g = (nI + 63) / 64, cap = (int64_t)sm_count() * 2;
    k_asgn_drop<<<dim3((unsigned)(g < cap ? g : cap), ASGN_PARTS), 256, 0, st>>>(a, I, nI, keep);
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
    const unsigned g = (unsigned)((a.nnzA + ASGN_TILE - 1) / ASGN_TILE);
    if (a.vbytes == 8) k_asgn_fill_a<unsigned long long><<<g, ASGN_NT, 0, st>>>(a, at, x.nnz, S, keep);
    else if (a.vbytes == 4) k_asgn_fill_a<uint32_t><<<g, ASGN_NT, 0, st>>>(a, at, x.nnz, S, keep);
    else k_asgn_fill_a<NoVal><<<g, ASGN_NT, 0, st>>>(a, at, x.nnz, S, keep);
  }
  if (x.nnz > 0) {
    count_launch();
    k_asgn_fill_x<<<grid1(x.nnz), 256, 0, st>>>(x, a, at, src, S, keep);
  }
}

}  // namespace hs
