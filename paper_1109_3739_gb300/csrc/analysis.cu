// analysis.cu -- integer work ahead of the products: per-row flop counts,
// binning of rows, prefix sums and input validation.
//
// flops(A*B) for row i is the number of nonzero multiplications of that row
// (Section 2 notation): sum over stored A(i,k) of nnz(B(k,:)).  Rows with no
// products are left out of every bin, so no later kernel does work for empty
// rows: the dimension-independent work list of the doubly compressed format
// (Section 2.2), built on the fly.
#include <mutex>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace hs {

static int g_sms = 0;
static unsigned long long g_launches = 0;
void count_launch() { __atomic_add_fetch(&g_launches, 1ull, __ATOMIC_RELAXED); }
unsigned long long launch_total() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }
cudaError_t &attr_error() {
  static thread_local cudaError_t e = cudaSuccess;
  return e;
}
void launch_sm_count_init() {
  if (g_sms) return;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
  if (g_sms <= 0) g_sms = 1;
}
int sm_count() {
  launch_sm_count_init();
  return g_sms;
}

int kernel_fit(const void *kernel, int threads, size_t smem) {
  struct Fit {
    const void *kernel;
    int dev, threads, ctas;
    size_t smem;
  };
  static std::mutex mu;
  static std::vector<Fit> fits;  // one per kernel, size and device: a few dozen
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  size_t limit = 0;  // the limit set so far (never lowered: other sizes of the kernel may need it)
  for (const Fit &f : fits) {
    if (f.kernel != kernel || f.dev != dev) continue;
    if (f.threads == threads && f.smem == smem) return f.ctas;
    if (f.smem > limit) limit = f.smem;
  }
  if (e == cudaSuccess && smem > limit && smem > 0)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int n = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem);
  if (e != cudaSuccess) {
    attr_error() = e;
    cudaGetLastError();
    return 1;
  }
  if (n < 1) n = 1;
  fits.push_back(Fit{kernel, dev, threads, n, smem});
  return n;
}

static int grid_for(int64_t items, int per_block, int max_per_sm) {
  int64_t g = (items + per_block - 1) / per_block;
  int64_t cap = (int64_t)sm_count() * max_per_sm;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

// ------------------------------------------------------- tiles and last block
// Inclusive scan of NT*PER values held PER to a thread, value u of thread x at
// position u*NT + x; s_tot holds PER*NT/32 words (64).  Returns the total.
// One barrier; the caller separates two uses of s_tot.
constexpr int TL_NT = 256, TL_PER = 8, TL_TILE = TL_NT * TL_PER, TL_NW = TL_NT / 32;
static_assert(TL_PER * TL_NW == 64, "two warp totals per lane");
__device__ __forceinline__ long long tile_scan(long long (&v)[TL_PER], long long *s_tot) {
  const int lane = lane_id(), w = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    v[u] = warp_incl_scan(v[u]);
    if (lane == 31) s_tot[u * TL_NW + w] = v[u];
  }
  __syncthreads();
  const long long x0 = s_tot[lane], x1 = s_tot[lane + 32];
  const long long i0 = warp_incl_scan(x0), t0 = __shfl_sync(FULL, i0, 31);
  const long long i1 = warp_incl_scan(x1) + t0;
  const long long e0 = i0 - x0, e1 = i1 - x1;
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) v[u] += __shfl_sync(FULL, u < 4 ? e0 : e1, (u * TL_NW + w) & 31);
  return __shfl_sync(FULL, i1, 31);
}
// True in every thread of the block that finishes last (its reads then see
// what all blocks wrote before).
__device__ __forceinline__ bool last_block(int *ticket, int *s_flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *s_flag = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!*s_flag) return false;
  __threadfence();
  return true;
}
// one warp: exclusive scan of the NKEYS counters into offsets and cursors;
// with `hub`, which hub rows are moved, and the counts with them there
__device__ __forceinline__ void key_offsets(const int *cnt, int *off, int *cur, HubRows *hub = nullptr) {
  static_assert(HUB_KEYS <= 32, "a key per lane");
  const int lane = lane_id();
  int a = __ldcg(cnt + 2 * lane), b = __ldcg(cnt + 2 * lane + 1);
  if (hub) {  // (uniform)
    int rows[HUB_LEVELS], mine[HUB_LEVELS];  // of all keys, of key KEY_TINY + 1 + lane
    const int any = __ldcg(&hub->any);
#pragma unroll
    for (int l = 0; l < HUB_LEVELS; ++l) rows[l] = mine[l] = lane < HUB_KEYS ? __ldcg(&hub->n[l][lane]) : 0;
    if (any) {  // (else `from` stays zero: no row reaches a level)
#pragma unroll
      for (int l = 0; l < HUB_LEVELS; ++l) rows[l] = warp_sum(rows[l]);
      const int from = hub_from(rows);
      if (lane == 0) hub->from = from;
      int moved = 0;
#pragma unroll
      for (int l = 0; l < HUB_LEVELS; ++l) moved += l >= from ? mine[l] : 0;
      const int all = warp_sum(moved);
      // (lanes from HUB_KEYS on hold none)
      a -= __shfl_sync(FULL, moved, (2 * lane - KEY_TINY - 1) & 31) * (2 * lane > KEY_TINY && 2 * lane < KEY_SPA);
      b -= __shfl_sync(FULL, moved, (2 * lane - KEY_TINY) & 31) * (2 * lane + 1 > KEY_TINY && 2 * lane + 1 < KEY_SPA);
      a += 2 * lane == KEY_LARGE ? all : 0;
      b += 2 * lane + 1 == KEY_LARGE ? all : 0;
    }
  }
  const int incl = warp_incl_scan(a + b);
  const int ex = incl - a - b;
  off[2 * lane] = ex;
  off[2 * lane + 1] = ex + a;
  cur[2 * lane] = ex;
  cur[2 * lane + 1] = ex + a;
  if (lane == 31) off[NKEYS] = incl;
}
static_assert(NKEYS == 64, "key_offsets assumes 64 keys");

// ------------------------------------------------------------------ flops
// f[r] = sum over the row's entries of nnz(B(A.j[q], :)), f zeroed before.
// A block takes TL_TILE consecutive entries of A, so that a hub row costs what
// its entries cost: their counts are scanned in shared memory and every row
// that has entries in the tile takes the difference of two scanned values (a
// row that crosses a tile's border adds its parts by atomics).  The rows at
// the tile's ends are found by a search of the offsets while the entries are
// on their way.  One read of A's columns and B's offsets and no array of
// counts per entry, which was written and passed over four times: the whole
// analysis of R-MAT scale 20 (8.2M entries) 0.22 -> 0.10 ms, of a 128^3
// Galerkin product (10.4M entries) 0.26 -> 0.14 ms; bound by the latency of
// column -> offset, not by its 0.2 GB.  zeros counts the entries
// whose B row is empty (they make no product).
__global__ void __launch_bounds__(TL_NT) k_entry_flops(RowSet A, RightOp B, int64_t *f, unsigned long long *zeros) {
  __shared__ long long S[TL_TILE], s_tot[64];
  __shared__ int64_t s_row[2];
  // offsets are trusted only inside A's arrays
  const int64_t lo = max(A.p[0], (int64_t)0), hi = min(A.p[A.nslots], A.nnz);
  const int64_t t0 = lo + (int64_t)blockIdx.x * TL_TILE, t1 = min(t0 + TL_TILE, hi);
  if (t0 >= hi) return;
  long long v[TL_PER];
  int z = 0;
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t q = t0 + u * TL_NT + threadIdx.x;
    const int k = q < t1 ? A.j[q] : -1;
    v[u] = 0;
    if (q < t1 && HS_G(A.dbg, k >= 0 && k < B.m, 52, k)) v[u] = B.p[k + 1] - B.p[k];
    z += q < t1 && v[u] == 0;
  }
  if (threadIdx.x < 64) {  // the rows that hold the tile's first and last entry
    const int which = threadIdx.x >> 5;
    const int64_t r = warp_upper_bound(A.p, A.nslots + 1, which ? t1 - 1 : t0) - 1;
    if (lane_id() == 0) s_row[which] = r;
  }
  tile_scan(v, s_tot);
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) S[u * TL_NT + threadIdx.x] = v[u];
  z = warp_sum(z);
  if (lane_id() == 0 && z) atomicAdd(zeros, (unsigned long long)z);
  __syncthreads();
  const int64_t r0 = max(s_row[0], (int64_t)0), r1 = min(s_row[1], A.nslots - 1);
  auto put = [&](int64_t r) {
    const int64_t q0 = A.p[r], q1 = A.p[r + 1];
    const int64_t a = max(q0, t0), b = min(q1, t1);
    if (a >= b) return;
    const long long x = S[b - 1 - t0] - (a > t0 ? S[a - 1 - t0] : 0);
    if (q0 >= t0 && q1 <= t1) f[r] = x;
    else atomicAdd(reinterpret_cast<unsigned long long *>(f + r), (unsigned long long)x);
  };
  if (r1 - r0 < 8 * TL_TILE) {
    for (int64_t r = r0 + threadIdx.x; r <= r1; r += TL_NT) put(r);
  } else {  // far more rows than entries (most are empty): every entry looks for its row, its first entry reports it
    for (int64_t q = t0 + threadIdx.x; q < t1; q += TL_NT) {
      int64_t l = r0, h = r1 + 1;  // last row that starts at or before q
      while (h - l > 1) {
        const int64_t mid = (l + h) >> 1;
        if (A.p[mid] <= q) l = mid;
        else h = mid;
      }
      if (max(A.p[l], t0) == q) put(l);
    }
  }
}
void launch_flops(const RowSet &A, const RightOp &B, int64_t *f, unsigned long long *zeros, cudaStream_t st) {
  if (A.nslots == 0 || A.nnz == 0) return;
  count_launch();
  k_entry_flops<<<(unsigned)((A.nnz + TL_TILE - 1) / TL_TILE), TL_NT, 0, st>>>(A, B, f, zeros);
}

// Rows per key, and (the last block) the keys' offsets.  stats[0] += total
// flops, stats[1] = max row flops, stats[2] = max row nnz of A, stats[3] +=
// min(f, n) over rows of the symbolic heavy bin, stats[4] += products of the
// tiny rows.  cnt (CSR only): the output
// counts, all set to zero here.
__global__ void __launch_bounds__(TL_NT) k_row_keys(RowSet A, const int64_t *f, int64_t *cnt, BinCounters c,
                                                    unsigned long long *stats, BinCfg bins, int64_t bn) {
  __shared__ int hist[NKEYS], s_last;
  __shared__ unsigned long long s_stats[5];  // (a block's atomics on the four words; one per warp took most of the kernel)
  for (int i = threadIdx.x; i < NKEYS; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x < 5) s_stats[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long my_tot = 0, my_max = 0, my_amax = 0, my_heavy = 0, my_tiny = 0;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < A.nslots;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t fr = f[r];
    if (cnt) cnt[r + 1] = 0;
    const int key = sym_key(fr, bins);
    if (key) atomicAdd(hist + key, 1);
    if (key >= KEY_HEAVY) my_heavy += (unsigned long long)min(fr, bn);
    if (key == KEY_TINY) my_tiny += (unsigned long long)fr;
    my_tot += (unsigned long long)fr;
    my_max = max(my_max, (unsigned long long)fr);
    my_amax = max(my_amax, (unsigned long long)max(A.p[r + 1] - A.p[r], (int64_t)0));
  }
  if (cnt && blockIdx.x == 0 && threadIdx.x == 0) cnt[0] = 0;
  my_tot = warp_sum(my_tot);
  my_heavy = warp_sum(my_heavy);
  my_tiny = warp_sum(my_tiny);
  my_max = warp_max(my_max);
  my_amax = warp_max(my_amax);
  if (lane_id() == 0) {
    if (my_tot) atomicAdd(s_stats + 0, my_tot);
    atomicMax(s_stats + 1, my_max);
    atomicMax(s_stats + 2, my_amax);
    if (my_heavy) atomicAdd(s_stats + 3, my_heavy);
    if (my_tiny) atomicAdd(s_stats + 4, my_tiny);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NKEYS; i += blockDim.x)
    if (hist[i]) atomicAdd(c.cnt + i, hist[i]);
  if (threadIdx.x < 5 && s_stats[threadIdx.x]) {
    if (threadIdx.x == 1 || threadIdx.x == 2) atomicMax(stats + threadIdx.x, s_stats[threadIdx.x]);
    else atomicAdd(stats + threadIdx.x, s_stats[threadIdx.x]);
  }
  if (last_block(c.ticket, &s_last) && threadIdx.x < 32) key_offsets(c.cnt, c.off, c.cur);
}
void launch_row_keys(const RowSet &A, const int64_t *f, int64_t *cnt, const BinCounters &c, unsigned long long *stats,
                     const BinCfg &bins, int64_t bn, cudaStream_t st) {
  if (A.nslots == 0) return;
  count_launch();
  k_row_keys<<<grid_for(A.nslots, TL_NT, 4), TL_NT, 0, st>>>(A, f, cnt, c, stats, bins, bn);
}

// Dropping the A entries whose B row is empty (their products are none, so
// C is unchanged): keep[q - lo] = 1 where nnz(B(A.j[q], :)) > 0; after an
// inclusive scan K of keep, entry q goes to K[q - lo] - 1 and row r starts at
// K[A.p[r] - 1 - lo].
__global__ void k_keep_flags(RowSet A, RightOp B, int64_t *keep) {
  const int64_t lo = A.p[0], n = min(A.p[A.nslots] - lo, A.nnz);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const int k = A.j[lo + x];
    keep[x] = HS_G(A.dbg, k >= 0 && k < B.m, 52, k) && B.p[k + 1] != B.p[k];
  }
}
__global__ void k_compact_entries(RowSet A, const int64_t *K, int32_t *j2, void *v2, int vb) {
  const int64_t lo = A.p[0], n = min(A.p[A.nslots] - lo, A.nnz);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t before = x > 0 ? K[x - 1] : 0;
    if (K[x] == before) continue;
    j2[before] = A.j[lo + x];
    if (vb == 8) reinterpret_cast<uint64_t *>(v2)[before] = reinterpret_cast<const uint64_t *>(A.v)[lo + x];
    else if (vb == 4) reinterpret_cast<uint32_t *>(v2)[before] = reinterpret_cast<const uint32_t *>(A.v)[lo + x];
  }
}
__global__ void k_compact_offsets(RowSet A, const int64_t *K, int64_t *p2) {
  const int64_t lo = A.p[0], n = min(A.p[A.nslots] - lo, A.nnz);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= A.nslots;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = min(max(A.p[r] - lo, (int64_t)0), n);
    p2[r] = x > 0 ? K[x - 1] : 0;
  }
}
void launch_compact_by_keep(const RowSet &A, const int64_t *K, int32_t *j2, void *v2, int vb, int64_t *p2,
                            cudaStream_t st) {
  count_launch();
  k_compact_entries<<<grid_for(A.nnz, 256, 8), 256, 0, st>>>(A, K, j2, v2, vb);
  count_launch();
  k_compact_offsets<<<grid_for(A.nslots + 1, 256, 8), 256, 0, st>>>(A, K, p2);
}
void launch_compact_a(const RowSet &A, const RightOp &B, int64_t *keep, int64_t *scan_tmp, int32_t *j2, void *v2,
                      int vb, int64_t *p2, cudaStream_t st) {
  count_launch();
  k_keep_flags<<<grid_for(A.nnz, 256, 8), 256, 0, st>>>(A, B, keep);
  launch_scan_i64(keep, A.nnz, scan_tmp, st);
  launch_compact_by_keep(A, keep, j2, v2, vb, p2, st);
}

// explicit zeros (value == 0; for floats +0 and -0 alike)
template <typename T> __global__ void k_keep_nonzero(const T *v, int64_t n, int64_t *keep) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
    keep[x] = v[x] != T(0);
}
void launch_keep_nonzero(const void *v, int dtype, int64_t n, int64_t *keep, cudaStream_t st) {
  if (n <= 0) return;
  count_launch();
  const int g = grid_for(n, 256, 8);
  switch (dtype) {
    case 0: k_keep_nonzero<<<g, 256, 0, st>>>(reinterpret_cast<const double *>(v), n, keep); break;
    case 1: k_keep_nonzero<<<g, 256, 0, st>>>(reinterpret_cast<const float *>(v), n, keep); break;
    case 2: k_keep_nonzero<<<g, 256, 0, st>>>(reinterpret_cast<const int32_t *>(v), n, keep); break;
    default: k_keep_nonzero<<<g, 256, 0, st>>>(reinterpret_cast<const int64_t *>(v), n, keep); break;
  }
}

// ---------------------------------------------------- B segment index
// Rows longer than min_len take the next table row and record, for every
// segment g = 0..nseg, the offset of their first entry with column >=
// g*SEG_W (nseg gives the row length).  Entry p fills the segments after its
// predecessor's up to its own; the last entry fills the rest.  A block takes
// 256 rows: a thread per row looks at its length, then a warp writes each
// longer row, and the whole block each row of more than BCI_LONG entries (a
// hub row of 4e4 entries walked by one warp set the kernel's time).
constexpr int BCI_NT = 256, BCI_LONG = 2048;
__device__ __forceinline__ void bci_row(const RightOp &B, int64_t b0, int len, int nseg, int32_t *row, int first,
                                        int step) {
  constexpr int U = 4;
  for (int q0 = first; q0 < len; q0 += U * step) {
    int c[U], cp[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u * step;
      c[u] = q < len ? __ldg(B.j + b0 + q) : 0;
      cp[u] = q > 0 && q < len ? __ldg(B.j + b0 + q - 1) : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u * step;
      if (q >= len) break;
      if (!HS_G(B.dbg, c[u] >= 0 && c[u] < B.n, 54, c[u])) continue;
      const int g = c[u] / SEG_W;
      const int gp = q ? (cp[u] >= 0 ? cp[u] / SEG_W : g) : -1;
      for (int x = gp + 1; x <= g && x <= nseg; ++x) row[x] = q;
      if (q == len - 1)
        for (int x = g + 1; x <= nseg; ++x) row[x] = len;
    }
  }
}
__global__ void __launch_bounds__(BCI_NT) k_build_bci(RightOp B, int nseg, int min_len, int64_t max_rows,
                                                      int32_t *bci_id, int32_t *bci, int *counter) {
  __shared__ int s_row[BCI_NT], s_long[BCI_NT], s_n, s_nlong;  // row within the block's 256
  __shared__ int s_t[BCI_NT];                                  // its table row
  const int64_t stride = (int64_t)nseg + 1;
  for (int64_t k0 = (int64_t)blockIdx.x * BCI_NT; k0 < B.m; k0 += (int64_t)gridDim.x * BCI_NT) {
    if (threadIdx.x == 0) s_n = s_nlong = 0;
    __syncthreads();
    const int64_t k = k0 + threadIdx.x;
    if (k < B.m) {
      const int64_t b0 = B.p[k], len = B.p[k + 1] - b0;
      int t = -1;
      if (len > min_len && len <= 0x7fffffffLL && HS_G(B.dbg, b0 >= 0 && b0 + len <= B.nnz, 53, b0)) {
        t = atomicAdd(counter, 1);
        if (t >= max_rows) t = -1;
      }
      bci_id[k] = t;
      s_t[threadIdx.x] = t;
      if (t >= 0) {
        if (len > BCI_LONG) s_long[atomicAdd(&s_nlong, 1)] = threadIdx.x;
        else s_row[atomicAdd(&s_n, 1)] = threadIdx.x;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x >> 5; i < s_n; i += BCI_NT / 32) {
      const int x = s_row[i];
      const int64_t b0 = B.p[k0 + x];
      bci_row(B, b0, (int)(B.p[k0 + x + 1] - b0), nseg, bci + s_t[x] * stride, lane_id(), 32);
    }
    for (int i = 0; i < s_nlong; ++i) {
      const int x = s_long[i];
      const int64_t b0 = B.p[k0 + x];
      bci_row(B, b0, (int)(B.p[k0 + x + 1] - b0), nseg, bci + s_t[x] * stride, threadIdx.x, BCI_NT);
    }
    __syncthreads();
  }
}

void launch_build_bci(const RightOp &B, int nseg, int min_len, int64_t max_rows, int32_t *bci_id, int32_t *bci,
                      int *counter, cudaStream_t st) {
  if (B.m <= 0) return;
  count_launch();
  k_build_bci<<<grid_for(B.m, BCI_NT, 8), BCI_NT, 0, st>>>(B, nseg, min_len, max_rows, bci_id, bci, counter);
}

// The tile's rows (row u*TL_NT + x of the tile with key key[u] of thread x;
// key 0: none) appended to the lists of their keys: counted per key in shared
// memory, one atomic per key and block.  s_cnt: NKEYS zeroed counters; two
// barriers.
__device__ __forceinline__ void append_tile(const int (&key)[TL_PER], int64_t r0, int *s_cnt, int *key_cur, int *list,
                                            int64_t cap, long long *dbg) {
  int at[TL_PER];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const unsigned grp = __match_any_sync(FULL, key[u]);
    const int leader = __ffs(grp) - 1;
    int base = 0;
    if (lane_id() == leader && key[u]) base = atomicAdd(s_cnt + key[u], __popc(grp));
    at[u] = __shfl_sync(FULL, base, leader) + __popc(grp & ((1u << lane_id()) - 1));
  }
  __syncthreads();
  if (threadIdx.x < NKEYS && s_cnt[threadIdx.x]) s_cnt[threadIdx.x] = atomicAdd(key_cur + threadIdx.x, s_cnt[threadIdx.x]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    if (!key[u]) continue;
    const int64_t x = (int64_t)s_cnt[key[u]] + at[u];
    if (HS_G(dbg, x >= 0 && x < cap, 52, x)) list[x] = (int)(r0 + u * TL_NT + threadIdx.x);
  }
}

__global__ void __launch_bounds__(TL_NT) k_scatter_sym(RowSet A, const int64_t *f, int *key_cur, int *list,
                                                       int32_t *hslot, int *nhist, BinCfg bins) {
  __shared__ int s_cnt[NKEYS], s_h;
  if (threadIdx.x < NKEYS) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == NKEYS) s_h = 0;
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  int key[TL_PER], slot[TL_PER];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    const int64_t fr = r < A.nslots ? f[r] : 0;
    key[u] = sym_key(fr, bins);
    // rows that may need column parts in the numeric pass (every row of the
    // bitmap kernel) get a histogram slot
    const bool h = fr > bins.sym_heavy_from;
    const unsigned hm = __ballot_sync(FULL, h);
    int base = 0;
    if (lane_id() == 0 && hm) base = atomicAdd(&s_h, __popc(hm));
    base = __shfl_sync(FULL, base, 0);
    slot[u] = h ? base + __popc(hm & ((1u << lane_id()) - 1)) : -1;
  }
  append_tile(key, r0, s_cnt, key_cur, list, A.nslots, A.dbg);
  if (threadIdx.x == 0 && s_h) s_h = atomicAdd(nhist, s_h);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    if (r < A.nslots) hslot[r] = slot[u] >= 0 ? s_h + slot[u] : -1;
  }
}

void launch_scatter_sym(const RowSet &A, const int64_t *f, int *key_cur, int *list, int32_t *hslot, int *nhist,
                        const BinCfg &bins, cudaStream_t st) {
  if (A.nslots == 0) return;
  count_launch();
  k_scatter_sym<<<(unsigned)((A.nslots + TL_TILE - 1) / TL_TILE), TL_NT, 0, st>>>(A, f, key_cur, list, hslot, nhist,
                                                                                 bins);
}

// ------------------------------------------- C's offsets and numeric bins
// Two kernels: the first counts the rows of every numeric key and sums the
// output counts of each tile of rows, and its last block turns both into
// offsets; the second scans each tile's counts from its offset into C's row
// offsets and, as it holds the counts, appends its rows to their lists.  (A
// scan of three to five kernels, a pass for the keys and a third for the
// lists made 18 launches of a 4096-row product; it now makes 10, 225 -> 187 us.)  For DCSR the rows
// of the lists are not those of the scan: the lists are written by a kernel of
// their own in between.
__device__ __forceinline__ int64_t raw_count(const RowSet &A, const int64_t *cnt, int64_t slot) {
  const int64_t o = A.ids ? (int64_t)A.ids[slot] : slot;
  return HS_G(A.dbg, o >= 0 && o < A.m, 30, o) ? cnt[o + 1] : 0;
}
__global__ void __launch_bounds__(TL_NT) k_num_count(RowSet A, const int64_t *f, const int64_t *cnt, BinCfg bins,
                                                     BinCounters c, int64_t *tsum, int64_t tiles, long long *nnz) {
  __shared__ int hist[NKEYS], s_last;
  __shared__ long long s_w[64];
  for (int i = threadIdx.x; i < NKEYS; i += TL_NT) hist[i] = 0;
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  long long sum = 0;
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    const int64_t n = r < A.m ? cnt[r + 1] : 0;
    sum += n;
    if (r < A.nslots) {
      const int64_t entries = A.p[r + 1] - A.p[r];
      const int key = row_key(f[r], A.ids ? raw_count(A, cnt, r) : n, entries, bins);
      if (key) atomicAdd(hist + key, 1);
      const int level = hub_level(key, entries);
      if (level >= 0) {  // (few: a row for every 4096 entries at most)
        atomicAdd(&c.hub->n[level][key - KEY_TINY - 1], 1);
        c.hub->any = 1;
      }
    }
  }
  sum = warp_sum(sum);
  if (lane_id() == 0) s_w[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < TL_NW; ++w) t += s_w[w];
    tsum[blockIdx.x] = t;
  }
  for (int i = threadIdx.x; i < NKEYS; i += TL_NT)
    if (hist[i]) atomicAdd(c.cnt + i, hist[i]);
  if (!last_block(c.ticket, &s_last)) return;
  if (threadIdx.x < 32) key_offsets(c.cnt, c.off, c.cur, c.hub);
  // exclusive scan of the tile sums, in place
  long long run = 0;
  for (int64_t b = 0; b < tiles; b += TL_TILE) {
    long long v[TL_PER], x[TL_PER];
#pragma unroll
    for (int u = 0; u < TL_PER; ++u) {
      const int64_t i = b + u * TL_NT + threadIdx.x;
      v[u] = x[u] = i < tiles ? __ldcg(tsum + i) : 0;
    }
    __syncthreads();  // s_w: the previous use is over
    const long long t = tile_scan(v, s_w);
#pragma unroll
    for (int u = 0; u < TL_PER; ++u) {
      const int64_t i = b + u * TL_NT + threadIdx.x;
      if (i < tiles) tsum[i] = run + v[u] - x[u];
    }
    run += t;
  }
  if (threadIdx.x == 0) *nnz = run;
}
template <bool LISTS>
__global__ void __launch_bounds__(TL_NT) k_num_offsets(RowSet A, const int64_t *f, int64_t *cnt, BinCfg bins,
                                                       BinCounters c, const int64_t *tsum, int *list) {
  __shared__ int s_cnt[NKEYS];
  __shared__ long long s_tot[64];
  if (threadIdx.x < NKEYS) s_cnt[threadIdx.x] = 0;
  const int from = c.hub->from;
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  long long v[TL_PER];
  int key[TL_PER];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    v[u] = r < A.m ? cnt[r + 1] : 0;
    key[u] = 0;
    if constexpr (LISTS)
      if (r < A.nslots) {
        const int64_t entries = A.p[r + 1] - A.p[r];
        key[u] = hub_key(row_key(f[r], v[u], entries, bins), entries, from);
      }
  }
  tile_scan(v, s_tot);
  const int64_t base = tsum[blockIdx.x];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    if (r < A.m) cnt[r + 1] = base + v[u];
  }
  if constexpr (LISTS) append_tile(key, r0, s_cnt, c.cur, list, A.nslots, A.dbg);
}
__global__ void __launch_bounds__(TL_NT) k_num_lists(RowSet A, const int64_t *f, const int64_t *cnt, BinCfg bins,
                                                     BinCounters c, int *list) {
  __shared__ int s_cnt[NKEYS];
  if (threadIdx.x < NKEYS) s_cnt[threadIdx.x] = 0;
  const int from = c.hub->from;
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  int key[TL_PER];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t r = r0 + u * TL_NT + threadIdx.x;
    const int64_t entries = r < A.nslots ? A.p[r + 1] - A.p[r] : 0;
    key[u] = r < A.nslots ? hub_key(row_key(f[r], raw_count(A, cnt, r), entries, bins), entries, from) : 0;
  }
  append_tile(key, r0, s_cnt, c.cur, list, A.nslots, A.dbg);
}
void launch_num_bins(const RowSet &A, const int64_t *f, int64_t *cnt, const BinCfg &bins, const BinCounters &c,
                     int64_t *tsum, long long *nnz, int *list, cudaStream_t st) {
  const int64_t rows = A.m > A.nslots ? A.m : A.nslots;
  if (rows <= 0) return;
  const int64_t tiles = (rows + TL_TILE - 1) / TL_TILE;
  count_launch();
  k_num_count<<<(unsigned)tiles, TL_NT, 0, st>>>(A, f, cnt, bins, c, tsum, tiles, nnz);
  if (A.ids) {
    count_launch();
    k_num_lists<<<(unsigned)((A.nslots + TL_TILE - 1) / TL_TILE), TL_NT, 0, st>>>(A, f, cnt, bins, c, list);
    count_launch();
    k_num_offsets<false><<<(unsigned)tiles, TL_NT, 0, st>>>(A, f, cnt, bins, c, tsum, list);
  } else {
    count_launch();
    k_num_offsets<true><<<(unsigned)tiles, TL_NT, 0, st>>>(A, f, cnt, bins, c, tsum, list);
  }
}

// ------------------------------------------------------------------- scan
// Inclusive prefix sum of an int64 array, in place, by two kernels: the sums
// of tiles of TL_TILE elements, then every tile's scan from the sum of the
// tiles before it.  Each block of the second kernel adds those sums itself
// (an array of up to 2^12 tiles, 8.4e6 elements, is a few coalesced reads
// from L2); for longer arrays they are scanned by a recursion.
constexpr int64_t SCAN_FLAT = 1 << 12;
__global__ void __launch_bounds__(TL_NT) k_scan_sums(const int64_t *a, int64_t n, int64_t *tot) {
  __shared__ long long s_w[TL_NW];
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  long long s = 0;
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t i = r0 + u * TL_NT + threadIdx.x;
    s += i < n ? a[i] : 0;
  }
  s = warp_sum(s);
  if (lane_id() == 0) s_w[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < TL_NW; ++w) t += s_w[w];
    tot[blockIdx.x] = t;
  }
}
// tot: the tiles' sums (flat) or their inclusive scan; null: a single tile
__global__ void __launch_bounds__(TL_NT) k_scan_apply(int64_t *a, int64_t n, const int64_t *tot, bool flat) {
  __shared__ long long s_tot[64], s_w[TL_NW];
  const int64_t r0 = (int64_t)blockIdx.x * TL_TILE;
  long long v[TL_PER];
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t i = r0 + u * TL_NT + threadIdx.x;
    v[u] = i < n ? a[i] : 0;
  }
  long long base = 0;
  if (tot && flat) {
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += TL_NT) base += tot[i];
    base = warp_sum(base);
    if (lane_id() == 0) s_w[threadIdx.x >> 5] = base;
  } else if (tot && blockIdx.x) {
    base = tot[blockIdx.x - 1];
  }
  tile_scan(v, s_tot);  // (its barrier also publishes s_w)
  if (tot && flat) {
    base = 0;
    for (int w = 0; w < TL_NW; ++w) base += s_w[w];
  }
#pragma unroll
  for (int u = 0; u < TL_PER; ++u) {
    const int64_t i = r0 + u * TL_NT + threadIdx.x;
    if (i < n) a[i] = base + v[u];
  }
}

int64_t scan_tmp_elems(int64_t n) {
  int64_t t = 0;
  while (n > TL_TILE) {
    n = (n + TL_TILE - 1) / TL_TILE;
    t += n;
  }
  return t + 1;
}

void launch_scan_i64(int64_t *a, int64_t n, int64_t *tmp, cudaStream_t st) {
  if (n <= 0) return;
  const int64_t tiles = (n + TL_TILE - 1) / TL_TILE;
  if (tiles > 1) {
    count_launch();
    k_scan_sums<<<(unsigned)tiles, TL_NT, 0, st>>>(a, n, tmp);
    if (tiles > SCAN_FLAT) launch_scan_i64(tmp, tiles, tmp + tiles, st);
  }
  count_launch();
  k_scan_apply<<<(unsigned)tiles, TL_NT, 0, st>>>(a, n, tiles > 1 ? tmp : nullptr, tiles <= SCAN_FLAT);
}

// -------------------------------------------------------------- validation
// flag bit 1: a column id outside [0, ncols); bit 2: a row not strictly
// increasing; bit 4: row offsets decreasing.
__global__ void k_validate(const int64_t *p, const int32_t *j, int64_t rows, int64_t ncols, int *flag) {
  const int lane = lane_id();
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t r = blockIdx.x * wpb + (threadIdx.x >> 5); r < rows; r += (int64_t)gridDim.x * wpb) {
    const int64_t q0 = p[r], q1 = p[r + 1];
    if (q1 < q0) {
      if (lane == 0) atomicOr(flag, 4);
      continue;
    }
    int bad = 0;
    for (int64_t q = q0 + lane; q < q1; q += 32) {
      const int c = j[q];
      if (c < 0 || c >= ncols) bad |= 1;
      if (q > q0 && j[q - 1] >= c) bad |= 2;
    }
    bad = __reduce_or_sync(FULL, bad);
    if (lane == 0 && bad) atomicOr(flag, bad);
  }
}

void launch_validate(const int64_t *p, const int32_t *j, int64_t rows, int64_t ncols, int *flag, cudaStream_t st) {
  if (rows <= 0) return;
  count_launch();
  k_validate<<<grid_for(rows, 8, 16), 256, 0, st>>>(p, j, rows, ncols, flag);
}

// ------------------------------------------------------- heavy row parts
// A heavy row's columns are cut into parts of whole SEG_W-column segments:
// a part takes segments in order while its outputs stay within caph and its
// span within `span` segments (a segment holds at most SEG_W <= caph
// outputs, so every segment fits a part of its own; were one to hold more,
// its part would carry its true count, which the numeric kernel rejects);
// parts without outputs are dropped.  One warp per row: the warp stages the
// row's segment counts in shared memory, WP_STAGE at a time, and lane 0 walks
// them (the greedy cut is sequential; plain shared loads keep its chain
// short); `emit(part, seg_lo, seg_hi, pc, done)` runs on lane 0 (done: the
// row's outputs before the part).  Every lane returns the part count.
constexpr int WP_NT = 256;     // threads of the planning kernels
constexpr int WP_STAGE = 256;  // segment counts staged per warp at a time
template <class Emit>
__device__ __forceinline__ int walk_parts(const uint32_t *hist, int nseg, int caph, int span, uint32_t *stage,
                                          Emit &&emit) {
  const int lane = lane_id();
  int start = 0, sum = 0, parts = 0;
  long long done = 0;
  for (int g0 = 0; g0 < nseg; g0 += WP_STAGE) {
    const int lim = min(WP_STAGE, nseg - g0);
    __syncwarp();  // lane 0 is done with the previous counts
    for (int j = lane; j < lim; j += 32) stage[j] = hist[g0 + j];
    __syncwarp();
    if (lane == 0) {
#pragma unroll 8
      for (int j = 0; j < lim; ++j) {
        const int x = (int)stage[j];
        const int g = g0 + j;
        if (g - start >= span || sum + x > caph) {
          if (sum > 0) {
            emit(parts, start, g, sum, done);
            ++parts;
            done += sum;
          }
          start = g;
          sum = 0;
        }
        sum += x;
      }
    }
  }
  if (lane == 0 && sum > 0) {
    emit(parts, start, nseg, sum, done);
    ++parts;
  }
  return __shfl_sync(FULL, parts, 0);
}

__global__ void k_count_parts(RowSet A, const int *list, const int *key_off, int key_lo, const int32_t *hslot,
                              const uint32_t *hist, const int64_t *loff, int nseg, int caph, int span, int64_t nmax,
                              int64_t *cnt, int64_t *cap) {
  const int lane = lane_id();
  const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int lo = key_off[key_lo];
  const int64_t count = key_off[NKEYS] - lo;
  __shared__ uint32_t s_stage[WP_NT / 32][WP_STAGE];
  uint32_t *stage = s_stage[threadIdx.x >> 5];
  for (int64_t w = wid; w < nmax; w += nw) {
    int64_t parts = 0, room = 0;
    if (w < count) {
      const int r = list[lo + w];
      const int h = (r >= 0 && r < A.nslots) ? hslot[r] : -1;
      if (h >= 0 && loff[r] >= 0) {
        parts = walk_parts(hist + (int64_t)h * nseg, nseg, caph, span, stage, [](int, int, int, int, long long) {});
        room = parts * (A.p[r + 1] - A.p[r]);
      }
    }
    if (lane == 0) {
      cnt[w] = parts;
      cap[w] = room;
    }
  }
}

void launch_count_parts(const RowSet &A, const int *list, const int *key_off, int key_lo, const int32_t *hslot,
                        const uint32_t *hist, const int64_t *loff, int nseg, int caph, int span, int64_t nmax,
                        int64_t *cnt, int64_t *cap, cudaStream_t st) {
  if (nmax <= 0) return;
  count_launch();
  k_count_parts<<<grid_for(nmax, WP_NT / 32, 16), WP_NT, 0, st>>>(A, list, key_off, key_lo, hslot, hist, loff, nseg, caph,
                                                       span, nmax, cnt, cap);
}

__global__ void k_plan_parts(RowSet A, const int *list, int count, const int32_t *hslot, const uint32_t *hist,
                             const int64_t *loff, const int64_t *Cp, int nseg, int caph, int span,
                             const int64_t *off, const int64_t *poff, HeavyUnit *units) {
  const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ uint32_t s_stage[WP_NT / 32][WP_STAGE];
  uint32_t *stage = s_stage[threadIdx.x >> 5];
  for (int64_t w = wid; w < count; w += nw) {
    const int r = list[w];
    const int h = (r >= 0 && r < A.nslots) ? hslot[r] : -1;
    if (h < 0 || loff[r] < 0) continue;
    const int64_t base = w ? off[w - 1] : 0;
    const int64_t end = off[w];
    const int64_t pbase = w ? poff[w - 1] : 0;
    const int64_t nq = A.p[r + 1] - A.p[r];
    const int64_t o = A.ids ? (int64_t)A.ids[r] : (int64_t)r;
    const int64_t cb = Cp[o], c = Cp[o + 1] - cb, lb = loff[r];
    walk_parts(hist + (int64_t)h * nseg, nseg, caph, span, stage, [&](int p, int s0, int s1, int pc, long long done) {
      // a part must lie inside its row (else pc 0: the numeric kernel rejects the unit)
      const bool fits = HS_G(A.dbg, done + pc <= c, 74, done);
      if (base + p < end)
        units[base + p] = HeavyUnit{r, s0, s1, fits ? pc : 0, done, pbase + p * nq, 0, 0, cb + done,
                                    lb + (lb & LIST_BITS ? (long long)s0 * (SEG_W / 32) : done)};
    });
  }
}

void launch_plan_parts(const RowSet &A, const int *list, int count, const int32_t *hslot, const uint32_t *hist,
                       const int64_t *loff, const int64_t *Cp, int nseg, int caph, int span, const int64_t *off,
                       const int64_t *poff, HeavyUnit *units, cudaStream_t st) {
  if (count <= 0) return;
  count_launch();
  k_plan_parts<<<grid_for(count, WP_NT / 32, 16), WP_NT, 0, st>>>(A, list, count, hslot, hist, loff, Cp, nseg, caph, span, off,
                                                       poff, units);
}

// The B segments of the units.  A warp takes `group` consecutive units; those
// of one row are filled together, from one pass over the row's A entries, 32
// at a time: a lane holds an entry's B row and the end of its last segment,
// and every unit of the row takes the entry's next segment up to the unit's
// last column (from the segment index, whose offsets of neighbouring
// segments share a cache line, or by a short search of a B row without one),
// the non-empty ones compacted by ballot.  Bound by the instructions per
// (entry, unit) and the latency of the entry -> B row -> index chain: one
// warp per unit went through the entries and B offsets again for each of a
// row's units, and scanned the products of its segments, which the unit
// kernel now does as it copies them.  The searches of many units run at
// once, so their latency is hidden here instead of sitting on the numeric
// kernel's path.  A row with more than long_from entries of A is left to
// k_build_pairs_long: a block per unit, four entries per thread at a time
// (the few units of a product with 1e5-entry rows of A would keep one warp
// each busy long after the others are done).
constexpr int PAIR_NT = 256, PAIR_U = 4, PAIR_GROUP = 8, PAIR_LONG = 1024, PAIR_SHARE = 2;
// consecutive units per warp: as few as leave no warp of the GPU a second group
static int64_t pair_warps() { return (int64_t)sm_count() * 40; }
static int pair_group(int64_t nunits) {
  const int64_t g = (nunits + pair_warps() - 1) / pair_warps();
  return (int)(g < 1 ? 1 : (g > PAIR_GROUP ? PAIR_GROUP : g));
}
// A row is long when a warp's group of its units is more than PAIR_SHARE times
// the warp's share of the whole layout (`entries`, summed over the units): rows
// that are all long keep every warp as busy as blocks do, and are gone through
// once for several units (3000 rows of 5000 / 10,000 entries, eight units each:
// a numeric pass 1.39 / 2.63 ms, by blocks 1.77 / 3.28, the warps in one and a
// third rounds of smaller groups 1.74 / 3.49; R-MAT scale 20, whose rows have up
// to 23,000 entries: the layout 4.6 -> 2.5 ms, the product 67.9 -> 65.8 ms).  At
// four times the share, 300 such rows took 377 / 704 us, by blocks 207 / 360.
int64_t pair_long_from(int64_t nunits, int64_t entries, int64_t longest) {
  const int64_t share = PAIR_SHARE * (entries / (pair_warps() * pair_group(nunits)));
  const int64_t from = share > PAIR_LONG ? share : PAIR_LONG;
  return longest > from ? from : INT64_MAX;
}
template <int AB> struct PairVal {
  using T = typename std::conditional<AB == 8, unsigned long long, unsigned>::type;
};
// evict-first: the pairs are read once, later; B and the segment index stay
// in L2 for this kernel and the unit kernel after it
template <int AB>
__device__ __forceinline__ void pair_put(int64_t at, int64_t s0, int len, typename PairVal<AB>::T av, int64_t *pseg,
                                         void *paval) {
  __stcs(reinterpret_cast<long long *>(pseg) + at, (long long)pair_pack(s0, len));
  if constexpr (AB > 0) __stcs(reinterpret_cast<typename PairVal<AB>::T *>(paval) + at, av);
}
__device__ __forceinline__ bool unit_ok(const RowSet &A, const HeavyUnit &u, int nseg, int64_t ui) {
  return HS_G(A.dbg, u.row >= 0 && u.row < A.nslots && u.seg_lo >= 0 && u.seg_lo < u.seg_hi && u.seg_hi <= nseg, 75,
              ui);
}
// B row of A entry q (false: none), and its row of the segment index
__device__ __forceinline__ bool pair_row(const RowSet &A, const RightOp &B, int64_t q, const int32_t *bci_id,
                                         int64_t &base, int64_t &end, int &t) {
  if (!HS_G(A.dbg, q >= 0 && q < A.nnz, 1, q)) return false;
  const int k = __ldg(A.j + q);
  if (!HS_G(A.dbg, k >= 0 && k < B.m, 2, k)) return false;
  base = __ldg(B.p + k);
  end = __ldg(B.p + k + 1);
  t = bci_id ? __ldg(bci_id + k) : -1;
  return HS_G(A.dbg, base >= 0 && base <= end && end <= B.nnz, 3, end);
}
// first entry of the B row at or after s whose segment is >= seg
__device__ __forceinline__ int64_t pair_end(const RightOp &B, int64_t base, int64_t s, int64_t end, int t, int seg,
                                            const int32_t *bci, int64_t bstride) {
  if (t >= 0) return base + __ldg(bci + (int64_t)t * bstride + seg);
  const int64_t x = (int64_t)seg * SEG_W;
  return x > 0x7fffffffLL ? end : gallop_lower_bound(B.j, s, end, (int)x);
}

template <int AB>
__global__ void __launch_bounds__(PAIR_NT) k_build_pairs(RowSet A, RightOp B, HeavyUnit *units, int64_t nunits,
                                                         const int32_t *bci_id, const int32_t *bci, int nseg,
                                                         int64_t *pseg, void *paval, int group, int64_t long_from) {
  using VT = typename PairVal<AB>::T;
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t bstride = (int64_t)nseg + 1;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g * group < nunits; g += nw) {
    const int64_t ua = g * group;
    const int cnt = (int)min((int64_t)group, nunits - ua);
    // lane j holds unit ua + j: its row (-1: skipped), segments and the next
    // free place of its slice
    int row = -1, slo = 0, shi = 0;
    int64_t at = 0, poff = 0;
    if (lane < cnt) {
      const HeavyUnit u = units[ua + lane];
      if (unit_ok(A, u, nseg, ua + lane)) row = u.row;
      slo = u.seg_lo;
      shi = u.seg_hi;
      at = poff = u.poff;
    }
    for (int j0 = 0; j0 < cnt;) {
      const int r = __shfl_sync(FULL, row, j0);
      const unsigned same = __ballot_sync(FULL, lane >= j0 && lane < cnt && row == r) >> j0;
      const int run = __ffs(~same) - 1;  // consecutive units of row r (group <= 8, so ~same is not 0)
      const int j1 = j0 + run;
      const int64_t q0 = r >= 0 ? A.p[r] : 0, q1 = r >= 0 ? A.p[r + 1] : 0;
      if (q1 - q0 <= long_from) {
        const int lo0 = __shfl_sync(FULL, slo, j0);
        for (int64_t qb = q0; qb < q1; qb += 32) {
          const int64_t q = qb + lane;
          int64_t base = 0, end = 0, s = 0;
          int t = -1;
          VT av = 0;
          if (q < q1 && pair_row(A, B, q, bci_id, base, end, t)) {
            s = lo0 ? pair_end(B, base, base, end, t, lo0, bci, bstride) : base;
            if (!HS_G(A.dbg, s >= base && s <= end, 65, s)) s = end;
            if constexpr (AB > 0)
              if (s < end) av = __ldg(reinterpret_cast<const VT *>(A.v) + q);
          }
          // the index's offsets for all units of the run first: their loads are in flight together
          int off[PAIR_GROUP];
#pragma unroll
          for (int i = 0; i < PAIR_GROUP; ++i) {
            const int hi = __shfl_sync(FULL, shi, (j0 + i) & 31);
            off[i] = i < run && t >= 0 ? __ldg(bci + (int64_t)t * bstride + hi) : 0;
          }
#pragma unroll
          for (int i = 0; i < PAIR_GROUP; ++i) {
            if (i >= run) break;
            const int hi = __shfl_sync(FULL, shi, j0 + i);
            const int64_t to = __shfl_sync(FULL, at, j0 + i);
            int64_t e = s;
            if (s < end) {
              e = t >= 0 ? base + off[i] : pair_end(B, base, s, end, -1, hi, bci, bstride);
              if (!HS_G(A.dbg, e >= s && e <= end, 65, e)) e = s;
            }
            const unsigned m = __ballot_sync(FULL, e > s);
            if (e > s) pair_put<AB>(to + __popc(m & ((1u << lane) - 1u)), s, (int)(e - s), av, pseg, paval);
            if (lane == j0 + i) at += __popc(m);
            s = e;
          }
        }
        if (lane >= j0 && lane < j1) units[ua + lane].npairs = (int32_t)(at - poff);
      }
      j0 = j1;
    }
  }
}

template <int AB>
__global__ void __launch_bounds__(PAIR_NT) k_build_pairs_long(RowSet A, RightOp B, HeavyUnit *units, int64_t nunits,
                                                              const int32_t *bci_id, const int32_t *bci, int nseg,
                                                              int64_t *pseg, void *paval, int64_t long_from) {
  using VT = typename PairVal<AB>::T;
  constexpr int NW = PAIR_NT / 32;
  __shared__ int s_long[PAIR_NT], s_n;
  __shared__ int s_w[NW];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const int64_t bstride = (int64_t)nseg + 1;
  // units are dealt to the blocks one by one (a hub row's units are
  // neighbours): block b looks at units b, b + gridDim, ...
  for (int64_t v0 = 0; v0 * gridDim.x < nunits; v0 += PAIR_NT) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t mine = (v0 + threadIdx.x) * gridDim.x + blockIdx.x;
    if (mine < nunits) {
      const HeavyUnit u = units[mine];
      if (unit_ok(A, u, nseg, mine) && A.p[u.row + 1] - A.p[u.row] > long_from)
        s_long[atomicAdd(&s_n, 1)] = threadIdx.x;
    }
    __syncthreads();
    const int n = s_n;
    for (int i = 0; i < n; ++i) {
      const int64_t vi = (v0 + s_long[i]) * gridDim.x + blockIdx.x;
      const HeavyUnit u = units[vi];
      const int64_t q0 = A.p[u.row], q1 = A.p[u.row + 1];
      int out = 0;
      for (int64_t qb = q0; qb < q1; qb += PAIR_U * PAIR_NT) {
        int64_t s[PAIR_U];
        int len[PAIR_U];
        VT av[PAIR_U];
        int c = 0;
#pragma unroll
        for (int k = 0; k < PAIR_U; ++k) {
          const int64_t q = qb + k * PAIR_NT + threadIdx.x;
          int64_t base = 0, end = 0;
          int t = -1;
          s[k] = 0;
          len[k] = 0;
          av[k] = 0;
          if (q < q1 && pair_row(A, B, q, bci_id, base, end, t) && base < end) {
            s[k] = u.seg_lo ? pair_end(B, base, base, end, t, u.seg_lo, bci, bstride) : base;
            const int64_t e = pair_end(B, base, s[k], end, t, u.seg_hi, bci, bstride);
            if (HS_G(A.dbg, base <= s[k] && s[k] <= e && e <= end, 65, e)) len[k] = (int)(e - s[k]);
            if constexpr (AB > 0)
              if (len[k] > 0) av[k] = __ldg(reinterpret_cast<const VT *>(A.v) + q);
          }
          c += len[k] > 0;
        }
        const int incl = warp_incl_scan(c);
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        int before = incl - c, all = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          before += w < warp ? s_w[w] : 0;
          all += s_w[w];
        }
        int64_t to = u.poff + out + before;
#pragma unroll
        for (int k = 0; k < PAIR_U; ++k)
          if (len[k] > 0) pair_put<AB>(to++, s[k], len[k], av[k], pseg, paval);
        out += all;
        __syncthreads();
      }
      if (threadIdx.x == 0) units[vi].npairs = out;
    }
    __syncthreads();
  }
}

void launch_build_pairs(const RowSet &A, const RightOp &B, HeavyUnit *units, int64_t nunits, const int32_t *bci_id,
                        const int32_t *bci, int nseg, int a_bytes, int64_t long_from, int64_t *pseg, void *paval,
                        cudaStream_t st) {
  if (nunits <= 0) return;
  const int group = pair_group(nunits);
  const int g = grid_for((nunits + group - 1) / group, PAIR_NT / 32, 16);
  const int gl = grid_for(nunits, 1, 4);
#define HS_PAIRS(AB)                                                                                              \
  do {                                                                                                            \
    count_launch();                                                                                               \
    k_build_pairs<AB><<<g, PAIR_NT, 0, st>>>(A, B, units, nunits, bci_id, bci, nseg, pseg, paval, group, long_from); \
    if (long_from < INT64_MAX) {                                                                                             \
      count_launch();                                                                                             \
      k_build_pairs_long<AB><<<gl, PAIR_NT, 0, st>>>(A, B, units, nunits, bci_id, bci, nseg, pseg, paval, long_from); \
    }                                                                                                             \
  } while (0)
  if (a_bytes == 8) HS_PAIRS(8);
  else if (a_bytes == 4) HS_PAIRS(4);
  else HS_PAIRS(0);
#undef HS_PAIRS
}

}  // namespace hs
