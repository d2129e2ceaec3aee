// symbolic.cu -- output nonzeros per row of C = A*B (structure only).
//
// The row-wise form of Algorithm 1 with the sparse accumulator of Figure 1
// reduced to its occupancy part: each row's distinct output columns are
// counted by the accumulator its bin selects.
//   tiny  (f <= 32)    several rows to a warp, one product per lane, equal
//                      columns of a row found with __match_any_sync;
//   warp  (f <= 1024)  one warp, private shared-memory hash set; or a bitmap
//                      of B's columns where they fit its room, else, for at
//                      most 64 products, a sort in registers;
//   mid   (f <= 4096)  one CTA, shared hash set of 2f slots (at most 8192) or
//                      a bitmap;
//   large (f <= min(16384, cap_large), so f <= 8192)
//                      one CTA, shared hash set of up to 16384 slots;
//   heavy (larger f)   one CTA, a bitmap over 2^20 columns (occupancy SPA in
//                      shared memory), rows handed out largest first.  The
//                      bitmap is read out in column order, so the kernel also
//                      writes the row's sorted column list (a dense row's
//                      bitmap) for the numeric pass, which then only has to
//                      place values.
// Rows with more than cap_large products also get per-column-segment counts
// (4096-column segments) from which the numeric pass plans its column parts.
// Counts go to cnt[row + 1] so an inclusive scan turns them into row offsets.
#include "common.cuh"
#include "internal.h"
#include "sortrow.cuh"

namespace hs {

using StructSR = Semiring<OR_AND, NoVal>;

__device__ __forceinline__ DevCsr dev_a(const RowSet &A) { return DevCsr{A.p, A.j, A.v, A.nslots, A.nnz, A.dbg}; }
__device__ __forceinline__ DevCsr dev_b(const RightOp &B) { return DevCsr{B.p, B.j, B.v, B.m, B.nnz, B.dbg}; }
// count of output row o goes to cnt[o + 1]
__device__ __forceinline__ void put_count(const SymArgs &a, int64_t o, int64_t v) {
  if (HS_G(a.A.dbg, o >= 0 && o < a.A.m, 30, o)) a.cnt[o + 1] = v;
}
__device__ __forceinline__ int64_t out_row(const RowSet &A, int r) { return A.ids ? (int64_t)A.ids[r] : (int64_t)r; }

// --------------------------------------------------------------- tiny
constexpr int TINY_WPB = 8;
__global__ void __launch_bounds__(TINY_WPB * 32, 4) k_sym_tiny(SymArgs a) {
  __shared__ int scol[TINY_WPB][32];
  const int w = threadIdx.x >> 5, lane = lane_id();
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int step = gridDim.x * TINY_WPB;
  int idx = blockIdx.x * TINY_WPB + w;
  RowAhead<StructSR> x, nx;
  x.all(A, B, a.list, idx, a.count);
  for (; idx < a.count; idx += step) {
    nx.row(A, a.list, idx + step, a.count);
    auto put = [&](int col, NoVal, int p) {
      if (HS_G(a.A.dbg, p < 32, 34, p)) scol[w][p] = col;
    };
    const int nprod = x.r >= 0 ? warp_products_of<StructSR>(A, B, x, put) : 0;
    nx.range(A);
    __syncwarp();
    const bool have = lane < nprod && lane < 32;
    const int col = have ? scol[w][lane] : 0;
    nx.entries(A);
    const unsigned act = __ballot_sync(FULL, have);
    bool first = false;
    if (have) {
      const unsigned grp = __match_any_sync(act, col);
      first = lane == __ffs(grp) - 1;
    }
    const int cnt = __popc(__ballot_sync(FULL, first));
    nx.segments(B);
    if (lane == 0 && x.r >= 0) {
      put_count(a, out_row(a.A, x.r), cnt);
      if (nprod > 32) atomicExch(a.err, 2);
    }
    __syncwarp();
    x = nx;
  }
}

// the same rows, several to a warp at a time (tiny_group): for long lists of
// rows of few products (tiny_group_pays)
__global__ void __launch_bounds__(TINY_WPB * 32, 4) k_sym_tiny_group(SymArgs a) {
  __shared__ int scol[TINY_WPB][32];
  const int w = threadIdx.x >> 5, lane = lane_id();
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int per = (a.count + gridDim.x * TINY_WPB - 1) / (gridDim.x * TINY_WPB);
  const int64_t first = (int64_t)(blockIdx.x * TINY_WPB + w) * per;
  const int end = (int)min(first + per, (int64_t)a.count);
  int idx = (int)min(first, (int64_t)a.count);
  TinyWindow win;
  win.ids(A, a.list, idx, end, 0);
  win.ranges(A, a.f, 0);
  while (idx < end) {
    TinyGroup<StructSR> g = tiny_group<StructSR>(A, B, a.list, idx, end, a.f, win);
    if (g.rows == 0) {  // more than 32 entries of A for at most 32 products
      RowAhead<StructSR> x;
      x.all(A, B, a.list, idx, end);
      auto put = [&](int col, NoVal, int p) {
        if (HS_G(a.A.dbg, p < 32, 34, p)) scol[w][p] = col;
      };
      const int nprod = x.r >= 0 ? warp_products_of<StructSR>(A, B, x, put) : 0;
      __syncwarp();
      g.rows = 1;
      const int from = win.slide(1);
      win.ids(A, a.list, idx + 1, end, from);
      win.ranges(A, a.f, from);
      g.nprod = min(nprod, 32);
      g.r = lane == 0 ? x.r : -1;
      g.mask = lane == 0 && g.nprod ? 0xffffffffu >> (32 - g.nprod) : 0u;
      g.row = 0;
      g.col = lane < g.nprod ? scol[w][lane] : 0;
      if (lane == 0 && nprod > 32) atomicExch(a.err, 2);
      __syncwarp();
    }
    const bool have = lane < g.nprod;
    // a lane without a product matches nobody's (row, column)
    const unsigned long long key = have ? ((unsigned long long)(unsigned)g.row << 32) | (unsigned)g.col
                                        : ~0ull - (unsigned)lane;
    const unsigned grp = __match_any_sync(FULL, key);
    const unsigned lead = __ballot_sync(FULL, have && lane == __ffs(grp) - 1);
    if (lane < g.rows && g.r >= 0) put_count(a, out_row(a.A, g.r), __popc(lead & g.mask));
    idx += g.rows;
  }
}

// --------------------------------------------------------------- warp
// one warp per row, a private table of 2f slots (at most SLOTS): rows of at
// most 512 products (1024 slots) and, in their own launch, of 513..1024
// products (2048 slots).  BITS: B's columns fit the table's room as a bitmap
// (32 columns a slot), which replaces the hash set: one atomic a product
// instead of hash, probe and compare-and-swap.  Without one, rows of at most
// 64 products sort their columns, two a lane, and count the changes: 21
// stages without a branch, against probes that the lanes of a warp, and
// repeated columns among them, wait for one another in.
constexpr int WARP_WPB = 8;
constexpr int F_SYM_SORT = 64;
template <int SLOTS, bool BITS>
__global__ void __launch_bounds__(WARP_WPB * 32, 4) k_sym_warp(SymArgs a) {
  extern __shared__ __align__(16) int tables[];
  const int w = threadIdx.x >> 5, lane = lane_id();
  int *keys = tables + w * SLOTS;
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int n = (int)a.B.n;
  const int step = gridDim.x * WARP_WPB;
  int idx = blockIdx.x * WARP_WPB + w;
  RowAhead<StructSR> x, nx;
  x.all(A, B, a.list, idx, a.count);
  int fr = !BITS && x.r >= 0 ? (int)a.f[x.r] : 0;
  for (; idx < a.count; idx += step) {
    nx.row(A, a.list, idx + step, a.count);
    const int slots = max(64, min(SLOTS, next_pow2(2 * fr)));
    const bool sorts = !BITS && SLOTS <= 2 * F_WARP && fr <= F_SYM_SORT;
    if constexpr (BITS) bitmap_clear<WarpGroup>(keys, n);
    else if (!sorts)
      for (int s = lane; s < slots; s += 32) keys[s] = EMPTY;
    __syncwarp();
    int cnt = 0;
    const unsigned mask = slots - 1;
    nx.range(A);
    if constexpr (!BITS) fr = nx.r >= 0 ? (int)__ldg(a.f + nx.r) : 0;
    auto put = [&](int col, NoVal, int p) {
      if constexpr (BITS) {
        if (HS_G(a.A.dbg, col >= 0 && col < n, 33, col)) cnt += bitmap_insert(keys, col);
      } else if (sorts) {
        if (HS_G(a.A.dbg, p < F_SYM_SORT, 34, p)) keys[p] = col;
      } else {
        cnt += hash_insert_key(keys, mask, col);
      }
    };
    const int got = x.r >= 0 ? warp_products_of<StructSR>(A, B, x, put) : 0;
    nx.entries(A);
    if (sorts) {
      __syncwarp();
      uint32_t k[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) k[i] = 2 * lane + i < got ? (uint32_t)keys[(2 * lane + i) & (F_SYM_SORT - 1)] : 0xffffffffu;
      warp_bitonic_flat<2>(k);
      const uint32_t before = __shfl_up_sync(FULL, k[1], 1);
      cnt = (k[0] != 0xffffffffu && (lane == 0 || k[0] != before)) + (k[1] != 0xffffffffu && k[1] != k[0]);
    }
    cnt = warp_sum(cnt);
    nx.segments(B);
    if (lane == 0 && x.r >= 0) put_count(a, out_row(a.A, x.r), cnt);
    __syncwarp();
    x = nx;
  }
}

// ------------------------------------------------------------- dense SPA
// Products whose B has at most SPA_COLS_4 columns: one warp per row sets an
// occupancy flag per product (a byte per column of all n columns, plain
// stores: lanes that hit one column do not queue on an atomic) and counts
// the flags (the occupancy half of Figure 1's sparse accumulator).
constexpr int SPA_WPB = 8;
__global__ void __launch_bounds__(SPA_WPB * 32) k_sym_spa(SymArgs a) {
  __shared__ unsigned flags_all[SPA_WPB][SPA_COLS_4 / 4];
  const int w = threadIdx.x >> 5, lane = lane_id();
  unsigned *flag4 = flags_all[w];
  unsigned char *flag = reinterpret_cast<unsigned char *>(flag4);
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int n = (int)a.B.n;
  const int fwords = (n + 3) >> 2;
  for (int i = lane; i < fwords; i += 32) flag4[i] = 0u;
  __syncwarp();
  for (int idx = blockIdx.x * SPA_WPB + w; idx < a.count; idx += gridDim.x * SPA_WPB) {
    const int r = a.list[idx];
    if (!HS_G(a.A.dbg, r >= 0 && r < a.A.nslots, 35, r)) continue;
    warp_products<StructSR>(A, B, A.p[r], A.p[r + 1], [&](int col, NoVal, int) {
      if (HS_G(a.A.dbg, col >= 0 && col < n, 84, col)) flag[col] = 1;
    });
    __syncwarp();
    int cnt = 0;
    for (int i = lane; i < fwords; i += 32) {
      cnt += __popc(flag4[i] & 0x01010101u);
      flag4[i] = 0u;
    }
    cnt = warp_sum(cnt);
    if (lane == 0) put_count(a, out_row(a.A, r), cnt);
    __syncwarp();
  }
}

// ----------------------------------------------------------- mid / large
constexpr int CH = 1024;   // A entries per expansion round (heavy)
constexpr int CHM = 256;   // the same for the hash kernels: smaller staging, more CTAs per SM

template <int SLOTS> struct SymCtaSmem {
  alignas(16) int keys[SLOTS];
  CtaExpandSmem<NoVal, CHM> ex;
  int wtmp[33];
  int total;
};

template <int SLOTS, int NT, bool BITS>  // BITS: as for k_sym_warp; 1536 threads an SM, as its shared memory allows
__global__ void __launch_bounds__(NT, 1536 / NT) k_sym_cta(SymArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto &sm = *reinterpret_cast<SymCtaSmem<SLOTS> *>(smem_raw);
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int n = (int)a.B.n;
  for (int idx = blockIdx.x; idx < a.count; idx += gridDim.x) {
    const int r = a.list[idx];
    if (!HS_G(a.A.dbg, r >= 0 && r < a.A.nslots, 35, r)) continue;
    const int slots = max(64, min(SLOTS, next_pow2(2 * (int)a.f[r])));
    const unsigned mask = slots - 1;
    if constexpr (BITS) bitmap_clear<CtaGroup>(sm.keys, n);
    else
      for (int s = threadIdx.x; s < slots; s += blockDim.x) sm.keys[s] = EMPTY;
    if (threadIdx.x == 0) sm.total = 0;
    __syncthreads();
    int cnt = 0;
    cta_products<StructSR, CHM>(A, B, A.p[r], A.p[r + 1], false, 0, 0, sm.ex, sm.wtmp,
                                [&](int col, NoVal, int) {
                                  if constexpr (BITS) {
                                    if (HS_G(a.A.dbg, col >= 0 && col < n, 33, col)) cnt += bitmap_insert(sm.keys, col);
                                  } else {
                                    cnt += hash_insert_key(sm.keys, mask, col);
                                  }
                                });
    cnt = warp_sum(cnt);
    if (lane_id() == 0 && cnt) atomicAdd(&sm.total, cnt);
    __syncthreads();
    if (threadIdx.x == 0) put_count(a, out_row(a.A, r), sm.total);
    __syncthreads();
  }
}

// --------------------------------------------------------------- heavy
// Per row and per chunk of 2^20 columns: the products set their bits (an OR
// whose old value nobody waits for), then each 4096-column segment's bits are
// counted by popcount.  The segment counts give the chunk's histogram and,
// scanned, each segment's place in the row's sorted column list.  Each warp then walks pairs of
// segments, every lane eight consecutive words: the lanes' bit counts are
// scanned across the warp, the columns go to a per-warp staging buffer in
// ascending order and leave it in coalesced stores.  A pair with more columns
// than the buffer holds is read again as eight steps of 1024 columns, lane l
// on the step's word l, so each step's columns also run in lane order and
// gather in the buffer (per-lane stores of the long runs measured 2.3 ms
// slower on R-MAT scale 20).
constexpr int SH_COLS = BITMAP_COLS;          // columns per chunk (one bitmap)
constexpr int SH_SEGS = SH_COLS / SEG_W;      // segments per chunk (256)
// Threads of the CTA: 1024, one CTA an SM, for a full bitmap; 512, two CTAs an
// SM, where B's columns need at most half of it and there are SH_ROWS_HALF rows
// an SM, so that one row's barriers and claims are filled by the other's
// products (200,003 columns: the pass 2.37 -> 1.83 ms; with few rows the
// longest one decides, and 512 threads made a product of 256 columns 27 us
// slower).
constexpr int SH_NT = 1024, SH_NT_HALF = 512, SH_COLS_HALF = SH_COLS / 2, SH_ROWS_HALF = 4;
constexpr int SH_BUF = 384;                   // per-warp list staging entries
static_assert(SEG_W == 4096, "two segments are 256 words: eight per lane");

// Product visitor: sets the column's bit; the old word is not needed (the
// segment counts come from the finished bitmap), so no lane waits for it.
// (Reading the word first and skipping the atomic when the bit is already set
// measured slower on R-MAT scale 20: 27.7 against 24.3 ms.)
struct SymHeavyBit {
  unsigned *bitmap;
  int lo;
  unsigned span;
  long long *dbg;
  __device__ __forceinline__ void operator()(int col, NoVal, int) const {
    const unsigned x = (unsigned)(col - lo);
    if (HS_G(dbg, x < span, 33, col)) atomicOr(bitmap + (x >> 5), 1u << (x & 31));
  }
};

template <int NT> struct SymHeavySmem {
  static constexpr int WARPS = NT / 32;
  static constexpr int PPW = SH_SEGS / 2 / WARPS;  // segment pairs per warp
  static_assert(PPW * WARPS * 2 == SH_SEGS, "the warps' pairs cover a chunk's segments");
  CtaExpandSmem<NoVal, CH> ex;
  int wtmp[33];
  int row;
  long long loff;        // the row's list in the pool, or -1
  int scnt[SH_SEGS + 1];  // new columns per segment of the chunk, then their exclusive scan and total
  int wbuf[WARPS][SH_BUF];
  alignas(16) unsigned bitmap[SH_COLS / 32];
};


// The eight bitmap words of a lane in a segment pair (words w0 .. w0 + 7),
// zero past the chunk's last word.
__device__ __forceinline__ void sh_load8(const unsigned *bitmap, int w0, int words, unsigned long long (&b)[4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int w = w0 + 4 * h;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (w + 3 < words) v = *reinterpret_cast<const uint4 *>(bitmap + w);
    else if (w < words) {
      v.x = bitmap[w];
      if (w + 1 < words) v.y = bitmap[w + 1];
      if (w + 2 < words) v.z = bitmap[w + 2];
    }
    b[2 * h] = ((unsigned long long)v.y << 32) | v.x;
    b[2 * h + 1] = ((unsigned long long)v.w << 32) | v.z;
  }
}
// Clears the same eight words (the bitmap is left empty for the next row).
__device__ __forceinline__ void sh_clear8(unsigned *bitmap, int w0, int words) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int w = w0 + 4 * h;
    if (w + 3 < words) *reinterpret_cast<uint4 *>(bitmap + w) = make_uint4(0u, 0u, 0u, 0u);
    else
      for (int k = w; k < words && k < w + 4; ++k) bitmap[k] = 0u;
  }
}

template <int NT>
__global__ void __launch_bounds__(NT, SH_NT / NT) k_sym_heavy(SymArgs a) {
  using L = SymHeavySmem<NT>;
  constexpr int SH_PPW = L::PPW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto &sm = *reinterpret_cast<L *>(smem_raw);
  const DevCsr A = dev_a(a.A), B = dev_b(a.B);
  const int64_t n = a.B.n;
  const int nchunk = (int)((n + SH_COLS - 1) / SH_COLS);
  const int lane = lane_id(), warp = threadIdx.x >> 5, nw = L::WARPS;
  int *buf = sm.wbuf[warp];
  // the first chunk is the widest: clearing its words once leaves the whole
  // bitmap empty, and every chunk clears the words it read afterwards
  {
    const int words0 = (int)((min(n, (int64_t)SH_COLS) + 31) >> 5);
    for (int wd = threadIdx.x; wd < words0; wd += NT) sm.bitmap[wd] = 0u;
  }
  while (true) {
    if (threadIdx.x == 0) sm.row = atomicAdd(a.dyn, 1);
    __syncthreads();
    const int idx = sm.row;
    if (idx >= a.count) break;
    const int r0 = a.list[idx];
    // a bad row id (guarded builds) runs no chunk, so the loop still reaches its closing barriers
    const bool r_ok = HS_G(a.A.dbg, r0 >= 0 && r0 < a.A.nslots, 35, r0);
    const int r = r_ok ? r0 : 0;
    const int h = r_ok ? a.hslot[r] : -1;
    uint32_t *hist = h >= 0 ? a.hist + (int64_t)h * a.nseg : nullptr;
    int32_t *lst = nullptr;  // the row's list, once its room is taken (first chunk)
    const int64_t lmax = r_ok ? min(a.f[r], n) : 0;  // the list's room: min(f, n) entries bound its output
    int64_t written = 0;  // columns of the earlier chunks
    bool as_bits = false;
    for (int ch = 0; ch < (r_ok ? nchunk : 0); ++ch) {
      const int lo = ch * SH_COLS;
      const int hi = (int)min((int64_t)lo + SH_COLS, n);
      const int words = (hi - lo + 31) >> 5;
      const int nsc = (hi - lo + SEG_W - 1) / SEG_W;
      cta_products<StructSR, CH, 4>(A, B, A.p[r], A.p[r + 1], nchunk > 1, lo, hi, sm.ex, sm.wtmp,
                                    SymHeavyBit{sm.bitmap, lo, (unsigned)(hi - lo), a.A.dbg});
      // columns per segment, by pairs of segments (8192 columns, eight words
      // per lane; warp w takes pairs w, w + 32, ...): each lane's count and
      // its inclusive scan over the warp are kept for the list pass.  The
      // row's list room is taken from the pool meanwhile (thread 0 issues the
      // atomic first and reads its answer after its counts)
      unsigned long long at_l = 0ull;
      const bool take = threadIdx.x == 0 && ch == 0 && a.glist;
      if (take) at_l = atomicAdd(a.lpool, (unsigned long long)lmax);
      int keep[SH_PPW];  // (inclusive scan << 16) | lane count
#pragma unroll
      for (int i = 0; i < SH_PPW; ++i) {
        const int g = 2 * (warp + nw * i);
        keep[i] = 0;
        if (g < nsc) {  // warp-uniform
          const int wb = g * (SEG_W / 32) + 8 * lane;
          unsigned long long b[4];
          sh_load8(sm.bitmap, wb, words, b);
          const int pcl = __popcll(b[0]) + __popcll(b[1]) + __popcll(b[2]) + __popcll(b[3]);
          const int incl = warp_incl_scan(pcl);
          const int first = __shfl_sync(FULL, incl, 15);  // lanes 0..15 hold segment g
          const int tot = __shfl_sync(FULL, incl, 31);
          if (lane == 0) {
            sm.scnt[g] = first;
            if (g + 1 < nsc) sm.scnt[g + 1] = tot - first;
          }
          keep[i] = (incl << 16) | pcl;
          if (!a.glist) sh_clear8(sm.bitmap, wb, words);  // no list pass reads them again
        }
      }
      if (threadIdx.x == 0 && ch == 0) sm.loff = (take && (long long)at_l + lmax <= a.lcap) ? (long long)at_l : -1;
      __syncthreads();
      if (ch == 0 && sm.loff >= 0) lst = a.glist + sm.loff;
      // one warp: the counts out to the segment histogram, then their
      // exclusive scan (at most eight per lane), the chunk's total in the last slot
      if (warp == 0) {
        const int per = (nsc + 31) / 32;
        const int gb = min(nsc, lane * per), ge = min(nsc, gb + per);
        int cs = 0;
        for (int g = gb; g < ge; ++g) {
          const int c = sm.scnt[g];
          cs += c;
          if (hist && HS_G(a.A.dbg, lo / SEG_W + g < a.nseg, 32, g)) hist[lo / SEG_W + g] = (uint32_t)c;
        }
        const int ci = warp_incl_scan(cs);
        int run = ci - cs;
        for (int g = gb; g < ge; ++g) {
          const int c = sm.scnt[g];
          sm.scnt[g] = run;
          run += c;
        }
        if (lane == 31) sm.scnt[SH_SEGS] = ci;
      }
      __syncthreads();
      const int ctotal = sm.scnt[SH_SEGS];
      // a row that is dense enough leaves its bitmap as it is, if its room in the pool holds it
      as_bits = lst && nchunk == 1 && ctotal >= a.bits_min && lmax >= words;
      if (as_bits) {
        for (int w0 = threadIdx.x; w0 < words; w0 += 4 * NT) {
          unsigned x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = w0 + u * NT < words ? sm.bitmap[w0 + u * NT] : 0u;
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (w0 + u * NT < words) {
              __stcs(lst + w0 + u * NT, (int32_t)x[u]);
              sm.bitmap[w0 + u * NT] = 0u;
            }
        }
      }
      // list: the same pairs, read again (a row that found no room in the
      // pool only clears them)
      if (!lst && a.glist) {
#pragma unroll
        for (int i = 0; i < SH_PPW; ++i) {
          const int g = 2 * (warp + nw * i);
          if (g < nsc) sh_clear8(sm.bitmap, g * (SEG_W / 32) + 8 * lane, words);
        }
      }
      if (lst && !as_bits) {
#pragma unroll
        for (int i = 0; i < SH_PPW; ++i) {
          const int g = 2 * (warp + nw * i);
          if (g >= nsc) break;  // warp-uniform
          const int wb = g * (SEG_W / 32) + 8 * lane;
          unsigned long long b[4];
          sh_load8(sm.bitmap, wb, words, b);
          const int pcl = keep[i] & 0xffff, incl = keep[i] >> 16;
          const int tot = __shfl_sync(FULL, incl, 31);
          // the pair's columns start where segment g's do (g + 1 follows it)
          const int64_t at0 = written + sm.scnt[g];
          const int cbase = lo + (wb << 5);
          if (!HS_G(a.A.dbg, at0 + tot <= lmax, 34, at0 + tot)) {
            // nothing is written; the words are still cleared below
          } else if (tot <= SH_BUF) {
            // the lane's columns one per iteration over all eight words (the
            // warp runs as many iterations as its fullest lane has columns);
            // the next non-empty word is read again when the current one is spent
            unsigned m = 0u;  // the lane's non-empty words
#pragma unroll
            for (int q = 0; q < 4; ++q)
              m |= ((unsigned)((unsigned)b[q] != 0u) << (2 * q)) | ((unsigned)((unsigned)(b[q] >> 32) != 0u) << (2 * q + 1));
            int p = incl - pcl;
            unsigned cur = 0u;
            int cw = 0;
            for (int k = 0; k < pcl; ++k) {
              if (cur == 0u) {
                const int j = __ffs(m) - 1;
                m &= m - 1;
                cur = sm.bitmap[wb + j];
                cw = cbase + 32 * j;
              }
              buf[p++] = cw + __ffs(cur) - 1;
              cur &= cur - 1;
            }
            __syncwarp();
            for (int i2 = lane; i2 < tot; i2 += 32) __stcs(lst + at0 + i2, buf[i2]);  // evict-first: B stays in L2
          } else {
            // dense pair: re-read as eight steps of 1024 columns, lane l on the
            // step's word l, so a step's columns run in lane order; the steps
            // gather in the staging buffer and leave it in coalesced stores
            const int gw = g * (SEG_W / 32);
            int fill = 0;       // staged entries
            int64_t at = at0;   // list position of buf[0]
            for (int s2 = 0; s2 < 8; ++s2) {
              const int wd = gw + 32 * s2 + lane;
              unsigned bb = wd < words ? sm.bitmap[wd] : 0u;
              const int pc = __popc(bb);
              const int inc = warp_incl_scan(pc);
              const int st = __shfl_sync(FULL, inc, 31);
              if (fill + st > SH_BUF) {  // warp-uniform
                __syncwarp();
                for (int i2 = lane; i2 < fill; i2 += 32) __stcs(lst + at + i2, buf[i2]);
                __syncwarp();
                at += fill;
                fill = 0;
              }
              const int c0 = lo + (wd << 5);
              if (st <= SH_BUF) {
                int p = fill + inc - pc;
                while (bb) {
                  buf[p++] = c0 + __ffs(bb) - 1;
                  bb &= bb - 1;
                }
                fill += st;
              } else {  // more than SH_BUF columns in 1024: each lane's few go straight out
                int64_t q = at + inc - pc;
                while (bb) {
                  __stcs(lst + q++, c0 + __ffs(bb) - 1);
                  bb &= bb - 1;
                }
                at += st;
              }
            }
            __syncwarp();
            for (int i2 = lane; i2 < fill; i2 += 32) __stcs(lst + at + i2, buf[i2]);
          }
          __syncwarp();  // every lane's reads of the pair's words (and of buf) are done
          sh_clear8(sm.bitmap, wb, words);
        }
      }
      written += ctotal;
      __syncthreads();
    }
    if (threadIdx.x == 0 && r_ok) {
      put_count(a, out_row(a.A, r), written);
      if (a.loff) a.loff[r] = lst ? sm.loff | (as_bits ? LIST_BITS : 0) : -1;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------- launchers
static int grid_cap(int items, int per_block, int per_sm) {
  int g = (items + per_block - 1) / per_block;
  int cap = sm_count() * per_sm;
  return g < cap ? (g < 1 ? 1 : g) : cap;
}

void launch_sym_tiny(const SymArgs &a, cudaStream_t st) {
  if (a.count <= 0) return;
  auto k = a.tiny_group ? k_sym_tiny_group : k_sym_tiny;
  const int fit = fit_per_sm(k, TINY_WPB * 32, 0);
  count_launch();
  k<<<grid_cap(a.count, TINY_WPB, fit), TINY_WPB * 32, 0, st>>>(a);
}
// A table of `slots` words holds a bitmap of all of B's columns up to 32 a
// slot; on both sides of the line the kernel needs the same shared memory, so
// the line lies where the room ends.
static bool fits_bitmap(const SymArgs &a, int64_t slots) { return a.B.n <= 32 * slots; }
template <int SLOTS, bool BITS> static void launch_sym_warp_as(const SymArgs &a, cudaStream_t st) {
  const size_t bytes = sizeof(int) * WARP_WPB * SLOTS;
  auto k = k_sym_warp<SLOTS, BITS>;
  const int fit = fit_per_sm(k, WARP_WPB * 32, bytes);
  count_launch();
  k<<<grid_cap(a.count, WARP_WPB, fit), WARP_WPB * 32, bytes, st>>>(a);
}
template <int SLOTS> static void launch_sym_warp_slots(const SymArgs &a, cudaStream_t st) {
  if (a.count <= 0) return;
  if (fits_bitmap(a, SLOTS)) launch_sym_warp_as<SLOTS, true>(a, st);
  else launch_sym_warp_as<SLOTS, false>(a, st);
}
// (up to 2^16 columns the short rows take the larger table for its bitmap)
void launch_sym_warp(const SymArgs &a, cudaStream_t st) {
  if (!fits_bitmap(a, 2 * F_WARP) && fits_bitmap(a, 2 * F_MID_S)) launch_sym_warp_slots<2 * F_MID_S>(a, st);
  else launch_sym_warp_slots<2 * F_WARP>(a, st);
}
void launch_sym_spa(const SymArgs &a, cudaStream_t st) {
  if (a.count <= 0) return;
  count_launch();
  k_sym_spa<<<grid_cap(a.count, SPA_WPB, fit_per_sm(k_sym_spa, SPA_WPB * 32, 0)), SPA_WPB * 32, 0, st>>>(a);
}

template <int SLOTS, int NT, bool BITS> static void launch_sym_cta_as(const SymArgs &a, cudaStream_t st) {
  const size_t bytes = sizeof(SymCtaSmem<SLOTS>);
  auto k = k_sym_cta<SLOTS, NT, BITS>;
  const int fit = fit_per_sm(k, NT, bytes);
  count_launch();
  k<<<grid_cap(a.count, 1, fit), NT, bytes, st>>>(a);
}
template <int SLOTS, int NT> static void launch_sym_cta(const SymArgs &a, cudaStream_t st) {
  if (a.count <= 0) return;
  if (fits_bitmap(a, SLOTS)) launch_sym_cta_as<SLOTS, NT, true>(a, st);
  else launch_sym_cta_as<SLOTS, NT, false>(a, st);
}
// table capacity 2f: mid rows have f <= 4096, large rows f <= min(16384, cap_large) = 8192 at most
void launch_sym_mid_s(const SymArgs &a, cudaStream_t st) { launch_sym_warp_slots<2 * F_MID_S>(a, st); }
void launch_sym_mid(const SymArgs &a, cudaStream_t st) { launch_sym_cta<2 * F_MID, 256>(a, st); }
void launch_sym_large(const SymArgs &a, cudaStream_t st) { launch_sym_cta<16384, 512>(a, st); }

template <int NT> static void launch_sym_heavy_as(const SymArgs &a, cudaStream_t st) {
  const size_t bytes = offsetof(SymHeavySmem<NT>, bitmap) + sizeof(unsigned) * (size_t)sym_bitmap_words(a.B.n);
  const int fit = fit_per_sm(k_sym_heavy<NT>, NT, bytes);
  count_launch();
  k_sym_heavy<NT><<<grid_cap(a.count, 1, fit), NT, bytes, st>>>(a);
}
void launch_sym_heavy(const SymArgs &a, cudaStream_t st) {
  if (a.count <= 0) return;
  if (a.B.n <= SH_COLS_HALF && a.count >= SH_ROWS_HALF * sm_count()) launch_sym_heavy_as<SH_NT_HALF>(a, st);
  else launch_sym_heavy_as<SH_NT>(a, st);
}

}  // namespace hs
