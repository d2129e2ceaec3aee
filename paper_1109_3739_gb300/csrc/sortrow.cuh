// sortrow.cuh -- one row of C by one warp, by sorting its products.
//
// Rows whose products seldom share a column (output count close to the
// product count, as in products of random sparse matrices) gain little from
// a hash table: every product still claims a slot, and the table must be
// sorted afterwards.  Here the warp lays the row's products (column, value)
// out in shared memory in product order, sorts packed keys
// (column - kmin) << PB | product index in registers with Batcher's bitonic
// network (32*K keys, K per lane), and folds runs of equal columns in the
// sorted order: Algorithm 1's row-wise accumulation
// done as expand, sort, compress.  The row leaves in ascending column order,
// its values summed (or minimised, or-ed) with the semiring's add.  A row
// whose column span does not fit the packed key sorts 64-bit keys
// column << 32 | product index instead (WIDE; the host keeps rows of more
// than 256 products out of the sort tiers when the matrix is that wide, so
// the larger tiers need not hold 64-bit keys in registers).
#pragma once
#include "common.cuh"

namespace hs {

// padded shared-memory index: one spare word per 32, so that a lane reading
// its K consecutive elements and 32 lanes reading consecutive elements both
// hit 32 distinct banks
__device__ __forceinline__ int sr_pad(int e) { return e + (e >> 5); }
__host__ __device__ constexpr int sr_pad_len(int n) { return n + (n >> 5); }

template <int N> struct ILog2 {
  static constexpr int v = 1 + ILog2<N / 2>::v;
};
template <> struct ILog2<1> {
  static constexpr int v = 0;
};

// the semiring's identity, or nothing for structure-only products
template <class SR> __device__ __forceinline__ typename SR::val_t sr_identity() {
  if constexpr (SR::has_val) return SR::identity();
  else return typename SR::val_t{};
}

template <typename T> __device__ __forceinline__ T shfl_up_val(T x, int d) { return __shfl_up_sync(FULL, x, d); }
template <typename T> __device__ __forceinline__ T shfl_down_val(T x, int d) { return __shfl_down_sync(FULL, x, d); }
template <> __device__ __forceinline__ NoVal shfl_down_val<NoVal>(NoVal x, int) { return x; }

// compare-exchange: a takes the smaller key, b the larger
template <typename KT> __device__ __forceinline__ void ce_up(KT &a, KT &b) {
  const KT lo = a < b ? a : b, hi = a < b ? b : a;
  a = lo;
  b = hi;
}

// bitonic stages of sizes 2 .. K/2 inside each lane (directions fixed by i)
template <int K, typename KT> __device__ __forceinline__ void bitonic_in_lane(KT (&key)[K]) {
#pragma unroll
  for (int size = 2; size < K; size <<= 1)
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
      for (int i = 0; i < K; ++i)
        if ((i & stride) == 0) {
          if ((i & size) == 0) ce_up(key[i], key[i | stride]);
          else ce_up(key[i | stride], key[i]);
        }
}

// the in-lane strides K/2 .. 1 of an ascending bitonic merge
template <int K, typename KT> __device__ __forceinline__ void merge_in_lane(KT (&key)[K]) {
#pragma unroll
  for (int stride = K >> 1; stride > 0; stride >>= 1)
#pragma unroll
    for (int i = 0; i < K; ++i)
      if ((i & stride) == 0) ce_up(key[i], key[i | stride]);
}

// Ascending bitonic sort of the warp's 32*K keys, element e = lane*K + i held
// in key[i] of lane `lane` (blocked layout).  Merges of blocks of K or more
// elements run as a loop over the block size: a block that the network
// sorts descending holds its keys complemented for that merge, so every
// comparator takes the smaller key to the lower element; comparator pairs
// closer than K elements sit in one lane's registers, the others are one
// shuffle apart.  The loop keeps the code small (a fully unrolled network of
// 1024 keys would not fit the instruction cache).
template <int K, typename KT> __device__ __forceinline__ void warp_bitonic(KT (&key)[K]) {
  constexpr int N = 32 * K;
  const int lane = lane_id();
  bitonic_in_lane<K>(key);
#pragma unroll 1
  for (int size = K; size <= N; size <<= 1) {
    const KT flip = ((lane * K) & size) ? ~KT(0) : KT(0);
#pragma unroll
    for (int i = 0; i < K; ++i) key[i] ^= flip;
#pragma unroll 1
    for (int stride = size >> 1; stride >= K; stride >>= 1) {
      const int lm = stride / K;
      const bool lower = (lane & lm) == 0;
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const KT o = __shfl_xor_sync(FULL, key[i], lm);
        const KT x = key[i];
        key[i] = (lower == (o < x)) ? o : x;
      }
    }
    merge_in_lane<K>(key);
#pragma unroll
    for (int i = 0; i < K; ++i) key[i] ^= flip;
  }
}

// The same network for few keys a lane, fully unrolled (no loop, and a
// descending block compares the other way round instead of holding its keys
// complemented): K = 2 is 21 stages in some 170 instructions.
template <int K, typename KT> __device__ __forceinline__ void warp_bitonic_flat(KT (&key)[K]) {
  constexpr int N = 32 * K;
  const int lane = lane_id();
  bitonic_in_lane<K>(key);
#pragma unroll
  for (int size = K; size <= N; size <<= 1) {
    const bool desc = ((lane * K) & size) != 0;
#pragma unroll
    for (int stride = size >> 1; stride >= K; stride >>= 1) {
      const bool small = ((lane & (stride / K)) == 0) != desc;
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const KT o = __shfl_xor_sync(FULL, key[i], stride / K);
        key[i] = small ? min(key[i], o) : max(key[i], o);
      }
    }
#pragma unroll
    for (int stride = K >> 1; stride > 0; stride >>= 1)
#pragma unroll
      for (int i = 0; i < K; ++i)
        if ((i & stride) == 0) {
          const KT lo = min(key[i], key[i | stride]), hi = max(key[i], key[i | stride]);
          key[i] = desc ? hi : lo;
          key[i | stride] = desc ? lo : hi;
        }
  }
}

// The products of the row held by x by one warp, in product order, to
// shared memory (columns at s_col[sr_pad(p)], values at s_val[p], at most
// nmax of them); returns their number (warp-uniform) and the least and
// greatest column in *kmn, *kmx.  Shared by every register width, so a kernel
// that sorts rows of several widths holds one copy of the expansion.
template <class SR>
__device__ __forceinline__ int sort_expand(const DevCsr &A, const DevCsr &B, const RowAhead<SR> &x, int nmax,
                                           int *s_col, typename SR::val_t *s_val, int *kmn_out, int *kmx_out) {
  using T = typename SR::val_t;
  int kmn = 0x7fffffff, kmx = -1;
  auto put = [&](int col, T v, int p) {
    if (HS_G(A.dbg, p >= 0 && p < nmax, 90, p)) {
      s_col[sr_pad(p)] = col;
      if constexpr (SR::has_val) s_val[p] = v;
    }
    kmn = min(kmn, col);
    kmx = max(kmx, col);
  };
  const int got = warp_products_of<SR>(A, B, x, put);
  __syncwarp();
  *kmn_out = warp_min(kmn);
  *kmx_out = warp_max(kmx);
  return got;
}

// The runs of more than four equal columns among a row's F sorted keys (column
// - kmn) << pb | product index: a segmented scan of each round of 32 in which
// one begins (a bit of long_in) or goes on, written from the run's last
// element at its rank (lane i of `before`: columns before round i).
template <class SR>
__device__ __forceinline__ void sum_long_runs(int F, int pb, int c, int kmn, unsigned long_in, int before,
                                           const int *s_col, const typename SR::val_t *s_val, int32_t *out_j,
                                           typename SR::val_t *out_v, long long *dbg) {
  using T = typename SR::val_t;
  const int lane = lane_id();
  const unsigned le = 0xffffffffu >> (31 - lane), at = (1u << pb) - 1u;
  auto key_at = [&](int e) { return e < F ? (uint32_t)s_col[sr_pad(e)] : 0xffffffffu; };  // (no element's column)
  bool open = false;  // a long run reaches into the round
  T carry = SR::identity();
  for (int i = 0; i * 32 < F; ++i) {
    if (!open && !((long_in >> i) & 1u)) continue;
    const int e = i * 32 + lane;
    const uint32_t kk = key_at(e);
    const bool valid = e < F;
    const bool head = valid && (e == 0 || (key_at(e - 1) >> pb) != (kk >> pb));
    const bool tail = valid && (key_at(e + 1) >> pb) != (kk >> pb);
    const unsigned hm = __ballot_sync(FULL, head);
    const unsigned lm = __ballot_sync(FULL, head && (key_at(e + 4) >> pb) == (kk >> pb));
    T x = valid ? s_val[kk & at] : SR::identity();
    bool fl = head;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const T y = shfl_up_val<T>(x, d);
      const bool g = __shfl_up_sync(FULL, (int)fl, d) != 0;
      if (lane >= d) {
        if (!fl) x = SR::add(y, x);
        fl = fl || g;
      }
    }
    if (!fl && valid) x = SR::add(carry, x);  // continues the run that came in
    carry = shfl_val<T>(x, 31);
    const unsigned upto = hm & le;
    const bool in_long = upto ? (lm >> (31 - __clz(upto))) & 1u : open;
    const int pos = __shfl_sync(FULL, before, i) + __popc(upto) - 1;
    if (in_long && tail && HS_G(dbg, pos >= 0 && pos < c, 91, pos)) {
      __stcs(out_j + pos, (int)(kk >> pb) + kmn);
      __stcs(out_v + pos, x);
    }
    open = __shfl_sync(FULL, (int)(in_long && !tail), 31) != 0;
  }
}

// out of line, for the persistent kernel, which holds sort_finish for four K:
// with 4-byte values a copy for each cost it 1.3 %, with 8-byte values the call
// 2.8 % (64 products: 5.75 against 5.62 ms; 5.60 without either)
template <class SR>
__device__ __noinline__ void sum_long_runs_call(int F, int pb, int c, int kmn, unsigned long_in, int before,
                                                const int *s_col, const typename SR::val_t *s_val, int32_t *out_j,
                                                typename SR::val_t *out_v, long long *dbg) {
  sum_long_runs<SR>(F, pb, c, kmn, long_in, before, s_col, s_val, out_j, out_v, dbg);
}

// Sort and fold a row whose F products (F <= 32*K) sort_expand laid out,
// writing its c outputs at out_j / out_v.  An output count other than c
// sets *err (the structure disagrees with the symbolic pass).  OUT_OF_LINE:
// long runs by a call.
template <class SR, int K, bool WIDE, bool OUT_OF_LINE = false>
__device__ __forceinline__ void sort_finish(int F, int c, int kmn, int kmx, int *s_col,
                                            const typename SR::val_t *s_val, int32_t *out_j,
                                            typename SR::val_t *out_v, int *err, long long *dbg) {
  using T = typename SR::val_t;
  constexpr int N = 32 * K;
  constexpr int PB = ILog2<N>::v;
  const int lane = lane_id();
  if (F <= 0) return;
  const unsigned span = (unsigned)kmx - (unsigned)kmn;
  if (span < (1u << (32 - PB)) - 1u) {
    // 2. packed keys, sorted
    uint32_t key[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int e = lane * K + i;
      key[i] = e < F ? (((uint32_t)(s_col[sr_pad(e)] - kmn)) << PB) | (uint32_t)e : 0xffffffffu;
    }
    if constexpr (K <= 4) warp_bitonic_flat<K>(key);
    else warp_bitonic<K>(key);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < K; ++i) s_col[sr_pad(lane * K + i)] = (int)key[i];
    __syncwarp();
    // 3. runs of equal columns, 32 elements a round (lane l takes element
    // 32*i + l), at the run's rank among the row's columns.  Most runs are one
    // or a few elements long: their head adds them up.  Runs of more than four
    // are left to a segmented scan of the rounds that they touch.
    // (A head that walked any run kept the warp waiting for the longest one,
    // and the sum's error grew with the run's length: half of a row's 256 /
    // 512 / 1024 products on one column took 246 / 468 / 1039 us a numeric
    // pass, 201 / 370 / 788 now; a scan of every round takes five shuffle-and-add
    // steps of two words each whatever the runs: 146 / 255 / 512 us without
    // repeats, 116 / 200 / 403 this way.)
    const unsigned le = 0xffffffffu >> (31 - lane);  // lanes <= this one
    auto key_at = [&](int e) { return e < F ? (uint32_t)s_col[sr_pad(e)] : 0xffffffffu; };  // (no element's column)
    int outb = 0, before = 0;  // columns so far; lane i: before round i
    unsigned long_in = 0;      // rounds in which a long run of this lane begins
    uint32_t last = 0;         // the previous round's last key
    for (int i = 0; i * 32 < F; ++i) {
      const int e = i * 32 + lane;
      const bool valid = e < F;
      const uint32_t kk = key_at(e);
      uint32_t kp = __shfl_up_sync(FULL, kk, 1);
      if (lane == 0) kp = last;
      last = __shfl_sync(FULL, kk, 31);
      const bool head = valid && (e == 0 || (kk >> PB) != (kp >> PB));
      const unsigned hm = __ballot_sync(FULL, head);
      const int pos = outb + __popc(hm & le) - 1;
      if (lane == i) before = outb;
      if (head) {
        T v{};
        bool more = false;
        if constexpr (SR::has_val) {
          v = s_val[kk & (N - 1)];
          const uint32_t k1 = key_at(e + 1);
          if ((k1 >> PB) == (kk >> PB)) {  // (nested: a loop of up to three steps took 1 % longer)
            v = SR::add(v, s_val[k1 & (N - 1)]);
            const uint32_t k2 = key_at(e + 2);
            if ((k2 >> PB) == (kk >> PB)) {
              v = SR::add(v, s_val[k2 & (N - 1)]);
              const uint32_t k3 = key_at(e + 3);
              if ((k3 >> PB) == (kk >> PB)) {
                v = SR::add(v, s_val[k3 & (N - 1)]);
                more = (key_at(e + 4) >> PB) == (kk >> PB);
              }
            }
          }
        }
        if (more) long_in |= 1u << i;
        else if (HS_G(dbg, pos >= 0 && pos < c, 91, pos)) {
          __stcs(out_j + pos, (int)(kk >> PB) + kmn);
          if constexpr (SR::has_val) __stcs(out_v + pos, v);
        }
      }
      outb += __popc(hm);
    }
    if constexpr (SR::has_val) {
      long_in = __reduce_or_sync(FULL, long_in);
      if (long_in) {
        if constexpr (OUT_OF_LINE) sum_long_runs_call<SR>(F, PB, c, kmn, long_in, before, s_col, s_val, out_j, out_v, dbg);
        else sum_long_runs<SR>(F, PB, c, kmn, long_in, before, s_col, s_val, out_j, out_v, dbg);
      }
    }
    if (outb != c && lane == 0) atomicExch(err, 13);
    return;
  }
  if constexpr (!WIDE) {
    if (lane == 0) atomicExch(err, 14);  // a span the host should have kept out of this tier
    return;
  }
  // wide rows: 64-bit keys column << 32 | product index, sorted, then folded
  // in the blocked layout (lane l holds sorted elements l*K .. l*K+K-1)
  unsigned long long key[K];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int e = lane * K + i;
    key[i] = e < F ? (((unsigned long long)(unsigned)s_col[sr_pad(e)]) << 32) | (unsigned)e : ~0ull;
  }
  warp_bitonic<K>(key);
  const unsigned long long before = __shfl_up_sync(FULL, key[K - 1], 1);  // element lane*K - 1
  int nh = 0;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const bool valid = key[i] != ~0ull;
    const unsigned long long pk = i ? key[i - 1] : before;
    nh += (valid && ((lane == 0 && i == 0) || (pk >> 32) != (key[i] >> 32))) ? 1 : 0;
  }
  const int hincl = warp_incl_scan(nh);
  const int total = __shfl_sync(FULL, hincl, 31);
  int outi = hincl - nh - 1;  // index of the run being summed
  T acc = sr_identity<SR>();
  T pre = acc;         // elements before this lane's first head (a run begun in an earlier lane)
  bool seen = false;   // a head in this lane
  int curcol = 0;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const bool valid = key[i] != ~0ull;
    if (!valid) continue;
    const unsigned long long pk = i ? key[i - 1] : before;
    const bool head = (lane == 0 && i == 0) || (pk >> 32) != (key[i] >> 32);
    T v{};
    if constexpr (SR::has_val) v = s_val[(unsigned)(key[i] & 0xffffffffull)];
    if (head) {
      if (seen && HS_G(dbg, outi >= 0 && outi < c, 92, outi)) {  // the previous run of this lane is complete
        __stcs(out_j + outi, curcol);
        if constexpr (SR::has_val) __stcs(out_v + outi, acc);
      }
      ++outi;
      seen = true;
      curcol = (int)(key[i] >> 32);
      acc = v;
    } else if (seen) {
      if constexpr (SR::has_val) acc = SR::add(acc, v);
    } else {
      if constexpr (SR::has_val) pre = SR::add(pre, v);
    }
  }
  // the lane's last run continues into the next lanes up to the first lane
  // with a head of its own
  bool open = seen;
  for (int d = 1; d < 32; ++d) {
    const T pd = shfl_down_val<T>(pre, d);
    const bool hd = __shfl_down_sync(FULL, (int)seen, d) != 0;
    if (open && lane + d < 32) {
      if constexpr (SR::has_val) acc = SR::add(acc, pd);
      if (hd) open = false;
    }
  }
  if (seen && HS_G(dbg, outi >= 0 && outi < c, 93, outi)) {
    __stcs(out_j + outi, curcol);
    if constexpr (SR::has_val) __stcs(out_v + outi, acc);
  }
  if (total != c && lane == 0) atomicExch(err, 13);
}

}  // namespace hs
