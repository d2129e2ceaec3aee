// common.cuh -- device building blocks shared by the SpGEMM kernels.
//
// Contents
//   * semiring traits (Section 1: SpGEMM over a semiring; Section 3.1 selector
//     products), each a mul and an add that may run as a shared-memory atomic;
//   * warp/CTA "groups" so one routine serves a warp-per-row and a CTA-per-row
//     kernel;
//   * the product iterator: the row-wise form of Algorithm 1, C(i,:) +=
//     A(i,k) * B(k,:), with products spread one per lane (a warp-level
//     load-balanced expansion, so short and long rows of B keep every lane busy);
//   * shared-memory hash tables (symbolic: keys; numeric: keys + values);
//   * sorted emission: compaction of a table, a monotone bucket sort in shared
//     memory and coalesced stores of the finished row.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

namespace hs {

// Checked accesses: indices that come from data (row ids read from bin
// lists, column ids, offsets, hash/bucket positions, output ranks) are tested
// before the load or store they address.  A failed check records (code,
// index) in a device word pair that the host reads, and the access is
// skipped, so corrupt or inconsistent input can never turn into an
// out-of-range access on the GPU.
__device__ __forceinline__ bool hs_guard_fail(long long *dbg, int code, long long idx) {
  if (dbg && atomicCAS(reinterpret_cast<unsigned long long *>(dbg), 0ull, (unsigned long long)code) == 0ull)
    dbg[1] = idx;
  return false;
}
#define HS_G(dbg, cond, code, idx) ((cond) ? true : ::hs::hs_guard_fail((dbg), (code), (long long)(idx)))

constexpr unsigned FULL = 0xffffffffu;
constexpr int EMPTY = -1;

// ----------------------------------------------------------------- semirings
enum SrKind { PLUS_TIMES = 0, OR_AND = 1, MIN_PLUS = 2, SELECT2ND = 3, SELECT1ST = 4 };

// Minimum of floats by one integer atomic: floats without their sign bit order
// like integers, those with it the other way round among unsigned numbers, and
// any of them lies below any float without one (a compare-and-swap loop took
// two shared accesses and a branch per attempt).  A NaN is never the smaller
// value and changes nothing; -0 lies below +0.
__device__ __forceinline__ void atomic_min_f32(float *p, float v) {
  const int b = __float_as_int(v);
  if (v != v) return;
  if (b >= 0) atomicMin(reinterpret_cast<int *>(p), b);
  else atomicMax(reinterpret_cast<unsigned *>(p), (unsigned)b);
}

// A semiring over value type T.  mul() is applied to one stored pair,
// add_atomic() folds a product into an accumulator slot that was initialised
// to identity() (the identity is only ever a slot's starting content: every
// slot that is emitted received at least one product, and identity (+) x == x
// exactly for each semiring below).
template <int KIND, typename T> struct Semiring;

template <typename T> struct Semiring<PLUS_TIMES, T> {
  using val_t = T;
  static constexpr bool has_val = true, needs_a = true, needs_b = true;
  __device__ static T identity() { return T(0); }
  __device__ static T mul(T a, T b) { return a * b; }
  __device__ static T add(T x, T y) { return x + y; }
  __device__ static void add_atomic(T *p, T v) { atomicAdd(p, v); }
};
template <> struct Semiring<PLUS_TIMES, int64_t> {
  using val_t = int64_t;
  static constexpr bool has_val = true, needs_a = true, needs_b = true;
  __device__ static int64_t identity() { return 0; }
  // two's complement products and sums, wrapping modulo 2^64
  __device__ static int64_t mul(int64_t a, int64_t b) {
    return (int64_t)((unsigned long long)a * (unsigned long long)b);
  }
  __device__ static int64_t add(int64_t x, int64_t y) {
    return (int64_t)((unsigned long long)x + (unsigned long long)y);
  }
  __device__ static void add_atomic(int64_t *p, int64_t v) {
    atomicAdd(reinterpret_cast<unsigned long long *>(p), (unsigned long long)v);
  }
};
template <> struct Semiring<MIN_PLUS, float> {
  using val_t = float;
  static constexpr bool has_val = true, needs_a = true, needs_b = true;
  __device__ static float identity() { return __int_as_float(0x7f800000); }  // +inf
  __device__ static float mul(float a, float b) { return __fadd_rn(a, b); }
  __device__ static float add(float x, float y) { return y < x ? y : x; }
  __device__ static void add_atomic(float *p, float v) { atomic_min_f32(p, v); }
};
template <> struct Semiring<MIN_PLUS, int32_t> {
  using val_t = int32_t;
  static constexpr bool has_val = true, needs_a = true, needs_b = true;
  __device__ static int32_t identity() { return 0x7fffffff; }
  __device__ static int32_t mul(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }
  __device__ static int32_t add(int32_t x, int32_t y) { return y < x ? y : x; }
  __device__ static void add_atomic(int32_t *p, int32_t v) { atomicMin(p, v); }
};
// structure only: no values at all
struct NoVal {};
template <> struct Semiring<OR_AND, NoVal> {
  using val_t = NoVal;
  static constexpr bool has_val = false, needs_a = false, needs_b = false;
};
// selectors: the value of the non-selector operand is copied; T is a bit
// container of the value's width (uint32_t or unsigned long long)
template <typename T> struct Semiring<SELECT2ND, T> {
  using val_t = T;
  static constexpr bool has_val = true, needs_a = false, needs_b = true;
  __device__ static T identity() { return T(0); }
  __device__ static T mul(T, T b) { return b; }
  __device__ static T add(T x, T) { return x; }
  __device__ static void add_atomic(T *p, T v) { *reinterpret_cast<volatile T *>(p) = v; }
};
template <typename T> struct Semiring<SELECT1ST, T> {
  using val_t = T;
  static constexpr bool has_val = true, needs_a = true, needs_b = false;
  __device__ static T identity() { return T(0); }
  __device__ static T mul(T a, T) { return a; }
  __device__ static T add(T x, T) { return x; }
  __device__ static void add_atomic(T *p, T v) { *reinterpret_cast<volatile T *>(p) = v; }
};

// ------------------------------------------------------------------ groups
struct WarpGroup {
  __device__ __forceinline__ static int size() { return 32; }
  __device__ __forceinline__ static int rank() { return threadIdx.x & 31; }
  __device__ __forceinline__ static int nwarps() { return 1; }
  __device__ __forceinline__ static int warp() { return 0; }
  __device__ __forceinline__ static void sync() { __syncwarp(); }
};
struct CtaGroup {
  __device__ __forceinline__ static int size() { return blockDim.x; }
  __device__ __forceinline__ static int rank() { return threadIdx.x; }
  __device__ __forceinline__ static int nwarps() { return blockDim.x >> 5; }
  __device__ __forceinline__ static int warp() { return threadIdx.x >> 5; }
  __device__ __forceinline__ static void sync() { __syncthreads(); }
};

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

template <typename T> __device__ __forceinline__ T warp_incl_scan(T v) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T u = __shfl_up_sync(FULL, v, d);
    if (lane_id() >= d) v += u;
  }
  return v;
}
template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
  return v;
}
__device__ __forceinline__ int warp_min(int v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v = min(v, __shfl_xor_sync(FULL, v, d));
  return v;
}
__device__ __forceinline__ int warp_max(int v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v = max(v, __shfl_xor_sync(FULL, v, d));
  return v;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v = max(v, __shfl_xor_sync(FULL, v, d));
  return v;
}

// Exclusive scan of a[0..n) in shared memory by a whole group; returns the
// total.  tmp needs 32 ints (CTA groups only); the closing barrier also ends
// every read of tmp.
template <class G> __device__ int group_excl_scan(int *a, int n, int *tmp) {
  const int gs = G::size(), r = G::rank();
  const int per = (n + gs - 1) / gs;
  const int b = min(n, r * per), e = min(n, b + per);
  int s = 0;
  for (int i = b; i < e; ++i) s += a[i];
  int incl = warp_incl_scan(s);
  int total;
  if (G::nwarps() == 1) {
    total = __shfl_sync(FULL, incl, 31);
  } else {
    // the warp totals are published once and every warp scans them itself
    // (nwarps <= 32), so one barrier separates the two levels
    if (lane_id() == 31) tmp[G::warp()] = incl;
    G::sync();
    const int w = lane_id() < G::nwarps() ? tmp[lane_id()] : 0;
    const int wi = warp_incl_scan(w);
    total = __shfl_sync(FULL, wi, 31);
    incl += __shfl_sync(FULL, wi - w, G::warp());
  }
  int run = incl - s;
  for (int i = b; i < e; ++i) {
    int x = a[i];
    a[i] = run;
    run += x;
  }
  G::sync();
  return total;
}

// ---------------------------------------------------------------- operands
struct DevCsr {
  const int64_t *p;  // row offsets (indexed by row slot)
  const int32_t *j;  // column ids
  const void *v;     // values (may be null)
  int64_t rows;      // row slots
  int64_t nnz;       // entries
  long long *dbg;    // guard record (guarded builds)
};

// lower_bound of x in j[s..e) (first position with j >= x)
__device__ __forceinline__ int64_t lower_bound_col(const int32_t *j, int64_t s, int64_t e, int x) {
  while (s < e) {
    int64_t mid = s + ((e - s) >> 1);
    if (__ldg(j + mid) < x) s = mid + 1;
    else e = mid;
  }
  return s;
}

// a[i] <= x holds for exactly the first returned entries of the non-decreasing
// a[0..n); a whole warp searches, 32 probes a step (every lane returns it)
__device__ __forceinline__ int64_t warp_upper_bound(const int64_t *a, int64_t n, int64_t x) {
  int64_t lo = 0, hi = n;
  while (hi - lo > 32) {
    const int64_t s = (hi - lo) >> 5;
    const int c = __popc(__ballot_sync(FULL, __ldg(a + lo + (lane_id() + 1) * s - 1) <= x));
    if (c < 32) hi = lo + (c + 1) * s - 1;
    lo += c * s;
  }
  const int64_t p = lo + lane_id();
  return lo + __popc(__ballot_sync(FULL, p < hi && __ldg(a + p) <= x));
}

template <typename T> __device__ __forceinline__ T load_val(const void *v, int64_t q) {
  return __ldg(reinterpret_cast<const T *>(v) + q);
}
template <> __device__ __forceinline__ NoVal load_val<NoVal>(const void *, int64_t) { return NoVal{}; }

// A visitor may split its work in two: prep(col) does the reads (and any
// atomic whose result it needs) and returns a state; commit(state, value)
// does the final write.  The long-segment loop then preps all of a step's
// products before committing any, so their shared-memory round trips overlap
// instead of queueing behind each other's atomics.
template <class V, class = void> struct two_stage : std::false_type {};
template <class V> struct two_stage<V, std::void_t<decltype(V::kTwoStage)>> : std::bool_constant<V::kTwoStage> {};

template <typename T> __device__ __forceinline__ T shfl_val(T x, int src) { return __shfl_sync(FULL, x, src); }
template <> __device__ __forceinline__ NoVal shfl_val<NoVal>(NoVal x, int) { return x; }

// Visitors that want a product's index in its row: batch() is told how many
// products of the round come before those of the next warp_expand, round() how
// many the round had.
template <class V, class = void> struct flat_visit : std::false_type {};
template <class V> struct flat_visit<V, std::enable_if_t<V::kFlat>> : std::true_type {};

// Visit the products of up to 32 B-row segments (one per lane: start s,
// length len, left value a).  Segments of at least 32 products are walked by
// the whole warp, one segment at a time, with consecutive lanes on
// consecutive entries of B (coalesced, no search).  The remaining short
// segments are dealt one product per lane: lane l takes product base+l of
// their concatenation and finds its segment by a binary search over the
// inclusive length scan (shuffles only).  SB such rounds are taken at once,
// their B loads all issued before the first visit, so a lane has SB
// independent reads in flight instead of one round trip per round.
// visit(col, prod, p) runs on every lane that holds a product, p being the
// product's index in the order of the segments (as if they were walked lane
// by lane).  Returns the number of products.  All 32 lanes must call this
// together.
template <class SR, int U = 2, int SB = 4, class Visit>
__device__ __forceinline__ int warp_expand(const DevCsr &B, int64_t s, int len, typename SR::val_t a,
                                            Visit &visit) {
  using T = typename SR::val_t;
  using VisitT = std::decay_t<Visit>;
  const int lane = lane_id();
  const int incl = warp_incl_scan(len);
  const int total = __shfl_sync(FULL, incl, 31);
  const int ex_full = incl - len;
  // long segments: the whole warp on one segment, U entries per lane per
  // step (all loads of a step issued before the first visit)
  unsigned longm = __ballot_sync(FULL, len >= 32);
  while (longm) {
    const int l = __ffs(longm) - 1;
    longm &= longm - 1;
    const int64_t sl = __shfl_sync(FULL, s, l);
    const int ll = __shfl_sync(FULL, len, l);
    const int el = __shfl_sync(FULL, ex_full, l);
    const T al = shfl_val<T>(a, l);
    if (!HS_G(B.dbg, sl >= 0 && sl + ll <= B.nnz, 4, sl)) continue;
    const int32_t *bj = B.j + sl;
    const T *bv = reinterpret_cast<const T *>(B.v) + sl;
    for (int off = lane; off < ll; off += 32 * U) {
      int c[U];
      T b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool ok = off + 32 * u < ll;
        c[u] = ok ? __ldg(bj + off + 32 * u) : 0;
        b[u] = T{};
        if constexpr (SR::needs_b)
          if (ok) b[u] = __ldg(bv + off + 32 * u);
      }
      if constexpr (two_stage<VisitT>::value) {
        typename VisitT::State st[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (off + 32 * u < ll) st[u] = visit.prep(c[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (off + 32 * u >= ll) break;
          if constexpr (SR::has_val) visit.commit(st[u], SR::mul(al, b[u]));
          else visit.commit(st[u], NoVal{});
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (off + 32 * u >= ll) break;
          if constexpr (SR::has_val) visit(c[u], SR::mul(al, b[u]), el + off + 32 * u);
          else visit(c[u], NoVal{}, el + off + 32 * u);
        }
      }
    }
  }
  // short segments: one product per lane, SB rounds of 32 at a time
  const int slen = len < 32 ? len : 0;
  const int sincl = warp_incl_scan(slen);
  const int stotal = __shfl_sync(FULL, sincl, 31);
  const int sexcl = sincl - slen;
  for (int base = 0; base < stotal; base += 32 * SB) {
    int col[SB], pidx[SB];
    T pv[SB];
    bool ok[SB];
#pragma unroll
    for (int u = 0; u < SB; ++u) {
      ok[u] = false;
      col[u] = 0;
      pidx[u] = 0;
      pv[u] = T{};
      if (base + 32 * u < stotal) {  // warp-uniform: the shuffles below see every lane
        const int p = base + 32 * u + lane;
        int src = 0;  // number of lanes whose inclusive end is <= p
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
          const int v = __shfl_sync(FULL, sincl, src + step - 1);
          if (v <= p) src += step;
        }
        const int64_t ss = __shfl_sync(FULL, s, src);
        const int sex = __shfl_sync(FULL, sexcl, src);
        const int fex = __shfl_sync(FULL, ex_full, src);
        const T aa = shfl_val<T>(a, src);
        if (p < stotal) {
          const int64_t pos = ss + (p - sex);
          if (HS_G(B.dbg, pos >= 0 && pos < B.nnz, 4, pos)) {
            ok[u] = true;
            col[u] = __ldg(B.j + pos);
            pidx[u] = fex + (p - sex);
            if constexpr (SR::has_val) {
              T b{};
              if constexpr (SR::needs_b) b = load_val<T>(B.v, pos);
              pv[u] = SR::mul(aa, b);
            }
          }
        }
      }
    }
    if constexpr (two_stage<VisitT>::value) {
      typename VisitT::State st[SB];
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) st[u] = visit.prep(col[u]);
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) visit.commit(st[u], pv[u]);
    } else {
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) visit(col[u], pv[u], pidx[u]);
    }
  }
  return total;
}

// B-row segment of A entry q: [s, e) of B(k,:), restricted to columns
// [lo, hi) when restrict_cols.
__device__ __forceinline__ void entry_segment(const DevCsr &A, const DevCsr &B, int64_t q, bool restrict_cols,
                                              int lo, int hi, int64_t &s, int64_t &e) {
  s = e = 0;
  if (!HS_G(A.dbg, q >= 0 && q < A.nnz, 1, q)) return;
  const int k = __ldg(A.j + q);
  if (!HS_G(A.dbg, k >= 0 && k < B.rows, 2, k)) return;
  s = __ldg(B.p + k);
  e = __ldg(B.p + k + 1);
  if (!HS_G(A.dbg, s >= 0 && s <= e && e <= B.nnz, 3, e)) {
    s = e = 0;
    return;
  }
  if (restrict_cols && s < e) {
    s = lower_bound_col(B.j, s, e, lo);
    e = lower_bound_col(B.j, s, e, hi);
  }
}

// Every product of one row, by one warp: A entries [q0, q1) in chunks of 32.
template <class SR, class Visit>
__device__ __forceinline__ void warp_products(const DevCsr &A, const DevCsr &B, int64_t q0, int64_t q1,
                                              Visit &&visit) {
  using T = typename SR::val_t;
  for (int64_t qb = q0; qb < q1; qb += 32) {
    const int64_t q = qb + lane_id();
    int64_t s = 0, e = 0;
    T a{};
    if (q < q1) {
      entry_segment(A, B, q, false, 0, 0, s, e);
      if constexpr (SR::needs_a) a = load_val<T>(A.v, q);
    }
    warp_expand<SR>(B, s, (int)(e - s), a, visit);
  }
}

// position of the (r + 1)-th set bit of m (r < popc(m))
__device__ __forceinline__ int nth_bit(unsigned m, int r) {
  int pos = 0;
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const int c = __popc((m >> pos) & ((1u << w) - 1u));
    if (c <= r) {
      r -= c;
      pos += w;
    }
  }
  return pos;
}

// warp_expand for the kernels that give a row to a warp.  The short segments
// are moved to the lowest lanes (empty ones drop out) and a round's segment
// starts are or-ed into one word (__reduce_or_sync), so that a lane's segment
// is the number of starts at or below it instead of a search over the length
// scan; the check against B's size is made once per segment.  (R-MAT scale
// 20: warp rows of the symbolic pass 0.36 -> 0.30 ms, a batch of random
// products 1.53 -> 1.38 ms.  In the kernels that give a row to a block, which
// hold more registers, the search measured faster: rows of 1024 to 4096
// products 1.52 against 1.58 ms, the bitmap kernel 23.8 against 24.2 ms.)
// visit and the result as for warp_expand; a segment outside B (a failed
// check) makes no products.
template <class SR, int U = 2, int SB = 4, class Visit>
__device__ __forceinline__ int warp_expand_row(const DevCsr &B, int64_t s, int len, typename SR::val_t a,
                                            Visit &visit) {
  using T = typename SR::val_t;
  using VisitT = std::decay_t<Visit>;
  const int lane = lane_id();
  if (len > 0 && !HS_G(B.dbg, s >= 0 && s + len <= B.nnz, 4, s)) len = 0;
  const int incl = warp_incl_scan(len);
  const int total = __shfl_sync(FULL, incl, 31);
  const int ex_full = incl - len;
  // long segments: the whole warp on one segment, U entries per lane per
  // step (all loads of a step issued before the first visit); a last step of
  // fewer than U * 32 entries runs only the sub-steps it has
  const unsigned long_all = __ballot_sync(FULL, len >= 32);
  for (unsigned longm = long_all; longm; longm &= longm - 1) {
    const int l = __ffs(longm) - 1;
    const int64_t sl = __shfl_sync(FULL, s, l);
    const int ll = __shfl_sync(FULL, len, l);
    const int el = __shfl_sync(FULL, ex_full, l);
    const T al = shfl_val<T>(a, l);
    const int32_t *bj = B.j + sl;
    const T *bv = reinterpret_cast<const T *>(B.v) + sl;
    for (int o0 = 0; o0 < ll; o0 += 32 * U) {
      const int off = o0 + lane;
      int c[U];
      T b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool ok = off + 32 * u < ll;
        c[u] = ok ? __ldg(bj + off + 32 * u) : 0;
        b[u] = T{};
        if constexpr (SR::needs_b)
          if (ok) b[u] = __ldg(bv + off + 32 * u);
      }
      if constexpr (two_stage<VisitT>::value) {
        typename VisitT::State st[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (off + 32 * u < ll) st[u] = visit.prep(c[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (o0 + 32 * u >= ll) break;
          if (off + 32 * u >= ll) continue;
          if constexpr (SR::has_val) visit.commit(st[u], SR::mul(al, b[u]));
          else visit.commit(st[u], NoVal{});
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (o0 + 32 * u >= ll) break;
          if (off + 32 * u >= ll) continue;
          if constexpr (SR::has_val) visit(c[u], SR::mul(al, b[u]), el + off + 32 * u);
          else visit(c[u], NoVal{}, el + off + 32 * u);
        }
      }
    }
  }
  // short segments: one product per lane, SB rounds of 32 at a time
  const unsigned shortm = __ballot_sync(FULL, len > 0 && len < 32);
  if (!shortm) return total;
  const int ns = __popc(shortm);
  int fex = ex_full;  // the segment's first product in the order of all segments
  int sex = ex_full;  // and among the short ones
  if (long_all) {
    const int slen = len < 32 ? len : 0;
    sex = warp_incl_scan(slen) - slen;
  }
  if (shortm & (shortm + 1)) {  // gaps: the short segments move to lanes 0 .. ns-1
    const int src = nth_bit(shortm, lane < ns ? lane : 0);
    s = __shfl_sync(FULL, s, src);
    a = shfl_val<T>(a, src);
    fex = __shfl_sync(FULL, fex, src);
    sex = __shfl_sync(FULL, sex, src);
    len = __shfl_sync(FULL, len, src);
  }
  const int stotal = __shfl_sync(FULL, sex + len, ns - 1);
  const int64_t place = s - sex;  // product p of the segment lies at place + p
  const unsigned le = 0xffffffffu >> (31 - lane);
  int before = 0;  // segments that start before the round
  for (int base = 0; base < stotal; base += 32 * SB) {
    int col[SB], pidx[SB];
    T pv[SB];
    bool ok[SB];
#pragma unroll
    for (int u = 0; u < SB; ++u) {
      ok[u] = false;
      col[u] = 0;
      pidx[u] = 0;
      pv[u] = T{};
      if (base + 32 * u < stotal) {  // warp-uniform: the shuffles below see every lane
        const int p = base + 32 * u + lane;
        const unsigned at = (unsigned)(sex - (base + 32 * u));
        const unsigned starts = __reduce_or_sync(FULL, lane < ns && at < 32u ? 1u << at : 0u);
        const int src = before + __popc(starts & le) - 1;
        before += __popc(starts);
        const int64_t pos = __shfl_sync(FULL, place, src) + p;
        const T aa = shfl_val<T>(a, src);
        if constexpr (!two_stage<VisitT>::value) {
          pidx[u] = p;
          if (long_all) pidx[u] += __shfl_sync(FULL, fex - sex, src);
        }
        if (p < stotal) {
          ok[u] = true;
          col[u] = __ldg(B.j + pos);
          if constexpr (SR::has_val) {
            T b{};
            if constexpr (SR::needs_b) b = load_val<T>(B.v, pos);
            pv[u] = SR::mul(aa, b);
          }
        }
      }
    }
    if constexpr (two_stage<VisitT>::value) {
      typename VisitT::State st[SB];
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) st[u] = visit.prep(col[u]);
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) visit.commit(st[u], pv[u]);
    } else {
#pragma unroll
      for (int u = 0; u < SB; ++u)
        if (ok[u]) visit(col[u], pv[u], pidx[u]);
    }
  }
  return total;
}

// The row a warp will take next, looked up in steps while it works on the
// present one: row id, its range of A, and for the first 32 entries of A
// their columns (with A's values) and B offsets.  Row kernels with one warp
// per row are a chain of five dependent loads before the first product; each
// step is issued one stage of the present row ahead of the next, so that only
// B's entries themselves are waited for.
template <class SR> struct RowAhead {
  using T = typename SR::val_t;
  int r = -1;
  int64_t q0 = 0, q1 = 0;
  int k = -1;
  T a{};
  int64_t s = 0;
  int len = 0;
  __device__ __forceinline__ void row(const DevCsr &A, const int *list, int idx, int count) {
    r = idx < count ? __ldg(list + idx) : -1;
    if (r >= 0 && !HS_G(A.dbg, r < A.rows, 35, r)) r = -1;
  }
  __device__ __forceinline__ void range(const DevCsr &A) {
    q0 = q1 = 0;
    if (r >= 0) {
      q0 = __ldg(A.p + r);
      q1 = __ldg(A.p + r + 1);
    }
  }
  __device__ __forceinline__ void entries(const DevCsr &A) {
    const int64_t q = q0 + lane_id();
    k = -1;
    if (q < q1 && HS_G(A.dbg, q >= 0 && q < A.nnz, 1, q)) {
      k = __ldg(A.j + q);
      if constexpr (SR::needs_a) a = load_val<T>(A.v, q);
    }
  }
  __device__ __forceinline__ void segments(const DevCsr &B) {
    s = 0;
    len = 0;
    if (q0 + lane_id() >= q1) return;
    if (!HS_G(B.dbg, k >= 0 && k < B.rows, 2, k)) return;
    s = __ldg(B.p + k);
    const int64_t e = __ldg(B.p + k + 1);
    if (HS_G(B.dbg, s >= 0 && s <= e && e <= B.nnz, 3, e)) len = (int)(e - s);
  }
  __device__ __forceinline__ void all(const DevCsr &A, const DevCsr &B, const int *list, int idx, int count) {
    row(A, list, idx, count);
    range(A);
    entries(A);
    segments(B);
  }
};

// Every product of the row held by `x`: its first 32 entries as looked up,
// the others as they come.  Returns their number.
template <class SR, class Visit>
__device__ __forceinline__ int warp_products_of(const DevCsr &A, const DevCsr &B, const RowAhead<SR> &x, Visit &visit) {
  using T = typename SR::val_t;
  int64_t s = x.s;
  int len = x.len, total = 0;
  T a = x.a;
  for (int64_t qb = x.q0;;) {
    const int done = total;
    auto at = [&](int col, T v, int p) { visit(col, v, done + p); };
    total += warp_expand_row<SR>(B, s, len, a, at);
    qb += 32;
    if (qb >= x.q1) return total;
    const int64_t q = qb + lane_id();
    int64_t e = 0;
    s = 0;
    if (q < x.q1) {
      entry_segment(A, B, q, false, 0, 0, s, e);
      if constexpr (SR::needs_a) a = load_val<T>(A.v, q);
    }
    len = (int)(e - s);
  }
}

// Rows of few products, several to a warp: as many of the next (at most
// eight) listed rows as hold at most 32 entries of A and 32 products together,
// their entries one per lane, then their products one per lane, row after row
// in product order.  A warp that takes such rows one by one spends some 250
// instructions a row on mostly idle lanes; taken together, the look-ups of a
// row do not run as far ahead.  7e5 rows of 5 products on average: symbolic
// 150 -> 82 us, numeric 210 -> 127 us; 1.1e5 rows of 32: 27 -> 38 us.
constexpr int TG_ROWS = 8;
// the next eight rows of the list, one per lane: as rows are taken the others
// move down, and the places that fall free are looked up while the taken rows
// are worked on
struct TinyWindow {
  int r = -1;         // row slot (-1: none, or an invalid id)
  int64_t q0 = 0, ne = 0;
  int f = 0;
  __device__ __forceinline__ void ids(const DevCsr &A, const int *list, int idx, int end, int from) {
    if (lane_id() < from) return;
    r = lane_id() < TG_ROWS && idx + lane_id() < end ? __ldg(list + idx + lane_id()) : -1;
    if (r >= 0 && !HS_G(A.dbg, r < A.rows, 35, r)) r = -1;
  }
  __device__ __forceinline__ void ranges(const DevCsr &A, const int64_t *fl, int from) {
    if (lane_id() < from) return;
    q0 = ne = 0;
    f = 0;
    if (r >= 0) {
      q0 = __ldg(A.p + r);
      ne = __ldg(A.p + r + 1) - q0;
      f = (int)__ldg(fl + r);
    }
  }
  // k rows taken: the first free place
  __device__ __forceinline__ int slide(int k) {
    r = __shfl_sync(FULL, r, (lane_id() + k) & 31);
    q0 = __shfl_sync(FULL, q0, (lane_id() + k) & 31);
    ne = __shfl_sync(FULL, ne, (lane_id() + k) & 31);
    f = __shfl_sync(FULL, f, (lane_id() + k) & 31);
    return TG_ROWS - k;
  }
};
template <class SR> struct TinyGroup {
  using T = typename SR::val_t;
  int rows;        // rows taken (uniform); 0: the first row has more than 32 entries
  int nprod;       // products (uniform)
  // lane l < rows: its row slot and the lanes that hold its products
  int r;
  unsigned mask;
  // lane l < nprod: its product's column, value and row (0 .. rows-1)
  int col, row;
  T v;
};
// the rows that fit, from the window win of rows idx .. idx+7; the window
// moves past them
template <class SR>
__device__ __forceinline__ TinyGroup<SR> tiny_group(const DevCsr &A, const DevCsr &B, const int *list, int idx, int end,
                                                    const int64_t *f, TinyWindow &win) {
  using T = typename SR::val_t;
  const int lane = lane_id();
  const unsigned le = 0xffffffffu >> (31 - lane);
  TinyGroup<SR> g{};
  g.r = lane < TG_ROWS ? win.r : -1;
  const int64_t q0 = win.q0, ne64 = win.ne;
  const int fr = lane < TG_ROWS ? win.f : 0;
  const int ne = lane < TG_ROWS ? (int)max(min(ne64, (int64_t)64), (int64_t)0) : 0;
  // entries (high half) and products of the rows so far; a listed row has
  // both, so the rows that still fit are the first ones (an invalid id takes
  // part as an empty row)
  const int both = (ne << 16) | min(max(fr, 0), 64);
  const int incl = warp_incl_scan(both);
  const bool fit = lane < TG_ROWS && idx + lane < end && (incl >> 16) <= 32 && (incl & 0xffff) <= 32;
  g.rows = __popc(__ballot_sync(FULL, fit));
  if (g.rows == 0) return g;
  const int from = win.slide(g.rows);
  win.ids(A, list, idx + g.rows, end, from);
  const int ex = incl - both;
  const int px = ex & 0xffff;
  g.mask = lane < g.rows && fr > 0 ? (0xffffffffu >> (32 - min(fr, 32))) << px : 0u;
  const int E = __shfl_sync(FULL, incl, g.rows - 1) >> 16;
  // rows without entries (invalid ids) own no lane: rows are found among those that do
  const unsigned starts = __reduce_or_sync(FULL, lane < g.rows && ne > 0 ? 1u << (ex >> 16) : 0u);
  const unsigned full = __ballot_sync(FULL, lane < g.rows && ne > 0);
  const int nth = __popc(starts & le) - 1;
  int row = (full & (full + 1)) ? nth_bit(full, nth < 0 ? 0 : nth) : nth;
  row = row < 0 ? 0 : row;
  const int64_t q = __shfl_sync(FULL, q0, row) + (lane - (__shfl_sync(FULL, ex, row) >> 16));
  int64_t s = 0;
  int len = 0;
  T a{};
  if (lane < E) {
    int64_t e = 0;
    entry_segment(A, B, q, false, 0, 0, s, e);
    len = (int)min(e - s, (int64_t)33);
    if constexpr (SR::needs_a) a = load_val<T>(A.v, q);
  }
  win.ranges(A, f, from);
  const int pincl = warp_incl_scan(len);
  const int total = __shfl_sync(FULL, pincl, 31);
  int sex = pincl - len;
  const unsigned nz = __ballot_sync(FULL, len > 0);
  const int ns = __popc(nz);
  if (nz & (nz + 1)) {
    const int src = nth_bit(nz, lane < ns ? lane : 0);
    s = __shfl_sync(FULL, s, src);
    a = shfl_val<T>(a, src);
    sex = __shfl_sync(FULL, sex, src);
    row = __shfl_sync(FULL, row, src);
  }
  g.nprod = min(total, 32);  // (more only if f does not belong to this A and B)
  const unsigned ps = __reduce_or_sync(FULL, lane < ns && sex < 32 ? 1u << sex : 0u);
  const int src = max(__popc(ps & le) - 1, 0);
  const int64_t pos = __shfl_sync(FULL, s - sex, src) + lane;
  const T aa = shfl_val<T>(a, src);
  g.row = __shfl_sync(FULL, row, src);
  g.col = 0;
  g.v = T{};
  if (lane < g.nprod) {
    g.col = __ldg(B.j + pos);
    if constexpr (SR::has_val) {
      T b{};
      if constexpr (SR::needs_b) b = load_val<T>(B.v, pos);
      g.v = SR::mul(aa, b);
    }
  }
  return g;
}

// Ask for [p, p + bytes) to be brought into L2 ahead of its reads (bulk
// prefetch, no completion to wait for).  The range is narrowed to 16-byte
// boundaries, so it never leaves the buffer, and issued in pieces of at most
// 64 KB.
__device__ __forceinline__ void prefetch_l2(const void *p, int64_t bytes) {
  if (bytes <= 0) return;
  uint64_t a = (uint64_t)__cvta_generic_to_global(p);
  const uint64_t e = (a + (uint64_t)bytes) & ~(uint64_t)15;
  a = (a + 15) & ~(uint64_t)15;
  while (a < e) {
    const uint64_t len = e - a < 65536 ? e - a : 65536;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)len) : "memory");
    a += len;
  }
}

// Asynchronous copy (cp.async, 16-byte pieces, completed by cp.async.wait_all
// and a barrier) of the global bytes [src, src + bytes) into shared memory at
// dst + off, off = src mod 16: the copy runs from the 16-byte boundary at or
// below src to the one at or above src + bytes, so dst needs bytes + 32 bytes
// of room and the source buffer 16 bytes of slack past its end.  Every
// thread of the group calls it with its rank.
__device__ __forceinline__ int async_copy16(void *dst, const void *src, int64_t bytes, int rank, int nthreads) {
  const uint64_t s = (uint64_t)src;
  const uint64_t s0 = s & ~(uint64_t)15;
  const int64_t chunks = (int64_t)((s + (uint64_t)bytes + 15 - s0) >> 4);
  const unsigned d0 = (unsigned)__cvta_generic_to_shared(dst);
  for (int64_t c = rank; c < chunks; c += nthreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + (unsigned)(c << 4)),
                 "l"(__cvta_generic_to_global((const void *)(s0 + (uint64_t)(c << 4))))
                 : "memory");
  return (int)(s - s0);
}
__device__ __forceinline__ void async_copy_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

__host__ __device__ __forceinline__ int next_pow2(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Shared-memory arrays for cta_products (CH A entries per round).
template <typename T, int CH> struct CtaExpandSmem {
  int excl[CH + 1];
  int64_t sbeg[CH];
  T aval[CH];
};

// The products of n staged B-row segments (start sbeg[e], exclusive length
// prefix excl[e], excl[n] = total, left values aval[e]) spread evenly over
// the warps of the CTA: each warp takes one contiguous range of the products
// and deals it one product per lane (warp_expand).  Reads the staged arrays
// only; all threads of the CTA must call it together.
// Each segment may also be charged K units of fixed cost (its setup in the
// warp loop): warps then split the cost, not just the products, so a warp
// whose range holds many short segments gets fewer products.  excl may hold
// a running prefix that starts at ebase instead of 0 (a batch of a longer
// list).
template <class SR, int U = 2, int K = 0, class Visit>
__device__ __forceinline__ void cta_expand_staged(const DevCsr &B, const int64_t *sbeg, const int *excl,
                                                  const typename SR::val_t *aval, int n, int total,
                                                  Visit &visit, int ebase = 0) {
  using T = typename SR::val_t;
  const int lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // entry e occupies [X_e, X_e+1) with X_e = excl[e] + K*e: K units of its
  // fixed cost, then its products
  const int64_t tcost = (int64_t)total + (int64_t)K * n;
  const int64_t pb = tcost * warp / nw, pe = tcost * (warp + 1) / nw;
  if (pb >= pe) return;
  // last entry whose start is <= pb (entry 0 starts at 0, so l >= 1)
  int l = 0, h = n;
  while (l < h) {
    const int mid = (l + h) >> 1;
    if (excl[mid] - ebase + (int64_t)K * mid <= pb) l = mid + 1;
    else h = mid;
  }
  for (int eb = l - 1; eb < n; eb += 32) {
    const int e = eb + lane;
    int64_t s = 0;
    int len = 0;
    T a{};
    if constexpr (flat_visit<std::decay_t<Visit>>::value) {  // products of the round before this batch
      const int64_t ahead = pb - (excl[eb] - ebase + (int64_t)K * eb + K);
      visit.batch(excl[eb] - ebase + (int)min(max(ahead, (int64_t)0), (int64_t)(excl[eb + 1] - excl[eb])));
    }
    if (e < n) {
      const int64_t x0 = excl[e] - ebase + (int64_t)K * e + K, x1 = excl[e + 1] - ebase + (int64_t)K * (e + 1);
      const int64_t cb = max(x0, pb), ce = min(x1, pe);
      if (ce > cb) {
        len = (int)(ce - cb);
        s = sbeg[e] + (cb - x0);
        if constexpr (SR::needs_a) a = aval[e];
      }
    }
    warp_expand<SR, U>(B, s, len, a, visit);
    if (eb + 32 >= n || excl[eb + 32] - ebase + (int64_t)K * (eb + 32) >= pe) break;
  }
}

// First position in [s, e) whose column is >= x.  Long ranges start with one
// interpolation probe (column ids of a row are close to uniform after a
// random relabelling) and narrow the bracket around it; then, as for short
// ranges, probe lo, lo+1, lo+3, lo+7, ... (galloping) and finish with a
// binary search, so the cost stays logarithmic for any distribution.
__device__ __forceinline__ int64_t gallop_lower_bound(const int32_t *j, int64_t s, int64_t e, int x);
__device__ __forceinline__ int64_t interp_lower_bound(const int32_t *j, int64_t s, int64_t e, int x) {
  if (e - s > 64) {
    const int c0 = __ldg(j + s), c1 = __ldg(j + e - 1);
    if (c0 >= x) return s;
    if (c1 < x) return e;
    // c0 < x <= c1: the answer is in (s, e-1]
    int64_t g = s + 1 + (int64_t)(((double)(x - c0) / (double)(c1 - c0 + 1)) * (double)(e - 2 - s));
    if (g > e - 1) g = e - 1;
    if (g <= s) g = s + 1;
    if (__ldg(j + g) >= x) {
      // answer in (s, g]: gallop leftwards from g
      int64_t hi = g, step = 1, lo = g - 1;
      while (lo > s && __ldg(j + lo) >= x) {
        hi = lo;
        step <<= 1;
        lo = g - step;
        if (lo < s) lo = s;
      }
      // j[lo] < x (or lo == s), j[hi] >= x
      int64_t a = lo + 1, b = hi;
      while (a < b) {
        const int64_t mid = a + ((b - a) >> 1);
        if (__ldg(j + mid) < x) a = mid + 1;
        else b = mid;
      }
      return a;
    }
    return gallop_lower_bound(j, g + 1, e, x);
  }
  return gallop_lower_bound(j, s, e, x);
}

// First position in [s, e) whose column is >= x: probe s, s+1, s+3, s+7, ...
// (galloping) and finish with a binary search, so a short distance costs few
// loads whatever the row's length.
__device__ __forceinline__ int64_t gallop_lower_bound(const int32_t *j, int64_t s, int64_t e, int x) {
  if (s >= e || __ldg(j + s) >= x) return s;
  int64_t lo = s + 1, step = 1, hi = s + 1;
  while (hi < e && __ldg(j + hi) < x) {
    lo = hi + 1;
    step <<= 1;
    hi = s + step;
  }
  if (hi > e) hi = e;
  while (lo < hi) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(j + mid) < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Every product of one row (or of the part of it inside columns [lo, hi)),
// spread evenly over the warps of the CTA.  A entries are taken CH at a time;
// their B segments' lengths are scanned across the CTA, the products of the
// round are cut into one contiguous range per warp, and each warp deals its
// range one product per lane (warp_expand).  Per-row product counts must stay
// below 2^31.  All threads of the CTA must call this together.
// SU: entries a thread looks up at a time (column, then B's offsets).
template <class SR, int CH, int U = 2, int SU = 1, class Visit>
__device__ __forceinline__ void cta_products(const DevCsr &A, const DevCsr &B, int64_t q0, int64_t q1, bool restrict_cols,
                             int lo, int hi, CtaExpandSmem<typename SR::val_t, CH> &sm, int *wtmp,
                             Visit &&visit) {
  using T = typename SR::val_t;
  const int tid = threadIdx.x;
  for (int64_t c0 = q0; c0 < q1; c0 += CH) {
    const int n = (int)min((int64_t)CH, q1 - c0);
    for (int e0 = tid; e0 < n; e0 += SU * blockDim.x) {
      int k[SU];
      int64_t s[SU], en[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int e = e0 + u * blockDim.x;
        k[u] = -1;
        if (e < n && HS_G(A.dbg, c0 + e >= 0 && c0 + e < A.nnz, 1, c0 + e)) k[u] = __ldg(A.j + c0 + e);
      }
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int e = e0 + u * blockDim.x;
        s[u] = en[u] = 0;
        if (e < n && HS_G(A.dbg, k[u] >= 0 && k[u] < B.rows, 2, k[u])) {
          s[u] = __ldg(B.p + k[u]);
          en[u] = __ldg(B.p + k[u] + 1);
        }
      }
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int e = e0 + u * blockDim.x;
        if (e >= n) break;
        if (!HS_G(A.dbg, s[u] >= 0 && s[u] <= en[u] && en[u] <= B.nnz, 3, en[u])) s[u] = en[u] = 0;
        if (restrict_cols && s[u] < en[u]) {
          s[u] = lower_bound_col(B.j, s[u], en[u], lo);
          en[u] = lower_bound_col(B.j, s[u], en[u], hi);
        }
        if constexpr (SR::needs_a) sm.aval[e] = load_val<T>(A.v, c0 + e);
        sm.excl[e] = (int)(en[u] - s[u]);
        sm.sbeg[e] = s[u];
      }
    }
    if (tid == 0) sm.excl[n] = 0;  // scanned with the entries, it becomes the round's total
    __syncthreads();
    // only the staged entries are scanned (a short row costs what it holds)
    const int total = group_excl_scan<CtaGroup>(sm.excl, n + 1, wtmp);
    cta_expand_staged<SR, U, 32>(B, sm.sbeg, sm.excl, sm.aval, n, total, visit);
    if constexpr (flat_visit<std::decay_t<Visit>>::value) visit.round(total);
    __syncthreads();
  }
}

// ------------------------------------------------------------ hash tables
__device__ __forceinline__ unsigned hash_slot(int key, unsigned mask) {
  return (unsigned)(key * 2654435761u) & mask;  // Knuth multiplicative hash
}

// Symbolic insert: returns 1 if the key was new.  The table holds at least
// twice the row's product count, so it cannot fill; the probe count is still
// bounded (a full table would return 0 after visiting every slot).
__device__ __forceinline__ int hash_insert_key(int *keys, unsigned mask, int key) {
  unsigned h = hash_slot(key, mask);
  for (unsigned probes = 0; probes <= mask; ++probes) {
    int k = reinterpret_cast<volatile int *>(keys)[h];
    if (k == key) return 0;
    if (k == EMPTY) {
      int old = atomicCAS(keys + h, EMPTY, key);
      if (old == EMPTY) return 1;
      if (old == key) return 0;
    }
    h = (h + 1) & mask;
  }
  return 0;
}

// Symbolic insert into a bitmap of all columns (when they fit the table's
// room): one atomic whose answer says whether the column was new, no probes.
__device__ __forceinline__ int bitmap_insert(int *words, int col) {
  const unsigned bit = 1u << (col & 31);
  return (atomicOr(reinterpret_cast<unsigned *>(words) + (col >> 5), bit) & bit) == 0u;
}
// the words of a bitmap of n columns, rounded up to 16-byte pieces, cleared by a group
template <class G> __device__ __forceinline__ void bitmap_clear(int *words, int n) {
  int4 *w4 = reinterpret_cast<int4 *>(words);
  for (int i = G::rank(); i < (n + 127) >> 7; i += G::size()) w4[i] = make_int4(0, 0, 0, 0);
}

// Numeric insert: fold v into the slot of key.  The table is sized from the
// symbolic count (at least twice the row's distinct keys), so it cannot fill;
// should it ever, the probe gives up after visiting every slot and raises
// *err instead of spinning.
template <class SR, typename T>
__device__ __forceinline__ void hash_insert_val(int *keys, T *vals, unsigned mask, int key, T v, int *err) {
  unsigned h = hash_slot(key, mask);
  for (unsigned probes = 0;; ++probes) {
    if (probes > mask) {
      atomicExch(err, 7);
      return;
    }
    int k = reinterpret_cast<volatile int *>(keys)[h];
    if (k == key) break;
    if (k == EMPTY) {
      int old = atomicCAS(keys + h, EMPTY, key);
      if (old == EMPTY || old == key) break;
    }
    h = (h + 1) & mask;
  }
  if constexpr (SR::has_val) SR::add_atomic(vals + h, v);
}

// ----------------------------------------------------------- sorted emit
// Shared-memory layout used by group_sort_emit (all offsets in bytes):
//   ck[cap] int32 | cv[cap] T           (compacted entries, arbitrary order)
//   work: bcnt[nb] int32 | sk[c] int32 | sv[c] T
// `work` may alias the hash table (it is free once compacted).
//
// Steps: (1) every occupied slot of the table is appended to ck/cv, and the
// key range [kmin, kmax] is found; (2) keys are distributed over nb buckets
// by the monotone map b = (key-kmin)*nb/(kmax-kmin+1); a histogram and an
// exclusive scan give every bucket its start, and the entries are put into
// their buckets; (3) an entry's final position is its bucket's start plus the
// number of keys in the bucket that are smaller (keys are distinct).  Rows of
// 2048..4096 entries spent half of their time on (3) when it ran over the
// unsorted entries, with ids in the buckets and the sorted row gathered in
// shared memory, every lane through a loop of its own length: R-MAT scale 20,
// these rows 5.04 -> 4.35 ms, those of 1024..2048 entries 2.56 -> 2.20 ms.
struct EmitScratch {
  int kmin, kmax, count;
};

// number of buckets for c entries: the largest power of two <= c
__host__ __device__ __forceinline__ int emit_buckets(int c) {
  int nb = 1;
  while (nb * 2 <= c) nb <<= 1;
  return nb;
}
// bytes of the `work` region for c entries with values of `vbytes` bytes
__host__ __device__ __forceinline__ size_t emit_work_bytes(int c, int vbytes) {
  return ((((size_t)(emit_buckets(c) + c) * 4 + 7) & ~(size_t)7)) + (size_t)c * vbytes;
}

// Steps (2) and (3): out(place, key, value) for the c entries of ck/cv.  DUPS:
// keys may be equal, and then keep some order among themselves; out may write
// to ck/cv, which are not read any more.  Step (3) takes as many steps as a
// bucket has entries: with DUPS, a row whose largest bucket holds more than
// `limit` is left as it is and false returned (*most: zeroed before).
template <class G, typename T, bool HAS_VAL, bool DUPS, class Out>
__device__ __forceinline__ bool group_bucket_sort(const int *ck, const T *cv, int c, int kmin, int kmax, void *work,
                                                  int *wtmp, long long *dbg, Out &&out, int *most_shared = nullptr,
                                                  int limit = 0) {
  constexpr int EU = 4;  // entries per thread per step: their shared-memory chains overlap
  const int gs = G::size(), r = G::rank(), lane = lane_id();
  const int nb = emit_buckets(c);
  int *bcnt = reinterpret_cast<int *>(work);
  int *sk = bcnt + nb;
  T *sv = reinterpret_cast<T *>(reinterpret_cast<char *>(work) + (((size_t)(nb + c) * 4 + 7) & ~(size_t)7));
  const uint64_t range = (uint64_t)(kmax - kmin) + 1;
  // monotone bucket map b = floor((key-kmin) * scale / 2^32), scale = floor(nb*2^32/range) < 2^32*nb/range
  const uint64_t scale = (((uint64_t)nb) << 32) / range;
  auto bucket = [&](int key) { return (int)(((uint64_t)(unsigned)(key - kmin) * scale) >> 32); };
  for (int b = r; b < nb; b += gs) bcnt[b] = 0;
  G::sync();
  for (int e = r; e < c; e += gs) {
    const int b = bucket(ck[e]);
    if (HS_G(dbg, b >= 0 && b < nb, 21, b)) atomicAdd(bcnt + b, 1);
  }
  G::sync();
  if constexpr (DUPS) {
    int n = 0;
    for (int b = r; b < nb; b += gs) n = max(n, bcnt[b]);
    n = warp_max(n);
    if (lane == 0 && n > limit) atomicMax(most_shared, n);
    G::sync();
    if (*most_shared > limit) return false;
  }
  group_excl_scan<G>(bcnt, nb, wtmp);
  // the entries into their buckets (arbitrary order inside a bucket); bcnt[b]
  // advances to the bucket's end
  for (int e0 = r; e0 < c; e0 += EU * gs) {
    int key[EU], at[EU];
#pragma unroll
    for (int u = 0; u < EU; ++u) {
      const int e = e0 + u * gs;
      key[u] = e < c ? ck[e] : 0;
    }
#pragma unroll
    for (int u = 0; u < EU; ++u) {
      at[u] = -1;
      const int b = e0 + u * gs < c ? bucket(key[u]) : -1;
      if (b >= 0 && HS_G(dbg, b < nb, 22, b)) at[u] = atomicAdd(bcnt + b, 1);
    }
#pragma unroll
    for (int u = 0; u < EU; ++u)
      if (at[u] >= 0 && HS_G(dbg, at[u] < c, 23, at[u])) {
        sk[at[u]] = key[u];
        if constexpr (HAS_VAL) sv[at[u]] = cv[e0 + u * gs];
      }
  }
  G::sync();
  // (3) position i's entry goes out at its bucket's start plus the number of
  // smaller keys in the bucket, a place or two from i: the lanes read the same
  // few words and their stores (evict-first: C is not read again here, B is)
  // fall into the same lines
  for (int w0 = r - lane; w0 < c; w0 += EU * gs) {  // (whole warps)
    int key[EU], bs[EU], len[EU], rank[EU];
    T v[EU];
    int most = 0;
#pragma unroll
    for (int u = 0; u < EU; ++u) {
      const int i = w0 + lane + u * gs;
      key[u] = i < c ? sk[i] : kmin;
      if constexpr (HAS_VAL) v[u] = i < c ? sv[i] : T{};
    }
#pragma unroll
    for (int u = 0; u < EU; ++u) {
      const int b = bucket(key[u]);
      bs[u] = b ? bcnt[b - 1] : 0;
      len[u] = w0 + lane + u * gs < c ? bcnt[b] - bs[u] : 0;
      if (!HS_G(dbg, bs[u] >= 0 && bs[u] + len[u] <= c, 24, bs[u])) len[u] = 0;
      rank[u] = bs[u];
      most = max(most, len[u]);
    }
    // every lane as many steps as the warp's largest bucket asks for: loops of
    // their own lengths left the lanes one behind the other
    most = warp_max(most);
    for (int t = 0; t < most; ++t) {
#pragma unroll
      for (int u = 0; u < EU; ++u) {
        const int k = t < len[u] ? sk[bs[u] + t] : 0x7fffffff;
        rank[u] += k < key[u] || (DUPS && k == key[u] && bs[u] + t < w0 + lane + u * gs);
      }
    }
#pragma unroll
    for (int u = 0; u < EU; ++u) {
      if (len[u] > 0) {
        out(rank[u], key[u], v[u]);
      }
    }
  }
  return true;
}

template <class G, typename T, bool HAS_VAL>
__device__ void group_sort_emit(const int *keys, const T *vals, int slots, int c, int *ck, T *cv,
                                void *work, int *wtmp, EmitScratch *es, int32_t *out_j, T *out_v,
                                int *err, int cap, long long *dbg, bool unsorted = false) {
  const int gs = G::size(), r = G::rank(), lane = lane_id();
  if (!HS_G(dbg, c >= 0 && c <= cap, 20, c)) {
    if (r == 0) atomicExch(err, 8);
    return;
  }
  if (r == 0) {
    es->kmin = 0x7fffffff;
    es->kmax = -1;
    es->count = 0;
  }
  G::sync();
  // (1) compaction: each warp counts its run of slots, reserves room once,
  // then copies the run's entries in order
  {
    const int nw = G::nwarps(), w = G::warp();
    const int per = ((slots + nw - 1) / nw + 31) & ~31;
    const int s0 = min(slots, w * per), s1 = min(slots, s0 + per);
    constexpr int CU = 4;  // slots per lane per step: their reads overlap
    int n = 0;
    for (int sb = s0; sb < s1; sb += 32 * CU) {
      int k[CU];
#pragma unroll
      for (int u = 0; u < CU; ++u) k[u] = sb + 32 * u + lane < s1 ? keys[sb + 32 * u + lane] : EMPTY;
#pragma unroll
      for (int u = 0; u < CU; ++u) n += k[u] != EMPTY;
    }
    n = warp_sum(n);
    int base = 0;
    if (lane == 0 && n) base = atomicAdd(&es->count, n);
    base = __shfl_sync(FULL, base, 0);
    int lmin = 0x7fffffff, lmax = -1;
    for (int sb = s0; sb < s1; sb += 32 * CU) {
      int k[CU];
#pragma unroll
      for (int u = 0; u < CU; ++u) k[u] = sb + 32 * u + lane < s1 ? keys[sb + 32 * u + lane] : EMPTY;
#pragma unroll
      for (int u = 0; u < CU; ++u) {
        const bool occ = k[u] != EMPTY;
        const unsigned m = __ballot_sync(FULL, occ);
        if (occ) {
          const int at = base + __popc(m & ((1u << lane) - 1));
          if (at < c) {
            ck[at] = k[u];
            if constexpr (HAS_VAL) cv[at] = vals[sb + 32 * u + lane];
          }
          lmin = min(lmin, k[u]);
          lmax = max(lmax, k[u]);
        }
        base += __popc(m);
      }
    }
    lmin = warp_min(lmin);
    lmax = warp_max(lmax);
    if (lane == 0) {
      atomicMin(&es->kmin, lmin);
      atomicMax(&es->kmax, lmax);
    }
  }
  G::sync();
  if (es->count != c) {  // structure disagrees with the symbolic count
    if (r == 0) atomicExch(err, 1);
    return;
  }
  if (c == 0) return;
  if (unsorted) {  // the caller takes the row in table order
    for (int e = r; e < c; e += gs) {
      __stcs(out_j + e, ck[e]);
      if constexpr (HAS_VAL) __stcs(out_v + e, cv[e]);
    }
    return;
  }
  group_bucket_sort<G, T, HAS_VAL, false>(ck, cv, c, es->kmin, es->kmax, work, wtmp, dbg, [&](int at, int k, T v) {
    __stcs(out_j + at, k);
    if constexpr (HAS_VAL) __stcs(out_v + at, v);
  });
  G::sync();
}

}  // namespace hs
