// spgemm.cu -- host driver and C ABI (include/hspgemm.h).
//
// hs_spgemm runs the phases of the row-wise SpGEMM on one stream:
//   1. flops per row and binning of the non-empty rows by flops
//      (one device->host read: bin sizes, total flops, validation flags);
//   2. symbolic pass per bin: output nonzeros per row;
//   3. inclusive scan of the counts into C's row offsets, binning of the rows
//      again by (flops, output count) for the numeric pass
//      (second device->host read: nnz(C) and the bin sizes);
//   4. allocation of C's column ids and values, numeric pass per bin.
// hs_spref and hs_spasgn build their 0/1 selection matrices on the device and
// call the same driver with the selector semirings (Section 3.1).
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/hspgemm.h"
#include "fan.h"
#include "internal.h"

namespace hs {

static thread_local int t_last_cuda = 0;
static thread_local char t_detail[256] = "";

// Checking mode: HS_DEBUG_SYNC=1 in the environment synchronises after every
// phase, so a CUDA error or a failed index check is attributed to the phase
// that raised it.  Without it, failed checks are reported at the product's
// second host synchronisation (or at the end with HS_FLAG_VALIDATE).
static bool debug_sync() {
  static int v = -1;
  if (v < 0) {
    const char *e = getenv("HS_DEBUG_SYNC");
    v = (e && *e && *e != '0') ? 1 : 0;
  }
  return v == 1;
}

// ---------------------------------------------------------------- profiling
struct Prof {
  std::mutex mu;
  bool on = false;
  std::vector<std::string> names;
  std::vector<double> ms;
  std::vector<int64_t> launches;
  struct Pending {
    int phase;
    cudaEvent_t a, b;
  };
  std::vector<Pending> pending;
  int phase_id(const char *nm) {
    for (size_t i = 0; i < names.size(); ++i)
      if (names[i] == nm) return (int)i;
    names.push_back(nm);
    ms.push_back(0);
    launches.push_back(0);
    return (int)names.size() - 1;
  }
  void drain() {
    for (auto &p : pending) {
      cudaEventSynchronize(p.b);
      float t = 0;
      cudaEventElapsedTime(&t, p.a, p.b);
      ms[p.phase] += t;
      launches[p.phase] += 1;
      cudaEventDestroy(p.a);
      cudaEventDestroy(p.b);
    }
    pending.clear();
  }
};
static Prof g_prof;

struct PhaseTimer {
  cudaEvent_t a = nullptr, b = nullptr;
  int phase = -1;
  cudaStream_t st;
  PhaseTimer(const char *nm, cudaStream_t s, bool active = true) : st(s) {
    if (!g_prof.on || !active) return;
    std::lock_guard<std::mutex> g(g_prof.mu);
    phase = g_prof.phase_id(nm);
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, st);
  }
  ~PhaseTimer() {
    if (phase < 0) return;
    cudaEventRecord(b, st);
    std::lock_guard<std::mutex> g(g_prof.mu);
    g_prof.pending.push_back({phase, a, b});
  }
};

// --------------------------------------------------------------- allocation
struct Mem {
  const hs_allocator *al;
  cudaStream_t st;
  cudaMemPool_t pool = nullptr;  // without an allocator: this pool if set, else the device's default pool
  struct Blk {
    void *p;
    size_t n;
  };
  std::vector<Blk> scratch;
  bool failed = false;
  // temporaries of at most SMALL bytes are cut from blocks of CHUNK bytes: a
  // call of the caller's allocator costs some 5 us, and a small operation
  // would make a dozen of them for a few KB each
  static constexpr size_t SMALL = 256 << 10, CHUNK = 1 << 20;
  char *chunk = nullptr;
  size_t chunk_left = 0;

  void *raw(size_t bytes) {
    if (bytes == 0) bytes = 16;
    void *p = nullptr;
    if (al && al->alloc) {
      p = al->alloc(bytes, (void *)st, al->ctx);
    } else if ((pool ? cudaMallocFromPoolAsync(&p, bytes, pool, st) : cudaMallocAsync(&p, bytes, st)) !=
               cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    if (!p) failed = true;
    return p;
  }
  void release(void *p, size_t bytes) {
    if (!p) return;
    if (bytes == 0) bytes = 16;
    if (al && al->free) al->free(p, bytes, (void *)st, al->ctx);
    else if (!al || !al->alloc) cudaFreeAsync(p, st);
  }
  template <typename T> T *tmp(size_t count) {
    const size_t bytes = sizeof(T) * count;
    if (bytes <= SMALL) {
      const size_t room = ((bytes ? bytes : 1) + 255) & ~(size_t)255;
      if (room > chunk_left) {
        chunk_left = 0;
        const bool before = failed;
        chunk = (char *)raw(CHUNK);
        if (!chunk) {  // an allocator of small blocks, or too little memory left: the block alone
          failed = before;
          T *p = (T *)raw(bytes);
          if (p) scratch.push_back({p, bytes});
          return p;
        }
        scratch.push_back({chunk, CHUNK});
        chunk_left = CHUNK;
      }
      T *p = (T *)chunk;
      chunk += room;
      chunk_left -= room;
      return p;
    }
    T *p = (T *)raw(bytes);
    if (p) scratch.push_back({p, bytes});
    return p;
  }
  // the temporaries taken since scratch.size() was n
  void release_from(size_t n) {
    for (size_t i = n; i < scratch.size(); ++i) release(scratch[i].p, scratch[i].n);
    scratch.resize(n);
    chunk_left = 0;  // (the shared block may be one of them)
  }
  ~Mem() { release_from(0); }
};

// A pool of the library's own for calls that allocate and free the same large
// blocks many times (hs_spgemm_to_host): it keeps freed memory mapped for the
// next block and the next call (hs_trim_memory returns it) instead of giving
// it back at every synchronisation.
static cudaMemPool_t own_pool() {
  static std::mutex mu;
  static cudaMemPool_t pools[64] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> g(mu);
  if (!pools[dev]) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    if (cudaMemPoolCreate(&pools[dev], &props) != cudaSuccess) {
      cudaGetLastError();
      pools[dev] = nullptr;
      return nullptr;
    }
    uint64_t keep = ~0ull;
    cudaMemPoolSetAttribute(pools[dev], cudaMemPoolAttrReleaseThreshold, &keep);
    cudaGetLastError();
  }
  return pools[dev];
}

static int vbytes_of(int dt) {
  switch (dt) {
    case HS_F64: case HS_I64: return 8;
    case HS_F32: case HS_I32: return 4;
    default: return 0;
  }
}

// pinned staging for the small device->host reads: one 8 KB page-locked
// buffer per thread, shared by every call on that thread.  A caller reads
// what it copied there before it calls another operation's implementation
// (SpAsgn runs two products, SpRef may build Q with sparse()), and copies
// into it again afterwards.
struct Pinned {
  void *p = nullptr;
  ~Pinned() {
    if (p) cudaFreeHost(p);
  }
};
static thread_local Pinned t_pin;
static void *pinned(size_t bytes) {
  if (!t_pin.p && cudaMallocHost(&t_pin.p, 8192) != cudaSuccess) {
    t_pin.p = nullptr;
    return nullptr;
  }
  return bytes <= 8192 ? t_pin.p : nullptr;
}

// the runtime as fan.h wants it: a failed call leaves no error behind
struct FanCuda {
  using Stream = cudaStream_t;
  using Event = cudaEvent_t;
  struct Capture {
    bool active;
    unsigned long long id;
  };
  static bool good(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
  }
  static bool device(int *d) { return good(cudaGetDevice(d)); }
  static bool priority(Stream s, int *p) { return good(cudaStreamGetPriority(s, p)); }
  static bool capture(Stream s, Capture *c) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    c->id = 0;
    if (!good(cudaStreamGetCaptureInfo(s, &st, &c->id)) || st == cudaStreamCaptureStatusInvalidated) return false;
    c->active = st == cudaStreamCaptureStatusActive;
    return true;
  }
  static bool create(Event *e) { return good(cudaEventCreateWithFlags(e, cudaEventDisableTiming)); }
  static bool create(Stream *s, int priority) {
    return good(cudaStreamCreateWithPriority(s, cudaStreamNonBlocking, priority));
  }
  static void destroy(Event e) { good(cudaEventDestroy(e)); }
  static void destroy(Stream s) { good(cudaStreamDestroy(s)); }
  static bool record(Event e, Stream s) { return good(cudaEventRecord(e, s)); }
  static bool wait(Stream s, Event e) { return good(cudaStreamWaitEvent(s, e, 0)); }
  static void synchronize(Stream s) { good(cudaStreamSynchronize(s)); }
};
using Fan = FanOf<FanCuda>;
static thread_local SidePool<FanCuda> t_sides;

// The bins of a pass over four streams: the caller's (group 0) and three
// beside it.  Bins of one pass work on different rows, and the larger ones end
// in tails of a few blocks (a row of very many entries or products), which the
// others fill (a contraction's two products 2.44 -> 1.76 ms, a narrow frontier
// product 1.43 -> 0.93 ms, a batch of random products 6.44 -> 6.15 ms).  In a
// product of more than FAN_PRODUCTS products the tails are nothing and the
// bins only take each other's cache (6.0e9 products: 72.4 against 72.2 ms;
// 6e8: 4.6 against 4.8 ms): its bins run one by one.
constexpr unsigned long long FAN_PRODUCTS = 1ull << 31;
// numeric kinds: heavy rows, large, mid, and the rows of a warp
static int num_group(int kind) { return kind == NUM_KINDS - 1 ? 1 : kind == 5 || kind == 6 ? 2 : kind == 3 || kind == 4 ? 3 : 0; }

#define CK(call)                          \
  do {                                    \
    cudaError_t e_ = (call);              \
    if (e_ != cudaSuccess) {              \
      t_last_cuda = (int)e_;              \
      cudaGetLastError();                 \
      return HS_ECUDA;                    \
    }                                     \
  } while (0)

static int check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && attr_error() != cudaSuccess) {
    e = attr_error();
    attr_error() = cudaSuccess;
  }
  if (e != cudaSuccess) {
    t_last_cuda = (int)e;
    snprintf(t_detail, sizeof(t_detail), "%s (%d)", cudaGetErrorName(e), (int)e);
    return HS_ECUDA;
  }
  return HS_OK;
}

struct SmallBlock;
static int phase_check(const char *phase, cudaStream_t st, const long long *dbg_dev);

static bool dtype_ok(int dt) { return dt >= HS_F64 && dt <= HS_BOOL; }

static void free_mat(hs_mat *M, Mem &mem) {
  if (!M) return;
  const int64_t rows = M->m;
  mem.release(M->ptr, sizeof(int64_t) * (size_t)(rows + 1));
  mem.release(M->idx, sizeof(int32_t) * (size_t)M->nnz);
  if (M->val) mem.release(M->val, (size_t)vbytes_of(M->dtype) * (size_t)M->nnz);
  memset(M, 0, sizeof(*M));
}

// ----------------------------------------------------------------- SpGEMM
struct SmallBlock {  // device counters, read back in one copy
  int key_cnt[2][NKEYS];  // symbolic, numeric
  int key_off[NKEYS + 1];
  int key_cur[NKEYS];
  int dyn[3];  // symbolic heavy rows, numeric heavy rows, numeric heavy units
  int nhist;
  int err;
  int valflag;
  int ticket[2];
  int pad;
  unsigned long long stats[5];
  unsigned long long lpool;  // heavy rows' column lists: pool entries handed out
  int bci_cnt;               // B segment index rows handed out
  int pad2;
  HubRows hub;
  long long nunits;          // numeric heavy units (column parts of rows with lists)
  long long npcap;           // their room in the pair arrays
  long long nnz;
  unsigned long long zeros;  // A entries whose B row is empty
  long long dbg[2];  // guarded builds: first failed check (code, index)
};

static int phase_check(const char *phase, cudaStream_t st, const long long *dbg_dev) {
  if (int e = check_launch()) {
    char tmp[sizeof(t_detail) + 64];
    snprintf(tmp, sizeof(tmp), "%.48s: %s", phase, t_detail);
    snprintf(t_detail, sizeof(t_detail), "%.*s", (int)sizeof(t_detail) - 1, tmp);
    return e;
  }
  if (!debug_sync()) return HS_OK;
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    t_last_cuda = (int)e;
    snprintf(t_detail, sizeof(t_detail), "%s: %s (%d)", phase, cudaGetErrorName(e), (int)e);
    cudaGetLastError();
    return HS_ECUDA;
  }
  if (dbg_dev) {
    long long d[2] = {0, 0};
    cudaMemcpy(d, dbg_dev, sizeof(d), cudaMemcpyDeviceToHost);
    if (d[0]) {
      snprintf(t_detail, sizeof(t_detail), "%s: guard %lld failed at index %lld", phase, d[0], d[1]);
      return HS_EINTERNAL;
    }
  }
  return HS_OK;
}

static bool numeric_supported(int sr, int adt, int bdt, int &out_dt) {
  switch (sr) {
    case HS_PLUS_TIMES:
      out_dt = adt;
      return adt == bdt && (adt == HS_F64 || adt == HS_F32 || adt == HS_I64);
    case HS_MIN_PLUS:
      out_dt = adt;
      return adt == bdt && (adt == HS_F32 || adt == HS_I32);
    case HS_OR_AND:
      out_dt = HS_BOOL;
      return true;
    case HS_SELECT2ND:
      out_dt = bdt;
      return true;
    case HS_SELECT1ST:
      out_dt = adt;
      return true;
  }
  return false;
}



// ----------------------------------------------------------------- tuning
static std::mutex g_tune_mu;
static const hs_tuning k_tune_default = {F_WARP_S, CAP_MID_S, 4096, F_MID_S, 0, F_SORT, 50, 0, 16, 0};
static hs_tuning g_tune = k_tune_default;

static int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

BinCfg bin_config(int value_bytes) {
  hs_tuning t;
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    t = g_tune;
  }
  BinCfg b;
  b.cap_large = value_bytes == 8 ? 4096 : 8192;
  b.warp_s_max = clampi(t.warp_s_max, F_TINY, F_WARP_S);
  b.mid_s_max = clampi(t.mid_s_max, 0, CAP_MID_S);
  b.large_s_max = clampi(t.large_s_max, CAP_MID, b.cap_large / 2 > CAP_MID ? b.cap_large / 2 : CAP_MID);
  b.sym_mid_s_max = clampi(t.sym_mid_s_max, F_WARP, F_MID_S);
  // 0: automatic.  With 4-byte values and bool, rows of more than 4096
  // products take the bitmap kernel and rows of more than 2048 outputs among
  // them the units (R-MAT scale 20: 77.8 ms against 79.0 ms with both at the
  // large capacity); 8-byte values keep the large capacity
  const bool narrow = value_bytes <= 4;
  b.sym_heavy_from = t.sym_heavy_from <= 0 ? (narrow ? F_MID : b.cap_large) : clampi(t.sym_heavy_from, 2 * F_MID_S, b.cap_large);
  b.sort_max = clampi(t.sort_max, F_TINY, F_SORT);
  b.sort_pct = clampi(t.sort_pct, 0, 101);
  b.spa_max = clampi(t.spa_max, 0, SPA_COLS_4);
  b.unit_kb = t.heavy_part_kb >= 32 ? 32 : 16;
  b.num_heavy_from =
      t.num_heavy_from <= 0 ? (narrow ? CAP_MID : b.cap_large) : clampi(t.num_heavy_from, CAP_MID, b.cap_large);
  b.spa = 0;
  return b;
}

static bool launch_num(int sr, int out_dt, int kind, const NumArgs &a, cudaStream_t st) {
  switch (sr) {
    case HS_PLUS_TIMES: return launch_numeric_pt(out_dt, kind, a, st);
    case HS_MIN_PLUS: return launch_numeric_mp(out_dt, kind, a, st);
    case HS_OR_AND: return launch_numeric_oa(kind, a, st);
    case HS_SELECT2ND: return launch_numeric_sel(1, vbytes_of(out_dt), kind, a, st);
    case HS_SELECT1ST: return launch_numeric_sel(0, vbytes_of(out_dt), kind, a, st);
  }
  return false;
}

}  // namespace hs

// A product's numeric pass, kept for re-execution (hs_plan_*): the numeric
// arguments with every scratch buffer, the row bins, and the buffers' owner.
struct hs_plan {
  int sr = 0, out_dt = 0;
  int64_t a_nnz = 0, b_nnz = 0, c_nnz = 0;
  hs::NumArgs na{};
  const int *list = nullptr;
  int off[hs::NUM_KINDS] = {0}, count[hs::NUM_KINDS] = {0};
  int *dyn = nullptr, *err = nullptr;
  long long *dbg = nullptr;
  hs_allocator al{};
  bool has_al = false;
  bool side_by_side = false;  // the bins run beside each other (hs::Fan)
  unsigned groups() const {
    unsigned g = 0;
    for (int kind = 0; kind < hs::NUM_KINDS; ++kind)
      if (side_by_side && count[kind] > 0) g |= 1u << hs::num_group(kind);
    return g;
  }
  // streams of the plan's own, so that plans on different streams of a thread
  // stay independent and an execution makes none (it may be captured)
  std::unique_ptr<hs::SideSet<hs::FanCuda>> sides;
  std::vector<hs::Mem::Blk> blocks;
};

namespace hs {

// Where C's column ids and values go when the caller places them (device
// pointers to memory of at least cap entries, e.g. host memory the GPU maps).
struct OutPlace {
  int32_t *idx;
  void *val;
  int64_t cap;
};

static int spgemm_impl(int sr, const hs_mat *A, const hs_mat *B, hs_mat *C, Mem &mem, Mem &outmem,
                       uint32_t flags, hs_plan *plan = nullptr, const OutPlace *place = nullptr) {
  cudaStream_t st = mem.st;
  if (!A || !B || !C) return HS_EINVAL;
  if (A->fmt != HS_CSR && A->fmt != HS_DCSR) return HS_EINVAL;
  if (B->fmt != HS_CSR) return HS_EINVAL;
  if (!dtype_ok(A->dtype) || !dtype_ok(B->dtype)) return HS_EINVAL;
  if (A->n != B->m || A->m < 0 || B->n < 0 || A->nnz < 0 || B->nnz < 0) return HS_EINVAL;
  if (B->n > 0x7fffffffLL || A->n > 0x7fffffffLL) return HS_EINVAL;
  int out_dt = 0;
  if (!numeric_supported(sr, A->dtype, B->dtype, out_dt)) return HS_EINVAL;
  const int vb = vbytes_of(out_dt);
  if ((sr == HS_PLUS_TIMES || sr == HS_MIN_PLUS) && ((A->nnz && !A->val) || (B->nnz && !B->val))) return HS_EINVAL;
  if (sr == HS_SELECT2ND && vb && B->nnz && !B->val) return HS_EINVAL;
  if (sr == HS_SELECT1ST && vb && A->nnz && !A->val) return HS_EINVAL;
  const int64_t m = A->m, n = B->n;
  const int64_t nslots = A->fmt == HS_DCSR ? A->nzr : A->m;
  if (nslots < 0 || (A->fmt == HS_DCSR && nslots > 0 && !A->ids)) return HS_EINVAL;
  if ((nslots > 0 && !A->ptr) || (B->m >= 0 && !B->ptr && B->m > 0)) return HS_EINVAL;
  if ((A->nnz > 0 && !A->idx) || (B->nnz > 0 && !B->idx)) return HS_EINVAL;
  if (nslots > 0x7fffffffLL) return HS_EUNSUPPORTED;

  memset(C, 0, sizeof(*C));
  C->fmt = HS_CSR;
  C->dtype = out_dt;
  C->m = m;
  C->n = n;
  int64_t *Cp = (int64_t *)outmem.raw(sizeof(int64_t) * (size_t)(m + 1));
  if (!Cp) return HS_ENOMEM;
  C->ptr = Cp;
  const bool none = nslots == 0 || A->nnz == 0 || B->nnz == 0 || n == 0;
  if (none || A->fmt == HS_DCSR)  // (a CSR product's counts are cleared as its rows are binned)
    CK(cudaMemsetAsync(Cp, 0, sizeof(int64_t) * (size_t)(m + 1), st));
  if (plan) {
    plan->sr = sr;
    plan->out_dt = out_dt;
    plan->a_nnz = A->nnz;
    plan->b_nnz = B->nnz;
  }
  if (none) {
    if (place) {  // nothing to write
      C->idx = place->idx;
      C->val = place->val;
      return check_launch();
    }
    C->idx = (int32_t *)outmem.raw(4);
    if (!C->idx) return HS_ENOMEM;
    if (vb) {  // typed outputs always carry a (here empty) value array
      C->val = outmem.raw((size_t)vb);
      if (!C->val) return HS_ENOMEM;
    }
    return check_launch();
  }

  const BinCfg bins = product_bins(bin_config(vb), n, vb);
  // the counters and, behind them, the rows' product counts: cleared together
  const size_t sb_bytes = (sizeof(SmallBlock) + 15) & ~(size_t)15;
  char *zeroed = mem.tmp<char>(sb_bytes + sizeof(int64_t) * (size_t)nslots);
  SmallBlock *sb = (SmallBlock *)zeroed;
  int64_t *f = zeroed ? (int64_t *)(zeroed + sb_bytes) : nullptr;
  int *list = mem.tmp<int>(nslots);
  int32_t *hslot = mem.tmp<int32_t>(nslots);
  int64_t *scan_tmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(m > nslots ? m : nslots));
  if (mem.failed) return HS_ENOMEM;
  RowSet rs{A->ptr, A->idx, A->val, A->fmt == HS_DCSR ? A->ids : nullptr, nslots, A->nnz, m, sb->dbg};
  RightOp rb{B->ptr, B->idx, B->val, n, B->m, B->nnz, sb->dbg};
  SmallBlock *hb = (SmallBlock *)pinned(sizeof(SmallBlock));
  if (!hb) return HS_ECUDA;
  CK(cudaMemsetAsync(zeroed, 0, sb_bytes + sizeof(int64_t) * (size_t)nslots, st));
  const BinCounters sym_c{sb->key_cnt[0], sb->key_off, sb->key_cur, &sb->ticket[0], nullptr};
  const BinCounters num_c{sb->key_cnt[1], sb->key_off, sb->key_cur, &sb->ticket[1], &sb->hub};
  {
    PhaseTimer t("analysis", st);
    if (flags & HS_FLAG_VALIDATE) {
      launch_validate(A->ptr, A->idx, nslots, A->n, &sb->valflag, st);
      launch_validate(B->ptr, B->idx, B->m, B->n, &sb->valflag, st);
    }
    launch_flops(rs, rb, f, &sb->zeros, st);
    launch_row_keys(rs, f, rs.ids ? nullptr : Cp, sym_c, sb->stats, bins, n, st);
    launch_scatter_sym(rs, f, sb->key_cur, list, hslot, &sb->nhist, bins, st);
  }
  if (int e = phase_check("analysis", st, sb->dbg)) return e;
  CK(cudaMemcpyAsync(hb, sb, sizeof(SmallBlock), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (hb->valflag & 4) return HS_EINVAL;
  if (hb->valflag & 1) return HS_EINVAL;
  if (hb->valflag & 2) return HS_ENONCANON;
  if (hb->stats[1] >= (1ull << 31)) return HS_EUNSUPPORTED;  // one row's products must fit int32
  int key_off[NKEYS + 1];
  memcpy(key_off, hb->key_off, sizeof(key_off));
  const int nhist = hb->nhist;
  const int tiny_group = tiny_group_pays(key_off[KEY_TINY + 1] - key_off[KEY_TINY], hb->stats[4]);
  const bool side_by_side = hb->stats[0] <= FAN_PRODUCTS;
  SideSet<FanCuda> *sides = nullptr;
  auto sides_for = [&](unsigned groups) {
    if (!sides && (groups & (groups - 1))) sides = t_sides.of(st);
    return sides;
  };
  const int64_t longest = (int64_t)hb->stats[2];  // (read before hb is copied to again)
  const int nseg = (int)((n + SEG_W - 1) / SEG_W);

  // A entries whose B row is empty make no products.  When they are most of
  // a large A (a very sparse B, as in the tall-skinny products of Section 4),
  // the passes below read a copy of A without them: rows keep their product
  // counts, bins and results, and a long row of A with few products no longer
  // costs a walk over all its entries.  Not for plans, whose execute reads A's
  // values in place.
  if (!plan && A->nnz >= (1 << 20) && hb->zeros * 2 > (unsigned long long)A->nnz) {
    const int64_t kept = A->nnz - (int64_t)hb->zeros;
    const int va = A->val ? vbytes_of(A->dtype) : 0;
    int64_t *keep = mem.tmp<int64_t>((size_t)A->nnz);
    int32_t *j2 = mem.tmp<int32_t>((size_t)(kept > 0 ? kept : 1));
    void *v2 = va ? (void *)mem.tmp<char>((size_t)va * (size_t)(kept > 0 ? kept : 1)) : nullptr;
    int64_t *p2 = mem.tmp<int64_t>((size_t)nslots + 1);
    int64_t *ktmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(A->nnz));
    if (!mem.failed) {
      PhaseTimer t("compact_a", st);
      launch_compact_a(rs, rb, keep, ktmp, j2, v2, va, p2, st);
      rs.p = p2;
      rs.j = j2;
      rs.v = v2;
      rs.nnz = kept;
      if (int e = phase_check("compact_a", st, sb->dbg)) return e;
    }
    mem.failed = false;
  }

  uint32_t *hist = nullptr;
  if (nhist > 0) {
    hist = mem.tmp<uint32_t>((size_t)nhist * nseg);
    if (!hist) return HS_ENOMEM;
    CK(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * (size_t)nhist * nseg, st));
  }

  // the symbolic heavy rows write their sorted column lists for the numeric
  // pass into a pool of sum(min(f, n)) entries, as much of it as fits a
  // quarter of the free device memory (at most 32 GiB); rows that find no
  // room are left to the numeric pass's own bitmap build
  int32_t *glist = nullptr;
  int64_t *loff = nullptr;
  int64_t lcap = 0;
  {
    const int64_t nsh = key_off[NKEYS] - key_off[KEY_HEAVY];
    size_t free_b = 0, total_b = 0;
    if (nsh > 0 && hb->stats[3] > 0 && cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) {
      const size_t budget = free_b / 4 < ((size_t)32 << 30) ? free_b / 4 : ((size_t)32 << 30);
      const size_t want = (size_t)hb->stats[3] * 4;
      const size_t bytes = want < budget ? want : budget;
      if (bytes >= 4) {
        // (16 bytes of slack: the numeric units copy their slices in 16-byte pieces)
        glist = (int32_t *)mem.raw(bytes + 16);
        loff = glist ? (int64_t *)mem.raw(sizeof(int64_t) * (size_t)nslots) : nullptr;
        if (glist) mem.scratch.push_back({glist, bytes + 16});
        if (loff) mem.scratch.push_back({loff, sizeof(int64_t) * (size_t)nslots});
        mem.failed = false;  // optional buffers
        if (!loff) glist = nullptr;
        else {
          lcap = (int64_t)(bytes / 4);
          CK(cudaMemsetAsync(loff, 0xff, sizeof(int64_t) * (size_t)nslots, st));
        }
      }
    }
    cudaGetLastError();
  }

  // the B segment index: for every B row longer than min_len, the offset of
  // its first entry in each SEG_W-column segment (the table kept within an
  // eighth of the free memory, at most 4 GiB): its room is taken here, the
  // numeric pass fills it
  int32_t *bci_id = nullptr, *bci = nullptr;
  int64_t bci_min_len = 32, bci_rows = 0;
  auto alloc_bci = [&]() {
    if (B->nnz <= 0) return;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) {
      const size_t budget = free_b / 8 < ((size_t)4 << 30) ? free_b / 8 : ((size_t)4 << 30);
      const int64_t row_bytes = ((int64_t)nseg + 1) * 4;
      const int64_t need = (B->nnz * row_bytes + (int64_t)budget - 1) / (int64_t)(budget ? budget : 1);
      if (need > bci_min_len) bci_min_len = need;
      bci_rows = B->nnz / (bci_min_len + 1);
      if (bci_rows > (int64_t)(budget / row_bytes)) bci_rows = (int64_t)(budget / row_bytes);
      if (bci_rows > 0 && bci_min_len < 0x7fffffff) {
        bci_id = (int32_t *)mem.raw(sizeof(int32_t) * (size_t)B->m);
        bci = bci_id ? (int32_t *)mem.raw((size_t)bci_rows * (size_t)row_bytes) : nullptr;
        if (bci_id) mem.scratch.push_back({bci_id, sizeof(int32_t) * (size_t)B->m});
        if (bci) mem.scratch.push_back({bci, (size_t)bci_rows * (size_t)row_bytes});
        mem.failed = false;  // optional: without it the part ends are searched
        if (!bci) bci_id = nullptr;
      }
    }
    cudaGetLastError();
  };

  // ---- symbolic
  // Rows whose values will be added up by units, and with an output for every
  // second bitmap word or more, leave the bitmap: writing and reading 128 KB
  // (2^20 columns) costs no more bytes than the list of 16,384 outputs or
  // more, the units need the bits anyway, and the columns are walked out of
  // them where five CTAs share an SM instead of one (R-MAT scale 20: the
  // symbolic rows 23.7 -> 20.4 ms, the units 32.5 -> 33.6 ms; twice or a third of
  // this line measured the same).  Without values
  // the units only copy the list.
  const int64_t half_words = (n + 63) / 64;
  const int64_t bits_min = !vb ? INT64_MAX
                               : (half_words > bins.num_heavy_from + 1 ? half_words : (int64_t)bins.num_heavy_from + 1);
  SymArgs sa{rs, rb, f, nullptr, 0, Cp, hslot, hist, nseg, &sb->dyn[0], &sb->err, glist, loff, &sb->lpool, lcap, tiny_group,
             bits_min};
  {
    struct SymBin {
      const char *name;
      int k0, k1, group;
      void (*launch)(const SymArgs &, cudaStream_t);
    };
    // the longest first; the rows of a warp stay on the caller's stream
    const SymBin bins_[] = {{"symbolic_heavy", KEY_HEAVY, NKEYS, 1, launch_sym_heavy},
                            {"symbolic_large", KEY_LARGE, KEY_LARGE + 1, 2, launch_sym_large},
                            {"symbolic_mid", KEY_MID, KEY_MID + 1, 2, launch_sym_mid},
                            {"symbolic_mid_s", KEY_MID_S, KEY_MID_S + 1, 3, launch_sym_mid_s},
                            {"symbolic_tiny", KEY_TINY, KEY_TINY + 1, 0, launch_sym_tiny},
                            {"symbolic_warp", KEY_WARP, KEY_WARP + 1, 0, launch_sym_warp},
                            {"symbolic_spa", KEY_SPA, KEY_SPA + 1, 0, launch_sym_spa}};
    unsigned groups = 0;
    for (const SymBin &x : bins_)
      if (side_by_side && key_off[x.k1] > key_off[x.k0]) groups |= 1u << x.group;
    PhaseTimer t("symbolic", st);
    Fan fan(st, groups, sides_for(groups), true);
    for (const SymBin &x : bins_) {
      sa.list = list + key_off[x.k0];
      sa.count = key_off[x.k1] - key_off[x.k0];
      if (sa.count <= 0) continue;
      const cudaStream_t bst = fan.stream(x.group);
      {
        PhaseTimer t2(x.name, bst);
        x.launch(sa, bst);
      }
      if (int e = phase_check(x.name, bst, sb->dbg)) return e;
    }
    if (!fan.join()) return HS_ECUDA;
  }

  // ---- offsets and numeric bins
  {
    PhaseTimer t("scan_bin", st);
    launch_num_bins(rs, f, Cp, numeric_bins(bins, n), num_c, scan_tmp, &sb->nnz, list, st);
  }
  // numeric heavy rows that have a sorted column list run as units (column
  // parts spread over the SMs): their parts are counted now, so that the
  // number of units comes back with nnz(C); the numeric heavy rows are a
  // subset of the symbolic heavy rows, whose number bounds the count array
  int64_t *pcnt = nullptr, *pcap = nullptr;
  const int64_t nsh_rows = key_off[NKEYS] - key_off[KEY_HEAVY];
  const int ucap = unit_part_cap(vb, bins.unit_kb);
  if (glist && nsh_rows > 0) {
    pcnt = mem.tmp<int64_t>((size_t)nsh_rows);
    pcap = pcnt ? mem.tmp<int64_t>((size_t)nsh_rows) : nullptr;
    int64_t *ptmp = pcap ? mem.tmp<int64_t>((size_t)scan_tmp_elems(nsh_rows)) : nullptr;
    mem.failed = false;  // optional: without units the heavy rows run one CTA per row
    if (!ptmp) pcnt = nullptr;
    if (pcnt) {
      PhaseTimer t("scan_bin", st);
      launch_count_parts(rs, list, sb->key_off, KEY_HEAVY, hslot, hist, loff, nseg, ucap, HU_SPAN_SEGS, nsh_rows,
                         pcnt, pcap, st);
      launch_scan_i64(pcnt, nsh_rows, ptmp, st);
      launch_scan_i64(pcap, nsh_rows, ptmp, st);
      CK(cudaMemcpyAsync(&sb->nunits, pcnt + nsh_rows - 1, sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
      CK(cudaMemcpyAsync(&sb->npcap, pcap + nsh_rows - 1, sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
    }
    cudaGetLastError();
  }

  if (int e = phase_check("scan_bin", st, sb->dbg)) return e;
  CK(cudaMemcpyAsync(hb, sb, sizeof(SmallBlock), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (hb->dbg[0]) {
    snprintf(t_detail, sizeof(t_detail), "index check %lld failed at %lld", hb->dbg[0], hb->dbg[1]);
    return HS_EINTERNAL;
  }
  if (hb->err) {
    snprintf(t_detail, sizeof(t_detail), "device consistency check %d", hb->err);
    return HS_EINTERNAL;
  }
  const int64_t nnz = hb->nnz;
  memcpy(key_off, hb->key_off, sizeof(key_off));
  C->nnz = nnz;
  if (place) {
    if (nnz > place->cap) return HS_ECAPACITY;
    C->idx = place->idx;
    C->val = vb ? place->val : nullptr;
  } else {
    C->idx = (int32_t *)outmem.raw(sizeof(int32_t) * (size_t)nnz);
    if (!C->idx) return HS_ENOMEM;
    if (vb) {
      C->val = outmem.raw((size_t)vb * (size_t)nnz);
      if (!C->val) return HS_ENOMEM;
    }
  }

  // ---- numeric
  // heavy bin: units, planned from the segment counts of the rows with lists
  // and, for semirings with values, each unit's B segments (place and left
  // value) laid out by launch_build_pairs once the segment index exists (below)
  HeavyUnit *units = nullptr;
  int64_t *pseg = nullptr;
  void *paval = nullptr;
  const int64_t nunits = pcnt ? hb->nunits : 0;
  const int64_t npcap = pcnt ? hb->npcap : 0;
  const int64_t pair_long = pair_long_from(nunits, npcap, longest);
  const int nheavy = key_off[NKEYS] - key_off[KEY_HEAVY];
  const int a_bytes = (sr == HS_PLUS_TIMES || sr == HS_MIN_PLUS || sr == HS_SELECT1ST) ? vb : 0;
  if (nheavy > 0 && nunits > 0) {
    units = mem.tmp<HeavyUnit>((size_t)nunits);
    if (units && vb) {  // 16 bytes of slack each: the units copy their slices in 16-byte pieces
      pseg = (int64_t *)mem.tmp<char>((size_t)npcap * 8 + 16);
      paval = a_bytes ? (void *)mem.tmp<char>((size_t)npcap * a_bytes + 16) : nullptr;
      if (!pseg || (a_bytes && !paval)) units = nullptr;
    }
    mem.failed = false;  // optional, as above
    if (units) {
      PhaseTimer t("scan_bin", st);
      launch_plan_parts(rs, list + key_off[KEY_HEAVY], nheavy, hslot, hist, loff, Cp, nseg, ucap, HU_SPAN_SEGS,
                        pcnt, pcap, units, st);
    }
    cudaGetLastError();
  }
  // rows that a unit does not cover (no list): one CTA per row, with
  // per-A-entry cursors into B rows (relative offsets)
  const bool lists_partial = lcap < (int64_t)hb->stats[3];
  int32_t *gcur = nullptr, *gend = nullptr;
  if (nheavy > 0 && (!units || lists_partial)) {
    gcur = mem.tmp<int32_t>((size_t)A->nnz);
    gend = mem.tmp<int32_t>((size_t)A->nnz);
    if (!gcur || !gend) return HS_ENOMEM;
  }
  unsigned groups = 0;
  for (int kind = 0; kind < NUM_KINDS; ++kind) {
    const int k0 = KEY_TINY + kind, k1 = kind == NUM_KINDS - 1 ? NKEYS : k0 + 1;
    if (side_by_side && key_off[k1] > key_off[k0]) groups |= 1u << num_group(kind);
  }
  if (nheavy > 0) alloc_bci();  // (every allocation before the streams part: they are ordered on the caller's)
  std::unique_ptr<PhaseTimer> t_num(new PhaseTimer("numeric", st));
  Fan fan(st, groups, sides_for(groups), true);
  // heavy bin: the B segment index, and the units' B segments
  const cudaStream_t hst = nheavy > 0 ? fan.stream(num_group(NUM_KINDS - 1)) : st;
  if (bci) {
    PhaseTimer t("bci", hst);
    launch_build_bci(rb, nseg, (int)bci_min_len, bci_rows, bci_id, bci, &sb->bci_cnt, hst);
    if (int e = phase_check("bci", hst, sb->dbg)) return e;
  }
  if (units && vb) {
    PhaseTimer t("heavy_pairs", hst);
    launch_build_pairs(rs, rb, units, nunits, bci_id, bci, nseg, a_bytes, pair_long, pseg, paval, hst);
    if (int e = phase_check("heavy_pairs", hst, sb->dbg)) return e;
  }
  NumArgs na{rs, rb,   f,    nullptr, 0,    Cp,    C->idx, C->val, hslot,
             hist, nseg, &sb->dyn[1], &sb->err, gcur, gend, glist, loff, bci_id, bci};
  na.unsorted = (flags & HS_FLAG_UNSORTED) ? 1 : 0;
  na.units = units;
  na.nunits = units ? nunits : 0;
  na.udyn = &sb->dyn[2];
  na.lists_partial = lists_partial ? 1 : 0;
  na.pseg = pseg;
  na.paval = paval;
  na.pair_abytes = a_bytes;
  na.pair_long = pair_long;
  na.unit_kb = bins.unit_kb;
  na.tiny_group = tiny_group;
  const char *names[NUM_KINDS] = {"numeric_tiny",   "numeric_warp_s", "numeric_warp",   "numeric_mid_s",
                                  "numeric_mid",    "numeric_large_s", "numeric_large", "numeric_sort_xs",
                                  "numeric_sort_s", "numeric_sort_m",  "numeric_sort",  "numeric_spa",
                                  "numeric_heavy"};
  static_assert(KEY_TINY + NUM_KINDS - 1 == KEY_HEAVY, "one key per numeric kind before the heavy keys");
  for (int i = 0; i < NUM_KINDS; ++i) {
    const int kind = NUM_KINDS - 1 - i;  // the longest first
    const int k0 = KEY_TINY + kind, k1 = kind == NUM_KINDS - 1 ? NKEYS : k0 + 1;
    na.list = list + key_off[k0];
    na.count = key_off[k1] - key_off[k0];
    if (plan) {
      plan->off[kind] = key_off[k0];
      plan->count[kind] = na.count;
    }
    if (na.count <= 0) continue;
    const cudaStream_t bst = fan.stream(num_group(kind));
    {
      PhaseTimer t2(names[kind], bst);
      if (!launch_num(sr, out_dt, kind, na, bst)) return HS_EINVAL;
    }
    if (int e = phase_check(names[kind], bst, sb->dbg)) return e;
  }
  if (!fan.join()) return HS_ECUDA;
  t_num.reset();
  if (flags & HS_FLAG_VALIDATE) {
    CK(cudaMemcpyAsync(hb, sb, sizeof(SmallBlock), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (hb->dbg[0]) {
      snprintf(t_detail, sizeof(t_detail), "index check %lld failed at %lld", hb->dbg[0], hb->dbg[1]);
      return HS_EINTERNAL;
    }
    if (hb->err) {
      snprintf(t_detail, sizeof(t_detail), "device consistency check %d", hb->err);
      return HS_EINTERNAL;
    }
  }
  // explicit zeros on request: entries whose (+,x) sum is exactly zero are
  // removed by one compaction of C (the symbolic pass counts structure only,
  // so this cannot happen earlier)
  if ((flags & HS_FLAG_PRUNE_ZEROS) && sr == HS_PLUS_TIMES && !plan && !place && nnz > 0) {
    int64_t *keep = mem.tmp<int64_t>((size_t)nnz);
    int64_t *ktmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(nnz));
    if (mem.failed) return HS_ENOMEM;
    {
      PhaseTimer t("prune_zeros", st);
      launch_keep_nonzero(C->val, out_dt, nnz, keep, st);
      launch_scan_i64(keep, nnz, ktmp, st);
    }
    CK(cudaMemcpyAsync(&hb->nnz, keep + nnz - 1, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const int64_t kept = hb->nnz;
    if (kept < nnz) {
      int64_t *p2 = (int64_t *)outmem.raw(sizeof(int64_t) * (size_t)(m + 1));
      int32_t *j2 = (int32_t *)outmem.raw(sizeof(int32_t) * (size_t)(kept > 0 ? kept : 1));
      void *v2 = outmem.raw((size_t)vb * (size_t)(kept > 0 ? kept : 1));
      if (!p2 || !j2 || !v2) {
        if (p2) outmem.release(p2, sizeof(int64_t) * (size_t)(m + 1));
        if (j2) outmem.release(j2, sizeof(int32_t) * (size_t)(kept > 0 ? kept : 1));
        if (v2) outmem.release(v2, (size_t)vb * (size_t)(kept > 0 ? kept : 1));
        return HS_ENOMEM;
      }
      const RowSet cs{Cp, C->idx, C->val, nullptr, m, nnz, m, sb->dbg};
      {
        PhaseTimer t("prune_zeros", st);
        launch_compact_by_keep(cs, keep, j2, v2, vb, p2, st);
      }
      outmem.release(C->ptr, sizeof(int64_t) * (size_t)(m + 1));
      outmem.release(C->idx, sizeof(int32_t) * (size_t)nnz);
      outmem.release(C->val, (size_t)vb * (size_t)nnz);
      C->ptr = p2;
      C->idx = j2;
      C->val = v2;
      C->nnz = kept;
    }
    if (int e = check_launch()) return e;
  }
  if (plan) {  // the plan takes over every scratch buffer
    plan->c_nnz = nnz;
    plan->na = na;
    plan->side_by_side = side_by_side;
    plan->list = list;
    plan->dyn = &sb->dyn[1];
    plan->err = &sb->err;
    plan->dbg = sb->dbg;
    plan->blocks = std::move(mem.scratch);
    mem.scratch.clear();
  }
  return HS_OK;
}

// runs fn; on failure releases whatever fn allocated for C
template <class F> static int with_output(hs_mat *C, Mem &outmem, F &&fn) {
  int e = fn();
  if (e != HS_OK && C) free_mat(C, outmem);
  return e;
}

static int sparse_impl(const int32_t *I, const int32_t *J, const void *V, int64_t nnz, int64_t m, int64_t n,
                       int dtype, int sr, hs_mat *C, Mem &mem, Mem &outmem, uint32_t flags);

// B = A(I, J) (Section 3.1's SpRef), the triple product R*A*Q evaluated
// without forming R*A: the rows I[t] are gathered end to end and each gathered
// entry (t, c, v) yields (t, p, v) for every p with J[p] == c (Q's row c).
// When J repeats no index, Q is the inverse map of J: an entry yields one
// tuple or none, the tuples lie row by row, and only the rows are sorted (not
// even those when J is increasing); two host synchronisations.  When J
// repeats indices the tuples are ordered by (t, p) with the radix sort of
// sparse(); five host synchronisations.  So they are, with three, where many
// long rows meet a wide J (spref_by_radix).
static int spref_impl(const hs_mat *A, const int32_t *I, int64_t nI, const int32_t *J, int64_t nJ, hs_mat *Bout,
                      Mem &mem, Mem &outmem, uint32_t flags) {
  cudaStream_t st = mem.st;
  if (!A || !Bout || A->fmt != HS_CSR || nI < 0 || nJ < 0) return HS_EINVAL;
  if ((nI > 0 && !I) || (nJ > 0 && !J)) return HS_EINVAL;
  if (nI > 0x7fffffffLL || nJ > 0x7fffffffLL) return HS_EUNSUPPORTED;
  if (!dtype_ok(A->dtype) || (A->m > 0 && !A->ptr)) return HS_EINVAL;
  if (A->dtype != HS_BOOL && A->nnz > 0 && !A->val) return HS_EINVAL;
  const int vb = A->dtype == HS_BOOL ? 0 : vbytes_of(A->dtype);
  const int64_t n = A->n;
  struct Small {  // device counters, read back in one copy
    int flag[2];
    int count[5];
    int pad;
    unsigned long long lmax, qmax, longs[3];
    int64_t total;
    long long dbg[2];
  };
  Small *sb = mem.tmp<Small>(1);
  Small *hb = (Small *)pinned(sizeof(Small));
  int32_t *pos = mem.tmp<int32_t>(n > 0 ? n : 1);
  int64_t *G = mem.tmp<int64_t>(nI + 1);
  int64_t *scan_tmp = mem.tmp<int64_t>(scan_tmp_elems((n + 1) > (nI + 1) ? (n + 1) : (nI + 1)));
  if (mem.failed || !hb) return HS_ENOMEM;
  // index ranges are always checked, and before any kernel uses I or J as an
  // address of its own (the look itself skips bad ones)
  {
    PhaseTimer t("spref_gather", st);
    CK(cudaMemsetAsync(sb, 0, sizeof(Small), st));
    CK(cudaMemsetAsync(pos, 0xff, sizeof(int32_t) * (size_t)n, st));
    if (nI == 0) CK(cudaMemsetAsync(G, 0, sizeof(int64_t), st));
    launch_spref_begin(A->ptr, A->m, n, I, nI, J, nJ, pos, G, sb->flag, &sb->lmax, st);
    if (flags & HS_FLAG_VALIDATE) launch_validate(A->ptr, A->idx, A->m, A->n, &sb->flag[1], st);
    launch_scan_i64(G, nI + 1, scan_tmp, st);
    CK(cudaMemcpyAsync(&sb->total, G + nI, 8, cudaMemcpyDeviceToDevice, st));
  }
  CK(cudaMemcpyAsync(hb, sb, sizeof(Small), cudaMemcpyDeviceToHost, st));
  if (int e = check_launch()) return e;
  CK(cudaStreamSynchronize(st));
  const int fl = hb->flag[0], vf = hb->flag[1];
  if (fl & 1) return HS_EINVAL;
  if (vf & 5) return HS_EINVAL;
  if (vf & 2) return HS_ENONCANON;
  const bool repeats = fl & 2, increasing = !(fl & 4);
  const int64_t total = hb->total, lmax = (int64_t)hb->lmax;

  auto out_ptr = [&]() {
    memset(Bout, 0, sizeof(*Bout));
    Bout->fmt = HS_CSR;
    Bout->dtype = A->dtype;
    Bout->m = nI;
    Bout->n = nJ;
    Bout->ptr = (int64_t *)outmem.raw(sizeof(int64_t) * (size_t)(nI + 1));
    return Bout->ptr != nullptr;
  };
  auto out = [&](int64_t nnz) {
    Bout->nnz = nnz;
    Bout->idx = (int32_t *)outmem.raw(sizeof(int32_t) * (size_t)(nnz > 0 ? nnz : 1));
    Bout->val = vb ? outmem.raw((size_t)vb * (size_t)(nnz > 0 ? nnz : 1)) : nullptr;
    return Bout->idx && (!vb || Bout->val);
  };
  auto empty_out = [&]() -> int {
    if (!out_ptr() || !out(0)) return HS_ENOMEM;
    CK(cudaMemsetAsync(Bout->ptr, 0, sizeof(int64_t) * (size_t)(nI + 1), st));
    return check_launch();
  };
  if (total == 0 || nJ == 0) return empty_out();
  // every (t, p) occurs once, so the combining operation of the radix sort
  // never acts: values are copied bit for bit whatever the operation
  const int sr = A->dtype == HS_BOOL ? HS_OR_AND : A->dtype == HS_I32 ? HS_MIN_PLUS : HS_PLUS_TIMES;

  if (!repeats) {
    const int64_t nw = (total + 31) / 32;
    int32_t *P = mem.tmp<int32_t>((size_t)total);
    void *V = vb ? (void *)mem.tmp<char>((size_t)vb * (size_t)total) : nullptr;
    uint32_t *keep = mem.tmp<uint32_t>((size_t)nw + 1);
    int64_t *S = mem.tmp<int64_t>((size_t)nw);
    int64_t *stmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(nw));
    if (mem.failed) return HS_ENOMEM;
    const SprefArgs a{A->ptr, A->idx, A->val, vb, I, nI, n, G, total, pos, P, V, keep, S};
    // B's offsets are needed now only where spref_by_radix may say yes
    const bool look = !increasing && lmax > SR_CTA && nJ > BITMAP_COLS;
    {
      PhaseTimer t("spref_gather", st);
      launch_spref_gather(a, st);
      launch_scan_i64(S, nw, stmp, st);
      if (look) {
        if (!out_ptr()) return HS_ENOMEM;
        launch_spref_offsets(a, Bout->ptr, sb->longs, st);
      }
    }
    if (look) CK(cudaMemcpyAsync(hb->longs, sb->longs, sizeof(sb->longs), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(&hb->total, S + nw - 1, 8, cudaMemcpyDeviceToHost, st));
    if (int e = check_launch()) return e;
    CK(cudaStreamSynchronize(st));
    const int64_t ntup = hb->total;
    if (ntup == 0 && !look) return empty_out();
    if (!increasing && ntup > 0x7fffffffLL) return HS_EUNSUPPORTED;
    const bool radix = look && spref_by_radix((int64_t)hb->longs[0], (int64_t)hb->longs[1], ntup, nI, nJ);
    if (!look && !out_ptr()) return HS_ENOMEM;
    if (!radix && !out(ntup)) return HS_ENOMEM;
    if (ntup == 0) return check_launch();  // (the offsets are all zero)
    std::unique_ptr<PhaseTimer> t(new PhaseTimer("spref_emit", st));
    if (!look) launch_spref_offsets(a, Bout->ptr, sb->longs, st);
    if (increasing) {
      launch_spref_emit(a, Bout->idx, Bout->val, st);
      return check_launch();
    }
    int32_t *tp = mem.tmp<int32_t>((size_t)ntup);
    void *tv = vb ? (void *)mem.tmp<char>((size_t)vb * (size_t)ntup) : nullptr;
    if (mem.failed) return HS_ENOMEM;
    launch_spref_emit(a, tp, tv, st);
    if (radix) {
      const size_t kept = mem.scratch.size();
      int32_t *ti = mem.tmp<int32_t>((size_t)ntup);
      hs_mat sorted;
      memset(&sorted, 0, sizeof(sorted));
      int e = HS_ENOMEM;
      if (ti) {
        launch_spref_row_ids(Bout->ptr, nI, ntup, ti, st);
        t.reset();
        if (int e2 = check_launch()) return e2;
        e = sparse_impl(ti, tp, tv, ntup, nI, nJ, A->dtype, sr, &sorted, mem, outmem, flags);
      }
      if (e != HS_ENOMEM) {
        free_mat(Bout, outmem);
        *Bout = sorted;
        return e;
      }
      free_mat(&sorted, outmem);  // no room for it: the bitmaps need less
      mem.release_from(kept);
      mem.failed = outmem.failed = false;
      if (!out(ntup)) return HS_ENOMEM;
    }
    int32_t *list = mem.tmp<int32_t>((size_t)(2 * nI));
    if (mem.failed) return HS_ENOMEM;
    launch_spref_rows(vb, Bout->ptr, nI, nJ, tp, tv, Bout->idx, Bout->val, lmax, sb->count, list, sb->dbg, st);
    if (!(flags & HS_FLAG_VALIDATE)) return check_launch();
    CK(cudaMemcpyAsync(hb, sb, sizeof(Small), cudaMemcpyDeviceToHost, st));  // the row sort's own checks
    if (int e = check_launch()) return e;
    CK(cudaStreamSynchronize(st));
    if (!hb->dbg[0] && !hb->count[4]) return HS_OK;
    snprintf(t_detail, sizeof(t_detail), "row sort check %d, index check %lld failed at %lld", hb->count[4],
             (long long)hb->dbg[0], (long long)hb->dbg[1]);
    return HS_EINTERNAL;
  }

  // Q = sparse(J, 1:len(J), 1, n, len(J)): row k holds every p with J[p] == k,
  // increasing.  Short rows (at most 32 repetitions of an index): counted,
  // filled by atomics and sorted in place; otherwise built by the stable
  // radix sort of sparse() itself
  int64_t *Qp = mem.tmp<int64_t>(n + 1);
  int64_t *Qcur = mem.tmp<int64_t>(n + 1);
  int32_t *Qj = mem.tmp<int32_t>(nJ);
  if (mem.failed) return HS_ENOMEM;
  CK(cudaMemsetAsync(Qp, 0, sizeof(int64_t) * (size_t)(n + 1), st));
  launch_build_Q_count(J, nJ, n, Qp, st);
  launch_max_count(Qp, n + 1, &sb->qmax, st);
  CK(cudaMemcpyAsync(&hb->qmax, &sb->qmax, 8, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  struct QGuard {
    hs_mat q{};
    Mem &m;
    ~QGuard() { free_mat(&q, m); }
  } qg{hs_mat{}, mem};
  if (hb->qmax <= 32) {
    PhaseTimer t("spref_build", st);
    launch_scan_i64(Qp, n + 1, scan_tmp, st);
    CK(cudaMemcpyAsync(Qcur, Qp, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyDeviceToDevice, st));
    launch_build_Q_fill(J, nJ, Qcur, Qj, st);
    launch_sort_short_rows(Qp, Qj, n, st);
  } else {
    int32_t *pidx = mem.tmp<int32_t>((size_t)nJ);
    if (!pidx) return HS_ENOMEM;
    launch_iota_i32(pidx, nJ, st);
    if (int e = sparse_impl(J, pidx, nullptr, nJ, n, nJ, HS_BOOL, HS_OR_AND, &qg.q, mem, mem, 0)) return e;
    Qp = qg.q.ptr;
    Qj = qg.q.idx;
  }
  int64_t *inc = mem.tmp<int64_t>((size_t)total);
  int64_t *W = mem.tmp<int64_t>((size_t)total);
  int64_t *scan_g = mem.tmp<int64_t>(scan_tmp_elems(total));
  if (mem.failed) return HS_ENOMEM;
  GatherArgs ga{A->ptr, A->idx, A->val, vb, I, G, inc, Qp, Qj, total, n};
  {
    PhaseTimer t("spref_gather", st);
    CK(cudaMemsetAsync(inc, 0, sizeof(int64_t) * (size_t)total, st));
    launch_row_starts(G, nI, total, inc, st);
    launch_scan_i64(inc, total, scan_g, st);
    launch_gather_w(ga, W, st);
    launch_scan_i64(W, total, scan_g, st);
  }
  CK(cudaMemcpyAsync(&hb->total, W + total - 1, 8, cudaMemcpyDeviceToHost, st));
  if (int e = check_launch()) return e;
  CK(cudaStreamSynchronize(st));
  const int64_t ntup = hb->total;
  if (ntup == 0) return empty_out();
  if (ntup > 0x7fffffffLL) return HS_EUNSUPPORTED;
  int32_t *ti = mem.tmp<int32_t>((size_t)ntup);
  int32_t *pj = mem.tmp<int32_t>((size_t)ntup);
  void *tv = vb ? (void *)mem.tmp<char>((size_t)vb * (size_t)ntup) : nullptr;
  if (mem.failed) return HS_ENOMEM;
  {
    PhaseTimer t("spref_gather", st);
    launch_gather_fill(ga, W, ti, pj, tv, st);
  }
  if (int e = check_launch()) return e;
  return sparse_impl(ti, pj, tv, ntup, nI, nJ, A->dtype, sr, Bout, mem, outmem, flags);
}

// C = sparse(i, j, v, m, n) (Section 2's constructor).  Every tuple is the
// key (i << bits(n-1)) | j, so that ascending keys are CSR order; a stable
// radix sort of the keys, carrying v, puts the tuples of one position next to
// each other in input order, and each run of equal keys becomes one entry of
// C, its values folded with the semiring's add (kernels in sparse.cu).  One
// host synchronisation: after the sort, to learn nnz(C) and whether an index
// was out of range.
static int bits_of(int64_t x) { return x > 0 ? 64 - __builtin_clzll((unsigned long long)x) : 0; }

// Failure-detection test setting for the next sparse() sort on this host
// thread (hs_test_lookback_expiry): a short look-back poll limit and a tile
// that never publishes its counts.  Consumed by one call.
static thread_local int t_sp_spin = 0;             // 0: the production limit
static thread_local long long t_sp_withhold = -1;  // -1: every tile publishes

static int sparse_impl(const int32_t *I, const int32_t *J, const void *V, int64_t nnz, int64_t m, int64_t n,
                       int dtype, int sr, hs_mat *C, Mem &mem, Mem &outmem, uint32_t) {
  cudaStream_t st = mem.st;
  if (!C || nnz < 0 || m < 0 || n < 0) return HS_EINVAL;
  int op = -1;
  if (sr == HS_PLUS_TIMES) op = dtype == HS_F64 ? 0 : dtype == HS_F32 ? 1 : dtype == HS_I64 ? 2 : -1;
  else if (sr == HS_MIN_PLUS) op = dtype == HS_F32 ? 3 : dtype == HS_I32 ? 4 : -1;
  else if (sr == HS_OR_AND) op = dtype == HS_BOOL ? 5 : -1;
  if (op < 0) return HS_EINVAL;
  if (nnz > 0 && (!I || !J || (dtype != HS_BOOL && !V))) return HS_EINVAL;
  if (nnz > 0x7fffffffLL || m > 0x7fffffffLL || n > 0x7fffffffLL) return HS_EUNSUPPORTED;
  const int vb = vbytes_of(dtype);
  memset(C, 0, sizeof(*C));
  C->fmt = HS_CSR;
  C->dtype = dtype;
  C->m = m;
  C->n = n;
  C->ptr = (int64_t *)outmem.raw(sizeof(int64_t) * (size_t)(m + 1));
  if (!C->ptr) return HS_ENOMEM;
  CK(cudaMemsetAsync(C->ptr, 0, sizeof(int64_t) * (size_t)(m + 1), st));
  if (nnz == 0) {
    C->idx = (int32_t *)outmem.raw(4);
    C->val = vb ? outmem.raw((size_t)vb) : nullptr;
    if (!C->idx || (vb && !C->val)) return HS_ENOMEM;
    return check_launch();
  }
  const int nbj = bits_of(n - 1), nbi = bits_of(m - 1);
  const int rb = sp_radix_bits();
  int passes = (nbi + nbj + rb - 1) / rb;
  if (passes < 1) passes = 1;
  if (passes > sp_max_passes()) return HS_EINTERNAL;
  const int64_t tiles = sp_tiles(nnz);
  const int64_t longcap = sp_long_capacity(nnz);
  const int64_t chunks = sp_chunks(nnz);
  const int64_t scan_n = chunks > m + 1 ? chunks : m + 1;
  uint64_t *kbuf[2] = {mem.tmp<uint64_t>((size_t)nnz), mem.tmp<uint64_t>((size_t)nnz)};
  void *vbuf[2] = {nullptr, nullptr};
  if (vb) {
    vbuf[0] = mem.tmp<char>((size_t)nnz * vb);
    vbuf[1] = mem.tmp<char>((size_t)nnz * vb);
  }
  unsigned long long *status = mem.tmp<unsigned long long>((size_t)(tiles << rb));
  unsigned long long *ghist = mem.tmp<unsigned long long>((size_t)passes << rb);
  int *ticket = mem.tmp<int>((size_t)passes);
  int64_t *theads = mem.tmp<int64_t>((size_t)chunks);
  int64_t *scan_tmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(scan_n));
  int64_t *longlist = vb ? mem.tmp<int64_t>((size_t)(2 * longcap)) : nullptr;
  int *flags = mem.tmp<int>(2);  // [0] index out of range, [1] long runs
  int64_t *host = (int64_t *)pinned(16);
  if (mem.failed || !host) return HS_ENOMEM;
  CK(cudaMemsetAsync(flags, 0, 8, st));
  CK(cudaMemsetAsync(status, 0, sizeof(unsigned long long) * (size_t)(tiles << rb), st));
  CK(cudaMemsetAsync(ghist, 0, sizeof(unsigned long long) * ((size_t)passes << rb), st));
  CK(cudaMemsetAsync(ticket, 0, sizeof(int) * (size_t)passes, st));
  int cur = 0;
  const int spin = t_sp_spin > 0 ? t_sp_spin : sp_spin_limit();
  const long long withhold = t_sp_withhold;
  t_sp_spin = 0;
  t_sp_withhold = -1;
  {
    PhaseTimer t("sparse_sort", st);
    launch_sp_allhist(I, J, nnz, nbj, m, n, passes, ghist, flags, st);
    for (int p = 0; p < passes; ++p) {
      const bool first = p == 0;
      const uint64_t *kin = first ? nullptr : kbuf[cur];
      const void *vin = first ? V : vbuf[cur];
      const int out = first ? 0 : cur ^ 1;
      PhaseTimer tp("sparse_pass", st);
      launch_sp_pass(vb, kin, I, J, vin, nnz, nbj, m, n, p, ghist + ((size_t)p << rb), status, ticket + p, tiles,
                     kbuf[out], vbuf[out], flags, spin, withhold, st);
      cur = out;
    }
    launch_sp_heads(kbuf[cur], nnz, theads, st);
    launch_scan_i64(theads, chunks, scan_tmp, st);
  }
  if (int e = check_launch()) return e;
  CK(cudaMemcpyAsync(host, theads + chunks - 1, 8, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(host + 1, flags, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  const int fl = *(int *)(host + 1);
  if (fl & 1) return HS_EINVAL;
  if (fl & 2) return HS_ETIMEDOUT;
  const int64_t U = host[0];
  C->nnz = U;
  C->idx = (int32_t *)outmem.raw(sizeof(int32_t) * (size_t)U);
  C->val = vb ? outmem.raw((size_t)vb * (size_t)U) : nullptr;
  if (!C->idx || (vb && !C->val)) return HS_ENOMEM;
  {
    PhaseTimer t("sparse_emit", st);
    launch_sp_emit(op, kbuf[cur], vbuf[cur], nnz, nbj, theads, C->idx, C->val, C->ptr, longlist, flags + 1, st);
    launch_scan_i64(C->ptr, m + 1, scan_tmp, st);
  }
  return check_launch();
}

// C = A .* not(S*A*T) + R*B*Q (assignment) or A + R*B*Q (extend-add), merged
// entry by entry (index.cu).  X = R*B*Q is B itself with its rows and columns
// relabelled, as long as every row of B keeps its column order under J (which
// the device checks); otherwise X is computed as the two products, which sort
// it.  One host synchronisation, to learn nnz(C) and the outcome of the
// checks (with the products: theirs, and one more).
static int spasgn_impl(const hs_mat *A, const int32_t *I, int64_t nI, const int32_t *J, int64_t nJ,
                       const hs_mat *B, int accumulate, int add_sr, hs_mat *C, Mem &mem, Mem &outmem,
                       uint32_t flags) {
  cudaStream_t st = mem.st;
  if (!A || !B || !C || A->fmt != HS_CSR || B->fmt != HS_CSR) return HS_EINVAL;
  if (nI < 0 || nJ < 0 || B->m != nI || B->n != nJ || A->dtype != B->dtype) return HS_EINVAL;
  if ((nI > 0 && !I) || (nJ > 0 && !J)) return HS_EINVAL;
  if (accumulate && A->dtype != HS_BOOL && add_sr != HS_PLUS_TIMES && add_sr != HS_MIN_PLUS) return HS_EINVAL;
  if (!dtype_ok(A->dtype) || A->m < 0 || A->n < 0 || A->nnz < 0 || B->nnz < 0) return HS_EINVAL;
  const int vb = vbytes_of(A->dtype);
  if ((A->m > 0 && !A->ptr) || (B->m > 0 && !B->ptr)) return HS_EINVAL;
  if ((A->nnz > 0 && (!A->idx || (vb && !A->val))) || (B->nnz > 0 && (!B->idx || (vb && !B->val)))) return HS_EINVAL;
  const int64_t m = A->m, n = A->n;
  if (nI > 0x7fffffffLL || nJ > 0x7fffffffLL || n > 0x7fffffffLL) return HS_EINVAL;
  if (m > 0x7fffffffLL) return HS_EUNSUPPORTED;
  const int64_t nnzA = m > 0 ? A->nnz : 0, nx = nI > 0 ? B->nnz : 0;
  const int64_t nw = (nnzA + 31) / 32;
  struct Small {  // device counters, read back in one copy
    int flag[2];
    unsigned long long viol[2];
    long long dbg[2];
    int64_t nnz, xtot;
  };
  Small *sb = mem.tmp<Small>(1);
  Small *hb = (Small *)pinned(sizeof(Small));
  int32_t *rpos = mem.tmp<int32_t>(m > 0 ? m : 1);
  int32_t *cpos = mem.tmp<int32_t>(n > 0 ? n : 1);
  int64_t *XB = mem.tmp<int64_t>((size_t)m + 1);
  int64_t *S = mem.tmp<int64_t>((size_t)(nw > 0 ? nw : 1));
  uint32_t *keep = mem.tmp<uint32_t>((size_t)nw + 1);  // (K(q) at A's end may look at the word past the last)
  int64_t *at = mem.tmp<int64_t>((size_t)(nx > 0 ? nx : 1));
  int64_t *src = mem.tmp<int64_t>((size_t)(nx > 0 ? nx : 1));
  int64_t *scan_tmp = mem.tmp<int64_t>((size_t)scan_tmp_elems(m + 1 > nw ? m + 1 : nw));
  if (mem.failed || !hb) return HS_ENOMEM;
  memset(C, 0, sizeof(*C));
  C->fmt = HS_CSR;
  C->dtype = A->dtype;
  C->m = m;
  C->n = n;
  C->ptr = (int64_t *)outmem.raw(sizeof(int64_t) * (size_t)(m + 1));
  if (!C->ptr) return HS_ENOMEM;
  AsgnArgs aa{A->ptr, A->idx, A->val, B->val, cpos, m, n, nnzA, vb, accumulate, add_sr, A->dtype,
              C->ptr, 0, nullptr, nullptr, sb->dbg};
  AsgnX x{B->ptr, B->idx, I, J, nI, nJ, nx};
  // everything up to C's offsets (xb: X's row offsets)
  auto offsets = [&](const int64_t *xb) -> int {
    PhaseTimer t("spasgn_merge", st);
    CK(cudaMemsetAsync(keep, 0xff, sizeof(uint32_t) * ((size_t)nw + 1), st));
    launch_asgn_keep(x, aa, I, nI, xb, at, src, keep, S, nw, st);
    launch_scan_i64(S, nw, scan_tmp, st);
    if (m > 0) launch_asgn_offsets(aa, xb, S, keep, st);
    else CK(cudaMemsetAsync(C->ptr, 0, sizeof(int64_t), st));
    CK(cudaMemcpyAsync(&sb->nnz, C->ptr + m, 8, cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(&sb->xtot, xb + m, 8, cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(hb, sb, sizeof(Small), cudaMemcpyDeviceToHost, st));
    if (int e = check_launch()) return e;
    CK(cudaStreamSynchronize(st));
    return HS_OK;
  };
  {
    PhaseTimer t("spasgn_build", st);
    CK(cudaMemsetAsync(sb, 0, sizeof(Small), st));
    CK(cudaMemsetAsync(rpos, 0xff, sizeof(int32_t) * (size_t)m, st));
    CK(cudaMemsetAsync(cpos, 0xff, sizeof(int32_t) * (size_t)n, st));
    launch_mark_positions(I, nI, m, rpos, sb->flag, st);
    launch_mark_positions(J, nJ, n, cpos, sb->flag, st);
    CK(cudaMemsetAsync(XB, 0, sizeof(int64_t) * (size_t)(m + 1), st));
    launch_asgn_rows(x, m, n, XB, sb->viol, sb->dbg, st);
    launch_scan_i64(XB, m + 1, scan_tmp, st);
  }
  // (a bad or repeated index of I or J is known only after this: until then
  // such indices are skipped or land inside the buffers)
  if (int e = offsets(XB)) return e;
  if (hb->flag[0] & 1) return HS_EINVAL;
  if (hb->flag[0] & 2) return HS_EDUP;
  auto internal = [&]() {
    snprintf(t_detail, sizeof(t_detail), "index check %lld failed at %lld", hb->dbg[0], hb->dbg[1]);
    return HS_EINTERNAL;
  };
  if (hb->dbg[0]) return internal();
  hs_mat X;
  memset(&X, 0, sizeof(X));
  struct Guard {
    hs_mat &x;
    Mem &m;
    ~Guard() { free_mat(&x, m); }
  } guard{X, mem};
  if (hb->viol[0] != hb->viol[1] || hb->xtot != nx) {
    // X by the products R*B and (R*B)*Q, R = sparse(I, 1:mb, 1, ma, mb) and
    // Q = sparse(1:nb, J, 1, nb, na)
    int64_t *Rp = mem.tmp<int64_t>(m + 1);
    int32_t *Rj = mem.tmp<int32_t>(nI > 0 ? nI : 1);
    int64_t *Qp = mem.tmp<int64_t>(nJ + 1);
    if (mem.failed) return HS_ENOMEM;
    {
      PhaseTimer t("spasgn_build", st);
      CK(cudaMemsetAsync(Rp, 0, sizeof(int64_t), st));
      launch_rows_from_pos(rpos, m, Rp, st);
      launch_scan_i64(Rp, m + 1, scan_tmp, st);
      launch_fill_from_pos(rpos, m, Rp, Rj, st);
      launch_iota_i64(Qp, nJ + 1, st);
    }
    hs_mat R{HS_CSR, HS_BOOL, m, nI, nI, 0, Rp, Rj, nullptr, nullptr};
    hs_mat Q{HS_CSR, HS_BOOL, nJ, n, nJ, 0, Qp, const_cast<int32_t *>(J), nullptr, nullptr};
    hs_mat RB;
    memset(&RB, 0, sizeof(RB));
    // the products feed the merge, which needs canonical rows
    const uint32_t pf = flags & ~(HS_FLAG_VALIDATE | HS_FLAG_UNSORTED | HS_FLAG_PRUNE_ZEROS);
    int e = spgemm_impl(HS_SELECT2ND, &R, B, &RB, mem, mem, pf);
    if (!e) e = spgemm_impl(HS_SELECT1ST, &RB, &Q, &X, mem, mem, pf);
    free_mat(&RB, mem);
    if (e) return e;
    if (X.nnz > nx) return HS_EINTERNAL;
    aa.Xv = X.val;
    x = AsgnX{X.ptr, X.idx, nullptr, nullptr, m, n, X.nnz};
    if (int e2 = offsets(X.ptr)) return e2;
    if (hb->dbg[0]) return internal();
  }
  C->nnz = hb->nnz;
  C->idx = (int32_t *)outmem.raw(sizeof(int32_t) * (size_t)C->nnz);
  if (vb) C->val = outmem.raw((size_t)vb * (size_t)C->nnz);
  if (!C->idx || (vb && !C->val)) return HS_ENOMEM;
  aa.nnzC = C->nnz;
  aa.Cj = C->idx;
  aa.Cv = C->val;
  {
    PhaseTimer t("spasgn_merge", st);
    launch_asgn_fill(x, aa, at, src, S, keep, st);
  }
  return check_launch();
}

}  // namespace hs

using namespace hs;

extern "C" {

int hs_spgemm(int semiring, const hs_mat *A, const hs_mat *B, hs_mat *C, const hs_allocator *al, void *stream,
              uint32_t flags) {
  if (!C) return HS_EINVAL;
  memset(C, 0, sizeof(*C));
  t_detail[0] = 0;
  Mem mem{al, (cudaStream_t)stream};
  Mem out{al, (cudaStream_t)stream};
  return with_output(C, out, [&] { return spgemm_impl(semiring, A, B, C, mem, out, flags); });
}

int hs_plan_create(int semiring, const hs_mat *A, const hs_mat *B, hs_mat *C, hs_plan **plan,
                   const hs_allocator *al, void *stream, uint32_t flags) {
  if (!C || !plan) return HS_EINVAL;
  memset(C, 0, sizeof(*C));
  *plan = nullptr;
  t_detail[0] = 0;
  hs_plan *P = new (std::nothrow) hs_plan();
  if (!P) return HS_ENOMEM;
  Mem mem{al, (cudaStream_t)stream};
  Mem out{al, (cudaStream_t)stream};
  const int e = with_output(C, out, [&] { return spgemm_impl(semiring, A, B, C, mem, out, flags, P); });
  if (e != HS_OK) {
    for (auto &b : P->blocks) mem.release(b.p, b.n);
    delete P;
    return e;
  }
  if (al) {
    P->al = *al;
    P->has_al = true;
  }
  if (const unsigned g = P->groups(); g & (g - 1)) {
    P->sides.reset(new (std::nothrow) SideSet<FanCuda>());
    if (P->sides && !P->sides->make((cudaStream_t)stream)) P->sides.reset();  // (the bins then run one by one)
  }
  *plan = P;
  return HS_OK;
}

int hs_plan_execute(const hs_plan *P, const void *A_val, const void *B_val, void *C_val, void *stream) {
  if (!P) return HS_EINVAL;
  const int vb = vbytes_of(P->out_dt);
  const bool need_a = P->sr == HS_PLUS_TIMES || P->sr == HS_MIN_PLUS || (P->sr == HS_SELECT1ST && vb);
  const bool need_b = P->sr == HS_PLUS_TIMES || P->sr == HS_MIN_PLUS || (P->sr == HS_SELECT2ND && vb);
  if ((need_a && P->a_nnz && !A_val) || (need_b && P->b_nnz && !B_val) || (vb && P->c_nnz && !C_val))
    return HS_EINVAL;
  if (P->c_nnz == 0) return HS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  NumArgs na = P->na;
  na.A.v = A_val;
  na.B.v = B_val;
  na.Cv = C_val;
  CK(cudaMemsetAsync(P->dyn, 0, 2 * sizeof(int), st));  // the heavy rows' and units' counters
  Fan fan(st, P->groups(), P->sides.get());
  // the heavy units' B segments carry A's values: laid out again from the new ones
  if (na.units && na.pseg && na.nunits > 0)
    launch_build_pairs(na.A, na.B, const_cast<HeavyUnit *>(na.units), na.nunits, na.bci_id, na.bci, na.nseg,
                       na.pair_abytes, na.pair_long, const_cast<int64_t *>(na.pseg), const_cast<void *>(na.paval),
                       fan.stream(num_group(NUM_KINDS - 1)));
  for (int i = 0; i < NUM_KINDS; ++i) {
    const int kind = NUM_KINDS - 1 - i;
    if (P->count[kind] <= 0) continue;
    na.list = P->list + P->off[kind];
    na.count = P->count[kind];
    if (!launch_num(P->sr, P->out_dt, kind, na, fan.stream(num_group(kind)))) return HS_EINVAL;
  }
  if (!fan.join()) return HS_ECUDA;
  return check_launch();
}

int hs_plan_status(const hs_plan *P, void *stream) {
  if (!P) return HS_EINVAL;
  if (!P->err) return HS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int *h = (int *)pinned(3 * sizeof(long long));
  if (!h) return HS_ECUDA;
  long long *hd = reinterpret_cast<long long *>(h) + 1;
  CK(cudaMemcpyAsync(h, P->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hd, P->dbg, 2 * sizeof(long long), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (hd[0]) {
    snprintf(t_detail, sizeof(t_detail), "index check %lld failed at %lld", hd[0], hd[1]);
    return HS_EINTERNAL;
  }
  if (h[0]) {
    snprintf(t_detail, sizeof(t_detail), "device consistency check %d", h[0]);
    return HS_EINTERNAL;
  }
  return HS_OK;
}

void hs_plan_destroy(hs_plan *P, void *stream) {
  if (!P) return;
  Mem mem{P->has_al ? &P->al : nullptr, (cudaStream_t)stream};
  for (auto &b : P->blocks) mem.release(b.p, b.n);
  P->blocks.clear();
  delete P;
}

int hs_spgemm_to_host(int semiring, const hs_mat *A, const hs_mat *B, int64_t nblocks, int64_t *h_ptr,
                      int32_t *h_idx, void *h_val, int64_t capacity, int64_t *nnz_out, void *stream,
                      uint32_t flags) {
  if (!A || !B || !h_ptr || !nnz_out || nblocks < 1 || capacity < 0) return HS_EINVAL;
  if (A->fmt != HS_CSR || A->m < 0) return HS_EINVAL;
  int out_dt = 0;
  if (!numeric_supported(semiring, A->dtype, B->dtype, out_dt)) return HS_EINVAL;
  const int vb = vbytes_of(out_dt);
  if ((capacity > 0 && !h_idx) || (vb && capacity > 0 && !h_val)) return HS_EINVAL;
  *nnz_out = 0;
  t_detail[0] = 0;
  cudaStream_t st = (cudaStream_t)stream;
  cudaStream_t cs = nullptr;  // copies of finished blocks run here, beside the next block's product
  CK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaEvent_t ev = nullptr;
  if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    cudaStreamDestroy(cs);
    return HS_ECUDA;
  }
  cudaMemPool_t pool = own_pool();
  const int64_t m = A->m;
  // Host arrays that the GPU maps (page-locked memory under unified
  // addressing; on NVLink-C2C systems the stores travel while the kernels
  // run): the numeric kernels write C's columns and values there directly,
  // so nothing is copied afterwards but the row offsets.
  auto mapped = [](const void *h) -> void * {
    if (!h) return nullptr;
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, h) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
  };
  int32_t *d_idx = (int32_t *)mapped(h_idx);
  void *d_val = vb ? mapped(h_val) : nullptr;
  if (nblocks == 1 && capacity > 0 && d_idx && (!vb || d_val) && !(flags & HS_FLAG_STAGE_ON_DEVICE)) {
    hs_mat Cd;
    memset(&Cd, 0, sizeof(Cd));
    Mem mem{nullptr, st, pool};
    Mem out{nullptr, st, pool};
    const OutPlace place{d_idx, d_val, capacity};
    int status = spgemm_impl(semiring, A, B, &Cd, mem, out, flags, nullptr, &place);
    *nnz_out = Cd.nnz;
    if (status == HS_OK) {
      if (cudaMemcpyAsync(h_ptr, Cd.ptr, sizeof(int64_t) * (size_t)(m + 1), cudaMemcpyDeviceToHost, st) !=
              cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        status = HS_ECUDA;
      }
    }
    if (Cd.ptr) out.release(Cd.ptr, sizeof(int64_t) * (size_t)(m + 1));
    cudaEventDestroy(ev);
    cudaStreamDestroy(cs);
    return status;
  }
  const int64_t rows_per = (m + nblocks - 1) / nblocks;
  int64_t base = 0;
  int status = HS_OK;
  for (int64_t r0 = 0; r0 < m || (m == 0 && r0 == 0); r0 += (rows_per ? rows_per : 1)) {
    const int64_t r1 = m == 0 ? 0 : (r0 + rows_per < m ? r0 + rows_per : m);
    // rows r0..r1 of A as a matrix of their own (offsets stay absolute)
    hs_mat Ab = *A;
    Ab.m = r1 - r0;
    Ab.ptr = A->ptr + r0;
    hs_mat Cb;
    memset(&Cb, 0, sizeof(Cb));
    Mem mem{nullptr, st, pool};
    Mem out{nullptr, st, pool};
    status = with_output(&Cb, out,
                         [&] { return spgemm_impl(semiring, &Ab, B, &Cb, mem, out, flags & ~HS_FLAG_PRUNE_ZEROS); });
    if (status != HS_OK) break;
    const int64_t rows = r1 - r0;
    if (base + Cb.nnz <= capacity) {
      if (base) launch_add_i64(Cb.ptr, rows + 1, base, st);
      if (cudaEventRecord(ev, st) != cudaSuccess || cudaStreamWaitEvent(cs, ev, 0) != cudaSuccess ||
          cudaMemcpyAsync(h_ptr + r0, Cb.ptr, sizeof(int64_t) * (size_t)(rows + 1), cudaMemcpyDeviceToHost, cs) !=
              cudaSuccess ||
          (Cb.nnz && cudaMemcpyAsync(h_idx + base, Cb.idx, sizeof(int32_t) * (size_t)Cb.nnz,
                                     cudaMemcpyDeviceToHost, cs) != cudaSuccess) ||
          (vb && Cb.nnz &&
           cudaMemcpyAsync(reinterpret_cast<char *>(h_val) + (size_t)base * vb, Cb.val, (size_t)vb * (size_t)Cb.nnz,
                           cudaMemcpyDeviceToHost, cs) != cudaSuccess)) {
        cudaGetLastError();
        status = HS_ECUDA;
      }
    } else if (cudaEventRecord(ev, st) != cudaSuccess || cudaStreamWaitEvent(cs, ev, 0) != cudaSuccess) {
      cudaGetLastError();
      status = HS_ECUDA;
    }
    // the block's output goes back to the pool on the copy stream, after its copies
    cudaFreeAsync(Cb.ptr, cs);
    cudaFreeAsync(Cb.idx, cs);
    if (Cb.val) cudaFreeAsync(Cb.val, cs);
    base += Cb.nnz;
    if (status != HS_OK || m == 0) break;
  }
  if (cudaStreamSynchronize(cs) != cudaSuccess && status == HS_OK) {
    cudaGetLastError();
    status = HS_ECUDA;
  }
  cudaEventDestroy(ev);
  cudaStreamDestroy(cs);
  *nnz_out = base;
  if (status == HS_OK && base > capacity) status = HS_ECAPACITY;
  return status;
}

int hs_trim_memory(void) {
  cudaMemPool_t pool = own_pool();
  if (!pool) return HS_ECUDA;
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemPoolTrimTo(pool, 0) != cudaSuccess) {
    cudaGetLastError();
    return HS_ECUDA;
  }
  return HS_OK;
}

int hs_spref(const hs_mat *A, const int32_t *I, int64_t nI, const int32_t *J, int64_t nJ, hs_mat *B,
             const hs_allocator *al, void *stream, uint32_t flags) {
  if (!B) return HS_EINVAL;
  memset(B, 0, sizeof(*B));
  Mem mem{al, (cudaStream_t)stream};
  Mem out{al, (cudaStream_t)stream};
  return with_output(B, out, [&] { return spref_impl(A, I, nI, J, nJ, B, mem, out, flags); });
}

int hs_sparse(const int32_t *i, const int32_t *j, const void *v, int64_t nnz, int64_t m, int64_t n, int dtype,
              int add_semiring, hs_mat *C, const hs_allocator *al, void *stream, uint32_t flags) {
  if (!C) return HS_EINVAL;
  memset(C, 0, sizeof(*C));
  Mem mem{al, (cudaStream_t)stream};
  Mem out{al, (cudaStream_t)stream};
  return with_output(C, out, [&] { return sparse_impl(i, j, v, nnz, m, n, dtype, add_semiring, C, mem, out, flags); });
}

int hs_spasgn(const hs_mat *A, const int32_t *I, int64_t nI, const int32_t *J, int64_t nJ, const hs_mat *B,
              int accumulate, int add_semiring, hs_mat *C, const hs_allocator *al, void *stream, uint32_t flags) {
  if (!C) return HS_EINVAL;
  memset(C, 0, sizeof(*C));
  Mem mem{al, (cudaStream_t)stream};
  Mem out{al, (cudaStream_t)stream};
  return with_output(C, out, [&] {
    return spasgn_impl(A, I, nI, J, nJ, B, accumulate, add_semiring, C, mem, out, flags);
  });
}

int hs_set_tuning(const hs_tuning *t) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  g_tune = t ? *t : k_tune_default;
  return HS_OK;
}

int hs_get_tuning(hs_tuning *t) {
  if (!t) return HS_EINVAL;
  std::lock_guard<std::mutex> g(g_tune_mu);
  *t = g_tune;
  return HS_OK;
}

void hs_mat_free(hs_mat *M, const hs_allocator *al, void *stream) {
  if (!M) return;
  Mem mem{al, (cudaStream_t)stream};
  free_mat(M, mem);
}

const char *hs_strerror(int s) {
  switch (s) {
    case HS_OK: return "success";
    case HS_EINVAL: return "invalid argument (shape, dtype, semiring, pointer or index)";
    case HS_ENONCANON: return "input matrix row not strictly increasing";
    case HS_EDUP: return "duplicate index in SpAsgn I or J";
    case HS_ENOMEM: return "allocation failed";
    case HS_ETIMEDOUT: return "bounded device wait expired";
    case HS_ECUDA: return "CUDA runtime error";
    case HS_EUNSUPPORTED: return "unsupported request";
    case HS_EINTERNAL: return "internal consistency check failed";
    case HS_ESCRATCH: return "product needs more scratch than the no-allocation entry point's fixed array";
    case HS_ECAPACITY: return "output capacity too small (C->nnz holds the size needed)";
  }
  return "unknown status";
}

int hs_last_cuda_error(void) { return t_last_cuda; }

const char *hs_last_error_detail(void) { return t_detail; }

int hs_version(void) { return 100; }

int64_t hs_launch_count(void) { return (int64_t)launch_total(); }

int hs_test_lookback_expiry(int spin_limit, int64_t withhold_tile) {
  if (spin_limit < 1 || withhold_tile < 0) return HS_EINVAL;
  t_sp_spin = spin_limit;
  t_sp_withhold = (long long)withhold_tile;
  return HS_OK;
}

void hs_profile_enable(int on) {
  std::lock_guard<std::mutex> g(g_prof.mu);
  g_prof.on = on != 0;
}

void hs_profile_reset(void) {
  std::lock_guard<std::mutex> g(g_prof.mu);
  g_prof.drain();
  for (auto &x : g_prof.ms) x = 0;
  for (auto &x : g_prof.launches) x = 0;
}

int hs_profile_read(double *ms, int64_t *launches, const char **names, int cap) {
  std::lock_guard<std::mutex> g(g_prof.mu);
  g_prof.drain();
  const int n = (int)g_prof.names.size();
  for (int i = 0; i < n && i < cap; ++i) {
    if (ms) ms[i] = g_prof.ms[i];
    if (launches) launches[i] = g_prof.launches[i];
    if (names) names[i] = g_prof.names[i].c_str();
  }
  return n;
}

}  // extern "C"
