// The C ABI (include/stc.h): argument checks, the key plan, stream-ordered memory, and the
// order of the stages of one contraction.
#include <algorithm>
#include <atomic>
#include <memory>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <mutex>
#include <string>
#include <vector>

#include "arena.h"
#include "launch.h"

using namespace stc;

// Autotuning of batches: per size bucket, each candidate is timed once with CUDA events around
// the accumulation kernels, read back without a sync on a later call of the same bucket; then
// the fastest is kept. A candidate sets three things: the group load factor (table sizes), the
// largest table a group may get in a warp of its own (group-per-warp granularity: groups above
// it take a CTA), and the expansion split of the CTA tables (products per lane per round).
struct TuneChoice {
  double alpha;
  int warp_max;  // slots of the largest warp-sized table used (256 or 1024)
  int depth;     // 0: the default expansion split, 1: half as many products per lane per round
};
constexpr TuneChoice kTune[] = {{0.5, 1024, 0}, {0.75, 1024, 0}, {0.9, 1024, 0}, {0.75, 256, 0}, {0.75, 1024, 1}};
constexpr int kTuneCand = 5;
constexpr TuneChoice kTuneDefault = {0.75, 1024, 0};
struct TuneEntry {
  int best = -1;
  float ms[kTuneCand] = {};
  bool done[kTuneCand] = {};
  bool pending[kTuneCand] = {};   // handed to a batch, not yet read back
  bool recorded[kTuneCand] = {};  // that batch has recorded both events
  cudaEvent_t ev0[kTuneCand] = {}, ev1[kTuneCand] = {};
};

struct stc_ctx : DevicePool {
  int device = 0;
  std::atomic<int64_t> live_results{0};
  int sms = 0;
  std::mutex tune_mu;
  std::map<int, TuneEntry> tune;
  // Problem shapes (shape_signature) whose last run here averaged at least kRowsMinPerOutput
  // products per output cell with output rows of at most kLaneRowMax keys: AUTO then groups X
  // and takes the lane-private dense rows for them (the product count is only known after the
  // survey, and the one-global-table path for small output key spaces never waits for it).
  std::mutex rows_mu;
  std::set<uint64_t> rows_shapes;
  // Page-locked blocks of kPinnedBytes for the counters that calls read back and the small
  // descriptors they send: as many as calls have run at once, given back with the context.
  std::mutex pin_mu;
  std::vector<void*> pins;
};
constexpr size_t kPinnedBytes = 2048;

namespace {
// Picks the load factor for a batch of this bucket; *measure is the candidate to time (or -1).
TuneChoice tune_pick(stc_ctx* ctx, int bucket, int* measure) {
  std::lock_guard<std::mutex> lk(ctx->tune_mu);
  TuneEntry& te = ctx->tune[bucket];
  *measure = -1;
  if (te.best >= 0) return kTune[te.best];
  // Only candidates whose batch has recorded both events are read: a batch of another thread
  // may still be between picking a candidate and recording its events (an event never
  // recorded reads as complete). A failed read is cleared so that it cannot surface as the
  // error of a later call on this thread, and the candidate is timed again.
  for (int c = 0; c < kTuneCand; c++) {
    if (!te.pending[c] || !te.recorded[c]) continue;
    const cudaError_t q = cudaEventQuery(te.ev1[c]);
    if (q == cudaErrorNotReady) {
      cudaGetLastError();
      continue;
    }
    const cudaError_t e = q == cudaSuccess ? cudaEventElapsedTime(&te.ms[c], te.ev0[c], te.ev1[c]) : q;
    if (e != cudaSuccess) cudaGetLastError();
    te.pending[c] = false;
    te.recorded[c] = false;
    te.done[c] = e == cudaSuccess;
  }
  int best = 0;
  bool all = true;
  for (int c = 0; c < kTuneCand; c++) {
    all = all && te.done[c];
    if (te.done[c] && te.ms[c] < te.ms[best]) best = c;
    if (te.done[c] && !te.done[best]) best = c;
  }
  if (all) {
    te.best = best;
    return kTune[best];
  }
  for (int c = 0; c < kTuneCand; c++) {
    if (!te.done[c] && !te.pending[c]) {
      if (!te.ev1[c]) {
        cudaEvent_t a = nullptr, b = nullptr;
        if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
          cudaGetLastError();
          if (a) cudaEventDestroy(a);
          return kTuneDefault;  // untimed
        }
        te.ev0[c] = a;
        te.ev1[c] = b;
      }
      *measure = c;
      te.pending[c] = true;
      te.recorded[c] = false;
      return kTune[c];
    }
  }
  return kTuneDefault;  // every remaining candidate is still being timed
}
void tune_mark(stc_ctx* ctx, int bucket, int cand, bool end, cudaStream_t s) {
  if (cand < 0) return;
  std::lock_guard<std::mutex> lk(ctx->tune_mu);
  TuneEntry& te = ctx->tune[bucket];
  if (cudaEventRecord(end ? te.ev1[cand] : te.ev0[cand], s) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  if (end) te.recorded[cand] = true;
}
// A batch that failed after picking a candidate gives it back.
void tune_abort(stc_ctx* ctx, int bucket, int cand) {
  if (cand < 0) return;
  std::lock_guard<std::mutex> lk(ctx->tune_mu);
  ctx->tune[bucket].pending[cand] = false;
  ctx->tune[bucket].recorded[cand] = false;
}
int log2_floor(uint64_t v) { return v ? 63 - __builtin_clzll(v) : 0; }
}  // namespace

// Device memory owned by one or more results (a batch's results share one block); returned to
// the context's pool, in the order of the stream it was made on, when the last owner goes.
struct DeviceBlock {
  stc_ctx* ctx = nullptr;
  cudaStream_t stream = nullptr;
  std::vector<std::pair<void*, size_t>> parts;
  ~DeviceBlock();
};

struct stc_result {
  stc_ctx* ctx = nullptr;
  cudaStream_t stream = nullptr;
  int64_t nnz = 0;
  int32_t order = 0;
  std::vector<int64_t> shape;
  int32_t* coords = nullptr;  // coordinates, or with keys_form the output keys (2 words each)
  double* vals = nullptr;
  bool keys_form = false;
  std::shared_ptr<DeviceBlock> mem;
  stc_stats stats{};
};

namespace {

thread_local std::string g_last_error;

stc_status fail(stc_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return s;
}

#define STC_CUDA(expr)                                                                          \
  do {                                                                                          \
    const cudaError_t e_ = (expr);                                                              \
    if (e_ != cudaSuccess)                                                                      \
      return fail(STC_ERR_CUDA, "%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, __LINE__); \
  } while (0)

#define STC_TRY(expr)                    \
  do {                                   \
    const stc_status s_ = (expr);        \
    if (s_ != STC_OK) return s_;         \
  } while (0)

// Makes the context's device current for the duration of a call, then restores the caller's.
struct DeviceGuard {
  int prev = -1;
  bool ok = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && (prev == dev || cudaSetDevice(dev) == cudaSuccess)) ok = true;
  }
  ~DeviceGuard() {
    if (ok && prev >= 0) cudaSetDevice(prev);
  }
};

// One page-locked block of the context's for the duration of a call. Copies to and from it are
// asynchronous, so it goes back only when the stream has passed them: calls wait for their stream
// before they return, and a call that fails in between waits here.
struct Pinned {
  stc_ctx* ctx;
  cudaStream_t s;
  void* p = nullptr;
  bool busy = false;  // a copy may be in flight
  Pinned(stc_ctx* c, cudaStream_t st) : ctx(c), s(st) {
    {
      std::lock_guard<std::mutex> lk(ctx->pin_mu);
      if (!ctx->pins.empty()) {
        p = ctx->pins.back();
        ctx->pins.pop_back();
      }
    }
    if (!p && cudaMallocHost(&p, kPinnedBytes) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
  }
  Pinned(const Pinned&) = delete;
  Pinned& operator=(const Pinned&) = delete;
  ~Pinned() {
    if (!p) return;
    if (busy) cudaStreamSynchronize(s);
    try {
      std::lock_guard<std::mutex> lk(ctx->pin_mu);
      ctx->pins.push_back(p);
    } catch (...) {
      cudaFreeHost(p);
    }
  }
};

bool is_pow2(uint64_t v) { return v && !(v & (v - 1)); }

// Output key spaces up to this size take the one-global-table strategy without a host read
// between the survey and the expansion: table and output sized from F (16 MB of table at most).
constexpr uint64_t kGlobalFromF = 1ull << 18;
// Lane-private dense rows (STC_ACC_ROWS): output rows of at most this many free keys, chosen by
// AUTO when the products average at least kRowsMinPerOutput per output cell.
constexpr uint64_t kLaneRowMax = 64;
constexpr uint64_t kRowsMinPerOutput = 64;
// Lanes that probe the one global table together when stc_opts.probe is 0.
constexpr int kDefaultProbe = 1;

// Moves the listed blocks from an arena into a shared block that results can own.
std::shared_ptr<DeviceBlock> adopt(Arena& ar, stc_ctx* ctx, cudaStream_t s, std::initializer_list<void*> ptrs) {
  auto blk = std::make_shared<DeviceBlock>();
  blk->ctx = ctx;
  blk->stream = s;
  for (void* p : ptrs)
    if (p) blk->parts.push_back({p, ar.keep(p)});
  return blk;
}

uint64_t pow2_at_least(uint64_t v) {
  uint64_t c = 1;
  while (c < v) c <<= 1;
  return c;
}

uint32_t log2_u64(uint64_t v) {
  uint32_t r = 0;
  while (v > 1) v >>= 1, r++;
  return r;
}

// The key plan of a contraction (Section 2.4.1 LN keys; the output mode order of Eq. 4).
struct Plan {
  KeyPlan kx{}, ky{};
  OutPlan op{};
  uint64_t K = 1, FX = 1, FY = 1, F = 1;
  uint64_t Kb = 1;         // bins that Y's contract keys are counted in: K, or with an id map n_Y
  bool id_map = false;     // contract keys replaced by dense ids through a bitmap (KeyPlan::idmap)
  bool report_ids = false; // ... in a call that is to report their number
  int32_t oz = 0;
  int32_t ocols = 0;      // int32 words per output entry: oz, or 2 for a 64-bit output key
  bool keys_out = false;  // outputs are keys (row-major over the output shape), not coordinates
  std::vector<int64_t> zshape;
};

stc_status check_coo(const stc_coo* t, const char* name) {
  if (!t) return fail(STC_ERR_INVALID_ARG, "%s is NULL", name);
  if (t->order < 0 || t->order > STC_MAX_ORDER)
    return fail(STC_ERR_INVALID_ARG, "%s.order = %d outside 0..%d", name, t->order, STC_MAX_ORDER);
  if (t->order > 0 && !t->shape) return fail(STC_ERR_INVALID_ARG, "%s.shape is NULL", name);
  for (int j = 0; j < t->order; j++)
    if (t->shape[j] < 1 || t->shape[j] > (int64_t)1 << 31)
      return fail(STC_ERR_INVALID_ARG, "%s.shape[%d] = %lld outside 1..2^31", name, j, (long long)t->shape[j]);
  if (t->nnz < 0 || t->nnz > STC_MAX_NNZ)
    return fail(STC_ERR_INVALID_ARG, "%s.nnz = %lld outside 0..%lld", name, (long long)t->nnz, STC_MAX_NNZ);
  if (t->nnz > 0 && (!t->vals || (t->order > 0 && !t->coords)))
    return fail(STC_ERR_INVALID_ARG, "%s has nnz > 0 but NULL coords or vals", name);
  return STC_OK;
}

// keys_out: outputs as 64-bit keys. xfree_sizes: when X is the split form of a tensor in key
// form, the lengths of that tensor's free modes, which the output's X part then has (the split
// form's free key is already the row-major index over them).
stc_status make_plan(const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx, const int32_t* cy,
                     const int32_t* out_order, Plan& pl, bool keys_out = false,
                     const std::vector<int64_t>* xfree_sizes = nullptr) {
  STC_TRY(check_coo(X, "X"));
  STC_TRY(check_coo(Y, "Y"));
  if (m < 0 || m > X->order || m > Y->order)
    return fail(STC_ERR_INVALID_ARG, "ncontract = %d outside 0..min(%d, %d)", m, X->order, Y->order);
  if (m > 0 && (!cx || !cy)) return fail(STC_ERR_INVALID_ARG, "cx or cy is NULL");
  bool xc[STC_MAX_ORDER] = {}, yc[STC_MAX_ORDER] = {};
  for (int i = 0; i < m; i++) {
    if (cx[i] < 0 || cx[i] >= X->order || cy[i] < 0 || cy[i] >= Y->order)
      return fail(STC_ERR_INVALID_ARG, "contract pair %d = (%d, %d) out of range", i, cx[i], cy[i]);
    if (xc[cx[i]] || yc[cy[i]]) return fail(STC_ERR_INVALID_ARG, "a mode is listed twice in cx or cy");
    xc[cx[i]] = yc[cy[i]] = true;
  }
  for (int i = 0; i < m; i++)
    if (X->shape[cx[i]] != Y->shape[cy[i]])
      return fail(STC_ERR_SHAPE_MISMATCH, "X mode %d has length %lld but Y mode %d has length %lld", cx[i],
                  (long long)X->shape[cx[i]], cy[i], (long long)Y->shape[cy[i]]);

  pl.kx = KeyPlan{};
  pl.ky = KeyPlan{};
  pl.kx.order = X->order;
  pl.ky.order = Y->order;
  pl.kx.nseg = pl.ky.nseg = 1;
  for (int j = 0; j < X->order; j++) pl.kx.size[j] = X->shape[j];
  for (int j = 0; j < Y->order; j++) pl.ky.size[j] = Y->shape[j];

  // Contract key: row-major over the contract list, first listed pair most significant.
  unsigned __int128 acc = 1;
  for (int i = m - 1; i >= 0; i--) {
    pl.kx.cstride[cx[i]] = (uint64_t)acc;
    pl.ky.cstride[cy[i]] = (uint64_t)acc;
    acc *= (unsigned __int128)X->shape[cx[i]];
    if (acc > (unsigned __int128)UINT64_MAX) return fail(STC_ERR_KEY_OVERFLOW, "contract key space exceeds 2^64");
  }
  pl.K = pl.Kb = (uint64_t)acc;

  // Free keys: row-major over the free modes in ascending order.
  std::vector<int> xf, yf;
  for (int j = 0; j < X->order; j++)
    if (!xc[j]) xf.push_back(j);
  for (int j = 0; j < Y->order; j++)
    if (!yc[j]) yf.push_back(j);
  acc = 1;
  for (int a = (int)xf.size() - 1; a >= 0; a--) {
    pl.kx.fstride[xf[a]] = (uint64_t)acc;
    acc *= (unsigned __int128)X->shape[xf[a]];
    if (acc > (unsigned __int128)UINT64_MAX) return fail(STC_ERR_KEY_OVERFLOW, "X free key space exceeds 2^64");
  }
  pl.FX = (uint64_t)acc;
  acc = 1;
  for (int b = (int)yf.size() - 1; b >= 0; b--) {
    pl.ky.fstride[yf[b]] = (uint64_t)acc;
    acc *= (unsigned __int128)Y->shape[yf[b]];
    if (acc > (unsigned __int128)UINT64_MAX) return fail(STC_ERR_KEY_OVERFLOW, "Y free key space exceeds 2^64");
  }
  pl.FY = (uint64_t)acc;
  const unsigned __int128 F = (unsigned __int128)pl.FX * pl.FY;
  // The all-ones key marks empty table slots, so the largest usable key is 2^64 - 2.
  if (F > (unsigned __int128)(UINT64_MAX - 1)) return fail(STC_ERR_KEY_OVERFLOW, "output key space exceeds 2^64 - 1");
  pl.F = (uint64_t)F;

  // Output: the concatenation (X free, Y free) is row-major in zkey = fX * FY + fY.
  std::vector<uint64_t> xs;
  if (xfree_sizes) {
    unsigned __int128 fx = 1;
    for (int64_t v : *xfree_sizes) xs.push_back((uint64_t)v), fx *= (unsigned __int128)v;
    if (fx > (unsigned __int128)pl.FX) return fail(STC_ERR_INVALID_ARG, "free modes do not fit the split key");
    const unsigned __int128 F2 = fx * pl.FY;
    if (F2 > (unsigned __int128)(UINT64_MAX - 1)) return fail(STC_ERR_KEY_OVERFLOW, "output key space exceeds 2^64 - 1");
    pl.F = (uint64_t)F2;
  } else {
    for (int a : xf) xs.push_back((uint64_t)X->shape[a]);
  }
  pl.oz = (int32_t)(xs.size() + yf.size());
  std::vector<uint64_t> csize(pl.oz), cstr(pl.oz);
  for (size_t a = 0; a < xs.size(); a++) csize[a] = xs[a];
  for (size_t b = 0; b < yf.size(); b++) csize[xs.size() + b] = (uint64_t)Y->shape[yf[b]];
  uint64_t st = 1;
  for (int t = pl.oz - 1; t >= 0; t--) {
    cstr[t] = st;
    st *= csize[t];
  }
  if (out_order) {
    std::vector<int> seen(pl.oz, 0);
    for (int q = 0; q < pl.oz; q++) {
      if (out_order[q] < 0 || out_order[q] >= pl.oz || seen[out_order[q]])
        return fail(STC_ERR_INVALID_ARG, "out_order is not a permutation of 0..%d", pl.oz - 1);
      seen[out_order[q]] = 1;
    }
  }
  pl.op = OutPlan{};
  pl.op.order = pl.oz;
  pl.op.pow2 = 1;
  pl.op.z32 = pl.F <= (1ull << 32);
  pl.op.ident = 1;
  pl.zshape.assign(pl.oz, 0);
  std::vector<int> pos_of(pl.oz);  // output position of concatenated mode t
  for (int q = 0; q < pl.oz; q++) {
    const int t = out_order ? out_order[q] : q;
    pos_of[t] = q;
    if (t != q) pl.op.ident = 0;
    pl.op.mod[q] = csize[t];
    pl.zshape[q] = (int64_t)csize[t];
    if (!is_pow2(csize[t])) pl.op.pow2 = 0;
  }
  for (int q = 0; q < pl.oz; q++) {
    const int t = out_order ? out_order[q] : q;
    pl.op.shift[q] = pl.op.pow2 ? log2_u64(cstr[t]) : 0;
  }
  // Digits least significant first: the last concatenated mode is the lowest digit.
  for (int j = 0; j < pl.oz; j++) {
    const int t = pl.oz - 1 - j;
    const uint64_t d = csize[t];
    const uint32_t l = d <= 1 ? 0 : 64 - (uint32_t)__builtin_clzll(d - 1);  // ceil(log2 d)
    const unsigned N = pl.op.z32 ? 32 : 64;
    const unsigned __int128 num = ((unsigned __int128)(((unsigned __int128)1 << l) - d)) << N;
    pl.op.magic[j] = (uint64_t)(num / d + 1);
    pl.op.magic32[j] = (uint32_t)(((((unsigned __int128)1 << l) - d) << 32) / d + 1);
    pl.op.dpos[j] = (uint8_t)pos_of[t];
    pl.op.dsh1[j] = (uint8_t)(l < 1 ? l : 1);
    pl.op.dsh2[j] = (uint8_t)(l > 1 ? l - 1 : 0);
  }
  pl.op.ny = (int32_t)yf.size();
  pl.op.split = pl.op.ident && !pl.op.pow2 && pl.oz >= 2 && pl.oz <= 8 &&
                pl.FX <= (1ull << 32) && pl.FY <= (1ull << 32);
  pl.ocols = pl.oz;
  pl.keys_out = keys_out;
  if (keys_out) {
    // The key itself, written by every output writer as two 32-bit "coordinates": the low and
    // the high half of zkey (a power-of-two plan of radix 2^32), i.e. one little-endian uint64.
    if (!pl.op.ident) return fail(STC_ERR_INVALID_ARG, "output_keys needs the output modes in concatenation order");
    OutPlan k{};
    k.order = 2;
    k.pow2 = 1;
    k.z32 = 0;
    k.ident = 1;
    k.mod[0] = k.mod[1] = 1ull << 32;
    k.shift[0] = 0;
    k.shift[1] = 32;
    pl.op = k;
    pl.ocols = 2;
  }
  return STC_OK;
}

stc_status status_word(uint32_t st) {
  if (st & kStatCoordRange) return fail(STC_ERR_COORD_OUT_OF_RANGE, "an input coordinate is outside its mode");
  if (st & kStatTableFull) return fail(STC_ERR_TABLE_FULL, "an accumulation table overflowed");
  if (st & kStatOutOverflow) return fail(STC_ERR_TABLE_FULL, "output capacity exceeded");
  if (st & kStatTimeout) return fail(STC_ERR_TIMEOUT, "a bounded wait gave up");
  if (st & kStatTooLarge) return fail(STC_ERR_UNSUPPORTED, "one X free group needs a table above 2^31 slots");
  return STC_OK;
}

// Small device counters of one call, in one allocation so one memset clears them.
struct Counters {
  u64 P;           // products
  u64 nz;          // output entries written
  unsigned ns;     // survivors
  uint32_t status; // kStat* bits
};

// Counters of the grouping and binning passes.
struct GroupCounters {
  uint32_t count[kMaxClasses + 4];
  unsigned nholes;       // pieces of reservations that hold no output
  u64 huge_slots;
  u64 out_cap;
  u64 holes;             // their positions
  u64 fill_counters[2];
  uint32_t ids;          // distinct contract keys of Y (with an id map)
};

// What a contraction reads back, in one copy.
struct CallCounters {
  Counters c;
  GroupCounters g;
};

// Per-stage CUDA events when timing is requested.
struct StageTimer {
  bool on = false;
  cudaStream_t s = nullptr;
  std::vector<cudaEvent_t> ev;
  int stage_of[16] = {};
  void start(bool enable, cudaStream_t st) {
    on = enable;
    s = st;
    if (on) mark(-1);
  }
  void mark(int stage) {
    if (!on) return;
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) {
      on = false;
      return;
    }
    cudaEventRecord(e, s);
    if (ev.size() > 16) {
      cudaEventDestroy(e);
      return;
    }
    if (stage >= 0 && stage < 8 && !ev.empty()) stage_of[ev.size() - 1] = stage;
    ev.push_back(e);
  }
  void collect(stc_stats& stats) {
    if (!on) return;
    if (!ev.empty()) cudaEventSynchronize(ev.back());  // stage times are a diagnostic: wait for them
    for (size_t i = 1; i < ev.size(); i++) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[i - 1], ev[i]);
      const int st = stage_of[i - 1];
      stats.stage_ms[st] += ms;
      stats.nstages = std::max(stats.nstages, st + 1);
    }
  }
  ~StageTimer() {
    for (auto e : ev) cudaEventDestroy(e);
  }
};

// The device state shared by the counting pass and the contraction: Y grouped by contract
// key, and X surveyed against it.
struct Prepared {
  KeyPlan kx{}, ky{};        // the plan's, with the id map
  uint32_t* yoff = nullptr;  // [K + 1]
  void* yfk = nullptr;       // [nY], Y free keys in contract-key order (u32 when key32, else u64)
  bool key32 = false;
  double* yv = nullptr;      // [nY]
  Survivors sv{};
  Counters* ctr = nullptr;   // of a CallCounters
  uint32_t* gcnt = nullptr;  // [FX] entries with a Y run per X free key (GROUPED only)
  bool dense = false;        // GROUPED without a survivor list (X re-read by the scatter)
  bool keep_ck = false;      // survivors keep their contract key (dense-row accumulation)
};

// How X is surveyed: a survivor list (GLOBAL), a survivor list plus per-group counts
// (GROUPED, few X entries have a Y run), or per-group counts alone (GROUPED, most do).
enum class Survey { kSurvivors, kSurvivorsGroups, kDenseGroups };

uint64_t survivor_blocks(int64_t nX) { return ((uint64_t)nX + kSurvivorBlock - 1) / kSurvivorBlock; }

stc_status prepare(stc_ctx* ctx, Arena& ar, const stc_coo* X, const stc_coo* Y, const Plan& pl, Survey mode,
                   cudaStream_t s, StageTimer& tm, Prepared& pr) {
  const bool groups = mode != Survey::kSurvivors;
  const uint64_t bins = pl.Kb * pl.ky.nseg;
  if (pl.Kb > kMaxDirectBins || bins > kMaxDirectBins)
    return fail(STC_ERR_UNSUPPORTED, "contract key space %llu exceeds %llu bins", (unsigned long long)pl.Kb,
                (unsigned long long)kMaxDirectBins);
  const int64_t nX = X->nnz, nY = Y->nnz;
  CallCounters* cc = nullptr;
  STC_TRY(ar.alloc(&cc, 1));
  pr.ctr = &cc->c;
  STC_CUDA(cudaMemsetAsync(cc, 0, sizeof(CallCounters), s));
  uint32_t* status = &pr.ctr->status;
  pr.kx = pl.kx;
  pr.ky = pl.ky;
  if (pl.id_map) {
    uint2* map = nullptr;
    uint32_t* scratch = nullptr;
    STC_TRY(ar.alloc(&map, (size_t)id_map_pairs(pl.K)));
    STC_TRY(ar.alloc(&scratch, (size_t)id_map_scratch(pl.K)));
    STC_CUDA(launch_id_map(Y->coords, nY, pl.ky, pl.K, map, scratch, &cc->g.ids, status, ctx->sms, s));
    pr.kx.idmap = pr.ky.idmap = map;
  }

  // Y: count per contract key, exclusive scan, scatter (Section 4.1.1 counting sort).
  uint32_t *ycnt = nullptr, *ycur = nullptr, *scr = nullptr;
  // The Y counts and, past them, the bitmap of contract keys with entries (one clearing).
  const uint64_t ne_words = (mode != Survey::kDenseGroups && pl.K <= kNonemptyMaxKeys) ? (pl.K + 31) / 32 : 0;
  // and, past that, the entries per X free key
  // or (one-table contractions of small output spaces) the products per block of survivors.
  const bool blocks = mode == Survey::kSurvivors && pl.F <= kGlobalFromF;
  const uint64_t lead = blocks ? 2 * survivor_blocks(nX) : 0;
  const uint64_t counts = lead + bins + ne_words + (groups ? pl.FX : 0);
  uint32_t* zeroed = nullptr;
  STC_TRY(ar.alloc(&zeroed, counts));
  if (blocks) pr.sv.bsum = reinterpret_cast<u64*>(zeroed);
  ycnt = zeroed + lead;
  if (groups) pr.gcnt = ycnt + bins + ne_words;
  STC_TRY(ar.alloc(&pr.yoff, bins + 1));
  STC_TRY(ar.alloc(&ycur, bins));
  STC_TRY(ar.alloc(&scr, (size_t)scan_scratch_elems((int64_t)bins)));
  pr.key32 = groups && pl.FY <= 0xffffffffull;
  if (pr.key32) {
    uint32_t* k32 = nullptr;
    STC_TRY(ar.alloc(&k32, (size_t)nY + 1));
    pr.yfk = k32;
  } else {
    u64* k64 = nullptr;
    STC_TRY(ar.alloc(&k64, (size_t)nY));
    pr.yfk = k64;
  }
  STC_TRY(ar.alloc(&pr.yv, (size_t)nY + 1));
  // X's arrays too, before any launch: the stages' events then enclose device work, not the
  // host's allocation calls.
  pr.sv.count = &pr.ctr->ns;
  pr.dense = mode == Survey::kDenseGroups;
  uint32_t* nonempty = nullptr;
  if (!pr.dense) {
    STC_TRY(ar.alloc(&pr.sv.fk, (size_t)nX));
    if (pr.keep_ck) STC_TRY(ar.alloc(&pr.sv.ck, (size_t)nX));
    STC_TRY(ar.alloc(&pr.sv.ystart, (size_t)nX));
    STC_TRY(ar.alloc(&pr.sv.w, (size_t)nX));
    STC_TRY(ar.alloc(&pr.sv.v, (size_t)nX));
    if (ne_words) nonempty = ycnt + bins;
  }
  STC_CUDA(cudaMemsetAsync(zeroed, 0, counts * sizeof(uint32_t), s));
  STC_CUDA(launch_y_count(Y->coords, nY, pr.ky, ycnt, status, ctx->sms, s, nonempty));
  STC_CUDA(scan_u32(ycnt, pr.yoff, (int64_t)bins, scr, s, ycur));
  STC_CUDA(launch_y_scatter(Y->coords, Y->vals, nY, pr.ky, pl.FY, ycur, pr.yfk, pr.key32, pr.yv, ctx->sms, s));
  tm.mark(0);

  // X: find each entry's Y run and count the products exactly (Section 4.3).
  if (pr.dense) {
    STC_CUDA(launch_x_count(X->coords, nX, pr.kx, pr.yoff, &pr.ctr->P, pr.gcnt, status, ctx->sms, s));
  } else {
    STC_CUDA(launch_x_survey(X->coords, X->vals, nX, pr.kx, pr.yoff, pl.K, pr.sv, &pr.ctr->P, pr.gcnt, status,
                             nonempty, ctx->sms, s, nonempty != nullptr));
  }
  tm.mark(1);
  return STC_OK;
}

// Reads the call's counters back and waits for the stream; the status word is the caller's to look at.
stc_status copy_counters(const Prepared& pr, Pinned& pin, CallCounters& h) {
  static_assert(sizeof(CallCounters) <= kPinnedBytes / 2, "a page-locked block holds the counters and a descriptor");
  CallCounters* const to = pin.p ? static_cast<CallCounters*>(pin.p) : &h;
  pin.busy = true;
  STC_CUDA(cudaMemcpyAsync(to, pr.ctr, sizeof(CallCounters), cudaMemcpyDeviceToHost, pin.s));
  STC_CUDA(cudaStreamSynchronize(pin.s));
  pin.busy = false;
  if (pin.p) h = *to;
  return STC_OK;
}

stc_status read_counters(const Prepared& pr, Pinned& pin, CallCounters& h) {
  STC_TRY(copy_counters(pr, pin, h));
  return status_word(h.c.status);
}

// The requests of prepare.
void count_prepare(ArenaBytes& b, const Plan& pl, int64_t nX, int64_t nY, Survey mode, bool keep_ck) {
  const bool groups = mode != Survey::kSurvivors;
  const uint64_t bins = pl.Kb * pl.ky.nseg, x = (uint64_t)nX, y = (uint64_t)nY;
  b.alloc(sizeof(CallCounters));
  if (pl.id_map) {
    b.alloc(id_map_pairs(pl.K) * sizeof(uint2));
    b.alloc((uint64_t)id_map_scratch(pl.K) * 4);
  }
  const uint64_t ne_words = (mode != Survey::kDenseGroups && pl.K <= kNonemptyMaxKeys) ? (pl.K + 31) / 32 : 0;
  const uint64_t lead = !groups && pl.F <= kGlobalFromF ? 2 * survivor_blocks(nX) : 0;
  b.alloc((lead + bins + ne_words + (groups ? pl.FX : 0)) * 4);
  b.alloc((bins + 1) * 4);
  b.alloc(bins * 4);
  b.alloc((uint64_t)scan_scratch_elems((int64_t)bins) * 4);
  b.alloc(groups && pl.FY <= 0xffffffffull ? (y + 1) * 4 : y * 8);
  b.alloc((y + 1) * 8);
  if (mode != Survey::kDenseGroups) {
    b.alloc(x * 8);
    if (keep_ck) b.alloc(x * 4);
    b.alloc(x * 4);
    b.alloc(x * 4);
    b.alloc(x * 8);
  }
}

// Whether the one-global-table strategy writes outputs as their keys are claimed, where the list of
// products that find their key claimed stays below 1 GB. It is the faster form whether products repeat
// keys or not (ms for the contraction, against accumulating in the table and passing over its slots):
// 3.2e6 products of 1.04 per key 0.71 against 0.79, 7.4e5 of 10.8 per key 0.28 against 0.29; 2e7 over a
// large key space of 1, 10, 1,000 and 1e5 per key 2.04 against 2.47, 1.13 against 1.69, 0.88 against
// 1.15, 0.74 against 0.99. The most it loses is 2e6 of 1,000 per key, 0.22 against 0.20. What counts is
// the table: it has twice the smaller of products and keys, so that in small key spaces there is little
// of it to pass over. 2e7 uniform products on F = 2, 1, 0.5 and 0.1 keys per product: 1.99 against 2.31,
// 1.87 against 2.22, 1.53 against 1.65, 0.95 against 0.60; 6e7: 6.09 against 6.41, 5.88 against 6.09,
// 5.33 against 4.95, 2.79 against 2.56. The line lies on the safe side, at two keys per product.
bool direct_global(uint64_t P, uint64_t F, uint64_t cap) {
  return P <= F / 2 && P <= (1ull << 26) && cap <= (1ull << 32);
}

// Cells of the array that holds an output space of F keys (launch_clear_space). The keys of smaller
// spaces than 2^15 are spread over as many cells, so that they share few lines: 4e7 products on 64 x 64
// keys take 0.61 ms for the contraction, on 4,096 cells 1.09, in a table 0.83; on 4 x 4 keys 5.6, 13.4
// and 15.6 (with tiles of 1,024 products). Under a budget no more than the table would take that the array stands for.
uint64_t space_cells(const stc_ctx* ctx, uint64_t F) {
  return pow2_at_least(std::max<uint64_t>(F, ctx->budget ? std::min<uint64_t>(2 * F, 1 << 15) : 1 << 15));
}

// Peak device bytes of the GLOBAL strategy for these counts.
uint64_t global_bytes(const stc_ctx* ctx, const Plan& pl, int64_t nX, int64_t nY, uint64_t ns, uint64_t P,
                      double alpha) {
  // Small output key spaces are sized from F itself (no host read of P), with products per block of X.
  const bool from_f = pl.F <= kGlobalFromF && nX > 0 && nY > 0;
  const uint64_t target = from_f ? pl.F : std::min<uint64_t>(P, pl.F);
  const uint64_t cap = pow2_at_least(std::max<uint64_t>(64, (uint64_t)((double)target / alpha) + 1));
  const uint64_t out = std::min(target, cap) * (4ull * pl.ocols + 8);
  ArenaBytes b(ctx);
  count_prepare(b, pl, nX, nY, Survey::kSurvivors, false);
  if (from_f) {
    b.alloc(space_cells(ctx, pl.F) * 8);
    b.alloc((survivor_blocks(nX) + 1) * 8);
    b.alloc_own(out);
    return b.held;
  }
  if (P == 0) return b.held;
  ArenaBytes table = b;  // the table of values, also where there is no memory for the list of repeats
  if (direct_global(P, pl.F, cap) && ctx->budget == 0) {
    b.alloc(cap * 8);
    b.alloc(cap * 4);
    b.alloc(P * 4);
    b.alloc(P * 8);
  } else {
    b = ArenaBytes(ctx);
  }
  table.alloc(cap * 8);
  table.alloc(cap * 8);
  for (ArenaBytes* t : {&b, &table}) {
    t->alloc((ns + 1) * 8);
    t->alloc((uint64_t)scan_scratch_elems((int64_t)ns) * 8);
    t->alloc_own(out);
  }
  return std::max(b.held, table.held);
}

// How GROUPED sweeps rows of bitmaps: F_Y in `nseg` segments of `seg` free keys; Y is grouped per
// (contract key, segment). For F_Y <= 2^20 and the bins' limit: for every group with the bitmap
// accumulator, for the groups beyond the warp-sized hash classes with AUTO.
bool dense_segments(const Plan& pl, int32_t accumulator, uint32_t& seg, uint32_t& nseg) {
  seg = nseg = 1;
  if (pl.FY > (1ull << 20) || (accumulator != STC_ACC_AUTO && accumulator != STC_ACC_DENSE)) return false;
  seg = (uint32_t)std::min<uint64_t>(kDenseSeg, pow2_at_least(std::max<uint64_t>(pl.FY, 64)));
  nseg = (uint32_t)((pl.FY + seg - 1) / seg);
  return pl.Kb * nseg <= kMaxDirectBins;
}

// Positions to be expected left over by `nstream` streamed groups: the last groups of the kernel's CTAs
// and the pieces that they drop.
uint64_t expected_holes(const stc_ctx* ctx, uint64_t nstream, uint64_t out_cap) {
  return std::min<uint64_t>(out_cap, std::min<uint64_t>(nstream, 4ull * ctx->sms) * stream_cap() + out_cap / 64);
}

// Peak device bytes of the GROUPED strategy with default options, the output at its bound, without the
// tables of groups that are too large for shared memory (F_Y above 2^20).
uint64_t grouped_bytes(const stc_ctx* ctx, Plan pl, int64_t nX, int64_t nY, uint64_t P, Survey mode) {
  uint32_t seg = 1, nseg = 1;
  const bool dense_rows = dense_segments(pl, STC_ACC_AUTO, seg, nseg);
  if (dense_rows) pl.ky.nseg = nseg;
  const uint64_t x = (uint64_t)nX, out = std::min<uint64_t>(P, pl.F);
  const uint64_t maxg = std::min<uint64_t>(pl.FX, (uint64_t)std::max<int64_t>(nX, 1));
  const bool wide = pl.FY > 0xffffffffull;
  ArenaBytes b(ctx);
  count_prepare(b, pl, nX, nY, mode, dense_rows);
  b.alloc((pl.FX + 1) * 4);
  b.alloc(pl.FX * 4);
  b.alloc((uint64_t)scan_scratch_elems((int64_t)pl.FX) * 4);
  b.alloc(x * 4);
  b.alloc(x * 4);
  b.alloc(x * 8);
  if (dense_rows) b.alloc(x * 4);
  for (int c = 0; c < (wide ? kNumClasses64 : kNumClasses32) + (dense_rows ? 3 : 0) + 1; c++) b.alloc(maxg * 4);
  b.alloc(maxg * 8);
  b.alloc(maxg * 8);
  if (P == 0) return b.held;
  b.alloc_own(out * 4ull * pl.ocols);
  b.alloc_own(out * 8);
  b.alloc(sizeof(BatchOut));
  if (dense_rows) {
    // Streamed groups have more products per segment than the warp classes have slots.
    const uint64_t nstream = std::min<uint64_t>(maxg, P / (kClassShapes32[1].slots / 2 * nseg));
    if (nstream) b.alloc(stream_max_holes((uint32_t)nstream, nseg) * sizeof(StreamHole));
    const uint64_t holes = expected_holes(ctx, nstream, out);
    if (ctx->budget == 0 && holes > x) b.alloc(holes * 4);  // under a budget only where there is room
  }
  return b.held;
}

// Whether GROUPED counts X without a survivor list: Y's runs cover the contract keys on average, or
// Y's keys were few enough beside its entries that ids are reported (ids cover them all).
bool x_dense(const Plan& pl, const stc_coo* Y) { return (uint64_t)Y->nnz >= pl.K || pl.report_ids; }

// GROUPED strategy (Sections 4.1 and 4.3): survivors are counting-sorted by X free key,
// each group is binned by its table size, and the class kernels accumulate one group per
// CTA in shared memory and write its outputs directly.
stc_status contract_grouped(stc_ctx* ctx, Arena& ar, const stc_coo* X, const stc_coo* Y, const Plan& plan_in,
                            const stc_opts& o, cudaStream_t s, StageTimer& tm, stc_result* r) {
  const int64_t nX = X->nnz;
  Plan pl = plan_in;
  if (o.accumulator == STC_ACC_ROWS && pl.FY > kLaneRowMax)
    return fail(STC_ERR_INVALID_ARG, "the ROWS accumulator takes at most %llu Y free keys, not %llu",
                (unsigned long long)kLaneRowMax, (unsigned long long)pl.FY);
  uint32_t seg = 1, nseg = 1;
  const bool dense_rows = dense_segments(pl, o.accumulator, seg, nseg);
  if (dense_rows) {
    pl.ky.nseg = pl.kx.nseg = nseg;
    pl.ky.seg_shift = log2_u64(seg);
  }
  Prepared pr;
  pr.keep_ck = dense_rows;
  // Dense when Y's runs cover the contract keys on average: then nearly every X entry has a
  // run and a survivor list would only be written and read back.
  const Survey mode = x_dense(pl, Y) ? Survey::kDenseGroups : Survey::kSurvivorsGroups;
  STC_TRY(prepare(ctx, ar, X, Y, pl, mode, s, tm, pr));

  const bool wide = pl.FY > 0xffffffffull;
  const int ncls = wide ? kNumClasses64 : kNumClasses32;
  const ClassShape* shapes = wide ? kClassShapes64 : kClassShapes32;
  const double ga = (o.group_load_factor > 0.0) ? o.group_load_factor : 0.75;
  const uint64_t maxg = std::min<uint64_t>(pl.FX, (uint64_t)std::max<int64_t>(nX, 1));

  uint32_t *goff = nullptr, *gcur = nullptr, *scr = nullptr;
  GroupedX gx{};
  Bins b{};
  Pinned pin(ctx, s);
  GroupCounters* const gc = &reinterpret_cast<CallCounters*>(pr.ctr)->g;
  STC_TRY(ar.alloc(&goff, pl.FX + 1));
  STC_TRY(ar.alloc(&gcur, pl.FX));
  STC_TRY(ar.alloc(&scr, (size_t)scan_scratch_elems((int64_t)pl.FX)));
  STC_TRY(ar.alloc(&gx.ystart, (size_t)nX));
  STC_TRY(ar.alloc(&gx.w, (size_t)nX));
  STC_TRY(ar.alloc(&gx.v, (size_t)nX));
  if (dense_rows) STC_TRY(ar.alloc(&gx.ck, (size_t)nX));
  b.nclasses = ncls;
  for (int c = 0; c < ncls; c++) {
    b.tmax[c] = (u64)(ga * shapes[c].slots);
    STC_TRY(ar.alloc(&b.list[c], maxg));
  }
  if (dense_rows) {
    // With AUTO, groups that fit the warp classes keep their hash tables (a bitmap sweep costs
    // a fixed amount per segment).
    b.dense_min = o.accumulator == STC_ACC_DENSE ? 0 : (b.tmax[1] + 1) * nseg;
    b.stream_cap = stream_cap();
    b.stash_cap = dense_stash_cap();
    for (int d = 0; d < 3; d++) STC_TRY(ar.alloc(&b.dense_list[d], maxg));
  }
  STC_TRY(ar.alloc(&b.huge_list, maxg));
  STC_TRY(ar.alloc(&b.huge_off, maxg));
  STC_TRY(ar.alloc(&b.huge_cap, maxg));
  b.count = gc->count;
  b.huge_slots = &gc->huge_slots;
  b.out_cap = &gc->out_cap;
  b.status = &pr.ctr->status;
  STC_CUDA(scan_u32(pr.gcnt, goff, (int64_t)pl.FX, scr, s, gcur));
  if (pr.dense) {
    STC_CUDA(launch_x_scatter_dense(X->coords, X->vals, nX, pr.kx, pr.yoff, gcur, gx, &pr.ctr->status, ctx->sms, s));
  } else {
    STC_CUDA(launch_x_group_scatter(pr.sv, gcur, gx, nX, ctx->sms, s));
  }
  STC_CUDA(launch_bin_groups(pl.FX, goff, gx.w, pl.FY, b, pr.dense ? &pr.ctr->ns : nullptr, ctx->sms, s));
  tm.mark(2);

  CallCounters hc{};
  STC_TRY(read_counters(pr, pin, hc));
  const Counters& h = hc.c;
  const GroupCounters hg = hc.g;
  tm.mark(3);
  r->stats.products = h.P;
  r->stats.survivors = h.ns;
  if (pl.report_ids) r->stats.contract_ids = hg.ids;
  uint64_t groups = 0, dense_groups = 0;
  for (int c = 0; c < kMaxClasses + 4; c++) groups += hg.count[c];
  dense_groups = hg.count[kMaxClasses + 1] + hg.count[kMaxClasses + 2] + hg.count[kMaxClasses + 3];
  r->stats.groups = groups;
  r->stats.table_slots = hg.huge_slots;
  r->stats.accumulator = dense_groups == 0 ? STC_ACC_HASH : (dense_groups == groups ? STC_ACC_DENSE : STC_ACC_AUTO);
  if (h.P == 0) return STC_OK;
  // Lane-private dense rows: asked for, or (AUTO) output rows of at most 64 keys that receive
  // on average kRowsMinPerOutput products or more per output cell.
  const bool lane_rows = !wide && pl.FY <= kLaneRowMax &&
                         (o.accumulator == STC_ACC_ROWS ||
                          (o.accumulator == STC_ACC_AUTO && h.P >= kRowsMinPerOutput * pl.FX * pl.FY));
  if (lane_rows) r->stats.accumulator = STC_ACC_ROWS;

  uint64_t out_cap = hg.out_cap;
  HugeGroups hh{};
  hh.count = lane_rows ? 0u : hg.count[kMaxClasses];
  hh.countp = gc->count + kMaxClasses;
  hh.list = b.huge_list;
  hh.off = b.huge_off;
  hh.cap = b.huge_cap;
  const uint32_t nstream = (dense_rows && !lane_rows) ? hg.count[kMaxClasses + 1] : 0u;
  bool direct = !wide && !lane_rows && out_cap < 0xffffffffull && o.accumulator != STC_ACC_HASH_SCAN;
  STC_TRY(ar.alloc_own(&r->coords, out_cap * (size_t)pl.ocols));
  STC_TRY(ar.alloc_own(&r->vals, out_cap));
  BatchOut* dbo = nullptr;
  STC_TRY(ar.alloc(&dbo, 1));
  if (hh.count) {
    STC_TRY(ar.alloc(&hh.keys, hg.huge_slots));
    STC_TRY(ar.alloc(&hh.vals, hg.huge_slots));
    STC_CUDA(cudaMemsetAsync(hh.keys, 0xff, hg.huge_slots * sizeof(u64), s));
    STC_CUDA(cudaMemsetAsync(hh.vals, 0, hg.huge_slots * sizeof(double), s));
  }
  BatchOut bo_here{};
  static_assert(sizeof(BatchOut) <= kPinnedBytes / 2, "a page-locked block holds the counters and a descriptor");
  BatchOut& hbo = pin.p ? *reinterpret_cast<BatchOut*>(static_cast<char*>(pin.p) + kPinnedBytes / 2) : bo_here;
  hbo = BatchOut{};
  hbo.FY = pl.FY;
  hbo.out_cap = out_cap;
  hbo.coords = r->coords;
  hbo.vals = r->vals;
  hbo.op = pl.op;
  pin.busy = true;
  STC_CUDA(cudaMemcpyAsync(dbo, &hbo, sizeof(BatchOut), cudaMemcpyHostToDevice, s));
  GroupArgs a{};
  a.goff = goff;
  a.gx = gx;
  a.yfk = pr.yfk;
  a.yv = pr.yv;
  a.FY = pl.FY;
  a.op = pl.op;
  a.coords = r->coords;
  a.vals = r->vals;
  a.out_cap = out_cap;
  a.nz = &pr.ctr->nz;
  a.status = &pr.ctr->status;
  a.bout = dbo;
  a.bnz = &pr.ctr->nz;
  StreamArgs sa{};
  if (nstream) {
    STC_TRY(ar.alloc(&sa.holes, stream_max_holes(nstream, nseg)));
    sa.nholes = &gc->nholes;
    sa.hole_total = &gc->holes;
    sa.ny_entries = (uint32_t)Y->nnz;
  }
  if (lane_rows) {
    STC_CUDA(launch_group_lanerow(a, pl.FX, (uint32_t)pl.FY, h.P, h.ns, ctx->sms, s));
  } else {
    STC_CUDA(launch_group_classes(a, wide, direct, b, hg.count, ctx->sms, s));
    STC_CUDA(launch_group_huge(a, hh, wide, ctx->sms, s));
  }
  if (dense_rows && !lane_rows) {
    STC_CUDA(launch_group_dense(a, pr.yoff, nseg, seg, b.dense_list[2], hg.count[kMaxClasses + 3], b.dense_list[1],
                                hg.count[kMaxClasses + 2], ctx->sms, s));
    STC_CUDA(launch_group_stream(a, pr.yoff, nseg, seg, b.dense_list[0], nstream, sa, ctx->sms, s));
  }
  tm.mark(4);
  // The holes are filled from the output's end before their number is known here, in one round for
  // as many positions as are to be expected; more take further rounds below. The scratch is one word
  // per position; where there is no memory for it, an array of the grouped X serves, which nothing
  // reads any more.
  HoleRound rd{};
  auto fill = [&]() -> stc_status {
    STC_CUDA(launch_hole_fill(sa.holes, sa.nholes, &pr.ctr->nz, &gc->holes, rd, gc->fill_counters, r->coords, r->vals,
                              pl.ocols, &pr.ctr->status, ctx->sms, s));
    tm.mark(5);
    return STC_OK;
  };
  if (nstream) {
    rd.win = expected_holes(ctx, nstream, out_cap);
    if (rd.win <= (uint64_t)nX || ar.alloc(&rd.dst, (size_t)rd.win) != STC_OK) {
      if (rd.win > (uint64_t)nX) g_last_error.clear();
      rd.win = std::min<uint64_t>(rd.win, (uint64_t)nX);
      rd.dst = gx.ystart;
    }
    STC_TRY(fill());
  }
  CallCounters hc2{};
  STC_TRY(read_counters(pr, pin, hc2));
  const u64 holes = hc2.g.holes;
  r->nnz = (int64_t)(hc2.c.nz - holes);
  for (rd.at = rd.win; rd.at < holes; rd.at += rd.win) {
    rd.base = hc2.g.fill_counters[1];
    STC_TRY(fill());
    STC_TRY(read_counters(pr, pin, hc2));
  }
  if (hc2.g.fill_counters[0] != hc2.g.fill_counters[1])
    return fail(STC_ERR_CUDA, "holes and entries to fill them do not match");
  r->stats.out_capacity = out_cap;
  r->mem = adopt(ar, ctx, s, {r->coords, r->vals});
  return STC_OK;
}

// AUTO: one global table when the output key space is small (the table stays in L2),
// per-group shared-memory tables when X's free keys can be counted directly.
// GROUPED pays per X free key (a counting sort over F_X bins) and per group (a table and an
// output reservation), so it needs groups with work in them: at most about two free keys per
// X entry, or up to sixteen when each X entry meets many Y entries (n_Y >= 16 K).
int pick_strategy(const Plan& pl, const stc_coo* X, const stc_coo* Y, int requested) {
  if (requested != STC_STRATEGY_AUTO) return requested;
  if (pl.F <= (1ull << 22)) return STC_STRATEGY_GLOBAL;
  if (pl.FX > kMaxDirectBins) return STC_STRATEGY_GLOBAL;
  const uint64_t nX = (uint64_t)X->nnz, nY = (uint64_t)Y->nnz;
  if (pl.FX <= 2 * nX + (1ull << 20)) return STC_STRATEGY_GROUPED;
  if (nY >= 16 * pl.K && pl.FX <= 16 * nX + (1ull << 20)) return STC_STRATEGY_GROUPED;
  return STC_STRATEGY_GLOBAL;
}

// FNV-1a over what fixes a contraction's shape: the operands' shapes and entry counts, the mode
// lists, the output order and form.
uint64_t shape_signature(const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx, const int32_t* cy,
                         const int32_t* out_order, int32_t oz, int32_t keys_out) {
  uint64_t h = 0xcbf29ce484222325ull;
  auto mix = [&](uint64_t v) {
    for (int i = 0; i < 8; i++) {
      h ^= (v >> (8 * i)) & 0xff;
      h *= 0x100000001b3ull;
    }
  };
  mix((uint64_t)X->order);
  for (int j = 0; j < X->order; j++) mix((uint64_t)X->shape[j]);
  mix((uint64_t)Y->order);
  for (int j = 0; j < Y->order; j++) mix((uint64_t)Y->shape[j]);
  mix((uint64_t)X->nnz);
  mix((uint64_t)Y->nnz);
  mix((uint64_t)m);
  for (int i = 0; i < m; i++) mix(((uint64_t)(uint32_t)cx[i] << 32) | (uint32_t)cy[i]);
  mix(out_order ? 1u : 0u);
  if (out_order)
    for (int q = 0; q < oz; q++) mix((uint64_t)(uint32_t)out_order[q]);
  mix((uint64_t)keys_out);
  return h;
}

bool rows_remembered(stc_ctx* ctx, uint64_t sig) {
  std::lock_guard<std::mutex> lk(ctx->rows_mu);
  return ctx->rows_shapes.count(sig) != 0;
}

void rows_note(stc_ctx* ctx, uint64_t sig, bool rows) {
  std::lock_guard<std::mutex> lk(ctx->rows_mu);
  if (!rows) {
    ctx->rows_shapes.erase(sig);
    return;
  }
  if (ctx->rows_shapes.size() >= 4096) ctx->rows_shapes.clear();  // a bound, not an eviction policy
  ctx->rows_shapes.insert(sig);
}

// Whether the contract keys are renumbered to dense ids before grouping (Section 4.1.2):
// always past the direct-counting limit, and under AUTO when the key space dwarfs the inputs
// (the K-bin histogram and scan would cost more than the renumbering).
bool use_dense_ids(const Plan& pl, const stc_coo* X, const stc_coo* Y, int mode) {
  if (pl.K > kMaxDirectBins) return true;
  if (pl.K <= 1 || mode == STC_IDS_DIRECT) return false;
  if (mode == STC_IDS_DENSE) return true;
  return pl.K > (1ull << 22) && pl.K > 8ull * (uint64_t)(X->nnz + Y->nnz);
}

// Whether AUTO numbers the contract keys through a bitmap of the key space instead (KeyPlan::idmap):
// the keys that would be renumbered, and those that direct counting would count in more than four
// times as many bins as Y has entries. Two bits per key of bitmap and ranks are cleared and scanned; past
// 2^28 keys, or 256 per entry, the table of id_insert_rows_kernel is the faster. Lengths 2,000 x 3,000 x
// 14,000 x 17,000, 3e6 entries, K = 4.2e7: 1.07 -> 0.80 ms for the contraction, by direct counting
// before; 63,891 x 63,890 x 1,847, 7.4e5 entries, K = 1.2e8: 0.42 -> 0.35, by the table. Two tensors of
// 2e6 entries each, by the map and by the table: K = 2^26 0.57 and 0.71, 2^28 0.65 and 0.67, 2^29 0.74
// and 0.67; of 4e6 each over 100 x 100 outputs 0.55 and 0.77, 0.64 and 0.76, 0.79 and 0.75.
bool use_id_map(const stc_ctx* ctx, const Plan& pl, const stc_coo* X, const stc_coo* Y, int mode, bool dense_ids) {
  const uint64_t nX = (uint64_t)X->nnz, nY = (uint64_t)Y->nnz;
  if (mode != STC_IDS_AUTO || nX == 0 || nY == 0 || nY >= kMaxDirectBins - 1) return false;
  if (pl.K <= (1ull << 22) || pl.K <= 4 * nY || pl.K > (1ull << 28) || pl.K > 256 * (nX + nY)) return false;
  // The map may take more memory than the table of the keys met: a budget that held the table holds.
  if (dense_ids && ctx->budget) return false;
  // Where the strategy depends on how many entries share a key, the table's count decides it.
  return !dense_ids || pl.FX <= 2 * nX + (1ull << 20) || pl.FX > 16 * nX + (1ull << 20);
}

// A contraction whose contract key space is too large to count directly, restated over
// dense ids (Section 4.1.2): the distinct contract keys of Y are numbered 0..D-1, and X and
// Y are rewritten with their free modes (ascending, lengths unchanged) followed by one
// paired mode of length D + 1 holding the id. X entries whose key Y lacks take the id D,
// which no Y entry has, so they form no products, as in Eq. 2. The free modes keep their
// order, so the output modes and out_order mean the same for the rewritten pair.
struct Relabelled {
  Arena ar;  // the rewritten coordinates
  StageTimer tm;
  std::vector<int64_t> xs, ys;
  stc_coo X{}, Y{};
  int32_t cx = 0, cy = 0;
  uint64_t ids = 0;  // D
  unsigned launches = 0;
  Relabelled(stc_ctx* c, cudaStream_t s) : ar(c, s) {}
};

stc_status relabel(stc_ctx* ctx, const stc_coo* X, const stc_coo* Y, const Plan& pl, bool record,
                   cudaStream_t s, Relabelled& rl) {
  rl.tm.start(record, s);
  const uint64_t slots = id_table_slots(Y->nnz);
  uint32_t fx = 0, fy = 0;
  int nfx = 0, nfy = 0;
  for (int j = 0; j < X->order; j++)
    if (pl.kx.cstride[j] == 0) fx |= 1u << j, rl.xs.push_back(X->shape[j]), nfx++;
  for (int j = 0; j < Y->order; j++)
    if (pl.ky.cstride[j] == 0) fy |= 1u << j, rl.ys.push_back(Y->shape[j]), nfy++;
  int32_t *xc = nullptr, *yc = nullptr;
  STC_TRY(rl.ar.alloc(&xc, (size_t)X->nnz * (nfx + 1)));
  STC_TRY(rl.ar.alloc(&yc, (size_t)Y->nnz * (nfy + 1)));
  uint32_t h[2] = {0, 0};
  {
    Arena tab(ctx, s);  // released (stream-ordered) once the rewrites are queued
    IdTable t{};
    uint32_t *scr = nullptr, *status = nullptr;
    t.slots = slots;
    STC_TRY(tab.alloc(&t.keys, slots));
    STC_TRY(tab.alloc(&t.flags, slots + 1));
    STC_TRY(tab.alloc(&t.prefix, slots + 2));
    STC_TRY(tab.alloc(&scr, (size_t)scan_scratch_elems((int64_t)slots + 1)));
    STC_TRY(tab.alloc(&status, 1));
    STC_CUDA(cudaMemsetAsync(t.keys, 0xff, slots * sizeof(u64), s));
    STC_CUDA(cudaMemsetAsync(t.flags + slots, 0, sizeof(uint32_t), s));
    STC_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
    STC_CUDA(launch_id_insert_rows(Y->coords, Y->nnz, pl.ky, t, status, ctx->sms, s));
    STC_CUDA(launch_id_number(t, scr, ctx->sms, s));
    STC_CUDA(launch_id_rewrite_rows(X->coords, X->nnz, pl.kx, fx, nfx, t, xc, status, ctx->sms, s));
    STC_CUDA(launch_id_rewrite_rows(Y->coords, Y->nnz, pl.ky, fy, nfy, t, yc, status, ctx->sms, s));
    STC_CUDA(cudaMemcpyAsync(&h[0], status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    STC_CUDA(cudaMemcpyAsync(&h[1], t.prefix + slots + 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    STC_CUDA(cudaStreamSynchronize(s));
  }
  rl.tm.mark(0);
  STC_TRY(status_word(h[0]));
  rl.ids = h[1];
  if (rl.ids + 1 > kMaxDirectBins)
    return fail(STC_ERR_UNSUPPORTED, "Y has %llu distinct contract keys; at most 2^26 - 1 are supported",
                (unsigned long long)rl.ids);
  rl.xs.push_back((int64_t)rl.ids + 1);
  rl.ys.push_back((int64_t)rl.ids + 1);
  rl.X = stc_coo{nfx + 1, rl.xs.data(), X->nnz, xc, X->vals};
  rl.Y = stc_coo{nfy + 1, rl.ys.data(), Y->nnz, yc, Y->vals};
  rl.cx = nfx;
  rl.cy = nfy;
  rl.launches = take_launches();
  return STC_OK;
}

}  // namespace

DeviceBlock::~DeviceBlock() {
  DeviceGuard g(ctx->device);
  for (auto& p : parts) {
    cudaFreeAsync(p.first, stream);
    ctx->held -= p.second;
  }
}

namespace stc {
// Lets other translation units of the library set the calling thread's last error.
stc_status report_error(stc_status s, const char* msg) { return fail(s, "%s", msg); }
int ctx_device(const stc_ctx* ctx) { return ctx->device; }
// Results handed out by a server outlive its streams: their memory is returned on the legacy
// default stream instead (their data is complete when they are handed out).
void result_release_on_default_stream(stc_result* r) {
  if (!r) return;
  r->stream = nullptr;
  if (r->mem) r->mem->stream = nullptr;
}
}  // namespace stc

namespace {

// ---------------------------------------------------------------- batches
// The device state of one batch of problems: descriptors and every scratch array, all sized
// from totals the host knows before any kernel runs (entries of X and Y, contract-key bins,
// problems). Filled by batch_setup, consumed by the launch sequence that follows.
struct BatchDev {
  int32_t n = 0;
  std::vector<Plan> plans;
  std::vector<BatchOut> hbo;  // per problem: F_Y and the output plan (positions filled later)
  BatchArgs ba{};
  GroupedX gx{};
  Bins b{};
  GroupCounters* gc = nullptr;
  Counters* ctr = nullptr;
  u64* per = nullptr;          // [3n]: products, output bound, output count per problem
  uint32_t* gprob = nullptr;
  u64* gfk = nullptr;
  BatchOut* dbo = nullptr;     // [n]
  int32_t* doz = nullptr;      // [n] output order per problem
  u64* offs = nullptr;         // [2n + 2] value and coordinate offsets of a captured run
  BatchLayoutArgs* dargs = nullptr;
  bool wide = false;
  int depth = 0;  // expansion split of the CTA tables (TuneChoice::depth)
  int64_t total_x = 0, total_y = 0;
  int tune_bucket = 0;
};

// Plans, descriptors and scratch of a batch (no kernel runs; the descriptors are copied on s).
stc_status batch_setup(stc_ctx* ctx, int32_t n, const stc_problem* problems, const stc_opts& o, Arena& ar,
                       cudaStream_t s, BatchDev& bd) {
  bd.n = n;
  bd.plans.assign(n, Plan{});
  std::vector<BatchProb> hb(n);
  std::vector<int64_t> xrow(n + 1, 0), yrow(n + 1, 0);
  std::vector<u64> fxoff(n + 1, 0);
  std::vector<int32_t> oz(n);
  unsigned __int128 bins = 0, fxsum = 0;
  bool key32 = true;
  for (int32_t i = 0; i < n; i++) {
    const stc_problem& q = problems[i];
    STC_TRY(make_plan(&q.X, &q.Y, q.ncontract, q.cx, q.cy, q.out_order, bd.plans[i]));
    const Plan& pl = bd.plans[i];
    if (pl.FY > 0xffffffffull) key32 = false;
    BatchProb& b = hb[i];
    b = BatchProb{};
    b.xc = q.X.coords;
    b.xv = q.X.vals;
    b.yc = q.Y.coords;
    b.yv = q.Y.vals;
    b.kx = pl.kx;
    b.ky = pl.ky;
    b.koff = (u64)bins;
    b.fxoff = (u64)fxsum;
    b.FY = pl.FY;
    oz[i] = pl.oz;
    bins += pl.K;
    fxsum += pl.FX;
    xrow[i + 1] = xrow[i] + q.X.nnz;
    yrow[i + 1] = yrow[i] + q.Y.nnz;
    fxoff[i + 1] = (u64)fxsum;
    if (bins > kMaxDirectBins) return fail(STC_ERR_UNSUPPORTED, "the batch's contract key spaces exceed 2^26 bins");
    if (fxsum >= ((unsigned __int128)1 << 63)) return fail(STC_ERR_KEY_OVERFLOW, "the batch's X free key spaces exceed 2^63");
    if (xrow[i + 1] > STC_MAX_NNZ || yrow[i + 1] > STC_MAX_NNZ)
      return fail(STC_ERR_INVALID_ARG, "the batch holds more than STC_MAX_NNZ entries of X or of Y");
  }
  bd.total_x = xrow[n];
  bd.total_y = yrow[n];
  bd.tune_bucket = log2_floor((uint64_t)(bd.total_x + bd.total_y)) * 32 + std::min(31, log2_floor((uint64_t)n));
  bd.hbo.assign(n, BatchOut{});
  for (int32_t i = 0; i < n; i++) {
    bd.hbo[i].FY = bd.plans[i].FY;
    bd.hbo[i].op = bd.plans[i].op;
  }

  BatchArgs& ba = bd.ba;
  ba = BatchArgs{};
  ba.n = n;
  ba.total_x = bd.total_x;
  ba.total_y = bd.total_y;
  ba.bins = (u64)bins;
  ba.key32 = key32;
  BatchProb* dpb = nullptr;
  int64_t *dxrow = nullptr, *dyrow = nullptr;
  u64* dfxoff = nullptr;
  STC_TRY(ar.alloc(&dpb, (size_t)n));
  STC_TRY(ar.alloc(&dxrow, (size_t)n + 1));
  STC_TRY(ar.alloc(&dyrow, (size_t)n + 1));
  STC_TRY(ar.alloc(&dfxoff, (size_t)n + 1));
  STC_TRY(ar.alloc(&bd.ctr, 1));
  STC_TRY(ar.alloc(&bd.per, 3 * (size_t)n));
  STC_TRY(ar.alloc(&bd.dbo, (size_t)n));
  STC_TRY(ar.alloc(&bd.doz, (size_t)n));
  STC_TRY(ar.alloc(&bd.offs, 2 * (size_t)n + 2));
  STC_TRY(ar.alloc(&bd.dargs, 1));
  STC_CUDA(cudaMemcpyAsync(dpb, hb.data(), n * sizeof(BatchProb), cudaMemcpyHostToDevice, s));
  STC_CUDA(cudaMemcpyAsync(dxrow, xrow.data(), (n + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  STC_CUDA(cudaMemcpyAsync(dyrow, yrow.data(), (n + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  STC_CUDA(cudaMemcpyAsync(dfxoff, fxoff.data(), (n + 1) * sizeof(u64), cudaMemcpyHostToDevice, s));
  STC_CUDA(cudaMemcpyAsync(bd.dbo, bd.hbo.data(), n * sizeof(BatchOut), cudaMemcpyHostToDevice, s));
  STC_CUDA(cudaMemcpyAsync(bd.doz, oz.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  ba.pb = dpb;
  ba.xrow = dxrow;
  ba.yrow = dyrow;
  ba.fxoff = dfxoff;
  ba.P = &bd.ctr->P;
  ba.Pp = bd.per;
  ba.pcap = bd.per + n;
  ba.status = &bd.ctr->status;

  const int64_t total_x = bd.total_x, total_y = bd.total_y;
  const u64 gcap = pow2_at_least(std::max<u64>(64, 2 * (u64)std::max<int64_t>(total_x, 1)));
  STC_TRY(ar.alloc(&ba.ycnt, ba.bins));
  STC_TRY(ar.alloc(&ba.yoff, ba.bins + 1));
  STC_TRY(ar.alloc(&ba.ycur, ba.bins));
  if (key32) {
    uint32_t* k = nullptr;
    STC_TRY(ar.alloc(&k, (size_t)total_y));
    ba.yfk = k;
    STC_TRY(ar.alloc(&ba.yuniq, (size_t)std::max<int64_t>(total_y, 1)));
  } else {
    u64* k = nullptr;
    STC_TRY(ar.alloc(&k, (size_t)total_y));
    ba.yfk = k;
  }
  STC_TRY(ar.alloc(&ba.yv, (size_t)total_y));
  STC_TRY(ar.alloc(&ba.sv.fk, (size_t)total_x));
  STC_TRY(ar.alloc(&ba.sv.ystart, (size_t)total_x));
  STC_TRY(ar.alloc(&ba.sv.w, (size_t)total_x));
  STC_TRY(ar.alloc(&ba.sv.v, (size_t)total_x));
  ba.sv.count = &bd.ctr->ns;
  STC_TRY(ar.alloc(&ba.idmap.keys, gcap));
  ba.idmap.mask = gcap - 1;
  STC_TRY(ar.alloc(&ba.gid, (size_t)total_x));
  STC_TRY(ar.alloc(&ba.gcnt, gcap));
  STC_TRY(ar.alloc(&ba.goff, gcap + 1));
  STC_TRY(ar.alloc(&ba.gcur, gcap));
  STC_TRY(ar.alloc(&ba.scan_scratch32, (size_t)std::max(scan_scratch_elems((int64_t)ba.bins),
                                                          scan_scratch_elems((int64_t)gcap))));

  // Grouped X, the class lists and counters.
  bd.wide = !key32;
  const int ncls = bd.wide ? kNumClasses64 : kNumClasses32;
  const size_t maxg = (size_t)std::max<int64_t>(total_x, 1);
  STC_TRY(ar.alloc(&bd.gx.ystart, maxg));
  STC_TRY(ar.alloc(&bd.gx.w, maxg));
  STC_TRY(ar.alloc(&bd.gx.v, maxg));
  STC_TRY(ar.alloc(&bd.gc, 1));
  STC_TRY(ar.alloc(&bd.gprob, gcap));
  STC_TRY(ar.alloc(&bd.gfk, gcap));
  Bins& b = bd.b;
  b = Bins{};
  b.nclasses = ncls;
  for (int c = 0; c < ncls; c++) STC_TRY(ar.alloc(&b.list[c], maxg));
  // The two-pass lists, unless the caller asks for scanned tables or a budget could refuse them (the
  // hash tables take the same groups).
  if (!bd.wide && o.accumulator != STC_ACC_HASH_SCAN && ctx->budget == 0)
    for (int d = 0; d < 3; d++) STC_TRY(ar.alloc(&b.dense_list[d], maxg));
  STC_TRY(ar.alloc(&b.huge_list, maxg));
  STC_TRY(ar.alloc(&b.huge_off, maxg));
  STC_TRY(ar.alloc(&b.huge_cap, maxg));
  b.count = bd.gc->count;
  b.huge_slots = &bd.gc->huge_slots;
  b.out_cap = &bd.gc->out_cap;
  b.status = &bd.ctr->status;
  return STC_OK;
}

// Class thresholds of a tuning choice: a group of bound t goes to the first class with
// t <= alpha * slots; with warp_max 256 the 1024-slot warp class takes no groups (its groups go
// to the CTA classes). depth selects the expansion split of the CTA tables.
void batch_set_choice(BatchDev& bd, const TuneChoice& ch) {
  const ClassShape* shapes = bd.wide ? kClassShapes64 : kClassShapes32;
  for (int c = 0; c < bd.b.nclasses; c++) bd.b.tmax[c] = (u64)(ch.alpha * shapes[c].slots);
  if (ch.warp_max < 1024) bd.b.tmax[1] = bd.b.tmax[0];
  bd.depth = ch.depth;
}

// The batch up to its per-group bins: counters cleared, Y grouped, X surveyed, grouped by
// (problem, X free key) and binned. Only enqueues work on s (no host reads).
stc_status batch_front(stc_ctx* ctx, BatchDev& bd, cudaStream_t s, StageTimer& tm) {
  BatchArgs& ba = bd.ba;
  const int32_t n = bd.n;
  STC_CUDA(cudaMemsetAsync(bd.ctr, 0, sizeof(Counters), s));
  STC_CUDA(cudaMemsetAsync(bd.per, 0, 3 * n * sizeof(u64), s));
  if (ba.bins) STC_CUDA(cudaMemsetAsync(ba.ycnt, 0, ba.bins * sizeof(uint32_t), s));
  STC_CUDA(cudaMemsetAsync(ba.idmap.keys, 0xff, (ba.idmap.mask + 1) * sizeof(u64), s));
  STC_CUDA(cudaMemsetAsync(ba.gcnt, 0, (ba.idmap.mask + 1) * sizeof(uint32_t), s));
  STC_CUDA(launch_batch_prepare(ba, ctx->sms, s));
  tm.mark(1);
  STC_CUDA(cudaMemsetAsync(bd.gc, 0, sizeof(GroupCounters), s));
  STC_CUDA(launch_batch_group(ba, bd.gx, bd.b, bd.gprob, bd.gfk, ctx->sms, s));
  tm.mark(2);
  return STC_OK;
}

// GroupArgs of the batch's accumulation kernels.
GroupArgs batch_group_args(const BatchDev& bd) {
  GroupArgs a{};
  a.goff = bd.ba.goff;
  a.gx = bd.gx;
  a.yfk = bd.ba.yfk;
  a.yv = bd.ba.yv;
  a.status = &bd.ctr->status;
  a.nz = &bd.ctr->nz;
  a.bout = bd.dbo;
  a.bnz = bd.per + 2 * bd.n;
  a.gprob = bd.gprob;
  a.gfk = bd.gfk;
  a.yuniq = bd.ba.yuniq;
  return a;
}

// One result per problem over a shared output block (offsets in elements).
void batch_results(stc_ctx* ctx, cudaStream_t s, const BatchDev& bd, const std::shared_ptr<DeviceBlock>& blk,
                   double* vals, int32_t* coords, const u64* voff, const u64* coff, const u64* hper,
                   const stc_stats& common, stc_result** outs) {
  const int32_t n = bd.n;
  for (int32_t i = 0; i < n; i++) {
    stc_result* r = new stc_result;
    r->ctx = ctx;
    r->stream = s;
    r->order = bd.plans[i].oz;
    r->shape = bd.plans[i].zshape;
    r->nnz = (int64_t)hper[2 * n + i];
    r->coords = coords ? coords + coff[i] : nullptr;
    r->vals = vals ? vals + voff[i] : nullptr;
    r->mem = blk;
    r->stats = common;
    r->stats.products = hper[i];
    r->stats.out_capacity = hper[n + i];
    ctx->live_results++;
    outs[i] = r;
  }
}

// Sizes one run of a batch needed, read back after it: what a captured run must provide.
struct BatchSizes {
  u64 vals = 0;     // output entries over all problems (sum of the exact bounds)
  u64 coords = 0;   // output coordinates over all problems
  u64 huge = 0;     // overflow-table slots
  u64 maxcap = 0;   // largest bound of one problem
};

// The rest of a batch with the host in the loop: the bins' counters are read back, one output
// block of the exact size is taken from `run`, the groups are accumulated, and the output
// counts are read back into hper[2n, 3n). bd.b.tmax must be set. tune_cand >= 0 times the
// accumulation for the autotuner.
stc_status batch_finish_eager(stc_ctx* ctx, BatchDev& bd, const stc_opts& o, Arena& run, cudaStream_t s,
                              StageTimer& tm, int tune_cand, bool* timed, std::vector<u64>& hper, BatchSizes& sz,
                              double** vals_out, int32_t** coords_out, std::vector<u64>& voff,
                              std::vector<u64>& coff) {
  const int32_t n = bd.n;
  Counters h{};
  GroupCounters hg{};
  hper.assign(3 * (size_t)n, 0);
  STC_CUDA(cudaMemcpyAsync(&hg, bd.gc, sizeof(GroupCounters), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaMemcpyAsync(hper.data(), bd.per, 2 * n * sizeof(u64), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaMemcpyAsync(&h, bd.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaStreamSynchronize(s));
  STC_TRY(status_word(h.status));
  tm.mark(3);

  // One output allocation: every problem's values, then every problem's coordinates.
  voff.assign(n + 1, 0);
  coff.assign(n + 1, 0);
  sz = BatchSizes{};
  for (int32_t i = 0; i < n; i++) {
    voff[i + 1] = voff[i] + hper[n + i];
    coff[i + 1] = coff[i] + hper[n + i] * (u64)bd.plans[i].oz;
    sz.maxcap = std::max<u64>(sz.maxcap, hper[n + i]);
  }
  sz.vals = voff[n];
  sz.coords = coff[n];
  sz.huge = hg.huge_slots;
  double* vals = nullptr;
  int32_t* coords = nullptr;
  STC_TRY(run.alloc_own(&vals, voff[n]));
  STC_TRY(run.alloc_own(&coords, coff[n]));
  std::vector<BatchOut> hbo = bd.hbo;
  for (int32_t i = 0; i < n; i++) {
    hbo[i].out_cap = hper[n + i];
    hbo[i].coords = coords ? coords + coff[i] : nullptr;
    hbo[i].vals = vals ? vals + voff[i] : nullptr;
  }
  STC_CUDA(cudaMemcpyAsync(bd.dbo, hbo.data(), n * sizeof(BatchOut), cudaMemcpyHostToDevice, s));
  HugeGroups hh{};
  hh.count = hg.count[kMaxClasses];
  hh.countp = bd.gc->count + kMaxClasses;
  hh.list = bd.b.huge_list;
  hh.off = bd.b.huge_off;
  hh.cap = bd.b.huge_cap;
  if (hh.count) {
    STC_TRY(run.alloc(&hh.keys, hg.huge_slots));
    STC_TRY(run.alloc(&hh.vals, hg.huge_slots));
    STC_CUDA(cudaMemsetAsync(hh.keys, 0xff, hg.huge_slots * sizeof(u64), s));
    STC_CUDA(cudaMemsetAsync(hh.vals, 0, hg.huge_slots * sizeof(double), s));
  }
  const GroupArgs a = batch_group_args(bd);
  if (h.P > 0) {
    const bool direct = !bd.wide && sz.maxcap < 0xffffffffull && o.accumulator != STC_ACC_HASH_SCAN;
    tune_mark(ctx, bd.tune_bucket, tune_cand, false, s);
    STC_CUDA(launch_group_classes(a, bd.wide, direct, bd.b, hg.count, ctx->sms, s, bd.depth));
    if (bd.b.dense_list[0]) STC_CUDA(launch_group_twopass(a, bd.b, hg.count, ctx->sms, s));
    STC_CUDA(launch_group_huge(a, hh, bd.wide, ctx->sms, s));
    tune_mark(ctx, bd.tune_bucket, tune_cand, true, s);
    if (timed) *timed = true;
  }
  tm.mark(4);
  STC_CUDA(cudaMemcpyAsync(hper.data() + 2 * n, bd.per + 2 * n, n * sizeof(u64), cudaMemcpyDeviceToHost, s));
  Counters h2{};
  STC_CUDA(cudaMemcpyAsync(&h2, bd.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaStreamSynchronize(s));
  STC_TRY(status_word(h2.status));
  *vals_out = vals;
  *coords_out = coords;
  return STC_OK;
}

}  // namespace

// A prepared batch: the problems' descriptors and every scratch array held on the device
// across runs, and, once the load factor is settled, the whole launch sequence of a run
// captured in one CUDA graph that each later run replays.
struct stc_batch_plan {
  stc_ctx* ctx = nullptr;
  stc_opts opts{};
  int32_t n = 0;
  std::vector<stc_problem> probs;
  std::vector<std::vector<int64_t>> shapes;
  std::vector<std::vector<int32_t>> modes;
  cudaStream_t stream = nullptr;  // scratch allocation and graph capture
  std::unique_ptr<Arena> scratch;
  BatchDev bd;
  BatchSizes sizes{};
  TuneChoice choice{0.0, 1024, 0};  // the settled choice the graph was captured with (alpha 0: none)
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  unsigned graph_launches = 0;
  u64* huge_keys = nullptr;
  double* huge_vals = nullptr;
  u64 huge_cap = 0;
  // pinned host mirrors written by the captured copies
  BatchLayoutArgs* h_args = nullptr;
  u64* h_per = nullptr;
  Counters* h_ctr = nullptr;
  u64* h_offs = nullptr;
  GroupCounters* h_gc = nullptr;
  int64_t runs = 0, graph_runs = 0;
};

namespace {

// Captures one run of the plan's batch on the plan's stream: the layout arguments copied in,
// the front of the batch, the device-side output layout, every class kernel with its count read
// on the device, and the copies of the counters the host reads after the run.
stc_status plan_capture(stc_batch_plan* pl) {
  BatchDev& bd = pl->bd;
  stc_ctx* ctx = pl->ctx;
  cudaStream_t ps = pl->stream;
  // The overflow groups' table is the plan's, sized by the last run.
  if (pl->sizes.huge > pl->huge_cap) {
    const u64 cap = std::max<u64>(pl->sizes.huge, 64);
    STC_TRY(pl->scratch->alloc(&pl->huge_keys, cap));
    STC_TRY(pl->scratch->alloc(&pl->huge_vals, cap));
    pl->huge_cap = cap;
    STC_CUDA(cudaStreamSynchronize(ps));
  }
  pl->h_args->huge_keys = pl->huge_keys;
  pl->h_args->huge_vals = pl->huge_vals;
  pl->h_args->huge_cap = pl->huge_cap;
  batch_set_choice(bd, pl->choice);
  if (pl->exec) cudaGraphExecDestroy(pl->exec);
  if (pl->graph) cudaGraphDestroy(pl->graph);
  pl->exec = nullptr;
  pl->graph = nullptr;
  take_launches();
  STC_CUDA(cudaStreamBeginCapture(ps, cudaStreamCaptureModeThreadLocal));
  auto body = [&]() -> stc_status {
    StageTimer tm;
    const int32_t n = bd.n;
    STC_CUDA(cudaMemcpyAsync(bd.dargs, pl->h_args, sizeof(BatchLayoutArgs), cudaMemcpyHostToDevice, ps));
    STC_TRY(batch_front(ctx, bd, ps, tm));
    STC_CUDA(launch_batch_layout(n, bd.per + n, bd.doz, bd.dbo, bd.dargs, bd.offs, &bd.gc->huge_slots,
                                 bd.gc->count + kMaxClasses, &bd.ctr->status, ctx->sms, ps));
    const GroupArgs a = batch_group_args(bd);
    const bool direct =
        !bd.wide && pl->sizes.maxcap < 0x7fffffffull && pl->opts.accumulator != STC_ACC_HASH_SCAN;
    STC_CUDA(launch_group_classes(a, bd.wide, direct, bd.b, nullptr, ctx->sms, ps, bd.depth));
    if (bd.b.dense_list[0]) STC_CUDA(launch_group_twopass(a, bd.b, nullptr, ctx->sms, ps));
    HugeGroups hh{};
    hh.count = kCountOnDevice;
    hh.countp = bd.gc->count + kMaxClasses;
    hh.list = bd.b.huge_list;
    hh.off = bd.b.huge_off;
    hh.cap = bd.b.huge_cap;
    hh.keys = pl->huge_keys;
    hh.vals = pl->huge_vals;
    STC_CUDA(launch_group_huge(a, hh, bd.wide, ctx->sms, ps));
    STC_CUDA(cudaMemcpyAsync(pl->h_per, bd.per, 3 * n * sizeof(u64), cudaMemcpyDeviceToHost, ps));
    STC_CUDA(cudaMemcpyAsync(pl->h_ctr, bd.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, ps));
    STC_CUDA(cudaMemcpyAsync(pl->h_offs, bd.offs, (2 * n + 2) * sizeof(u64), cudaMemcpyDeviceToHost, ps));
    STC_CUDA(cudaMemcpyAsync(pl->h_gc, bd.gc, sizeof(GroupCounters), cudaMemcpyDeviceToHost, ps));
    return STC_OK;
  };
  const stc_status st = body();
  cudaGraph_t g = nullptr;
  const cudaError_t e = cudaStreamEndCapture(ps, &g);  // ends the capture whatever happened
  if (st != STC_OK) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return st;
  }
  STC_CUDA(e);
  pl->graph = g;
  STC_CUDA(cudaGraphInstantiate(&pl->exec, g, 0));
  pl->graph_launches = take_launches();
  return STC_OK;
}

// One run with the host in the loop (the first runs, while the load factor is tuned, and any
// run whose sizes outgrew the captured layout). Captures the graph once the load factor is
// settled.
stc_status plan_run_eager(stc_batch_plan* pl, cudaStream_t s, stc_result** outs) {
  BatchDev& bd = pl->bd;
  stc_ctx* ctx = pl->ctx;
  int tune_cand = -1;
  const bool given = pl->opts.group_load_factor > 0.0;
  const TuneChoice ch =
      given ? TuneChoice{pl->opts.group_load_factor, 1024, 0} : tune_pick(ctx, bd.tune_bucket, &tune_cand);
  struct TuneGuard {
    stc_ctx* c;
    int b, k;
    bool armed = true;
    ~TuneGuard() {
      if (armed) tune_abort(c, b, k);
    }
  } tune_guard{ctx, bd.tune_bucket, tune_cand};
  batch_set_choice(bd, ch);
  Arena run(ctx, s);
  StageTimer tm;
  tm.start(pl->opts.record_times != 0, s);
  take_launches();
  STC_TRY(batch_front(ctx, bd, s, tm));
  std::vector<u64> hper, voff, coff;
  double* vals = nullptr;
  int32_t* coords = nullptr;
  bool timed = false;
  STC_TRY(batch_finish_eager(ctx, bd, pl->opts, run, s, tm, tune_cand, &timed, hper, pl->sizes, &vals, &coords, voff,
                             coff));
  if (timed) tune_guard.armed = false;
  stc_stats common{};
  tm.collect(common);
  common.launches = take_launches();
  common.strategy = STC_STRATEGY_GROUPED;
  common.accumulator = STC_ACC_HASH;
  auto blk = adopt(run, ctx, s, {vals, coords});
  batch_results(ctx, s, bd, blk, vals, coords, voff.data(), coff.data(), hper.data(), common, outs);
  // Capture once the choice is settled (given, or the tuner's pick for this bucket).
  TuneChoice settled{0.0, 1024, 0};
  if (given) {
    settled = ch;
  } else {
    int probe = -1;
    const TuneChoice pick = tune_pick(ctx, bd.tune_bucket, &probe);
    if (probe < 0) settled = pick;
    else tune_abort(ctx, bd.tune_bucket, probe);
  }
  const bool changed = settled.alpha != pl->choice.alpha || settled.warp_max != pl->choice.warp_max ||
                       settled.depth != pl->choice.depth;
  if (settled.alpha > 0.0 && (!pl->exec || changed || pl->sizes.huge > pl->huge_cap)) {
    pl->choice = settled;
    const stc_status st = plan_capture(pl);
    if (st != STC_OK) {
      // The results of this run stand; the plan keeps running with the host in the loop.
      cudaGetLastError();
      pl->exec = nullptr;
    }
  }
  return STC_OK;
}

}  // namespace

namespace {
stc_status contract_impl(stc_ctx* ctx, const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx,
                         const int32_t* cy, const int32_t* out_order, const stc_opts* opts, void* stream,
                         stc_result** out, const std::vector<int64_t>* xfree);
}  // namespace

extern "C" {

const char* stc_status_string(stc_status s) {
  switch (s) {
    case STC_OK: return "ok";
    case STC_ERR_INVALID_ARG: return "invalid argument";
    case STC_ERR_SHAPE_MISMATCH: return "paired modes have different lengths";
    case STC_ERR_KEY_OVERFLOW: return "key space exceeds 64 bits";
    case STC_ERR_OUT_OF_MEMORY: return "out of device memory or over budget";
    case STC_ERR_TABLE_FULL: return "accumulation table full";
    case STC_ERR_TIMEOUT: return "timeout";
    case STC_ERR_CUDA: return "CUDA error";
    case STC_ERR_COORD_OUT_OF_RANGE: return "coordinate out of range";
    case STC_ERR_UNSUPPORTED: return "unsupported";
    case STC_ERR_CANCELLED: return "cancelled";
  }
  return "unknown status";
}

const char* stc_last_error(void) { return g_last_error.c_str(); }

stc_status stc_create(stc_ctx** out, int device, size_t mem_budget_bytes) {
  if (!out) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  *out = nullptr;
  int ndev = 0;
  STC_CUDA(cudaGetDeviceCount(&ndev));
  if (device < 0 || device >= ndev) return fail(STC_ERR_INVALID_ARG, "device %d of %d", device, ndev);
  DeviceGuard g(device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", device);
  stc_ctx* c = new stc_ctx;
  c->device = device;
  c->budget = mem_budget_bytes;
  cudaError_t e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, device);
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = device;
  if (e == cudaSuccess) e = cudaMemPoolCreate(&c->pool, &props);
  if (e == cudaSuccess) {
    uint64_t keep_all = UINT64_MAX;
    e = cudaMemPoolSetAttribute(c->pool, cudaMemPoolAttrReleaseThreshold, &keep_all);
  }
  if (e != cudaSuccess) {
    if (c->pool) cudaMemPoolDestroy(c->pool);
    delete c;
    return fail(STC_ERR_CUDA, "context set-up failed: %s", cudaGetErrorString(e));
  }
  *out = c;
  return STC_OK;
}

stc_status stc_destroy(stc_ctx* ctx) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  if (ctx->live_results.load() != 0)
    return fail(STC_ERR_INVALID_ARG, "%lld results of this context are still alive",
                (long long)ctx->live_results.load());
  DeviceGuard g(ctx->device);
  cudaDeviceSynchronize();
  for (auto& kv : ctx->tune)
    for (int c = 0; c < kTuneCand; c++) {
      if (kv.second.ev0[c]) cudaEventDestroy(kv.second.ev0[c]);
      if (kv.second.ev1[c]) cudaEventDestroy(kv.second.ev1[c]);
    }
  for (void* p : ctx->pins) cudaFreeHost(p);
  cudaMemPoolDestroy(ctx->pool);
  delete ctx;
  return STC_OK;
}

stc_status stc_contract(stc_ctx* ctx, const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx,
                        const int32_t* cy, const int32_t* out_order, const stc_opts* opts, void* stream,
                        stc_result** out) {
  return contract_impl(ctx, X, Y, m, cx, cy, out_order, opts, stream, out, nullptr);
}

}  // extern "C"

namespace {
// stc_contract, and the contraction of the split form of a tensor in key form (xfree: the
// lengths of that tensor's free modes; the operands then keep their roles).
stc_status contract_impl(stc_ctx* ctx, const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx,
                         const int32_t* cy, const int32_t* out_order, const stc_opts* opts, void* stream,
                         stc_result** out, const std::vector<int64_t>* xfree) {
  if (!ctx || !out) return fail(STC_ERR_INVALID_ARG, "ctx or out is NULL");
  *out = nullptr;
  const stc_opts o = opts ? *opts : stc_opts{};
  Plan pl;
  STC_TRY(make_plan(X, Y, m, cx, cy, out_order, pl, o.output_keys != 0, xfree));
  const double alpha = (o.load_factor > 0.0) ? o.load_factor : 0.5;
  if (!(alpha > 0.0 && alpha <= 0.9)) return fail(STC_ERR_INVALID_ARG, "load_factor %g outside (0, 0.9]", alpha);
  if (o.strategy < 0 || o.strategy > STC_STRATEGY_GROUPED)
    return fail(STC_ERR_INVALID_ARG, "unknown strategy %d", o.strategy);
  if (o.accumulator < 0 || o.accumulator > STC_ACC_ROWS)
    return fail(STC_ERR_INVALID_ARG, "unknown accumulator %d", o.accumulator);
  if (o.group_load_factor < 0.0 || o.group_load_factor > 0.9)
    return fail(STC_ERR_INVALID_ARG, "group_load_factor %g outside (0, 0.9]", o.group_load_factor);
  if (o.contract_ids < 0 || o.contract_ids > STC_IDS_DENSE)
    return fail(STC_ERR_INVALID_ARG, "unknown contract_ids %d", o.contract_ids);
  if (o.operands < 0 || o.operands > STC_OPERANDS_SWAPPED)
    return fail(STC_ERR_INVALID_ARG, "unknown operands %d", o.operands);
  if (o.table_shrink < 0 || o.table_shrink > 30)
    return fail(STC_ERR_INVALID_ARG, "table_shrink %d outside 0..30", o.table_shrink);
  if (o.probe != 0 && o.probe != 1 && o.probe != 4 && o.probe != 8)
    return fail(STC_ERR_INVALID_ARG, "probe %d is none of 0, 1, 4, 8", o.probe);
  const int probe = o.probe ? o.probe : kDefaultProbe;
  // A swap permutes the output modes back, so outputs in key form keep the operands as given.
  if (!xfree && (o.operands == STC_OPERANDS_SWAPPED ||
                 (o.operands == STC_OPERANDS_AUTO && !o.output_keys && (uint64_t)Y->nnz > 4 * (uint64_t)X->nnz))) {
    // Y (x) X has output modes (Y free, X free); map each requested mode onto that order.
    const int nfx = X->order - m, nfy = Y->order - m;
    std::vector<int32_t> oo(nfx + nfy);
    for (int q = 0; q < nfx + nfy; q++) {
      const int t = out_order ? out_order[q] : q;
      oo[q] = t < nfx ? nfy + t : t - nfx;
    }
    stc_opts inner = o;
    inner.operands = STC_OPERANDS_AS_GIVEN;
    STC_TRY(stc_contract(ctx, Y, X, m, cy, cx, oo.data(), &inner, stream, out));
    (*out)->stats.swapped = 1;
    return STC_OK;
  }
  const bool dense_ids = !xfree && use_dense_ids(pl, X, Y, o.contract_ids);
  if (!xfree && use_id_map(ctx, pl, X, Y, o.contract_ids, dense_ids)) {
    pl.id_map = true;
    pl.report_ids = dense_ids;
    pl.Kb = (uint64_t)Y->nnz;
  } else if (dense_ids) {
    DeviceGuard g(ctx->device);
    if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
    Relabelled rl(ctx, static_cast<cudaStream_t>(stream));
    take_launches();
    STC_TRY(relabel(ctx, X, Y, pl, o.record_times != 0, static_cast<cudaStream_t>(stream), rl));
    stc_opts inner = o;
    inner.contract_ids = STC_IDS_DIRECT;
    STC_TRY(stc_contract(ctx, &rl.X, &rl.Y, 1, &rl.cx, &rl.cy, out_order, &inner, stream, out));
    (*out)->stats.launches += rl.launches;
    (*out)->stats.contract_ids = rl.ids;
    rl.tm.collect((*out)->stats);
    return STC_OK;
  }
  int strategy = pick_strategy(pl, X, Y, o.strategy);
  // AUTO: a shape whose last run here was rows-heavy is grouped again (lane-private rows).
  const uint64_t sig = shape_signature(X, Y, m, cx, cy, out_order, pl.oz, o.output_keys);
  const bool rows_shape = o.strategy == STC_STRATEGY_AUTO && pl.FY <= kLaneRowMax && pl.FX <= kMaxDirectBins &&
                          (o.accumulator == STC_ACC_AUTO || o.accumulator == STC_ACC_ROWS);
  const bool by_memory = rows_shape && strategy == STC_STRATEGY_GLOBAL && rows_remembered(ctx, sig);
  if (by_memory) strategy = STC_STRATEGY_GROUPED;
  if (strategy == STC_STRATEGY_GROUPED && pl.FX > kMaxDirectBins)
    return fail(STC_ERR_UNSUPPORTED, "X free key space %llu exceeds %llu bins", (unsigned long long)pl.FX,
                (unsigned long long)kMaxDirectBins);

  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  StageTimer tm;
  tm.start(o.record_times != 0, s);
  take_launches();

  if (strategy == STC_STRATEGY_GROUPED) {
    stc_result* r = new stc_result;
    r->ctx = ctx;
    r->stream = s;
    r->order = pl.oz;
    r->keys_form = pl.keys_out;
    r->shape = pl.zshape;
    r->stats.strategy = STC_STRATEGY_GROUPED;
    const stc_status st = contract_grouped(ctx, ar, X, Y, pl, o, s, tm, r);
    if (st != STC_OK) {
      delete r;
      return st;
    }
    if (by_memory && r->stats.accumulator != STC_ACC_ROWS) rows_note(ctx, sig, false);
    tm.collect(r->stats);
    r->stats.launches = take_launches();
    ctx->live_results++;
    *out = r;
    return STC_OK;
  }

  Prepared pr;
  Pinned pin(ctx, s);
  STC_TRY(prepare(ctx, ar, X, Y, pl, Survey::kSurvivors, s, tm, pr));
  if (pl.F <= kGlobalFromF && o.table_shrink == 0 && X->nnz > 0 && Y->nnz > 0) {
    // A small output key space: the table and the output are sized from F itself, and P and
    // the survivor count are read on the device, so the call waits once, at its end.
    // Unless a load factor or a way of probing is asked for, the table is an array of the whole
    // space: no hashing and no claims (4096 x 64 outputs, 1.6e6 products, X of 2e7 entries: expansion 33
    // against 48 us).
    const bool whole = o.probe == 0 && o.load_factor == 0.0;
    const uint64_t cap = whole ? space_cells(ctx, pl.F)
                               : pow2_at_least(std::max<uint64_t>(64, (uint64_t)((double)pl.F / alpha) + 1));
    const uint64_t out_cap = std::min<uint64_t>(pl.F, cap);
    const int64_t nX = X->nnz;
    stc_result* r = new stc_result;
    r->ctx = ctx;
    r->stream = s;
    r->order = pl.oz;
    r->keys_form = pl.keys_out;
    r->shape = pl.zshape;
    r->stats.strategy = STC_STRATEGY_GLOBAL;
    auto run = [&]() -> stc_status {
      GlobalTable t{};
      u64* bpre = nullptr;
      if (!whole) STC_TRY(ar.alloc(&t.keys, cap));
      STC_TRY(ar.alloc(&t.vals, cap));
      STC_TRY(ar.alloc(&bpre, survivor_blocks(nX) + 1));
      STC_TRY(ar.alloc_own(&r->coords, out_cap * (size_t)pl.ocols));
      STC_TRY(ar.alloc_own(&r->vals, out_cap));
      t.mask = cap - 1;
      if (whole) {
        STC_CUDA(launch_clear_space(t, ctx->sms, s));
      } else {
        STC_CUDA(cudaMemsetAsync(t.keys, 0xff, cap * sizeof(u64), s));
        STC_CUDA(cudaMemsetAsync(t.vals, 0, cap * sizeof(double), s));
      }
      tm.mark(3);
      STC_CUDA(launch_expand_blocks(pr.sv, bpre, static_cast<const u64*>(pr.yfk), pr.yv, pl.FY, t,
                                    &pr.ctr->status, ctx->sms, s, probe));
      tm.mark(4);
      STC_CUDA(launch_compact_global(t, pl.op, r->coords, r->vals, out_cap, &pr.ctr->nz, &pr.ctr->status,
                                     ctx->sms, s));
      tm.mark(5);
      CallCounters hc{};
      STC_TRY(read_counters(pr, pin, hc));
      const Counters& h = hc.c;
      r->nnz = (int64_t)h.nz;
      r->stats.products = h.P;
      r->stats.survivors = h.ns;
      if (pl.report_ids) r->stats.contract_ids = hc.g.ids;
      r->stats.table_slots = cap;
      r->stats.out_capacity = out_cap;
      return STC_OK;
    };
    const stc_status st = run();
    if (st != STC_OK) {
      delete r;
      return st;
    }
    if (rows_shape && r->stats.products >= kRowsMinPerOutput * pl.F) rows_note(ctx, sig, true);
    r->mem = adopt(ar, ctx, s, {r->coords, r->vals});
    tm.collect(r->stats);
    r->stats.launches = take_launches();
    ctx->live_results++;
    *out = r;
    return STC_OK;
  }
  CallCounters hc{};
  STC_TRY(read_counters(pr, pin, hc));
  const Counters& h = hc.c;
  tm.mark(3);
  if (rows_shape && h.P >= kRowsMinPerOutput * pl.F) rows_note(ctx, sig, true);

  stc_result* r = new stc_result;
  r->ctx = ctx;
  r->stream = s;
  r->order = pl.oz;
  r->keys_form = pl.keys_out;
  r->shape = pl.zshape;
  r->stats.products = h.P;
  r->stats.survivors = h.ns;
  if (pl.report_ids) r->stats.contract_ids = hc.g.ids;
  r->stats.strategy = STC_STRATEGY_GLOBAL;

  if (h.P > 0) {
    const uint64_t target = std::min<uint64_t>(h.P, pl.F);
    const uint64_t cap = pow2_at_least(std::max<uint64_t>(64, (uint64_t)((double)target / alpha) + 1));
    const uint64_t out_cap = std::min(target, cap);
    // Fault injection (stc_opts.table_shrink): the first attempt uses a smaller table.
    const uint64_t first_cap = std::max<uint64_t>(64, o.table_shrink > 0 ? cap >> o.table_shrink : cap);
    GlobalTable t{};
    u64* wpre = nullptr;
    u64* wscr = nullptr;
    stc_status st = STC_OK;
    auto run = [&]() -> stc_status {
      // (The list of repeats may take more than the table of values saves: not under a budget.)
      if (direct_global(h.P, pl.F, cap) && o.table_shrink == 0 && o.probe == 0 && ctx->budget == 0) {
        DirectTable dt{};
        dt.mask = cap - 1;
        dt.nreps = reinterpret_cast<u64*>(&reinterpret_cast<CallCounters*>(pr.ctr)->g.fill_counters[0]);
        if (ar.alloc(&dt.keys, cap) == STC_OK && ar.alloc(&dt.pos, cap) == STC_OK && ar.alloc(&dt.rep_slot, h.P) == STC_OK &&
            ar.alloc(&dt.rep_val, h.P) == STC_OK) {
          STC_TRY(ar.alloc(&wpre, (size_t)h.ns + 1));
          STC_TRY(ar.alloc(&wscr, (size_t)scan_scratch_elems((int64_t)h.ns)));
          STC_TRY(ar.alloc_own(&r->coords, out_cap * (size_t)pl.ocols));
          STC_TRY(ar.alloc_own(&r->vals, out_cap));
          STC_CUDA(scan_u32_u64(pr.sv.w, wpre, (int64_t)h.ns, wscr, s));
          STC_CUDA(cudaMemsetAsync(dt.keys, 0xff, cap * sizeof(u64), s));
          tm.mark(3);
          STC_CUDA(launch_expand_direct(wpre, (int64_t)h.ns, h.P, pr.sv, static_cast<const u64*>(pr.yfk), pr.yv, pl.FY,
                                        dt, pl.op, r->coords, r->vals, out_cap, &pr.ctr->nz, &pr.ctr->status, ctx->sms,
                                        s));
          tm.mark(4);
          CallCounters hc2{};
          STC_TRY(read_counters(pr, pin, hc2));
          r->nnz = (int64_t)hc2.c.nz;
          return STC_OK;
        }
        g_last_error.clear();  // no memory for the list of repeats: the table of values below
        ar.release(dt.keys);
        ar.release(dt.pos);
        ar.release(dt.rep_slot);
        ar.release(dt.rep_val);
      }
      STC_TRY(ar.alloc(&t.keys, cap));
      STC_TRY(ar.alloc(&t.vals, cap));
      STC_TRY(ar.alloc(&wpre, (size_t)h.ns + 1));
      STC_TRY(ar.alloc(&wscr, (size_t)scan_scratch_elems((int64_t)h.ns)));
      STC_TRY(ar.alloc_own(&r->coords, out_cap * (size_t)pl.ocols));
      STC_TRY(ar.alloc_own(&r->vals, out_cap));
      STC_CUDA(scan_u32_u64(pr.sv.w, wpre, (int64_t)h.ns, wscr, s));
      tm.mark(3);
      for (uint64_t c = first_cap;; c = cap) {
        t.mask = c - 1;
        STC_CUDA(cudaMemsetAsync(t.keys, 0xff, c * sizeof(u64), s));
        STC_CUDA(cudaMemsetAsync(t.vals, 0, c * sizeof(double), s));
        STC_CUDA(launch_expand_global(wpre, (int64_t)h.ns, h.P, pr.sv, static_cast<const u64*>(pr.yfk), pr.yv,
                                      pl.FY, t, &pr.ctr->status, ctx->sms, s, probe));
        tm.mark(4);
        STC_CUDA(launch_compact_global(t, pl.op, r->coords, r->vals, out_cap, &pr.ctr->nz, &pr.ctr->status,
                                       ctx->sms, s));
        tm.mark(5);
        CallCounters hc2{};
        STC_TRY(copy_counters(pr, pin, hc2));
        const Counters& h2 = hc2.c;
        // A table that overflowed lost products: run the expansion again at full capacity
        // (the compaction wrote at most out_cap entries, all of them overwritten now).
        if (h2.status == kStatTableFull && c < cap) {
          STC_CUDA(cudaMemsetAsync(&pr.ctr->nz, 0, sizeof(u64), s));
          STC_CUDA(cudaMemsetAsync(&pr.ctr->status, 0, sizeof(uint32_t), s));
          r->stats.retries++;
          continue;
        }
        STC_TRY(status_word(h2.status));
        r->nnz = (int64_t)h2.nz;
        return STC_OK;
      }
    };
    st = run();
    if (st != STC_OK) {
      delete r;  // its blocks are still owned by the arena and are released with it
      return st;
    }
    r->mem = adopt(ar, ctx, s, {r->coords, r->vals});
    r->stats.out_capacity = out_cap;
    r->stats.table_slots = cap;
  }
  tm.collect(r->stats);
  r->stats.launches = take_launches();
  ctx->live_results++;
  *out = r;
  return STC_OK;
}


}  // namespace

extern "C" {

stc_status stc_contract_batch(stc_ctx* ctx, int32_t n, const stc_problem* problems, const stc_opts* opts,
                              void* stream, stc_result** outs) {
  if (!ctx || n < 0 || (n > 0 && (!problems || !outs))) return fail(STC_ERR_INVALID_ARG, "bad batch arguments");
  for (int32_t i = 0; i < n; i++) outs[i] = nullptr;
  if (n == 0) return STC_OK;
  const stc_opts o = opts ? *opts : stc_opts{};
  if (o.group_load_factor < 0.0 || o.group_load_factor > 0.9)
    return fail(STC_ERR_INVALID_ARG, "group_load_factor %g outside (0, 0.9]", o.group_load_factor);
  if (o.output_keys) return fail(STC_ERR_UNSUPPORTED, "batches return coordinates (output_keys is for stc_contract)");
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  BatchDev bd;
  STC_TRY(batch_setup(ctx, n, problems, o, ar, s, bd));
  // Load factor: given, or picked by the autotuner for this size bucket (entries, problems).
  int tune_cand = -1;
  const TuneChoice ch =
      o.group_load_factor > 0.0 ? TuneChoice{o.group_load_factor, 1024, 0} : tune_pick(ctx, bd.tune_bucket, &tune_cand);
  struct TuneGuard {  // gives a picked candidate back if the batch fails before it is timed
    stc_ctx* c;
    int b, k;
    bool armed = true;
    ~TuneGuard() {
      if (armed) tune_abort(c, b, k);
    }
  } tune_guard{ctx, bd.tune_bucket, tune_cand};
  batch_set_choice(bd, ch);
  StageTimer tm;
  tm.start(o.record_times != 0, s);
  take_launches();
  STC_TRY(batch_front(ctx, bd, s, tm));
  std::vector<u64> hper, voff, coff;
  BatchSizes sz;
  double* vals = nullptr;
  int32_t* coords = nullptr;
  bool timed = false;
  STC_TRY(batch_finish_eager(ctx, bd, o, ar, s, tm, tune_cand, &timed, hper, sz, &vals, &coords, voff, coff));
  if (timed) tune_guard.armed = false;
  auto blk = adopt(ar, ctx, s, {vals, coords});
  stc_stats common{};
  tm.collect(common);
  common.launches = take_launches();
  common.strategy = STC_STRATEGY_GROUPED;
  common.accumulator = STC_ACC_HASH;
  batch_results(ctx, s, bd, blk, vals, coords, voff.data(), coff.data(), hper.data(), common, outs);
  return STC_OK;
}

stc_status stc_batch_plan_create(stc_ctx* ctx, int32_t n, const stc_problem* problems, const stc_opts* opts,
                                 stc_batch_plan** out) {
  if (!ctx || !out || n <= 0 || !problems) return fail(STC_ERR_INVALID_ARG, "bad batch plan arguments");
  *out = nullptr;
  const stc_opts o = opts ? *opts : stc_opts{};
  if (o.group_load_factor < 0.0 || o.group_load_factor > 0.9)
    return fail(STC_ERR_INVALID_ARG, "group_load_factor %g outside (0, 0.9]", o.group_load_factor);
  if (o.output_keys) return fail(STC_ERR_UNSUPPORTED, "batches return coordinates (output_keys is for stc_contract)");
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  std::unique_ptr<stc_batch_plan> pl(new stc_batch_plan);
  pl->ctx = ctx;
  pl->opts = o;
  pl->n = n;
  // The problems' host arrays are copied; their device arrays are the caller's.
  pl->probs.assign(problems, problems + n);
  pl->shapes.resize(2 * (size_t)n);
  pl->modes.resize(3 * (size_t)n);
  for (int32_t i = 0; i < n; i++) {
    stc_problem& q = pl->probs[i];
    STC_TRY(check_coo(&q.X, "X"));
    STC_TRY(check_coo(&q.Y, "Y"));
    if (q.ncontract < 0 || q.ncontract > q.X.order || q.ncontract > q.Y.order || (q.ncontract && (!q.cx || !q.cy)))
      return fail(STC_ERR_INVALID_ARG, "problem %d: bad contract mode lists", i);
    pl->shapes[2 * i].assign(q.X.shape, q.X.shape + q.X.order);
    pl->shapes[2 * i + 1].assign(q.Y.shape, q.Y.shape + q.Y.order);
    pl->modes[3 * i].assign(q.cx, q.cx + q.ncontract);
    pl->modes[3 * i + 1].assign(q.cy, q.cy + q.ncontract);
    const int oz = (q.X.order - q.ncontract) + (q.Y.order - q.ncontract);
    if (q.out_order) pl->modes[3 * i + 2].assign(q.out_order, q.out_order + oz);
    q.X.shape = pl->shapes[2 * i].data();
    q.Y.shape = pl->shapes[2 * i + 1].data();
    q.cx = pl->modes[3 * i].data();
    q.cy = pl->modes[3 * i + 1].data();
    q.out_order = q.out_order ? pl->modes[3 * i + 2].data() : nullptr;
  }
  STC_CUDA(cudaStreamCreateWithFlags(&pl->stream, cudaStreamNonBlocking));
  pl->scratch.reset(new Arena(ctx, pl->stream));
  stc_status st = batch_setup(ctx, n, pl->probs.data(), pl->opts, *pl->scratch, pl->stream, pl->bd);
  cudaError_t e = cudaSuccess;
  if (st == STC_OK) {
    e = cudaMallocHost(&pl->h_args, sizeof(BatchLayoutArgs));
    if (e == cudaSuccess) e = cudaMallocHost(&pl->h_per, 3 * (size_t)n * sizeof(u64));
    if (e == cudaSuccess) e = cudaMallocHost(&pl->h_ctr, sizeof(Counters));
    if (e == cudaSuccess) e = cudaMallocHost(&pl->h_offs, (2 * (size_t)n + 2) * sizeof(u64));
    if (e == cudaSuccess) e = cudaMallocHost(&pl->h_gc, sizeof(GroupCounters));
    if (e == cudaSuccess) e = cudaStreamSynchronize(pl->stream);
    if (e != cudaSuccess) st = fail(STC_ERR_CUDA, "batch plan set-up failed: %s", cudaGetErrorString(e));
  }
  if (st != STC_OK) {
    stc_batch_plan_destroy(pl.release());
    return st;
  }
  *out = pl.release();
  return STC_OK;
}

stc_status stc_batch_plan_run(stc_batch_plan* pl, void* stream, stc_result** outs) {
  if (!pl || !outs) return fail(STC_ERR_INVALID_ARG, "plan or outs is NULL");
  for (int32_t i = 0; i < pl->n; i++) outs[i] = nullptr;
  stc_ctx* ctx = pl->ctx;
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  pl->runs++;
  if (!pl->exec) return plan_run_eager(pl, s, outs);
  // Replay: one output block of the last run's exact size, the layout arguments written for
  // the graph's first copy, the graph, one wait.
  const int32_t n = pl->n;
  BatchDev& bd = pl->bd;
  const u64 vbytes = (pl->sizes.vals * 8 + 15) & ~15ull;
  const u64 bytes = vbytes + pl->sizes.coords * 4;
  Arena run(ctx, s);
  unsigned char* block = nullptr;
  STC_TRY(run.alloc_own(&block, (size_t)std::max<u64>(bytes, 16)));
  pl->h_args->out = block;
  pl->h_args->out_bytes = bytes;
  STC_CUDA(cudaGraphLaunch(pl->exec, s));
  STC_CUDA(cudaStreamSynchronize(s));
  const uint32_t status = pl->h_ctr->status;
  if (status & kStatOutOverflow) {
    // This run's bounds outgrew the captured layout (the inputs' contents changed): run it
    // again with the host in the loop, which also captures a layout of the new sizes.
    return plan_run_eager(pl, s, outs);
  }
  STC_TRY(status_word(status));
  pl->graph_runs++;
  const u64* offs = pl->h_offs;
  std::vector<u64> voff(offs, offs + n + 1), coff(offs + n + 1, offs + 2 * n + 2);
  double* vals = reinterpret_cast<double*>(block);
  int32_t* coords = reinterpret_cast<int32_t*>(block + vbytes);
  stc_stats common{};
  common.launches = pl->graph_launches;
  common.strategy = STC_STRATEGY_GROUPED;
  common.accumulator = STC_ACC_HASH;
  auto blk = adopt(run, ctx, s, {block});
  batch_results(ctx, s, bd, blk, vals, coords, voff.data(), coff.data(), pl->h_per, common, outs);
  return STC_OK;
}

stc_status stc_batch_plan_stats(const stc_batch_plan* pl, int64_t* runs, int64_t* graph_runs,
                                double* group_load_factor, int32_t* warp_table_max, int32_t* expansion_depth) {
  if (!pl) return fail(STC_ERR_INVALID_ARG, "plan is NULL");
  if (runs) *runs = pl->runs;
  if (graph_runs) *graph_runs = pl->graph_runs;
  if (group_load_factor) *group_load_factor = pl->exec ? pl->choice.alpha : 0.0;
  if (warp_table_max) *warp_table_max = pl->exec ? pl->choice.warp_max : 0;
  if (expansion_depth) *expansion_depth = pl->exec ? pl->choice.depth : 0;
  return STC_OK;
}

stc_status stc_batch_plan_destroy(stc_batch_plan* pl) {
  if (!pl) return STC_OK;
  DeviceGuard g(pl->ctx->device);
  if (pl->exec) cudaGraphExecDestroy(pl->exec);
  if (pl->graph) cudaGraphDestroy(pl->graph);
  if (pl->stream) cudaStreamSynchronize(pl->stream);
  pl->scratch.reset();  // scratch goes back to the pool in the plan stream's order
  if (pl->stream) {
    cudaStreamSynchronize(pl->stream);
    cudaStreamDestroy(pl->stream);
  }
  if (pl->h_args) cudaFreeHost(pl->h_args);
  if (pl->h_per) cudaFreeHost(pl->h_per);
  if (pl->h_ctr) cudaFreeHost(pl->h_ctr);
  if (pl->h_offs) cudaFreeHost(pl->h_offs);
  if (pl->h_gc) cudaFreeHost(pl->h_gc);
  delete pl;
  return STC_OK;
}

stc_status stc_ctx_stats(const stc_ctx* ctx, uint64_t* held_bytes, int64_t* live_results) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  if (held_bytes) *held_bytes = ctx->held.load();
  if (live_results) *live_results = ctx->live_results.load();
  return STC_OK;
}

stc_status stc_count(stc_ctx* ctx, const stc_coo* X, const stc_coo* Y, int32_t m, const int32_t* cx,
                     const int32_t* cy, void* stream, uint64_t* products, uint64_t* bytes_bound) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  Plan pl;
  STC_TRY(make_plan(X, Y, m, cx, cy, nullptr, pl));
  // Bound the orientation stc_contract's AUTO operand order will run (P is the same).
  if ((uint64_t)Y->nnz > 4 * (uint64_t)X->nnz)
    return stc_count(ctx, Y, X, m, cy, cx, stream, products, bytes_bound);
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool dense_ids = use_dense_ids(pl, X, Y, STC_IDS_AUTO);
  if (use_id_map(ctx, pl, X, Y, STC_IDS_AUTO, dense_ids)) {
    pl.id_map = true;
    pl.report_ids = dense_ids;
    pl.Kb = (uint64_t)Y->nnz;
  } else if (dense_ids) {
    Relabelled rl(ctx, s);
    STC_TRY(relabel(ctx, X, Y, pl, false, s, rl));
    uint64_t b = 0;
    STC_TRY(stc_count(ctx, &rl.X, &rl.Y, 1, &rl.cx, &rl.cy, stream, products, bytes_bound ? &b : nullptr));
    // The rewritten coordinates stay held beside the id table, then beside the contraction.
    const uint64_t slots = id_table_slots(Y->nnz);
    ArenaBytes rows(ctx), table(ctx);
    rows.alloc(4ull * (uint64_t)rl.X.order * (uint64_t)X->nnz);
    rows.alloc(4ull * (uint64_t)rl.Y.order * (uint64_t)Y->nnz);
    for (uint64_t n : {slots * 8, (slots + 1) * 4, (slots + 2) * 4, (uint64_t)scan_scratch_elems((int64_t)slots + 1) * 4,
                       (uint64_t)4})
      table.alloc(n);
    if (bytes_bound) *bytes_bound = rows.held + std::max(b, table.held);
    return STC_OK;
  }
  Arena ar(ctx, s);
  StageTimer tm;
  Prepared pr;
  const int strategy = pick_strategy(pl, X, Y, STC_STRATEGY_AUTO);
  const bool dense = strategy == STC_STRATEGY_GROUPED && x_dense(pl, Y);
  STC_TRY(prepare(ctx, ar, X, Y, pl, dense ? Survey::kDenseGroups : Survey::kSurvivors, s, tm, pr));
  Pinned pin(ctx, s);
  CallCounters hc{};
  STC_TRY(read_counters(pr, pin, hc));
  const Counters& h = hc.c;
  if (products) *products = h.P;
  if (!bytes_bound) return STC_OK;
  const Survey grouped = x_dense(pl, Y) ? Survey::kDenseGroups : Survey::kSurvivorsGroups;
  *bytes_bound = strategy == STC_STRATEGY_GROUPED ? grouped_bytes(ctx, pl, X->nnz, Y->nnz, h.P, grouped)
                                                  : global_bytes(ctx, pl, X->nnz, Y->nnz, h.ns, h.P, 0.5);
  // A shape that a run here finds to be rows-heavy is grouped from then on.
  if (strategy == STC_STRATEGY_GLOBAL && pl.FY <= kLaneRowMax && pl.FX <= kMaxDirectBins &&
      h.P >= kRowsMinPerOutput * pl.F)
    *bytes_bound = std::max(*bytes_bound, grouped_bytes(ctx, pl, X->nnz, Y->nnz, h.P, grouped));
  return STC_OK;
}

stc_status stc_linearize(stc_ctx* ctx, const stc_coo* T, int32_t nmodes, const int32_t* modes, uint64_t* keys_out,
                         void* stream) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  STC_TRY(check_coo(T, "T"));
  if (nmodes < 0 || nmodes > T->order || (nmodes > 0 && !modes))
    return fail(STC_ERR_INVALID_ARG, "bad mode list");
  if (T->nnz > 0 && !keys_out) return fail(STC_ERR_INVALID_ARG, "keys_out is NULL");
  KeyPlan p{};
  p.order = T->order;
  for (int j = 0; j < T->order; j++) p.size[j] = T->shape[j];
  bool seen[STC_MAX_ORDER] = {};
  unsigned __int128 acc = 1;
  for (int i = nmodes - 1; i >= 0; i--) {
    if (modes[i] < 0 || modes[i] >= T->order || seen[modes[i]]) return fail(STC_ERR_INVALID_ARG, "bad mode list");
    seen[modes[i]] = true;
    p.cstride[modes[i]] = (uint64_t)acc;
    acc *= (unsigned __int128)T->shape[modes[i]];
    if (acc > (unsigned __int128)UINT64_MAX) return fail(STC_ERR_KEY_OVERFLOW, "key space exceeds 2^64");
  }
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  uint32_t* status = nullptr;
  STC_TRY(ar.alloc(&status, 1));
  STC_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
  STC_CUDA(launch_linearize(T->coords, T->nnz, p, reinterpret_cast<u64*>(keys_out), status, ctx->sms, s));
  uint32_t h = 0;
  STC_CUDA(cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaStreamSynchronize(s));
  return status_word(h);
}

stc_status stc_group_keys(stc_ctx* ctx, const uint64_t* keys, int64_t n, uint64_t k, uint32_t* offsets_out,
                          uint32_t* perm_out, void* stream) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  if (n < 0 || n > STC_MAX_NNZ) return fail(STC_ERR_INVALID_ARG, "n = %lld out of range", (long long)n);
  if (k > kMaxDirectBins) return fail(STC_ERR_UNSUPPORTED, "k = %llu exceeds 2^26", (unsigned long long)k);
  if (!offsets_out || (n > 0 && (!keys || !perm_out))) return fail(STC_ERR_INVALID_ARG, "NULL pointer");
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  uint32_t *cnt = nullptr, *cur = nullptr, *scr = nullptr, *status = nullptr;
  STC_TRY(ar.alloc(&status, 1));
  STC_TRY(ar.alloc(&cnt, k));
  STC_TRY(ar.alloc(&cur, k));
  STC_TRY(ar.alloc(&scr, (size_t)scan_scratch_elems((int64_t)k)));
  STC_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
  if (k) STC_CUDA(cudaMemsetAsync(cnt, 0, k * sizeof(uint32_t), s));
  const u64* kk = reinterpret_cast<const u64*>(keys);
  STC_CUDA(launch_key_count(kk, n, k, cnt, status, ctx->sms, s));
  STC_CUDA(scan_u32(cnt, offsets_out, (int64_t)k, scr, s));
  if (k) STC_CUDA(cudaMemcpyAsync(cur, offsets_out, k * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  STC_CUDA(launch_key_scatter(kk, n, k, cur, perm_out, ctx->sms, s));
  uint32_t h = 0;
  STC_CUDA(cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaStreamSynchronize(s));
  return status_word(h);
}

stc_status stc_dense_ids(stc_ctx* ctx, const uint64_t* keys, int64_t n, uint32_t* ids_out, uint64_t* ndistinct,
                         void* stream) {
  if (!ctx) return fail(STC_ERR_INVALID_ARG, "ctx is NULL");
  if (n < 0 || n > STC_MAX_NNZ) return fail(STC_ERR_INVALID_ARG, "n = %lld out of range", (long long)n);
  if (!ndistinct || (n > 0 && (!keys || !ids_out))) return fail(STC_ERR_INVALID_ARG, "NULL pointer");
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  IdTable t{};
  uint32_t *scr = nullptr, *status = nullptr;
  t.slots = id_table_slots(n);
  STC_TRY(ar.alloc(&t.keys, t.slots));
  STC_TRY(ar.alloc(&t.flags, t.slots + 1));
  STC_TRY(ar.alloc(&t.prefix, t.slots + 2));
  STC_TRY(ar.alloc(&scr, (size_t)scan_scratch_elems((int64_t)t.slots + 1)));
  STC_TRY(ar.alloc(&status, 1));
  STC_CUDA(cudaMemsetAsync(t.keys, 0xff, t.slots * sizeof(u64), s));
  STC_CUDA(cudaMemsetAsync(t.flags + t.slots, 0, sizeof(uint32_t), s));
  STC_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
  const u64* kk = reinterpret_cast<const u64*>(keys);
  STC_CUDA(launch_id_insert_keys(kk, n, t, status, ctx->sms, s));
  STC_CUDA(launch_id_number(t, scr, ctx->sms, s));
  STC_CUDA(launch_id_lookup_keys(kk, n, t, ids_out, ctx->sms, s));
  uint32_t h[2] = {0, 0};
  STC_CUDA(cudaMemcpyAsync(&h[0], status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaMemcpyAsync(&h[1], t.prefix + t.slots + 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  STC_CUDA(cudaStreamSynchronize(s));
  *ndistinct = h[1];
  return status_word(h[0]);
}

stc_status stc_result_info(const stc_result* r, int64_t* nnz, int32_t* order, const int64_t** shape) {
  if (!r) return fail(STC_ERR_INVALID_ARG, "result is NULL");
  if (nnz) *nnz = r->nnz;
  if (order) *order = r->order;
  if (shape) *shape = r->shape.empty() ? nullptr : r->shape.data();
  return STC_OK;
}

stc_status stc_result_data(const stc_result* r, const int32_t** coords, const double** vals) {
  if (!r) return fail(STC_ERR_INVALID_ARG, "result is NULL");
  if (coords) *coords = r->coords;
  if (vals) *vals = r->vals;
  return STC_OK;
}

stc_status stc_result_stats(const stc_result* r, stc_stats* stats) {
  if (!r || !stats) return fail(STC_ERR_INVALID_ARG, "NULL argument");
  *stats = r->stats;
  return STC_OK;
}

stc_status stc_result_as_coo(const stc_result* r, stc_coo* out) {
  if (!r || !out) return fail(STC_ERR_INVALID_ARG, "NULL argument");
  if (r->keys_form) return fail(STC_ERR_INVALID_ARG, "the result is in key form (stc_result_as_keyed)");
  out->order = r->order;
  out->shape = r->shape.empty() ? nullptr : r->shape.data();
  out->nnz = r->nnz;
  out->coords = r->coords;
  out->vals = r->vals;
  return STC_OK;
}

stc_status stc_result_keys(const stc_result* r, const uint64_t** keys) {
  if (!r || !keys) return fail(STC_ERR_INVALID_ARG, "NULL argument");
  *keys = r->keys_form ? reinterpret_cast<const uint64_t*>(r->coords) : nullptr;
  return STC_OK;
}

stc_status stc_result_as_keyed(const stc_result* r, stc_keyed* out) {
  if (!r || !out) return fail(STC_ERR_INVALID_ARG, "NULL argument");
  if (!r->keys_form) return fail(STC_ERR_INVALID_ARG, "the result holds coordinates, not keys");
  out->order = r->order;
  out->shape = r->shape.empty() ? nullptr : r->shape.data();
  out->nnz = r->nnz;
  out->keys = reinterpret_cast<const uint64_t*>(r->coords);
  out->vals = r->vals;
  return STC_OK;
}

stc_status stc_contract_keyed(stc_ctx* ctx, const stc_keyed* X, const stc_coo* Y, int32_t m, const int32_t* cx,
                              const int32_t* cy, const int32_t* out_order, const stc_opts* opts, void* stream,
                              stc_result** out) {
  if (!ctx || !out || !X) return fail(STC_ERR_INVALID_ARG, "ctx, X or out is NULL");
  *out = nullptr;
  if (X->order < 1 || X->order > STC_MAX_ORDER || !X->shape)
    return fail(STC_ERR_INVALID_ARG, "X.order = %d outside 1..%d", X->order, STC_MAX_ORDER);
  if (X->nnz < 0 || X->nnz > STC_MAX_NNZ || (X->nnz > 0 && (!X->keys || !X->vals)))
    return fail(STC_ERR_INVALID_ARG, "bad X.nnz, keys or vals");
  if (m < 0 || m > X->order || (m > 0 && (!cx || !cy))) return fail(STC_ERR_INVALID_ARG, "bad contract mode lists");
  for (int j = 0; j < X->order; j++)
    if (X->shape[j] < 1 || X->shape[j] > (int64_t)1 << 31)
      return fail(STC_ERR_INVALID_ARG, "X.shape[%d] = %lld outside 1..2^31", j, (long long)X->shape[j]);
  // The contracted modes: a contiguous block at the end (or the start) of X's modes, in order.
  bool trailing = true, leading = true;
  for (int i = 0; i < m; i++) {
    trailing = trailing && cx[i] == X->order - m + i;
    leading = leading && cx[i] == i;
  }
  if (!trailing && !leading)
    return fail(STC_ERR_INVALID_ARG, "X's contracted modes must be its last (or first) %d modes, in order", m);
  KeySplit ks{};
  ks.m = m;
  ks.trailing = trailing ? 1 : 0;
  unsigned __int128 K = 1, F = 1;
  std::vector<int64_t> xfree;
  for (int j = 0; j < X->order; j++) {
    const bool contracted = trailing ? j >= X->order - m : j < m;
    if (contracted) K *= (unsigned __int128)X->shape[j];
    else F *= (unsigned __int128)X->shape[j], xfree.push_back(X->shape[j]);
  }
  for (int i = 0; i < m; i++) ks.csize[i] = X->shape[cx[i]];
  if (K * F > (unsigned __int128)UINT64_MAX) return fail(STC_ERR_KEY_OVERFLOW, "X's key space exceeds 2^64");
  if (K > kMaxDirectBins) return fail(STC_ERR_UNSUPPORTED, "X's contract key space exceeds 2^26");
  ks.K = (u64)K;
  ks.F = (u64)F;
  ks.FL = std::min<u64>(ks.F, 1ull << 30);
  const u64 FH = (ks.F + ks.FL - 1) / ks.FL;
  if (FH > (1ull << 31)) return fail(STC_ERR_UNSUPPORTED, "X's free key space exceeds 2^61");
  DeviceGuard g(ctx->device);
  if (!g.ok) return fail(STC_ERR_CUDA, "cannot make device %d current", ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Arena ar(ctx, s);
  int32_t* rows = nullptr;
  uint32_t* status = nullptr;
  STC_TRY(ar.alloc(&rows, (size_t)X->nnz * (2 + m)));
  STC_TRY(ar.alloc(&status, 1));
  STC_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), s));
  take_launches();
  STC_CUDA(launch_keyed_split(reinterpret_cast<const u64*>(X->keys), X->nnz, ks, rows, status, ctx->sms, s));
  const unsigned split_launches = take_launches();
  // The split form: modes (free / FL, free % FL, contracted modes), its free key the original
  // free index, paired on its last m modes.
  std::vector<int64_t> shape2 = {(int64_t)FH, (int64_t)ks.FL};
  std::vector<int32_t> cx2(m);
  for (int i = 0; i < m; i++) shape2.push_back(ks.csize[i]), cx2[i] = 2 + i;
  const stc_coo X2{2 + m, shape2.data(), X->nnz, rows, X->vals};
  stc_opts o = opts ? *opts : stc_opts{};
  o.operands = STC_OPERANDS_AS_GIVEN;
  o.contract_ids = STC_IDS_DIRECT;
  STC_TRY(contract_impl(ctx, &X2, Y, m, cx2.data(), cy, out_order, &o, stream, out, &xfree));
  uint32_t h = 0;
  const cudaError_t e1 = cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, s);
  const cudaError_t e2 = e1 == cudaSuccess ? cudaStreamSynchronize(s) : e1;
  const stc_status st = e2 != cudaSuccess ? fail(STC_ERR_CUDA, "%s", cudaGetErrorString(e2)) : status_word(h);
  if (st != STC_OK) {
    stc_result_free(*out);
    *out = nullptr;
    return st;
  }
  (*out)->stats.launches += split_launches;
  return STC_OK;
}

stc_status stc_result_free(stc_result* r) {
  if (!r) return STC_OK;
  r->ctx->live_results--;
  delete r;
  return STC_OK;
}

}  // extern "C"
