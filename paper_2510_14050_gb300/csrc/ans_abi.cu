// C ABI of libans.so: contexts, memory budget, scratch, matrices, the batch
// pipeline and completion tickets.  Host code only; the kernels live in the
// other ans_*.cu files.
//
// Pipeline of one batch of windows (every window of the batch in one fixed
// sequence of launches, independent of the number of windows):
//   sample sort of the packets (sample, count, scatter, local; long windows
//   split twice) -> run-length reduce to DCSR -> values, row statistics and
//   destination partition counts -> column pass (links scattered into the
//   partitions, each counted)
//   [-> time sum: the windows' links merged pairwise, or gathered and sorted
//   by 8 key/value passes, then their value prefix; or the packets sorted
//   again as one segment -> run-length reduce -> statistics -> column pass].
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "ans.h"
#include "ans_internal.cuh"

using namespace ans;

namespace {

thread_local std::string t_last_error;

int fail(int code, const std::string& msg) {
  t_last_error = msg;
  return code;
}

#define ANS_CUDA(expr)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (expr);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return fail(ANS_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_));        \
  } while (0)

#define ANS_TRY(expr)           \
  do {                          \
    int rc_ = (expr);           \
    if (rc_ != ANS_OK) return rc_; \
  } while (0)

constexpr size_t kAlign = 256;
constexpr uint64_t kMaxWindow = (1ull << 31) - 1;
constexpr int kStageSlots = 16;
constexpr int kErrSlots = 4096;
// Tickets of the look-back kernels, 32 per phase: window sort + RLE, time-sum
// sort + RLE + scan, window column pass, time-sum column pass.
constexpr int kTicketBlocks = 4;

size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }
uint64_t tiles_for(uint64_t n) { return (n + kTile - 1) / kTile; }

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    cudaGetDevice(&cur);
    if (prev >= 0 && cur != prev) cudaSetDevice(prev);
  }
};

// Scratch guards (debug mode, ANS_SCRATCH_GUARDS): while a GuardSink is in
// scope on this thread, every Layout region is followed by kGuardBytes whose
// offset the sink records.
thread_local std::vector<size_t>* t_guard_sink = nullptr;
struct GuardSink {
  std::vector<size_t>* prev;
  explicit GuardSink(std::vector<size_t>* sink) : prev(t_guard_sink) { t_guard_sink = sink; }
  ~GuardSink() { t_guard_sink = prev; }
};

// Two-phase bump layout: add() records sizes, bind() turns offsets into pointers.
struct Layout {
  size_t size = 0;
  size_t add(size_t bytes) {
    size_t off = size;
    size = align_up(size + std::max<size_t>(bytes, 1));
    if (t_guard_sink) {
      t_guard_sink->push_back(size);
      size += kGuardBytes;
    }
    return off;
  }
};
static_assert(kGuardBytes % kAlign == 0, "guards keep the regions aligned");

// Fill (err == nullptr) or check the guards at these device addresses.
cudaError_t run_guards(const std::vector<uint64_t>& addrs, uint32_t* err, cudaStream_t st) {
  GuardList g;
  for (size_t i = 0; i < addrs.size(); ++i) {
    g.addr[g.n++] = addrs[i];
    if (g.n == kGuardsPerLaunch || i + 1 == addrs.size()) {
      const cudaError_t e = launch_guards(g, err, st);
      if (e != cudaSuccess) return e;
      g.n = 0;
    }
  }
  return cudaSuccess;
}

}  // namespace

int ans::set_last_error(int code, const std::string& msg) { return fail(code, msg); }

struct Block;

struct ans_ctx {
  int device = 0;
  size_t budget = 0;
  ans_alloc_fn alloc_fn = nullptr;
  ans_free_fn free_fn = nullptr;
  void* user = nullptr;
  std::mutex mu;
  size_t live = 0;  // device bytes held: scratch + live matrix blocks
  // Lifetime: matrix blocks keep the context alive; ans_ctx_destroy releases
  // what only calls need and the last block to go frees the rest.
  size_t blocks = 0;
  bool closed = false;

  void* scratch = nullptr;
  size_t scratch_size = 0;
  // The device error word (bounded waits that gave up set bits here).
  uint32_t* d_err = nullptr;
  void* small_mem = nullptr;
  // Debug mode (ANS_SCRATCH_GUARDS at creation): guards after every region of
  // a batch's scratch and of its output blocks, checked after each batch.
  bool guards = false;

  // Pinned staging ring for plan uploads.
  struct Stage {
    void* h = nullptr;
    size_t size = 0;
    cudaEvent_t ev = nullptr;
  } stage[kStageSlots];
  int stage_next = 0;

  // Completion tickets.
  uint32_t* h_err_slots = nullptr;  // pinned
  int err_next = 0;
  struct Ticket {
    cudaEvent_t ev;
    int slot;
  };
  std::map<uint64_t, Ticket> tickets;
  uint64_t next_ticket = 1;
  cudaStream_t aux = nullptr;  // frees of matrix memory

  // Launch configurations of the families of radix passes (key_*: kept, unused) (set by
  // ans_set_tuning / ans_autotune).
  SortCfg cfg_keys, cfg_kv, cfg_col;
  // Window sort: 0 = on chip (one 8-CTA cluster per window of at most
  // kClusterWindowMax packets; larger windows take the sample sort),
  // 1 = the sample sort for every window (the default: faster on every
  // workload measured so far).  cfg_win: the cluster kernel's threads and
  // ranking mode.
  int win_path = 1;
  SortCfg cfg_win{1024, kRankMatch, 1};
  // Time sum: 0 = merge the matrices' sorted links pairwise, 1 = radix-sort
  // the gathered links (kv passes), 2 = sort a batch's packets again as one
  // segment (sums of given matrices: merged up to 256 of them).
  int sum_path = 0;
  int merge_tile = 4096;  // merge rounds: output positions per CTA (4096 or 2048)
  // Window aggregation: 0 = sort every packet's key, 1 = count links in
  // per-window hash tables and sort the distinct links.  The tables live in
  // their own arena, left empty by every call that used them (hash_dirty
  // marks one that may not have been).
  int agg_path = 0;
  // Column statistics: 1 = links in hash partitions (or, large time sums,
  // hash groups) of their destinations, 0 = the column sort.
  int col_hash = 1;
  int pageable = -1;  // does the device read pageable host memory (-1: not asked yet)
  // Packets a batch with device-resident offsets may hold (0: the call reads
  // the first and last offset back to size its scratch).
  uint64_t batch_cap = 0;
  // Batches replay their launch sequence as a CUDA graph (graph = 1): it is
  // captured on `cap` each call and applied to a cached executable graph of
  // the same shape by cudaGraphExecUpdate (re-instantiated if the topology
  // changed).  Off while per-kernel profiling is on.
  int graph = 1;
  cudaStream_t cap = nullptr;
  std::map<std::string, cudaGraphExec_t> graphs;
  // A batch's time sum orders its links (gather, merge rounds) on `side`,
  // beside the window column pass on the main stream: fork and join events.
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  void* hash_mem = nullptr;
  size_t hash_slots = 0;
  bool hash_dirty = false;
  // ans_batch_submit_windows on the paths that sort a batch's packets as one
  // segment: the windows' pairs gathered into one buffer (src words, then
  // dst words, then the windows' gather table), grown on demand.
  void* gather_mem = nullptr;
  size_t gather_bytes = 0;

  // Optional per-kernel timing: CUDA events recorded around each launch on
  // the launching stream, accumulated by name when read.
  struct Prof {
    bool on = false;
    struct Rec {
      const char* name;
      cudaEvent_t a, b;
    };
    std::vector<Rec> pending;
    std::vector<cudaEvent_t> spare;
    std::map<std::string, std::pair<double, uint64_t>> acc;
  } prof;
};

namespace {

cudaEvent_t prof_event(ans_ctx* c) {
  if (!c->prof.spare.empty()) {
    cudaEvent_t e = c->prof.spare.back();
    c->prof.spare.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return e;
}

// Times one kernel launch when profiling is on (records nothing otherwise).
struct KTime {
  ans_ctx* c;
  const char* name;
  cudaStream_t st;
  cudaEvent_t a = nullptr, b = nullptr;
  KTime(ans_ctx* c_, const char* name_, cudaStream_t st_) : c(c_), name(name_), st(st_) {
    if (!c->prof.on) return;
    a = prof_event(c);
    b = prof_event(c);
    if (a && b) cudaEventRecord(a, st);
  }
  ~KTime() {
    if (!a || !b) return;
    cudaEventRecord(b, st);
    c->prof.pending.push_back({name, a, b});
  }
};

template <class F>
cudaError_t timed(ans_ctx* c, const char* name, cudaStream_t st, F&& f) {
  KTime kt(c, name, st);
  return f();
}

void prof_collect(ans_ctx* c) {
  for (auto& r : c->prof.pending) {
    float ms = 0.f;
    if (cudaEventSynchronize(r.b) == cudaSuccess && cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) {
      auto& x = c->prof.acc[r.name];
      x.first += ms;
      x.second += 1;
    } else {
      cudaGetLastError();
    }
    c->prof.spare.push_back(r.a);
    c->prof.spare.push_back(r.b);
  }
  c->prof.pending.clear();
}

}  // namespace

// Device memory that holds one or more matrices (one per window of a batch,
// or a single time sum).
struct Block {
  ans_ctx* ctx = nullptr;
  void* mem = nullptr;
  size_t bytes = 0;
  uint32_t nseg = 0;
  std::vector<uint64_t> base;  // padded start per segment
  std::vector<uint64_t> cap;   // upper bound on nnz per segment
  uint32_t* col_ids = nullptr;
  uint64_t* vals = nullptr;
  uint32_t* row_ids = nullptr;
  uint64_t* row_ptr = nullptr;
  uint64_t* hdr = nullptr;
  ans_quantities* q = nullptr;
  uint32_t* status = nullptr;  // device error word captured at completion
  // A block of a batch planned on the device: the padded starts live in
  // d_base until the block completes; base and cap (then the exact link
  // counts) are filled by block_fill_cache.
  bool dev_plan = false;
  uint64_t* d_base = nullptr;
  cudaEvent_t done = nullptr;
  std::atomic<int> refs{0};
  std::mutex mu;
  std::vector<cudaEvent_t> readers;  // completion of library calls that read the block
  bool cached = false;
  std::vector<uint64_t> h_hdr;
  std::vector<ans_quantities> h_q;
  uint32_t h_status = 0;
  std::vector<uint64_t> guards;  // device addresses of its guards (debug mode)
};

struct ans_matrix {
  Block* blk;
  uint32_t seg;
};

namespace {

// Recordings of batches (run_launches) and waits for the whole device exclude
// one another across contexts and threads: the runtime refuses such a wait while
// a stream is being captured, and breaks the capture off.
struct Recordings {
  std::mutex mu;
  std::condition_variable cv;
  int running = 0, waits = 0;  // recordings under way; waits asked for or under way
};
Recordings g_rec;
struct RecordGuard {
  RecordGuard() {
    std::unique_lock<std::mutex> l(g_rec.mu);
    g_rec.cv.wait(l, [] { return g_rec.waits == 0; });
    ++g_rec.running;
  }
  ~RecordGuard() {
    std::lock_guard<std::mutex> l(g_rec.mu);
    --g_rec.running;
    g_rec.cv.notify_all();
  }
};
cudaError_t device_wait() {
  std::unique_lock<std::mutex> l(g_rec.mu);
  ++g_rec.waits;
  g_rec.cv.wait(l, [] { return g_rec.running == 0; });
  const cudaError_t e = cudaDeviceSynchronize();
  --g_rec.waits;
  g_rec.cv.notify_all();
  return e;
}

int dev_alloc(ans_ctx* c, size_t bytes, cudaStream_t st, void** out) {
  *out = nullptr;
  if (bytes == 0) return ANS_OK;
  if (c->budget && c->live + bytes > c->budget)
    return fail(ANS_ERR_BUDGET, "memory budget exceeded: holding " + std::to_string(c->live) +
                                    " bytes, need " + std::to_string(bytes) + " more, budget " +
                                    std::to_string(c->budget));
  void* p = nullptr;
  if (c->alloc_fn) {
    p = c->alloc_fn(bytes, (void*)st, c->user);
    if (!p) return fail(ANS_ERR_OOM, "allocator hook returned NULL for " + std::to_string(bytes) + " bytes");
  } else {
    cudaError_t e = cudaMallocAsync(&p, bytes, st);
    if (e == cudaErrorMemoryAllocation) {
      // The pool keeps freed memory (release threshold: unlimited); return it
      // to the device once everything queued has finished, and retry.
      cudaGetLastError();
      cudaMemPool_t pool = nullptr;
      if (device_wait() == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, c->device) == cudaSuccess)
        cudaMemPoolTrimTo(pool, 0);
      cudaGetLastError();
      e = cudaMallocAsync(&p, bytes, st);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(ANS_ERR_OOM, std::string("cudaMallocAsync(") + std::to_string(bytes) + "): " +
                                   cudaGetErrorString(e));
    }
  }
  c->live += bytes;
  *out = p;
  return ANS_OK;
}

void dev_free(ans_ctx* c, void* p, size_t bytes, cudaStream_t st) {
  if (!p) return;
  if (c->free_fn) c->free_fn(p, (void*)st, c->user);
  else cudaFreeAsync(p, st);
  c->live -= bytes;
}

int ensure_scratch(ans_ctx* c, size_t bytes, cudaStream_t st) {
  if (bytes <= c->scratch_size) return ANS_OK;
  size_t want = std::max(bytes, c->scratch_size + c->scratch_size / 4);
  dev_free(c, c->scratch, c->scratch_size, st);
  c->scratch = nullptr;
  c->scratch_size = 0;
  void* p = nullptr;
  int rc = dev_alloc(c, want, st, &p);
  if (rc != ANS_OK && want > bytes) rc = dev_alloc(c, bytes, st, &p), want = bytes;
  if (rc != ANS_OK) return rc;
  c->scratch = p;
  c->scratch_size = want;
  return ANS_OK;
}

// The hash tables' arena: `slots` slots of (uint64 key, uint32 count), all
// empty (keys all ones, counts 0) when this returns.
int ensure_hash(ans_ctx* c, size_t slots, cudaStream_t st) {
  if (slots > c->hash_slots) {
    dev_free(c, c->hash_mem, c->hash_slots * 12, st);
    c->hash_mem = nullptr;
    c->hash_slots = 0;
    void* p = nullptr;
    ANS_TRY(dev_alloc(c, slots * 12, st, &p));
    c->hash_mem = p;
    c->hash_slots = slots;
    c->hash_dirty = true;
  }
  if (c->hash_dirty) {
    ANS_CUDA(cudaMemsetAsync(c->hash_mem, 0xff, c->hash_slots * 8, st));
    ANS_CUDA(cudaMemsetAsync((char*)c->hash_mem + c->hash_slots * 8, 0, c->hash_slots * 4, st));
    c->hash_dirty = false;
  }
  return ANS_OK;
}

// All the small host arrays of one call (plans, matrix descriptors), staged
// together in one slot of the context's pinned ring and copied before the
// call's first kernel.  One slot per call lets kStageSlots calls be in flight
// before the host waits for the GPU.
struct UploadSet {
  struct Item {
    void* dst;
    size_t off, bytes;
  };
  std::vector<uint8_t> img;
  std::vector<Item> items;
  void add(void* dst, const void* src, size_t bytes) {
    if (bytes == 0) return;
    const size_t off = (img.size() + 15) & ~size_t(15);
    img.resize(off + bytes);
    std::memcpy(img.data() + off, src, bytes);
    items.push_back({dst, off, bytes});
  }
  int flush(ans_ctx* c, cudaStream_t st) {
    if (items.empty()) return ANS_OK;
    ans_ctx::Stage& s = c->stage[c->stage_next];
    c->stage_next = (c->stage_next + 1) % kStageSlots;
    ANS_CUDA(cudaEventSynchronize(s.ev));
    if (s.size < img.size()) {
      if (s.h) ANS_CUDA(cudaFreeHost(s.h));
      s.h = nullptr;
      s.size = 0;
      const size_t want = std::max<size_t>(align_up(img.size(), 1 << 16), 2 * s.size);
      ANS_CUDA(cudaHostAlloc(&s.h, want, cudaHostAllocDefault));
      s.size = want;
    }
    std::memcpy(s.h, img.data(), img.size());
    // copied by kernels reading the pinned slot in place: a copy-engine
    // transfer would queue behind bulk copies of other streams
    SmallCopyBatch b;
    for (const Item& it : items) {
      b.it[b.n++] = SmallCopyItem{it.dst, (const char*)s.h + it.off, it.bytes};
      if (b.n == kSmallCopyItems) {
        ANS_CUDA(launch_small_copy(b, st));
        b.n = 0;
      }
    }
    ANS_CUDA(launch_small_copy(b, st));
    ANS_CUDA(cudaEventRecord(s.ev, st));
    items.clear();
    img.clear();
    return ANS_OK;
  }
};

// Device layout of a block holding nseg matrices over `pad` padded items.
struct BlockLayout {
  size_t col_ids, vals, row_ids, row_ptr, hdr, q, status, base = 0, total;
  BlockLayout(uint64_t pad, uint32_t nseg, bool dev_base = false) {
    Layout L;
    col_ids = L.add(pad * 4);
    vals = L.add(pad * 8);
    row_ids = L.add(pad * 4);
    row_ptr = L.add((pad + nseg) * 8);
    hdr = L.add((size_t)nseg * 16);
    q = L.add((size_t)nseg * sizeof(ans_quantities));
    status = L.add(8);
    if (dev_base) base = L.add((size_t)nseg * 8);
    total = L.size;
  }
};

// dev_base: the segments' padded starts are computed on the device (base
// and cap stay empty until the block completes).
int make_block(ans_ctx* c, uint64_t pad, uint32_t nseg, std::vector<uint64_t> base, std::vector<uint64_t> cap,
               cudaStream_t st, Block** out, bool dev_base = false) {
  std::vector<size_t> goff;
  const BlockLayout bl = [&] {
    GuardSink gs(c->guards ? &goff : nullptr);
    return BlockLayout(pad, nseg, dev_base);
  }();
  void* mem = nullptr;
  ANS_TRY(dev_alloc(c, bl.total, st, &mem));
  std::vector<uint64_t> gaddr;
  for (size_t o : goff) gaddr.push_back((uint64_t)(uintptr_t)mem + o);
  if (!gaddr.empty()) {
    const cudaError_t ge = run_guards(gaddr, nullptr, st);
    if (ge != cudaSuccess) {
      dev_free(c, mem, bl.total, st);
      return fail(ANS_ERR_CUDA, std::string("guards: ") + cudaGetErrorString(ge));
    }
  }
  Block* b = new Block();
  b->ctx = c;
  b->mem = mem;
  b->bytes = bl.total;
  b->nseg = nseg;
  b->base = std::move(base);
  b->cap = std::move(cap);
  b->guards = std::move(gaddr);
  char* m = (char*)mem;
  b->col_ids = (uint32_t*)(m + bl.col_ids);
  b->vals = (uint64_t*)(m + bl.vals);
  b->row_ids = (uint32_t*)(m + bl.row_ids);
  b->row_ptr = (uint64_t*)(m + bl.row_ptr);
  b->hdr = (uint64_t*)(m + bl.hdr);
  b->q = (ans_quantities*)(m + bl.q);
  b->status = (uint32_t*)(m + bl.status);
  if (dev_base) {
    b->dev_plan = true;
    b->d_base = (uint64_t*)(m + bl.base);
  }
  cudaError_t e = cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    dev_free(c, mem, bl.total, st);
    delete b;
    return fail(ANS_ERR_CUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
  }
  ++c->blocks;  // callers hold c->mu
  *out = b;
  return ANS_OK;
}

// Note that work just enqueued on `st` reads block b: freeing b waits for it.
int note_read(Block* b, cudaStream_t st) {
  cudaEvent_t ev = nullptr;
  ANS_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  cudaError_t e = cudaEventRecord(ev, st);
  if (e != cudaSuccess) {
    cudaEventDestroy(ev);
    return fail(ANS_ERR_CUDA, std::string("cudaEventRecord: ") + cudaGetErrorString(e));
  }
  std::lock_guard<std::mutex> g(b->mu);
  b->readers.push_back(ev);
  return ANS_OK;
}

void ctx_finalize(ans_ctx* c);

void block_release(Block* b) {
  if (--b->refs > 0) return;
  ans_ctx* c = b->ctx;
  cudaEventSynchronize(b->done);
  {
    std::lock_guard<std::mutex> g(b->mu);
    for (cudaEvent_t ev : b->readers) {
      cudaEventSynchronize(ev);
      cudaEventDestroy(ev);
    }
    b->readers.clear();
  }
  bool last = false;
  {
    std::lock_guard<std::mutex> g(c->mu);
    DeviceGuard dg(c->device);
    dev_free(c, b->mem, b->bytes, c->aux);
    cudaEventDestroy(b->done);
    last = --c->blocks == 0 && c->closed;
  }
  delete b;
  if (last) ctx_finalize(c);
}

// Free what the context kept for its live matrices, and the context.
void ctx_finalize(ans_ctx* c) {
  DeviceGuard dg(c->device);
  cudaStreamSynchronize(c->aux);
  for (auto& s : c->stage) {
    if (s.h) cudaFreeHost(s.h);
    if (s.ev) cudaEventDestroy(s.ev);
  }
  if (c->h_err_slots) cudaFreeHost(c->h_err_slots);
  cudaStreamDestroy(c->aux);
  delete c;
}

// Discard a block that never left the library (error path).
void block_discard(Block* b, cudaStream_t st) {
  if (!b) return;
  cudaStreamSynchronize(st);
  dev_free(b->ctx, b->mem, b->bytes, st);
  cudaEventDestroy(b->done);
  --b->ctx->blocks;  // callers hold the context's lock and keep it open
  delete b;
}

int block_fill_cache(Block* b) {
  std::lock_guard<std::mutex> g(b->mu);
  if (b->cached) return ANS_OK;
  DeviceGuard dg(b->ctx->device);
  ANS_CUDA(cudaEventSynchronize(b->done));
  b->h_hdr.resize(2 * (size_t)b->nseg);
  b->h_q.resize(b->nseg);
  // headers, quantities and status lie one after another (BlockLayout): one
  // copy of the span instead of three synchronising ones (41 -> 17 us)
  const char* span = (const char*)b->hdr;
  std::vector<char> img((size_t)((const char*)b->status - span) + 4);
  ANS_CUDA(cudaMemcpy(img.data(), span, img.size(), cudaMemcpyDeviceToHost));
  std::memcpy(b->h_hdr.data(), img.data(), b->h_hdr.size() * 8);
  std::memcpy(b->h_q.data(), img.data() + ((const char*)b->q - span), b->h_q.size() * sizeof(ans_quantities));
  std::memcpy(&b->h_status, img.data() + ((const char*)b->status - span), 4);
  if (b->dev_plan) {
    b->base.resize(b->nseg);
    ANS_CUDA(cudaMemcpy(b->base.data(), b->d_base, (size_t)b->nseg * 8, cudaMemcpyDeviceToHost));
    b->cap.resize(b->nseg);
    for (uint32_t s = 0; s < b->nseg; ++s) b->cap[s] = b->h_hdr[2 * (size_t)s + 1];
  }
  b->cached = true;
  return ANS_OK;
}

// A block's host-side padded starts and link bounds (a block planned on the
// device learns them when it completes: this waits for it).
int block_plan(Block* b) { return b->dev_plan ? block_fill_cache(b) : ANS_OK; }

// The status code of a device error word.
int status_of_err(uint32_t err) {
  if (!err) return ANS_OK;
  if (err == kErrNegative) return fail(ANS_ERR_INVALID_ARG, "a signed combination left a negative count");
  if (err & kErrPlan)
    return fail(ANS_ERR_INVALID_ARG, "device batch offsets decrease, hold a window of 2^31 packets or more, "
                                     "or exceed the batch capacity");
  return fail(ANS_ERR_INTERNAL, "device check failed (code " + std::to_string(err) + ")");
}

// The device-side outcome recorded with a block's results.
int block_status(const Block* b) { return status_of_err(b->h_status); }

// Everything the statistics phases of one segment set need.
struct StatsBufs {
  uint32_t* col_ids;
  uint64_t* vals;
  uint32_t* row_ids;
  uint64_t* row_ptr;
  uint64_t* hdr;
  ans_quantities* q;
};

// Host-side plan of a set of segments.
struct HostPlan {
  std::vector<uint64_t> in_off, len, base;
  std::vector<uint64_t> src_at, dst_at;  // per-window array addresses (empty: one input stream)
  std::vector<uint32_t> first_tile;
  uint64_t pad = 0;   // padded items
  uint32_t ntiles = 0;
  void build(const std::vector<uint64_t>& lens, const std::vector<uint64_t>* offs) {
    const size_t n = lens.size();
    in_off.assign(n, 0);
    len = lens;
    base.resize(n);
    first_tile.resize(n + 1);
    uint64_t b = 0, t = 0;
    for (size_t s = 0; s < n; ++s) {
      if (offs) in_off[s] = (*offs)[s];
      base[s] = b;
      first_tile[s] = (uint32_t)t;
      const uint64_t k = tiles_for(lens[s]);
      t += k;
      b += k * kTile;
    }
    first_tile[n] = (uint32_t)t;
    pad = b;
    ntiles = (uint32_t)t;
  }
  // The segments `ids` of `all`, keeping their padded starts (so a pass over
  // this plan writes where one over `all` would).
  void subset(const HostPlan& all, const std::vector<uint32_t>& ids) {
    const size_t n = ids.size();
    in_off.resize(n);
    len.resize(n);
    base.resize(n);
    first_tile.resize(n + 1);
    uint64_t t = 0;
    src_at.clear();
    dst_at.clear();
    for (size_t i = 0; i < n; ++i) {
      in_off[i] = all.in_off[ids[i]];
      if (!all.src_at.empty()) {
        src_at.push_back(all.src_at[ids[i]]);
        dst_at.push_back(all.dst_at[ids[i]]);
      }
      len[i] = all.len[ids[i]];
      base[i] = all.base[ids[i]];
      first_tile[i] = (uint32_t)t;
      t += tiles_for(len[i]);
    }
    first_tile[n] = (uint32_t)t;
    pad = all.pad;
    ntiles = (uint32_t)t;
  }
};

struct DevPlan {
  size_t in_off, len, base, first_tile;
  size_t src_at = 0, dst_at = 0;
  bool addrs = false;
  void reserve(Layout& L, size_t nseg, bool with_addrs = false) {
    in_off = L.add(nseg * 8);
    len = L.add(nseg * 8);
    base = L.add(nseg * 8);
    first_tile = L.add((nseg + 1) * 4);
    addrs = with_addrs;
    if (addrs) {
      src_at = L.add(nseg * 8);
      dst_at = L.add(nseg * 8);
    }
  }
  SegPlan bind(char* m, const HostPlan& hp) const {
    SegPlan p;
    p.in_off = (const uint64_t*)(m + in_off);
    if (addrs) {
      p.src_at = (const uint64_t*)(m + src_at);
      p.dst_at = (const uint64_t*)(m + dst_at);
    }
    p.len = (const uint64_t*)(m + len);
    p.base = (const uint64_t*)(m + base);
    p.first_tile = (const uint32_t*)(m + first_tile);
    p.nseg = (uint32_t)hp.len.size();
    p.ntiles = hp.ntiles;
    return p;
  }
};

// Scratch needed by one sort + statistics pipeline over `pad` padded items and
// `ntiles` tiles.
struct PipeScratch {
  size_t keys_a, keys_b, vals_a, vals_b, seg_hist, st0, st1, lb, lb2, tickets, run_start, row_pos, pre;
  size_t ck_a, ck_b, cv_a, cv_b, col_hist, ulen, bnd;
  size_t cp_cnt, cp_cur, cp_start, cp_hkey, cp_hsum;  // hash partitions of the links by destination
  uint32_t cp_entries = 0;
  // hash-group column statistics of a time sum (buffers for up to
  // hgroup_links links, when reserved)
  size_t hbnd = 0, hitem = 0, higrp = 0, hpart = 0, hheavy = 0, hmeta = 0, hcnt = 0, hbuf = 0, hacc = 0;
  uint64_t hgroup_links = 0;
  uint32_t hgroup_cap = 0;  // parts of cut groups the buffers hold
  void reserve(Layout& L, uint64_t pad, uint32_t nseg, uint32_t ntiles, bool with_vals) {
    ck_a = L.add(pad * 4);
    ck_b = L.add(pad * 4);
    cv_a = L.add(pad * 8);
    cv_b = L.add(pad * 8);
    col_hist = L.add((size_t)nseg * kColPasses * kRadix * 4);
    ulen = L.add((size_t)nseg * 8);
    bnd = L.add((size_t)ntiles * sizeof(ColBnd));
    cp_entries = kColPerTile * ntiles;
    cp_cnt = L.add((size_t)cp_entries * 4);
    cp_cur = L.add((size_t)cp_entries * 4);
    cp_start = L.add((size_t)cp_entries * 4);
    cp_hkey = L.add((size_t)ntiles * kColHeavyPerTile * 4);
    cp_hsum = L.add((size_t)ntiles * kColHeavyPerTile * 16);
    if (with_vals && pad >= kHGroupMinLinks) {
      hgroup_links = pad;
      hgroup_cap = (uint32_t)(2 * (pad / kHGroupPartLinks) + 1);
      hbnd = L.add((size_t)kHGroupBounds * 4);
      hitem = L.add((size_t)kHGroupBounds * 4);
      higrp = L.add(((size_t)kHGroups + hgroup_cap) * 4);
      hpart = L.add((size_t)kHGroupBounds * 4);
      hheavy = L.add((size_t)kHGroups * 4);
      hmeta = L.add(16);
      hcnt = L.add((size_t)hgroup_cap * 4);
      hbuf = L.add((size_t)hgroup_cap * kHGroupPartWords * 4);
      hacc = L.add(3 * sizeof(ColPartAcc));
    }
    keys_a = L.add(pad * 8);
    keys_b = L.add(pad * 8);
    vals_a = with_vals ? L.add(pad * 8) : 0;
    vals_b = with_vals ? L.add(pad * 8) : 0;
    seg_hist = L.add((size_t)nseg * kPasses * kRadix * 4);
    st0 = L.add((size_t)ntiles * 2 * kRadix * 8);  // column passes may run two sub-tiles per tile
    st1 = L.add((size_t)ntiles * 2 * kRadix * 8);
    lb = L.add((size_t)ntiles * 8);
    lb2 = L.add((size_t)ntiles * 8);
    tickets = L.add(kTicketBlocks * 32 * 4);
    run_start = L.add((pad + nseg) * 4);
    row_pos = L.add((pad + nseg) * 4);
    pre = with_vals ? L.add((pad + nseg) * 8) : 0;
  }
};

template <typename T>
T* at(char* m, size_t off) {
  return reinterpret_cast<T*>(m + off);
}

// Sort the (key, value) pairs of the segments of `p` in place: 8 stable digit
// passes ping-ponging between a and b; the result ends in a.
int sort_segments(ans_ctx* c, const SegPlan& p, uint64_t* ka, uint64_t* kb, uint64_t* va, uint64_t* vb,
                  const uint32_t* seg_hist, uint64_t* st0, uint64_t* st1, uint32_t* tickets, cudaStream_t st,
                  const char* name = "onesweep_sum") {
  for (int pass = 0; pass < kPasses; ++pass) {
    const bool even = (pass % 2) == 0;
    KTime kt(c, name, st);
    ANS_CUDA(launch_onesweep(p, pass, even ? ka : kb, even ? kb : ka, even ? va : vb, even ? vb : va, seg_hist,
                             even ? st0 : st1, even ? st1 : st0, tickets + pass, c->d_err, c->cfg_kv, st));
  }
  return ANS_OK;
}

// Scratch of a segmented sample sort (ans_ssort.cu) over plans of up to
// `ntiles` tiles and `nseg` segments; with `two` also for a first split of
// the segments too long for one.
struct SsScratch {
  size_t tree[2] = {0, 0}, cnt[2] = {0, 0}, cur[2] = {0, 0}, bstart[2] = {0, 0}, eq[2] = {0, 0};
  size_t start2 = 0, len2 = 0, parent2 = 0, first_tile2 = 0, tile_seg2 = 0, count2 = 0;
  uint32_t nseg2 = 0, ntiles2 = 0;
  void reserve(Layout& L, uint32_t nseg, uint32_t ntiles, bool two) {
    const uint64_t l1 = two ? ss_level1_buckets((uint64_t)ntiles * kTile, nseg) : 0;
    nseg2 = (uint32_t)(nseg + l1);
    ntiles2 = (uint32_t)(ntiles + l1);
    for (int lv = 0; lv < (two ? 2 : 1); ++lv) {
      const size_t nb = (size_t)kSsPerTile * (lv ? ntiles : ntiles2);
      tree[lv] = L.add(nb * 2 * 8);
      cnt[lv] = L.add(nb * 4);
      cur[lv] = L.add(nb * 4);
      bstart[lv] = L.add(nb * 4);
      eq[lv] = L.add(nb);
    }
    if (two) {
      start2 = L.add((size_t)nseg2 * 8);
      len2 = L.add((size_t)nseg2 * 8);
      parent2 = L.add((size_t)nseg2 * 4);
      first_tile2 = L.add(((size_t)nseg2 + 1) * 4);
      tile_seg2 = L.add((size_t)ntiles2 * 4);
      count2 = L.add(8);
    }
  }
};

// The raw packets of the segments of `p`, packed and sorted into ka (kb and
// ids are scratch).  total and max_len bound the keys in all and the longest
// segment; `two`: some segments may be too long for one split (the scratch
// was reserved for it).
int sample_sort(ans_ctx* c, char* m, const SsScratch& ss, const SegPlan& p, const uint32_t* d_src,
                const uint32_t* d_dst, uint64_t total, uint64_t max_len, bool two, uint64_t* ka, uint64_t* kb,
                uint16_t* ids, cudaStream_t st) {
  SsArgs a;
  a.one_level = ss_one_level(total);
  a.plan = p;
  a.src = d_src;
  a.dst = d_dst;
  a.start = p.base;
  a.len = p.len;
  a.first_tile = p.first_tile;
  a.tile_seg = p.tile_seg;
  a.nseg = p.nseg;
  a.ntiles = p.ntiles;
  a.keys_split = kb;
  a.keys_out = ka;
  a.ids = ids;
  auto level = [&](int lv) {
    a.tree = at<uint64_t>(m, ss.tree[lv]);
    a.cnt = at<uint32_t>(m, ss.cnt[lv]);
    a.cur = at<uint32_t>(m, ss.cur[lv]);
    a.bstart = at<uint32_t>(m, ss.bstart[lv]);
    a.eq = at<uint8_t>(m, ss.eq[lv]);
  };
  if (two) {  // long segments into buckets of keys_a first
    level(1);
    a.level1 = true;
    a.keys_split = ka;
    SsSeg2 o;
    o.start = at<uint64_t>(m, ss.start2);
    o.len = at<uint64_t>(m, ss.len2);
    o.parent = at<uint32_t>(m, ss.parent2);
    o.first_tile = at<uint32_t>(m, ss.first_tile2);
    o.tile_seg = at<uint32_t>(m, ss.tile_seg2);
    o.count = at<uint32_t>(m, ss.count2);
    ANS_CUDA(timed(c, "ss_sample", st, [&] { return launch_ss_sample(a, max_len, st); }));
    ANS_CUDA(timed(c, "ss_count", st, [&] { return launch_ss_count(a, st); }));
    ANS_CUDA(timed(c, "ss_plan", st, [&] { return launch_ss_plan2(a, o, st); }));
    ANS_CUDA(timed(c, "ss_scatter", st, [&] { return launch_ss_scatter(a, st); }));
    a.level1 = false;
    a.keys_in = ka;
    a.keys_split = kb;
    a.start = o.start;
    a.len = o.len;
    a.first_tile = o.first_tile;
    a.tile_seg = o.tile_seg;
    a.parent = o.parent;
    a.nseg_d = o.count;
    a.ntiles_d = o.count + 1;
    a.nseg = ss.nseg2;
    a.ntiles = ss.ntiles2;
    max_len = a.one_level;
  }
  level(0);
  ANS_CUDA(timed(c, "ss_sample", st, [&] { return launch_ss_sample(a, max_len, st); }));
  ANS_CUDA(timed(c, "ss_count", st, [&] { return launch_ss_count(a, st); }));
  ANS_CUDA(timed(c, "ss_scatter", st, [&] { return launch_ss_scatter(a, st); }));
  ANS_CUDA(timed(c, "ss_local", st, [&] { return launch_ss_local(a, st); }));
  return ANS_OK;
}

// The segments whose links are grouped by hash partitions for the column
// statistics: of at most 2^25 links (max_len bounds them; known: on the host).
// Longer ones may meet many times kColMaxParts tables' worth of destinations,
// whose partitions are cut in memory (a batch planned on the device may hold
// such windows: 2^28 links of as many destinations in 25 ms, 44 with the column
// sort and the digit passes of before).  With `narrow` counts, one
// segment of 2^24 links or more takes the hash groups instead.
bool col_parts_ok(const ans_ctx* c, uint64_t max_len, bool known = true) {
  return c->col_hash && (!known || max_len <= (1ull << 25));
}
// Their partition counts and heavy sums over the plan `p` (to be cleared
// before k_finish).
void col_parts_begin(char* m, const PipeScratch& ps, const SegPlan& p, uint64_t max_len, StatsArgs* a, ZeroBatch* z) {
  a->cp.cnt = at<uint32_t>(m, ps.cp_cnt);
  a->cp.cur = at<uint32_t>(m, ps.cp_cur);
  a->cp.start = at<uint32_t>(m, ps.cp_start);
  a->cp.max_parts = col_parts(max_len, std::min<uint64_t>(kColMaxParts, (uint64_t)kColPerTile * p.ntiles));
  a->cp.hkey = at<uint32_t>(m, ps.cp_hkey);
  a->cp.hsum = at<unsigned long long>(m, ps.cp_hsum);
  a->cp.sdst = at<uint32_t>(m, ps.ck_b);
  a->cp.sval = at<uint64_t>(m, ps.cv_b);
  z->add(a->cp.cnt, (size_t)kColPerTile * p.ntiles * 4);
  z->add(a->cp.cur, (size_t)kColPerTile * p.ntiles * 4);
  if (max_len >= kColHeavyLinks) z->add(a->cp.hsum, (size_t)kColHeavyPerTile * p.ntiles * 16);
}
// Their heavy destinations, between the run reduction and k_finish.
int col_parts_heavy(ans_ctx* c, const SegPlan& p, uint64_t max_len, const StatsArgs& a, cudaStream_t st) {
  if (!a.cp.cnt || max_len < kColHeavyLinks) return ANS_OK;
  ANS_CUDA(timed(c, "col_heavy", st, [&] { return launch_col_heavy(p, a.cp, a.col_ids, a.hdr, st); }));
  return ANS_OK;
}

// Column statistics of the segments of a.plan after k_finish: by hash
// partitions (a.cp), or by the transpose-free column sort: the stored links
// (a.col_ids, a.vals) are sorted by destination in four 8-bit
// passes (in -> A -> B -> A -> B) and the destination runs reduced.  Expects
// k_finish to have filled col_hist and ulen and zeroed st0 and the tickets.
// With a.vals32 (counts below 2^32; k_finish wrote the copy into the value
// buffer B) the passes carry uint32 counts.  With a.col_hkeys
// (one segment, vals32: k_finish wrote the mixed destinations there and
// counted their bytes), the passes sort the mixed destinations, and after
// the first two the hash groups are counted (launch_hgroup_stats); if they
// all fit, the segment's length drops to 0 and the rest finds no work.
int column_pass(ans_ctx* c, const StatsArgs& a, const PipeScratch& ps, char* m, ans_quantities* q, cudaStream_t st) {
  const SegPlan& p = a.plan;
  uint64_t* ulen = a.ulen;
  const uint32_t* col_ids = a.col_ids;
  const uint64_t* vals = a.vals;
  const bool vals32 = a.vals32 != nullptr;
  const uint32_t* hkeys = a.col_hkeys;
  uint32_t* tickets = a.col_tickets;
  SegPlan cp = p;
  cp.len = ulen;
  if (a.cp.cnt) {
    uint32_t* pdst = at<uint32_t>(m, ps.ck_a);
    uint64_t* pval = at<uint64_t>(m, ps.cv_a);
    ANS_CUDA(timed(c, "col_scatter", st, [&] {
      return launch_col_scatter(cp, a.cp, col_ids, a.vals32, a.vals, pdst, pval, st);
    }));
    ANS_CUDA(timed(c, "col_count", st, [&] {
      return launch_col_count(cp, a.cp, col_ids, a.vals32, a.vals, pdst, pval, q, st);
    }));
    return ANS_OK;
  }
  uint32_t* ka = at<uint32_t>(m, ps.ck_a);
  uint32_t* kb = at<uint32_t>(m, ps.ck_b);
  uint64_t* va = at<uint64_t>(m, ps.cv_a);
  uint64_t* vb = at<uint64_t>(m, ps.cv_b);
  uint64_t* st0 = at<uint64_t>(m, ps.st0);
  uint64_t* st1 = at<uint64_t>(m, ps.st1);
  uint32_t* hist = at<uint32_t>(m, ps.col_hist);
  if (hkeys && (p.nseg != 1 || !vals32)) return fail(ANS_ERR_INTERNAL, "hash-group column statistics");
  for (int pass = 0; pass < kColPasses; ++pass) {
    if (hkeys && pass == 2) {  // the links grouped by the mix's low 16 bits (keys in B)
      HGroupBufs hb;
      hb.bnd = at<uint32_t>(m, ps.hbnd);
      hb.item_start = at<uint32_t>(m, ps.hitem);
      hb.item_group = at<uint32_t>(m, ps.higrp);
      hb.hpart = at<uint32_t>(m, ps.hpart);
      hb.heavy = at<uint32_t>(m, ps.hheavy);
      hb.meta = at<uint32_t>(m, ps.hmeta);
      hb.hcnt = at<uint32_t>(m, ps.hcnt);
      hb.hbuf = at<uint32_t>(m, ps.hbuf);
      hb.acc = at<ColPartAcc>(m, ps.hacc);
      ANS_CUDA(launch_zero(hb.acc, 3 * sizeof(ColPartAcc), st));
      ANS_CUDA(timed(c, "hgroup", st, [&] {
        return launch_hgroup_stats(kb, (const uint32_t*)vb, ulen, hb, ps.hgroup_cap, q, st);
      }));
    }
    const uint32_t* kin = pass == 0 ? (hkeys ? hkeys : col_ids) : (pass % 2 ? ka : kb);
    uint32_t* kout = pass % 2 ? kb : ka;
    ANS_CUDA(timed(c, "onesweep_col", st, [&] {
      if (vals32) {  // B (the copy, then pass 2's output) -> A -> B
        const uint32_t* vin = (const uint32_t*)(pass % 2 ? va : vb);
        uint32_t* vout = (uint32_t*)(pass % 2 ? vb : va);
        return launch_onesweep_col32(cp, pass, kin, kout, vin, vout, hist, pass % 2 ? st1 : st0,
                                     pass % 2 ? st0 : st1, tickets + pass, c->d_err, c->cfg_col, st);
      }
      const uint64_t* vin = pass == 0 ? vals : (pass % 2 ? va : vb);
      uint64_t* vout = pass % 2 ? vb : va;
      return launch_onesweep_col(cp, pass, kin, kout, vin, vout, hist, pass % 2 ? st1 : st0, pass % 2 ? st0 : st1,
                                 tickets + pass, c->d_err, c->cfg_col, st);
    }));
  }
  ANS_CUDA(timed(c, "colstat", st, [&] {
    if (vals32) return launch_colstat32(cp, kb, (const uint32_t*)vb, at<ColBnd>(m, ps.bnd), q, st);
    return launch_colstat(cp, kb, vb, at<ColBnd>(m, ps.bnd), q, st);
  }));
  return ANS_OK;
}

// A time sum (one segment at base 0) takes the hash-group column statistics
// when its counts are 32-bit, the column hashes are on, it may hold `least`
// or more links (smaller sums sort their 2^16 groups' worth of work faster)
// and the scratch holds the buffers for that many.
bool hgroup_ok(const ans_ctx* c, const SegPlan& p, bool narrow, const PipeScratch& ps,
               uint64_t least = kHGroupMinLinks) {
  const uint64_t links = (uint64_t)p.ntiles * kTile;
  return narrow && c->col_hash && p.nseg == 1 && links >= least && ps.hgroup_cap > 0 &&
         links <= ps.hgroup_links;
}

struct SumPlan {
  HostPlan gp, sp;
  SegPlan g, s;
  Block* blk = nullptr;
};

// The block of a time sum of at most total_cap input links.
int sum_block(ans_ctx* c, uint64_t total_cap, cudaStream_t st, SumPlan* out) {
  out->sp.build(std::vector<uint64_t>{total_cap}, nullptr);
  return make_block(c, out->sp.pad, 1, std::vector<uint64_t>{0}, std::vector<uint64_t>{total_cap}, st, &out->blk);
}

// caps: a bound on each input matrix's links (and the sum's block made by
// sum_block, unless that has been called).  dev_gather (optional): a
// device-resident plan whose segment s covers at least caps[s] items, used
// as the gather plan instead of one built from caps (a batch planned on the
// device: its window plan; caps then holds only the total).
int sum_prepare(ans_ctx* c, char* m, uint32_t k, const std::vector<uint64_t>& caps, size_t off_gplan,
                size_t off_splan, size_t off_lens, size_t off_total, UploadSet& us, cudaStream_t st, SumPlan* out,
                const SegPlan* dev_gather = nullptr) {
  if (!out->blk) {
    uint64_t total_cap = 0;
    for (uint64_t x : caps) total_cap += x;
    ANS_TRY(sum_block(c, total_cap, st, out));
  }
  if (dev_gather) {
    out->g = *dev_gather;
  } else {
    out->gp.build(caps, nullptr);
    DevPlan gdp{off_gplan, off_gplan + align_up(k * 8), off_gplan + 2 * align_up(k * 8),
                off_gplan + 3 * align_up(k * 8)};
    us.add(m + gdp.in_off, out->gp.in_off.data(), k * 8);
    us.add(m + gdp.base, out->gp.base.data(), k * 8);
    us.add(m + gdp.first_tile, out->gp.first_tile.data(), (k + 1) * 4);
    out->g = gdp.bind(m, out->gp);
  }
  out->g.len = at<uint64_t>(m, off_lens);
  DevPlan sdp{off_splan, off_splan + kAlign, off_splan + 2 * kAlign, off_splan + 3 * kAlign};
  us.add(m + sdp.in_off, out->sp.in_off.data(), 8);
  us.add(m + sdp.base, out->sp.base.data(), 8);
  us.add(m + sdp.first_tile, out->sp.first_tile.data(), 8);
  out->s = sdp.bind(m, out->sp);
  out->s.len = at<uint64_t>(m, off_total);
  return ANS_OK;
}

// The header and row pointer of a sum without a tile (every window empty),
// which no kernel of the sum writes.
void zero_empty(Block* blk, ZeroBatch* z) {
  z->add(blk->hdr, 16);
  z->add(blk->row_ptr, 8);
}

// Device half of the time sum of the matrices described by `d_mats` (device
// array of k MatDesc), written into plan->blk.  Uses scratch laid out by the
// caller at `m` / `ps` (which must provide vals buffers).  Only queues work
// on `st` (it may be capturing); on failure the caller discards plan->blk.
int links_to_block(ans_ctx* c, char* m, const PipeScratch& ps, const SegPlan& s, const uint64_t* fk,
                   const uint64_t* fv, Block* blk, cudaStream_t st, bool narrow = false, bool cols = true,
                   uint64_t group_links = kHGroupMinLinks);

// First half of the time sum: the input links gathered and ordered (merge
// rounds, or the kv passes with sum_path 1), left in (*fk, *fv).  Touches
// only the sum's own scratch (keys and values ping-pong, run offsets, the
// look-back words lb / lb2, the digit histograms, the tickets at 32..63) --
// with sum_path 0 none of what a window column pass uses, so it may run
// beside one (col_hist is cleared by the second half).  in_keys / in_vals /
// run_base (merge rounds only): the input links already lie as sorted runs
// at run_base[m] (the window statistics wrote their keys beside the stored
// values), so the gather is skipped and the first round reads them in
// place.  Only queues work.
int sum_order(ans_ctx* c, char* m, const PipeScratch& ps, const MatDesc* d_mats, uint32_t k, SumPlan* plan,
              size_t off_catoff, size_t off_lens, size_t off_total, cudaStream_t st, const uint64_t** fk_out,
              const uint64_t** fv_out, const uint64_t* run_base = nullptr, const uint64_t* in_keys = nullptr,
              const uint64_t* in_vals = nullptr) {
  const HostPlan& sp = plan->sp;
  const SegPlan& g = plan->g;
  const SegPlan& s = plan->s;
  int rc = ANS_OK;

  uint64_t* ka = at<uint64_t>(m, ps.keys_a);
  uint64_t* kb = at<uint64_t>(m, ps.keys_b);
  uint64_t* va = at<uint64_t>(m, ps.vals_a);
  uint64_t* vb = at<uint64_t>(m, ps.vals_b);
  uint32_t* seg_hist = at<uint32_t>(m, ps.seg_hist);
  uint32_t* tickets = at<uint32_t>(m, ps.tickets) + 32;

  auto fail_blk = [&](cudaError_t e, const char* what) {
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  cudaError_t e;
  if ((e = timed(c, "count_prefix", st, [&] { return launch_count_prefix(d_mats, k, at<uint64_t>(m, off_catoff), at<uint64_t>(m, off_lens),
                               at<uint64_t>(m, off_total), st); })) != cudaSuccess)
    return fail_blk(e, "count_prefix");
  // gather zeroes the tickets and, for the radix path, builds the sum
  // segment's histograms and zeroes the sort's first status words (the
  // gather plan has at least as many tiles as the sum plan)
  // sum_path 2 re-sorts a batch's packets; sums of given matrices then merge
  // their sorted links when there are few of them (ceil(log2 k) <= 8 rounds,
  // against the 8 kv passes) and take the kv passes otherwise
  const bool merge = c->sum_path == 0 || (c->sum_path == 2 && k <= 256);
  const uint64_t* cat_off = at<uint64_t>(m, off_catoff);
  const bool in_place = merge && run_base;
  ZeroBatch z;
  z.add(m + ps.lb, (size_t)sp.ntiles * 8);
  z.add(m + ps.lb2, (size_t)sp.ntiles * 8);
  if (!merge) z.add(seg_hist, kPasses * kRadix * 4);
  if (in_place) z.add(tickets, 32 * 4);
  if ((e = launch_zero_batch(z, st)) != cudaSuccess) return fail_blk(e, "memset");
  if (in_place) {
  } else if ((e = timed(c, "gather", st, [&] {
                return launch_gather(g, d_mats, cat_off, ka, va, merge ? nullptr : seg_hist,
                                     merge ? nullptr : at<uint64_t>(m, ps.st0), tickets, st);
              })) != cudaSuccess) {
    return fail_blk(e, "gather");
  }
  const uint64_t *fk = ka, *fv = va;  // the sorted links
  if (merge) {
    const uint64_t* rb = in_place ? run_base : nullptr;
    if (in_place) {
      fk = in_keys;
      fv = in_vals;
    }
    uint64_t *ok = in_place ? ka : kb, *ov = in_place ? va : vb;
    for (int round = 0; (1ull << round) < k; ++round) {
      if ((e = timed(c, "merge", st, [&] {
             return launch_merge(cat_off, rb, k, sp.pad, round, fk, fv, ok, ov, c->merge_tile, st);
           })) != cudaSuccess)
        return fail_blk(e, "merge");
      // the next round reads what this one wrote and writes the other pair
      // (never the window values the first round may have read in place)
      uint64_t *nk = ok == ka ? kb : ka, *nv = ov == va ? vb : va;
      fk = ok;
      fv = ov;
      ok = nk;
      ov = nv;
    }
  } else {
    rc = sort_segments(c, s, ka, kb, va, vb, seg_hist, at<uint64_t>(m, ps.st0), at<uint64_t>(m, ps.st1), tickets, st);
    if (rc != ANS_OK) return rc;
  }
  *fk_out = fk;
  *fv_out = fv;
  return ANS_OK;
}

// narrow: every count of the sum is known to stay below 2^32 (the column
// pass then carries 32-bit counts).
int sum_launch(ans_ctx* c, char* m, const PipeScratch& ps, const MatDesc* d_mats, uint32_t k, SumPlan* plan,
               size_t off_catoff, size_t off_lens, size_t off_total, cudaStream_t st, bool narrow = false,
               bool cols = true, uint64_t group_links = kHGroupMinLinks) {
  const uint64_t *fk = nullptr, *fv = nullptr;
  ANS_TRY(sum_order(c, m, ps, d_mats, k, plan, off_catoff, off_lens, off_total, st, &fk, &fv));
  return links_to_block(c, m, ps, plan->s, fk, fv, plan->blk, st, narrow, cols, group_links);
}

// From sorted (key, value) links (equal keys adjacent) of the single segment
// of `s` to a DCSR block: value prefix, run-length reduction, values as
// prefix differences, row statistics and the column pass (the time sum's
// statistics half).  cols false: without column statistics (a block that is
// only gathered again); group_links: as hgroup_ok's.  Only queues work on `st`.
int links_to_block(ans_ctx* c, char* m, const PipeScratch& ps, const SegPlan& s, const uint64_t* fk,
                   const uint64_t* fv, Block* blk, cudaStream_t st, bool narrow, bool cols, uint64_t group_links) {
  uint32_t* tickets = at<uint32_t>(m, ps.tickets) + 32;
  auto fail_blk = [&](cudaError_t e, const char* what) {
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  cudaError_t e;
  uint64_t* pre = at<uint64_t>(m, ps.pre);
  if ((e = timed(c, "scan_u64", st, [&] { return launch_scan_u64(s, fv, pre, at<uint64_t>(m, ps.lb2), tickets + kPasses + 1, c->d_err, st); })) !=
      cudaSuccess)
    return fail_blk(e, "scan");
  StatsArgs a;
  a.plan = s;
  a.hdr = blk->hdr;
  a.q = blk->q;
  a.keys = fk;
  a.col_ids = blk->col_ids;
  a.vals = blk->vals;
  a.row_ids = blk->row_ids;
  a.row_ptr = blk->row_ptr;
  a.run_start = at<uint32_t>(m, ps.run_start);
  a.row_pos = at<uint32_t>(m, ps.row_pos);
  a.pre = pre;
  a.lookback = at<uint64_t>(m, ps.lb);
  a.ticket = tickets + kPasses;
  a.col_hist = at<uint32_t>(m, ps.col_hist);
  a.ulen = at<uint64_t>(m, ps.ulen);
  a.col_st0 = at<uint64_t>(m, ps.st0);
  uint32_t* col_tickets = at<uint32_t>(m, ps.tickets) + 3 * 32;
  a.col_tickets = col_tickets;
  a.err = c->d_err;
  a.mode = kModeSum;
  if (narrow) a.vals32 = (uint32_t*)at<uint64_t>(m, ps.cv_b);
  a.no_cols = !cols;
  if (cols && hgroup_ok(c, s, narrow, ps, group_links)) a.col_hkeys = at<uint32_t>(m, ps.ck_b);
  const uint64_t most = (uint64_t)s.ntiles * kTile;
  ZeroBatch z;
  z.add(blk->q, sizeof(ans_quantities));
  if (s.ntiles == 0) zero_empty(blk, &z);
  if (cols && !a.col_hkeys && col_parts_ok(c, most)) col_parts_begin(m, ps, s, most, &a, &z);
  else z.add(m + ps.col_hist, kColPasses * kRadix * 4);
  if ((e = launch_zero_batch(z, st)) != cudaSuccess) return fail_blk(e, "memset");
  if ((e = timed(c, "rle", st, [&] { return launch_rle(a, st); })) != cudaSuccess) return fail_blk(e, "rle");
  ANS_TRY(col_parts_heavy(c, s, most, a, st));
  if ((e = timed(c, "finish", st, [&] { return launch_finish(a, st); })) != cudaSuccess) return fail_blk(e, "finish");
  return cols ? column_pass(c, a, ps, m, blk->q, st) : ANS_OK;
}

// Time sum of a batch from its packets (sum_path 2): every packet of the
// batch, as the one segment of `pk`, is sorted again, and the sorted keys are
// reduced like a window (counts = run lengths) into `blk`, with the sum's row
// and column statistics.  Runs after the window statistics, whose key
// buffers, status words and tickets it reuses.  Only queues work on `st`.
int sum_packets(ans_ctx* c, char* m, const PipeScratch& ps, const SegPlan& pk, const uint32_t* d_src,
                const uint32_t* d_dst, Block* blk, cudaStream_t st, bool narrow, const SsScratch& ss, uint64_t total,
                bool two) {
  uint64_t* ka = at<uint64_t>(m, ps.keys_a);
  uint64_t* kb = at<uint64_t>(m, ps.keys_b);
  uint32_t* tickets = at<uint32_t>(m, ps.tickets);
  auto cu = [&](cudaError_t e, const char* what) -> int {
    if (e == cudaSuccess) return ANS_OK;
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  int rc;
  StatsArgs a;
  if (hgroup_ok(c, pk, narrow, ps)) a.col_hkeys = at<uint32_t>(m, ps.ck_b);
  ZeroBatch z;
  z.add(m + ps.lb, (size_t)pk.ntiles * 8);
  z.add(blk->q, sizeof(ans_quantities));
  z.add(tickets, 32 * 4);
  if (pk.ntiles == 0) zero_empty(blk, &z);
  if (!a.col_hkeys && col_parts_ok(c, total)) col_parts_begin(m, ps, pk, total, &a, &z);
  else z.add(m + ps.col_hist, kColPasses * kRadix * 4);
  if ((rc = cu(launch_zero_batch(z, st), "memset")) ||
      (rc = sample_sort(c, m, ss, pk, d_src, d_dst, total, total, two, ka, kb, at<uint16_t>(m, ps.ck_a), st)))
    return rc;
  a.plan = pk;
  a.hdr = blk->hdr;
  a.q = blk->q;
  a.keys = ka;
  a.col_ids = blk->col_ids;
  a.vals = blk->vals;
  a.row_ids = blk->row_ids;
  a.row_ptr = blk->row_ptr;
  a.run_start = at<uint32_t>(m, ps.run_start);
  a.row_pos = at<uint32_t>(m, ps.row_pos);
  if (narrow) a.vals32 = (uint32_t*)at<uint64_t>(m, ps.cv_b);
  a.lookback = at<uint64_t>(m, ps.lb);
  a.ticket = tickets + kPasses;
  a.col_hist = at<uint32_t>(m, ps.col_hist);
  a.ulen = at<uint64_t>(m, ps.ulen);
  a.col_st0 = at<uint64_t>(m, ps.st0);
  a.col_tickets = tickets + 3 * 32;
  a.err = c->d_err;
  a.mode = kModeWindow;
  if ((rc = cu(timed(c, "rle", st, [&] { return launch_rle(a, st); }), "rle"))) return rc;
  ANS_TRY(col_parts_heavy(c, pk, total, a, st));
  if ((rc = cu(timed(c, "finish", st, [&] { return launch_finish(a, st); }), "finish"))) return rc;
  return column_pass(c, a, ps, m, blk->q, st);
}

// Snapshot the device error word into `dst` (device); reset_err clears it.
// (kernels: no copy engine, see UploadSet)
int capture_err(ans_ctx* c, uint32_t* dst_dev, cudaStream_t st) {
  ANS_CUDA(launch_copy_word(dst_dev, c->d_err, st));
  return ANS_OK;
}
int reset_err(ans_ctx* c, cudaStream_t st) {
  ANS_CUDA(launch_zero(c->d_err, 4, st));
  return ANS_OK;
}

// A ticket's word in the pinned ring, to receive the device error word before
// the ticket's event.
uint32_t take_err_slot(ans_ctx* c) {
  const uint32_t slot = (uint32_t)c->err_next;
  c->err_next = (c->err_next + 1) % kErrSlots;
  c->h_err_slots[slot] = 0;
  return slot;
}
int add_ticket(ans_ctx* c, cudaStream_t st, uint32_t slot, ans_ticket* out) {
  ans_ctx::Ticket t;
  ANS_CUDA(cudaEventCreateWithFlags(&t.ev, cudaEventDisableTiming));
  t.slot = (int)slot;
  ANS_CUDA(cudaEventRecord(t.ev, st));
  const uint64_t id = c->next_ticket++;
  c->tickets[id] = t;
  *out = id;
  return ANS_OK;
}
int new_ticket(ans_ctx* c, cudaStream_t st, ans_ticket* out) {
  const uint32_t slot = take_err_slot(c);
  ANS_CUDA(cudaMemcpyAsync(c->h_err_slots + slot, c->d_err, 4, cudaMemcpyDeviceToHost, st));
  return add_ticket(c, st, slot, out);
}

// `ptr` as kernels of this device can address it (its own memory, page-locked
// or managed host memory), or null.
void* addressable(void* ptr) {
  cudaPointerAttributes pa{};
  int dev = -1;
  const bool known = cudaPointerGetAttributes(&pa, ptr) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess;
  if (!known) cudaGetLastError();
  const bool ok = known && (pa.type == cudaMemoryTypeHost || pa.type == cudaMemoryTypeManaged ||
                            (pa.type == cudaMemoryTypeDevice && pa.device == dev));
  if (!ok) return nullptr;
  return pa.devicePointer ? pa.devicePointer : ptr;
}

// The quantities to the caller's array: by a kernel when the device can
// address it (see UploadSet for why not the copy engines), else by
// cudaMemcpyAsync.
int copy_quantities_out(ans_quantities* out, const ans_quantities* src, size_t n, cudaStream_t st) {
  if (!out || n == 0) return ANS_OK;
  if (void* dst = addressable(out)) {
    SmallCopyBatch b;
    b.it[b.n++] = SmallCopyItem{dst, src, n * sizeof(ans_quantities)};
    ANS_CUDA(launch_small_copy(b, st));
    return ANS_OK;
  }
  ANS_CUDA(cudaMemcpyAsync(out, src, n * sizeof(ans_quantities), cudaMemcpyDefault, st));
  return ANS_OK;
}

// Key of the cached executable graph for a batch: what decides its topology
// and kernel functions (the launch sequence zeroes scratch with kernels, so
// sizes only change node parameters, which cudaGraphExecUpdate applies).
std::string launch_sig(uint32_t flags, bool any_tiles, bool any_small, bool any_big, int rounds, const ans_ctx* c) {
  std::string k = std::to_string(flags) + "/" + std::to_string(any_tiles) + std::to_string(any_small) +
                  std::to_string(any_big) + "/" + std::to_string(rounds) + "/" + std::to_string(c->win_path) +
                  std::to_string(c->sum_path) + std::to_string(c->agg_path) + std::to_string(c->col_hash) + "/" +
                  std::to_string(c->merge_tile);
  for (const SortCfg* f : {&c->cfg_keys, &c->cfg_kv, &c->cfg_col, &c->cfg_win})
    k += "/" + std::to_string(f->threads) + std::to_string(f->rank) + std::to_string(f->blocks);
  return k;
}

// Run `fn(stream)` (which only queues work) on `st`, directly or through the
// context's graph cache.
template <typename F>
int run_launches(ans_ctx* c, cudaStream_t st, const std::string& key, F&& fn) {
  if (!c->side) ANS_CUDA(cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking));
  if (!c->ev_fork) ANS_CUDA(cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming));
  if (!c->ev_join) ANS_CUDA(cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming));
  if (!c->graph || c->prof.on) return fn(st);
  if (!c->cap) ANS_CUDA(cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking));
  cudaGraph_t g = nullptr;
  int rc = ANS_OK;
  cudaError_t e = cudaSuccess;
  {
    RecordGuard rg;
    ANS_CUDA(cudaStreamBeginCapture(c->cap, cudaStreamCaptureModeThreadLocal));
    rc = fn(c->cap);
    e = cudaStreamEndCapture(c->cap, &g);
  }
  if (rc != ANS_OK || e != cudaSuccess) {
    // (the caller's own wait for the device in another thread breaks a recording
    // off, too; nothing of it has run: launched directly, which reports what
    // else may be wrong)
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return fn(st);
  }
  auto it = c->graphs.find(key);
  if (it != c->graphs.end()) {
    cudaGraphExecUpdateResultInfo info;
    if (cudaGraphExecUpdate(it->second, g, &info) != cudaSuccess) {
      cudaGetLastError();
      cudaGraphExecDestroy(it->second);
      c->graphs.erase(it);
      it = c->graphs.end();
    }
  }
  if (it == c->graphs.end()) {
    if (c->graphs.size() >= 8) {  // keep a few shapes
      cudaGraphExecDestroy(c->graphs.begin()->second);
      c->graphs.erase(c->graphs.begin());
    }
    cudaGraphExec_t ex = nullptr;
    const cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
    if (ie != cudaSuccess) {
      cudaGraphDestroy(g);
      return fail(ANS_ERR_CUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(ie));
    }
    it = c->graphs.emplace(key, ex).first;
  }
  cudaGraphDestroy(g);
  ANS_CUDA(cudaGraphLaunch(it->second, st));
  return ANS_OK;
}

// Hash path: window s gets a table of 2^lg[s] >= 2 * lens[s] slots (at
// least one tile; none for an empty window); `tab` lays the tables out as
// segments of the arena.
void plan_tables(const std::vector<uint64_t>& lens, std::vector<uint32_t>* lg, HostPlan* tab) {
  std::vector<uint64_t> slots(lens.size());
  lg->resize(lens.size());
  for (size_t s = 0; s < lens.size(); ++s) {
    uint32_t l = 13;  // kTile slots
    while ((1ull << l) < 2 * lens[s]) ++l;
    (*lg)[s] = l;
    slots[s] = lens[s] ? (1ull << l) : 0;
  }
  tab->build(slots, nullptr);
}

// agg_path 3: the time sum comes from the batch's packets, sorted as one
// segment, for batches with a time sum, two or more windows (at most 2^16)
// and the packets in one stream.
bool agg_packets(const ans_ctx* c, uint32_t nseg, bool want_sum, bool addrs) {
  return c->agg_path == 3 && want_sum && nseg >= 2 && nseg <= kMaxPacketWindows && !addrs;
}

// Scratch layout of one batch (shared by run_windows and ans_batch_bytes).
struct WinLayout {
  DevPlan dp, dp_big;  // every window; the windows sorted by the sample sort
  size_t off_small = 0;  // ids of the windows sorted on chip
  size_t off_tileseg = 0; // the window plan's segment of every tile
  DevPlan dp_tab;        // hash path: the windows' tables as segments
  DevPlan dp_pk;         // sum_path 2: all packets of the batch as one segment
  size_t off_tlg = 0, off_special = 0, off_hulen = 0, off_nclaim = 0, off_claims = 0;
  PipeScratch ps;
  SsScratch ss;
  bool ss_two_win = false, ss_two_pk = false;  // windows, or the batch as one segment, beyond one split
  size_t s_col = 0, s_vals = 0, s_row = 0, s_rp = 0, s_hdr = 0, s_q = 0;
  size_t off_mats = 0, off_gplan = 0, off_splan = 0, off_catoff = 0, off_lens = 0, off_total = 0;
  size_t size = 0;
  // total, max_len: the batch's packets, its longest window (bounds, when
  // the batch is planned on the device).
  void reserve(const HostPlan& hp, uint32_t nseg, bool want_mats, bool want_sum, uint64_t total, uint64_t max_len,
               bool hash = false) {
    Layout L;
    const bool addrs = !hp.src_at.empty();
    dp.reserve(L, nseg, addrs);
    dp_big.reserve(L, nseg, addrs);
    off_small = L.add((size_t)nseg * 4);
    off_tileseg = L.add((size_t)hp.ntiles * 4);
    dp_pk.reserve(L, 1);
    if (hash) {
      dp_tab.reserve(L, nseg);
      off_tlg = L.add((size_t)nseg * 4);
      off_special = L.add((size_t)nseg * 8);
      off_hulen = L.add((size_t)nseg * 8);
      off_nclaim = L.add((size_t)nseg * 8);
      off_claims = L.add(hp.pad * 4);
    }
    ps.reserve(L, hp.pad, std::max<uint32_t>(nseg, 1), hp.ntiles, want_sum || hash);
    ss_two_win = max_len > ss_one_level(total);
    ss_two_pk = want_sum && total > ss_one_level(total);
    ss.reserve(L, std::max<uint32_t>(nseg, 1), hp.ntiles, ss_two_win || ss_two_pk);
    if (!want_mats) {  // the DCSR arrays are intermediate: keep them in scratch
      s_col = L.add(hp.pad * 4);
      s_vals = L.add(hp.pad * 8);
      s_row = L.add(hp.pad * 4);
      s_rp = L.add((hp.pad + nseg) * 8);
      s_hdr = L.add((size_t)nseg * 16);
      s_q = L.add((size_t)nseg * sizeof(ans_quantities));
    }
    if (want_sum) {
      off_mats = L.add((size_t)nseg * sizeof(MatDesc));
      off_gplan = L.add(4 * align_up((size_t)(nseg + 1) * 8));
      off_splan = L.add(4 * kAlign);
      off_catoff = L.add(((size_t)nseg + 1) * 8);
      off_lens = L.add((size_t)nseg * 8);
      off_total = L.add(8);
    }
    size = L.size;
  }
};

// The batch pipeline (also serves ans_build_window with nwin == 1).  feed (or
// empty) queues on `st` what fills the packet arrays, once all the batch's
// memory is held: a batch refused for memory leaves nothing queued that reads
// the caller's arrays.
int run_windows(ans_ctx* c, const uint32_t* d_src, const uint32_t* d_dst, const uint64_t* h_offsets,
                size_t nwin, uint32_t flags, ans_quantities* out, ans_matrix** per_window, ans_matrix** sum,
                ans_ticket* ticket, cudaStream_t st, const uint32_t* const* h_srcs = nullptr,
                const uint32_t* const* h_dsts = nullptr, const uint64_t* d_offsets = nullptr,
                uint64_t dev_cap = 0, const std::function<int()>& feed = {}) {
  // dev: the offsets live on the device and the batch is planned there
  // (launch_plan); the host sizes everything for dev_cap packets.
  const bool dev = d_offsets != nullptr;
  if (nwin > 0xFFFFFFF0ull) return fail(ANS_ERR_INVALID_ARG, "too many windows");
  std::vector<uint64_t> lens(nwin), offs(nwin);
  uint64_t total = dev_cap;
  if (!dev) {
    for (size_t w = 0; w < nwin; ++w) {
      if (h_offsets[w + 1] < h_offsets[w]) return fail(ANS_ERR_INVALID_ARG, "offsets must be nondecreasing");
      lens[w] = h_offsets[w + 1] - h_offsets[w];
      if (lens[w] > kMaxWindow) return fail(ANS_ERR_INVALID_ARG, "a window exceeds 2^31 - 1 packets");
      offs[w] = h_offsets[w];
    }
    total = h_offsets[nwin] - h_offsets[0];
  }
  uint64_t max_len = dev ? total : 0;
  bool maybe_empty = dev;  // segments without a tile, whose outputs no tile writes
  for (uint64_t l : lens) {
    max_len = std::max(max_len, l);
    maybe_empty = maybe_empty || l == 0;
  }
  if (total && !h_srcs && (!d_src || !d_dst)) return fail(ANS_ERR_INVALID_ARG, "NULL packet arrays");
  const bool want_mats = (flags & ANS_BATCH_MATRICES) != 0;
  const bool want_sum = (flags & ANS_BATCH_SUM) != 0;
  if (want_sum && total > kMaxWindow) return fail(ANS_ERR_INVALID_ARG, "a time sum is limited to 2^31 - 1 links");
  const uint32_t nseg = (uint32_t)nwin;

  HostPlan hp;
  if (dev) {  // a bound: every window may add up to one tile of padding
    const uint64_t nt = nseg ? tiles_for(total) + nseg : 0;
    if (nt > 0xFFFFFFF0ull) return fail(ANS_ERR_INVALID_ARG, "batch capacity too large");
    hp.in_off.assign(nseg, 0);
    hp.len.assign(nseg, 0);
    hp.base.assign(nseg, 0);
    hp.first_tile.assign(nseg + 1, 0);
    hp.ntiles = (uint32_t)nt;
    hp.pad = nt * kTile;
  } else {
    hp.build(lens, &offs);
  }
  if ((uint64_t)hp.ntiles * kTile != hp.pad) return fail(ANS_ERR_INTERNAL, "plan");
  if (h_srcs) {  // every window's own arrays
    hp.src_at.resize(nwin);
    hp.dst_at.resize(nwin);
    for (size_t w = 0; w < nwin; ++w) {
      hp.src_at[w] = (uint64_t)(uintptr_t)h_srcs[w];
      hp.dst_at[w] = (uint64_t)(uintptr_t)h_dsts[w];
    }
  }
  // Which windows are sorted on chip (one cluster each) and which by the
  // sample sort.
  std::vector<uint32_t> small_ids, big_ids;
  const int win_path = c->win_path;  // the caller holds c->mu
  const SortCfg cfg_win = c->cfg_win;
  const bool packets = agg_packets(c, nseg, want_sum, h_srcs != nullptr);
  const bool on_chip = !dev && win_path == 0 && !packets &&
                       cluster_sort_clusters(c->device) > 0;
  for (uint32_t s = 0; s < nseg; ++s) {
    if (on_chip && lens[s] <= kClusterWindowMax) small_ids.push_back(s);
    else big_ids.push_back(s);
  }
  HostPlan hp_big;
  if (dev) hp_big = hp;  // planned on the device: the sample sort takes every window
  else hp_big.subset(hp, big_ids);
  // Hash path: one table per window of 2^lg >= 2 * packets slots (at least
  // one tile; none for an empty window), as segments of the table arena.
  const bool hash = c->agg_path == 1 && nseg > 0;
  HostPlan hp_tab;
  std::vector<uint32_t> tab_lg;
  if (hash && dev) {  // a bound: 2^lg < max(2^13 + 1, 4 * packets)
    hp_tab.pad = (uint64_t)nseg * (1ull << 13) + 4 * total;
  } else if (hash) {
    plan_tables(lens, &tab_lg, &hp_tab);
  }

  // ---- scratch layout (with guards after every region in debug mode)
  WinLayout wl;
  std::vector<size_t> guard_off;
  {
    GuardSink gs(c->guards ? &guard_off : nullptr);
    wl.reserve(hp, nseg, want_mats, want_sum, total, max_len, hash);
  }
  const DevPlan& dp = wl.dp;
  const PipeScratch& ps = wl.ps;
  const size_t s_col = wl.s_col, s_vals = wl.s_vals, s_row = wl.s_row, s_rp = wl.s_rp, s_hdr = wl.s_hdr,
               s_q = wl.s_q;
  const size_t off_mats = wl.off_mats, off_gplan = wl.off_gplan, off_splan = wl.off_splan,
               off_catoff = wl.off_catoff, off_lens = wl.off_lens, off_total = wl.off_total;

  ANS_TRY(ensure_scratch(c, wl.size, st));
  if (hash) ANS_TRY(ensure_hash(c, hp_tab.pad, st));
  char* m = (char*)c->scratch;

  Block* blk = nullptr;
  if (want_mats && nseg > 0) {
    if (dev) {
      ANS_TRY(make_block(c, hp.pad, nseg, {}, {}, st, &blk, true));
    } else {
      std::vector<uint64_t> caps(lens);
      ANS_TRY(make_block(c, hp.pad, nseg, hp.base, caps, st, &blk));
    }
  }
  StatsBufs sb;
  if (blk) {
    sb = {blk->col_ids, blk->vals, blk->row_ids, blk->row_ptr, blk->hdr, blk->q};
  } else {
    sb = {at<uint32_t>(m, s_col), at<uint64_t>(m, s_vals), at<uint32_t>(m, s_row), at<uint64_t>(m, s_rp),
          at<uint64_t>(m, s_hdr), at<ans_quantities>(m, s_q)};
  }
  SumPlan sump;
  Block* sblk = nullptr;
  bool queued = false;  // work that reads the caller's arrays
  auto bail = [&](int rc) {
    if (queued) cudaStreamSynchronize(st);
    block_discard(blk, st);
    block_discard(sump.blk, st);
    block_discard(sblk, st);
    return rc;
  };

  int rc = ANS_OK;
  if (want_sum && nseg && (rc = sum_block(c, total, st, &sump))) return bail(rc);
  // (all the batch's memory is held; the rest of the planning runs beside the
  // filling: a served batch of 100 windows 845 us with the filling after it, 835
  // so; 827 with the filling before anything is asked for)
  if (feed) {
    queued = true;
    if ((rc = feed())) return bail(rc);
  }

  // ---- host-side preparation: plans and matrix descriptors; every small
  // array goes to the device in one staged upload.
  UploadSet us;
  if (nseg && !dev) {
    us.add(m + dp.in_off, hp.in_off.data(), nseg * 8);
    us.add(m + dp.len, hp.len.data(), nseg * 8);
    us.add(m + dp.base, hp.base.data(), nseg * 8);
    us.add(m + dp.first_tile, hp.first_tile.data(), (nseg + 1) * 4);
    if (dp.addrs) {
      us.add(m + dp.src_at, hp.src_at.data(), nseg * 8);
      us.add(m + dp.dst_at, hp.dst_at.data(), nseg * 8);
    }
  }
  if (!small_ids.empty()) us.add(m + wl.off_small, small_ids.data(), small_ids.size() * 4);
  // sum_path 2: all packets of the batch as one segment (device-planned
  // batches: its offset and length come from the planner, the tile count is
  // the capacity's)
  const bool sum_pk = want_sum && nseg && (c->sum_path == 2 || packets) && !h_srcs;
  HostPlan hp_pk;
  if (sum_pk) {
    std::vector<uint64_t> pk_off{dev ? 0 : h_offsets[0]};
    hp_pk.build(std::vector<uint64_t>{total}, &pk_off);
    if (!dev) {
      us.add(m + wl.dp_pk.in_off, hp_pk.in_off.data(), 8);
      us.add(m + wl.dp_pk.len, hp_pk.len.data(), 8);
    }
    us.add(m + wl.dp_pk.base, hp_pk.base.data(), 8);
    us.add(m + wl.dp_pk.first_tile, hp_pk.first_tile.data(), 8);
  }
  if (hash && !dev) {
    us.add(m + wl.dp_tab.base, hp_tab.base.data(), nseg * 8);
    us.add(m + wl.off_tlg, tab_lg.data(), nseg * 4);
  }
  if (!hash && !big_ids.empty() && !dev) {
    const size_t nb = big_ids.size();
    us.add(m + wl.dp_big.in_off, hp_big.in_off.data(), nb * 8);
    us.add(m + wl.dp_big.len, hp_big.len.data(), nb * 8);
    us.add(m + wl.dp_big.base, hp_big.base.data(), nb * 8);
    us.add(m + wl.dp_big.first_tile, hp_big.first_tile.data(), (nb + 1) * 4);
    if (wl.dp_big.addrs) {
      us.add(m + wl.dp_big.src_at, hp_big.src_at.data(), nb * 8);
      us.add(m + wl.dp_big.dst_at, hp_big.dst_at.data(), nb * 8);
    }
  }
  SegPlan p = dp.bind(m, hp);
  if (nseg > 1) p.tile_seg = at<uint32_t>(m, wl.off_tileseg);  // filled at the head of the launch sequence
  std::vector<MatDesc> md;
  if (want_sum && nseg && dev) {  // descriptors written by the device planner; the window plan gathers
    if ((rc = sum_prepare(c, m, nseg, std::vector<uint64_t>{total}, off_gplan, off_splan, off_lens, off_total, us,
                          st, &sump, &p)))
      return bail(rc);
  } else if (want_sum && nseg) {
    md.resize(nseg);
    for (uint32_t s = 0; s < nseg; ++s) {
      md[s].row_ids = sb.row_ids + hp.base[s];
      md[s].row_ptr = sb.row_ptr + hp.base[s] + s;
      md[s].col_ids = sb.col_ids + hp.base[s];
      md[s].vals = sb.vals + hp.base[s];
      md[s].hdr = sb.hdr + 2 * (size_t)s;
    }
    us.add(m + off_mats, md.data(), md.size() * sizeof(MatDesc));
    if ((rc = sum_prepare(c, m, nseg, lens, off_gplan, off_splan, off_lens, off_total, us, st, &sump)))
      return bail(rc);
  }
  if ((rc = us.flush(c, st))) return bail(rc);

  auto cu = [&](cudaError_t e, const char* what) -> int {
    if (e == cudaSuccess) return ANS_OK;
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  std::vector<uint64_t> guard_addr;
  for (size_t o : guard_off) guard_addr.push_back((uint64_t)(uintptr_t)(m + o));
  if ((rc = cu(run_guards(guard_addr, nullptr, st), "guards"))) return bail(rc);
  // Empty batch with a time sum: an empty sum matrix.
  if (want_sum && nseg == 0) {
    if ((rc = make_block(c, 0, 1, {0}, {0}, st, &sblk))) return bail(rc);
  }
  // ---- the launch sequence (every kernel and memset of the batch), run on
  // `ls`: the caller's stream, or a capture stream when it is recorded into a
  // CUDA graph.  Host-side state is only read here.
  auto launch_all = [&](cudaStream_t ls) -> int {
    int rc = ANS_OK;
    // With merge rounds, the sum's first half runs on the side stream from
    // the end of the window statistics, beside the window column pass.
    bool forked = false;
    const uint64_t *sfk = nullptr, *sfv = nullptr;
    uint64_t* ka = at<uint64_t>(m, ps.keys_a);
    uint64_t* kb = at<uint64_t>(m, ps.keys_b);
    uint32_t* seg_hist = at<uint32_t>(m, ps.seg_hist);
    uint32_t* tickets = at<uint32_t>(m, ps.tickets);
    if (nseg && dev) {  // the plan of the batch, from the device-resident offsets
      DevPlanOut o;
      o.in_off = at<uint64_t>(m, dp.in_off);
      o.len = at<uint64_t>(m, dp.len);
      o.base = at<uint64_t>(m, dp.base);
      o.first_tile = at<uint32_t>(m, dp.first_tile);
      if (hash) {
        o.tab_lg = at<uint32_t>(m, wl.off_tlg);
        o.tab_base = at<uint64_t>(m, wl.dp_tab.base);
      }
      if (blk) o.blk_base = blk->d_base;
      if (sum_pk) {
        o.pk_in_off = at<uint64_t>(m, wl.dp_pk.in_off);
        o.pk_len = at<uint64_t>(m, wl.dp_pk.len);
      }
      if (want_sum) {
        o.md = at<MatDesc>(m, off_mats);
        o.row_ids = sb.row_ids;
        o.row_ptr = sb.row_ptr;
        o.col_ids = sb.col_ids;
        o.vals = sb.vals;
        o.hdr = sb.hdr;
      }
      if ((rc = cu(timed(c, "plan", ls, [&] { return launch_plan(d_offsets, nseg, total, o, c->d_err, ls); }),
                   "plan")))
        return rc;
    }
    if (p.tile_seg && (rc = cu(launch_tile_seg(p, at<uint32_t>(m, wl.off_tileseg), ls), "tile segments")))
      return rc;
    if (nseg) {
      StatsArgs a;
      ZeroBatch z;
      z.add(sb.q, (size_t)nseg * sizeof(ans_quantities));
      z.add(m + ps.lb, (size_t)hp.ntiles * 8);
      z.add(tickets, 32 * 4);
      if (col_parts_ok(c, max_len, !dev)) col_parts_begin(m, ps, p, max_len, &a, &z);
      else z.add(m + ps.col_hist, (size_t)nseg * kColPasses * kRadix * 4);
      if ((rc = cu(launch_zero_batch(z, ls), "memset"))) return rc;
      SegPlan pw = p;  // the plan of the statistics phases
      int mode = kModeWindow;
      uint64_t* pre = nullptr;
      if (hash) {
        HashTabs h;
        h.keys = (uint64_t*)c->hash_mem;
        h.cnt = (uint32_t*)((char*)c->hash_mem + c->hash_slots * 8);
        h.off = at<uint64_t>(m, wl.dp_tab.base);
        h.lg = at<uint32_t>(m, wl.off_tlg);
        h.special = at<uint64_t>(m, wl.off_special);
        h.claims = at<uint32_t>(m, wl.off_claims);
        h.nclaim = at<uint64_t>(m, wl.off_nclaim);
        uint64_t* hulen = at<uint64_t>(m, wl.off_hulen);
        uint64_t* va = at<uint64_t>(m, ps.vals_a);
        uint64_t* vb = at<uint64_t>(m, ps.vals_b);
        pre = at<uint64_t>(m, ps.pre);
        if ((rc = cu(launch_zero(h.special, (size_t)nseg * 8, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(h.nclaim, (size_t)nseg * 8, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(hulen, (size_t)nseg * 8, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(seg_hist, (size_t)nseg * kPasses * kRadix * 4, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(m + ps.lb2, (size_t)hp.ntiles * 8, ls), "memset"))) return rc;
        c->hash_dirty = true;  // until the compaction that empties the tables is queued
        if ((rc = cu(timed(c, "hash_insert", ls, [&] { return launch_hash_insert(p, d_src, d_dst, h, c->d_err, ls); }),
                     "hash insert")))
          return rc;
        SegPlan pc = p;
        pc.len = h.nclaim;
        if ((rc = cu(timed(c, "hash_compact", ls, [&] {
                       return launch_hash_compact(pc, h, hulen, ka, va, seg_hist, at<uint64_t>(m, ps.st0), tickets, ls);
                     }), "hash compact")))
          return rc;
        c->hash_dirty = false;
        pw.len = hulen;
        if ((rc = sort_segments(c, pw, ka, kb, va, vb, seg_hist, at<uint64_t>(m, ps.st0), at<uint64_t>(m, ps.st1),
                                tickets, ls, "onesweep_hash")))
          return rc;
        if ((rc = cu(timed(c, "scan_u64", ls, [&] {
                       return launch_scan_u64(pw, va, pre, at<uint64_t>(m, ps.lb2), tickets + kPasses + 1, c->d_err, ls);
                     }), "scan")))
          return rc;
        mode = kModeSum;
      }
      if (!hash && !small_ids.empty()) {
        const uint32_t* ids = small_ids.size() == nseg ? nullptr : at<uint32_t>(m, wl.off_small);
        if ((rc = cu(timed(c, "cluster_sort", ls, [&] {
                       return launch_cluster_sort(p, ids, (uint32_t)small_ids.size(), d_src, d_dst, ka, tickets,
                                                  cfg_win, ls);
                     }), "cluster sort")))
          return rc;
      }
      if (!hash && !big_ids.empty()) {
        const SegPlan pb = dev || big_ids.size() == nseg ? p : wl.dp_big.bind(m, hp_big);
        if ((rc = sample_sort(c, m, wl.ss, pb, d_src, d_dst, total, max_len, wl.ss_two_win, ka, kb,
                              at<uint16_t>(m, ps.ck_a), ls)))
          return rc;
      }
      a.plan = pw;
      a.hdr = sb.hdr;
      a.q = sb.q;
      a.keys = ka;
      a.col_ids = sb.col_ids;
      a.vals = sb.vals;
      a.row_ids = sb.row_ids;
      a.row_ptr = sb.row_ptr;
      a.run_start = at<uint32_t>(m, ps.run_start);
      a.row_pos = at<uint32_t>(m, ps.row_pos);
      a.pre = pre;
      a.vals32 = (uint32_t*)at<uint64_t>(m, ps.cv_b);  // window counts fit 31 bits
      a.lookback = at<uint64_t>(m, ps.lb);
      a.ticket = tickets + kPasses;
      a.col_hist = at<uint32_t>(m, ps.col_hist);
      a.ulen = at<uint64_t>(m, ps.ulen);
      a.col_st0 = at<uint64_t>(m, ps.st0);
      a.col_tickets = tickets + 2 * 32;
      a.err = c->d_err;
      a.mode = mode;
      // With merge rounds, the run reduction also writes each link's key
      // beside its stored value (keys_b at the window's padded base): the
      // windows' links are then the time sum's sorted input runs in place.
      // (windows whose matrices nobody reads keep neither counts nor row ids)
      if (!want_mats && (!want_sum || sum_pk)) {
        a.vals = nullptr;
        a.row_ids = nullptr;
      }
      const bool in_place = want_sum && c->sum_path == 0 && !packets;
      if (in_place) a.sum_keys = kb;
      if (maybe_empty && (rc = cu(timed(c, "empty_fixup", ls, [&] { return launch_empty_fixup(a, ls); }), "empty")))
        return rc;
      if ((rc = cu(timed(c, "rle", ls, [&] { return launch_rle(a, ls); }), "rle"))) return rc;
      if ((rc = col_parts_heavy(c, pw, max_len, a, ls))) return rc;
      if ((rc = cu(timed(c, "finish", ls, [&] { return launch_finish(a, ls); }), "finish"))) return rc;
      if (in_place) {
        if ((rc = cu(cudaEventRecord(c->ev_fork, ls), "event")) ||
            (rc = cu(cudaStreamWaitEvent(c->side, c->ev_fork, 0), "event")))
          return rc;
        forked = true;
        rc = sum_order(c, m, ps, at<MatDesc>(m, off_mats), nseg, &sump, off_catoff, off_lens, off_total, c->side,
                       &sfk, &sfv, p.base, kb, sb.vals);
        const cudaError_t ej = cudaEventRecord(c->ev_join, c->side);
        if (rc == ANS_OK) rc = cu(ej, "event");
      }
      if (rc == ANS_OK) rc = column_pass(c, a, ps, m, sb.q, ls);
      if (forked) {  // join (also after a failure, so that a capture ends joined)
        const cudaError_t ew = cudaStreamWaitEvent(ls, c->ev_join, 0);
        if (rc == ANS_OK) rc = cu(ew, "event");
      }
      if (rc) return rc;
    }

    if (want_sum) {
      if (nseg == 0) {
        // an empty batch: an empty sum (its block is made before the launches)
        if ((rc = cu(launch_zero(sblk->row_ptr, 8, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(sblk->hdr, 16, ls), "memset"))) return rc;
        if ((rc = cu(launch_zero(sblk->q, sizeof(ans_quantities), ls), "memset"))) return rc;
      } else if (forked) {  // a sum of window counts stays below the batch's packets
        if ((rc = links_to_block(c, m, ps, sump.s, sfk, sfv, sump.blk, ls, total < (1ull << 32)))) return rc;
      } else if (sum_pk) {
        if ((rc = sum_packets(c, m, ps, wl.dp_pk.bind(m, hp_pk), d_src, d_dst, sump.blk, ls, total < (1ull << 32),
                              wl.ss, total, wl.ss_two_pk)))
          return rc;
      } else {
        rc = sum_launch(c, m, ps, at<MatDesc>(m, off_mats), nseg, &sump, off_catoff, off_lens, off_total, ls,
                        total < (1ull << 32));
        if (rc) return rc;
      }
    }
    return ANS_OK;
  };
  int rounds = 0;
  while ((1ull << rounds) < nseg) ++rounds;
  // (what else decides the kernels: one or two splits, the sort's launch
  // shapes, which column statistics, and theirs)
  const uint64_t pk_tiles = tiles_for(total);
  const std::string sig = launch_sig(flags, hp.ntiles > 0, !small_ids.empty(), !big_ids.empty(), rounds, c) + "/h" +
                          std::to_string(col_parts_ok(c, max_len, !dev)) + std::to_string(col_parts_ok(c, total)) +
                          std::to_string(max_len > kColPart) + std::to_string(total > kColPart) +
                          std::to_string(max_len > 512 * (uint64_t)kColPart) + std::to_string(total > 512 * (uint64_t)kColPart) +
                          std::to_string(max_len >= kColHeavyLinks) + std::to_string(total >= kColHeavyLinks) +
                          std::to_string(pk_tiles >= kHGroupMinLinks / kTile) + std::to_string(maybe_empty) + (dev ? "/d" : "") + "/s" +
                          std::to_string(wl.ss_two_win) + std::to_string(wl.ss_two_pk) +
                          std::to_string(ss_shape(hp.ntiles)) + std::to_string(ss_shape(wl.ss.ntiles2)) +
                          std::to_string(ss_shape((uint32_t)pk_tiles));
  queued = true;
  if ((rc = run_launches(c, st, sig, launch_all))) return bail(rc);
  if (sump.blk) {  // the time sum's block is filled
    sblk = sump.blk;
    sump.blk = nullptr;
  }

  // ---- completion
  if (c->guards) {  // debug mode: every guard of the scratch and the outputs intact
    for (const Block* b : {blk, sblk})
      if (b) guard_addr.insert(guard_addr.end(), b->guards.begin(), b->guards.end());
    if ((rc = cu(run_guards(guard_addr, c->d_err, st), "guards"))) return bail(rc);
  }
  BatchEnd end;
  end.err = c->d_err;
  if (blk) end.status[0] = blk->status;
  if (sblk) end.status[1] = sblk->status;
  // (whole words; an array off their alignment is copied by copy_quantities_out)
  if (out && nseg && (uintptr_t)out % 8 == 0 && (end.dst = (uint64_t*)addressable(out))) {
    end.src = (const uint64_t*)sb.q;
    end.words = (uint64_t)nseg * sizeof(ans_quantities) / 8;
  }
  uint32_t slot = 0;
  if (ticket) {
    slot = take_err_slot(c);
    end.status[2] = c->h_err_slots + slot;
  }
  if ((rc = cu(launch_batch_end(end, st), "batch end"))) return bail(rc);
  if (!end.dst && (rc = copy_quantities_out(out, sb.q, nseg, st))) return bail(rc);
  // (nothing may fail once the first handle has been given out)
  for (Block* b : {blk, sblk})
    if (b && (rc = cu(cudaEventRecord(b->done, st), "record"))) return bail(rc);
  if (ticket && (rc = add_ticket(c, st, slot, ticket))) return bail(rc);
  if (blk) {
    blk->refs = (int)nseg;
    for (uint32_t s = 0; s < nseg; ++s) per_window[s] = new ans_matrix{blk, s};
  }
  if (sblk) {
    sblk->refs = 1;
    *sum = new ans_matrix{sblk, 0};
  }
  if (flags & ANS_BATCH_SYNC) ANS_CUDA(cudaStreamSynchronize(st));
  return ANS_OK;
}

// The nine quantities of matrix (b, seg) recomputed from its stored DCSR
// into the device array q (kModeMatrix pipeline: value prefix, row
// statistics, column pass).  The caller holds c->mu and has ordered `st`
// after the matrix's completion.
int matrix_stats(ans_ctx* c, const Block* b, uint32_t seg, ans_quantities* q_out, cudaStream_t st) {
  const uint64_t cap = b->cap[seg];
  const uint64_t bs = b->base[seg];
  HostPlan hp;
  hp.build(std::vector<uint64_t>{cap}, nullptr);
  Layout L;
  DevPlan dp;
  dp.reserve(L, 1);
  const size_t off_pre = L.add((hp.pad + 1) * 8);
  const size_t off_lb = L.add((size_t)std::max<uint32_t>(hp.ntiles, 1) * 8);
  const size_t off_q = L.add(sizeof(ans_quantities));
  PipeScratch ps;
  ps.reserve(L, hp.pad, 1, std::max<uint32_t>(hp.ntiles, 1), false);
  ANS_TRY(ensure_scratch(c, L.size, st));
  char* m = (char*)c->scratch;
  UploadSet us;
  us.add(m + dp.base, hp.base.data(), 8);
  us.add(m + dp.first_tile, hp.first_tile.data(), 8);
  ANS_TRY(us.flush(c, st));
  SegPlan p = dp.bind(m, hp);
  uint64_t* hdr = b->hdr + 2 * (size_t)seg;
  p.len = hdr + 1;  // nnz, on the device
  ans_quantities* q = at<ans_quantities>(m, off_q);
  uint32_t* tickets = at<uint32_t>(m, ps.tickets);
  StatsArgs a;
  ZeroBatch z;
  z.add(q, sizeof(ans_quantities));
  z.add(m + off_lb, (size_t)std::max<uint32_t>(hp.ntiles, 1) * 8);
  z.add(tickets, 32 * 4);
  if (hp.ntiles && col_parts_ok(c, cap)) col_parts_begin(m, ps, p, cap, &a, &z);
  else z.add(m + ps.col_hist, kColPasses * kRadix * 4);
  ANS_CUDA(launch_zero_batch(z, st));
  uint64_t* pre = at<uint64_t>(m, off_pre);
  if (hp.ntiles) {
    ANS_CUDA(timed(c, "scan_u64", st, [&] { return launch_scan_u64(p, b->vals + bs, pre, at<uint64_t>(m, off_lb), tickets, c->d_err, st); }));
    a.plan = p;
    a.hdr = hdr;
    a.q = q;
    a.col_ids = b->col_ids + bs;
    a.vals = b->vals + bs;
    a.row_ids = b->row_ids + bs;
    a.row_ptr = b->row_ptr + bs + seg;
    a.pre = pre;
    a.col_hist = at<uint32_t>(m, ps.col_hist);
    a.ulen = at<uint64_t>(m, ps.ulen);
    a.col_st0 = at<uint64_t>(m, ps.st0);
    a.col_tickets = tickets + 32;
    a.err = c->d_err;
    a.mode = kModeMatrix;
    ANS_TRY(col_parts_heavy(c, p, cap, a, st));
    ANS_CUDA(timed(c, "finish", st, [&] { return launch_finish(a, st); }));
    ANS_TRY(column_pass(c, a, ps, m, q, st));
  }
  return copy_quantities_out(q_out, q, 1, st);
}

// Drop the stored zeros of a signed combination: the links of `blk` (one
// matrix, at most cap links; narrow: the result's counts stay below 2^32) are
// gathered as (key, value), the nonzero ones compacted in order, and the statistics rebuilt into a new block *out.  A
// negative count sets kErrNegative in the context's error word.
int drop_zeros(ans_ctx* c, Block* blk, uint64_t cap, bool narrow, cudaStream_t st, Block** out) {
  *out = nullptr;
  HostPlan sp;
  sp.build(std::vector<uint64_t>{cap}, nullptr);
  Layout L;
  PipeScratch ps;
  ps.reserve(L, sp.pad, 1, std::max<uint32_t>(sp.ntiles, 1), true);
  const size_t off_mats = L.add(sizeof(MatDesc));
  const size_t off_gplan = L.add(4 * align_up(2 * 8));
  const size_t off_splan = L.add(4 * kAlign);
  const size_t off_catoff = L.add(2 * 8);
  const size_t off_lens = L.add(8);
  const size_t off_total = L.add(8);
  const size_t off_count = L.add(8);
  ANS_TRY(ensure_scratch(c, L.size, st));
  char* m = (char*)c->scratch;
  MatDesc md{blk->row_ids, blk->row_ptr, blk->col_ids, blk->vals, blk->hdr};
  UploadSet us;
  us.add(m + off_mats, &md, sizeof(MatDesc));
  SumPlan plan;
  ANS_TRY(sum_prepare(c, m, 1, std::vector<uint64_t>{cap}, off_gplan, off_splan, off_lens, off_total, us, st, &plan));
  auto bail = [&](int rc) {
    block_discard(plan.blk, st);
    return rc;
  };
  int rc = us.flush(c, st);
  if (rc) return bail(rc);
  auto cu = [&](cudaError_t e, const char* what) -> int {
    if (e == cudaSuccess) return ANS_OK;
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  uint64_t* ka = at<uint64_t>(m, ps.keys_a);
  uint64_t* kb = at<uint64_t>(m, ps.keys_b);
  uint64_t* va = at<uint64_t>(m, ps.vals_a);
  uint64_t* vb = at<uint64_t>(m, ps.vals_b);
  uint32_t* tickets = at<uint32_t>(m, ps.tickets) + 32;
  uint64_t* flags = at<uint64_t>(m, ps.cv_a);  // free until the column pass
  uint64_t* pos = at<uint64_t>(m, ps.pre);     // and until the result's prefix
  uint64_t* count = at<uint64_t>(m, off_count);
  const uint64_t* cat_off = at<uint64_t>(m, off_catoff);
  const SegPlan& s = plan.s;
  if ((rc = cu(launch_count_prefix(at<MatDesc>(m, off_mats), 1, at<uint64_t>(m, off_catoff),
                                   at<uint64_t>(m, off_lens), at<uint64_t>(m, off_total), st), "count")) ||
      (rc = cu(launch_zero(m + ps.lb, (size_t)sp.ntiles * 8, st), "zero")) ||
      (rc = cu(launch_zero(m + ps.lb2, (size_t)sp.ntiles * 8, st), "zero")) ||
      (rc = cu(launch_gather(plan.g, at<MatDesc>(m, off_mats), cat_off, ka, va, nullptr, at<uint64_t>(m, ps.st0),
                             tickets, st), "gather")) ||
      (rc = cu(launch_nonzero_flags(s, va, flags, c->d_err, st), "flags")) ||
      (rc = cu(launch_scan_u64(s, flags, pos, at<uint64_t>(m, ps.lb2), tickets + kPasses + 1, c->d_err, st),
               "scan")) ||
      (rc = cu(launch_scatter_nonzero(s, ka, va, pos, kb, vb, count, st), "scatter")) ||
      // the statistics scan reuses this look-back array and ticket
      (rc = cu(launch_zero(m + ps.lb2, (size_t)sp.ntiles * 8, st), "zero")) ||
      (rc = cu(launch_zero(tickets + kPasses + 1, 4, st), "zero")))
    return bail(rc);
  SegPlan s2 = s;
  s2.len = count;
  if ((rc = links_to_block(c, m, ps, s2, kb, vb, plan.blk, st, narrow, true, kHGroupGivenLinks))) return bail(rc);
  *out = plan.blk;
  return ANS_OK;
}

// Sum of k matrices, each with sign +1 or -1 (signs null: all +1), into a
// new matrix *out (the body of ans_sum_windows and ans_combine).
int combine_matrices(ans_ctx* c, const ans_matrix* const* mats, const int* signs, size_t k, ans_matrix** out,
                     cudaStream_t st) {
  if (!c || !out || (k && !mats)) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  std::vector<uint64_t> caps;
  std::vector<MatDesc> md;
  uint64_t total_cap = 0;
  bool any_neg = false;
  // every count of the result stays below 2^32 if the inputs hold fewer
  // packets in all (known once they have been computed).  An input's packets
  // are counted modulo 2^62: they are taken at their word only where its links
  // times its largest count cannot reach that (imported counts may)
  uint64_t packets = 0;
  bool narrow = true;
  for (size_t i = 0; i < k; ++i) {
    const ans_matrix* x = mats[i];
    if (!x) return fail(ANS_ERR_INVALID_ARG, "NULL matrix");
    const Block* b = x->blk;
    if (b->ctx->device != c->device) return fail(ANS_ERR_INVALID_ARG, "matrix on another device");
    ANS_TRY(block_plan(const_cast<Block*>(b)));
    const uint64_t bs = b->base[x->seg];
    const bool neg = signs && signs[i] < 0;
    any_neg = any_neg || neg;
    md.push_back({b->row_ids + bs, b->row_ptr + bs + x->seg, b->col_ids + bs, b->vals + bs, b->hdr + 2 * x->seg,
                  neg ? 1ull : 0ull});
    // An input that has already been computed contributes its actual link
    // count to the output's capacity; one still running contributes its bound.
    uint64_t cap = b->cap[x->seg];
    if (cudaEventQuery(b->done) == cudaSuccess) {
      ANS_TRY(block_fill_cache(const_cast<Block*>(b)));
      cap = std::min<uint64_t>(cap, b->h_hdr[2 * (size_t)x->seg + 1]);
      const ans_quantities& hq = b->h_q[x->seg];
      const uint64_t held = hq.valid_packets;
      narrow = narrow && held < (1ull << 32) - packets &&
               (!hq.unique_links || hq.max_link_packets < (1ull << 62) / hq.unique_links);
      if (narrow) packets += held;
    } else {
      cudaGetLastError();
      narrow = false;
    }
    caps.push_back(cap);
    total_cap += cap;
    ANS_CUDA(cudaStreamWaitEvent(st, b->done, 0));
  }
  if (total_cap > kMaxWindow) return fail(ANS_ERR_INVALID_ARG, "a time sum is limited to 2^31 - 1 links");
  Block* sblk = nullptr;
  if (k == 0 || total_cap == 0) {
    ANS_TRY(make_block(c, 0, 1, {0}, {0}, st, &sblk));
    ANS_CUDA(cudaMemsetAsync(sblk->row_ptr, 0, 8, st));
    ANS_CUDA(cudaMemsetAsync(sblk->hdr, 0, 16, st));
    ANS_CUDA(cudaMemsetAsync(sblk->q, 0, sizeof(ans_quantities), st));
    ANS_CUDA(cudaMemsetAsync(sblk->status, 0, 4, st));
  } else {
    HostPlan sp;
    sp.build(std::vector<uint64_t>{total_cap}, nullptr);
    HostPlan gp;
    gp.build(caps, nullptr);
    Layout L;
    PipeScratch ps;
    ps.reserve(L, sp.pad, 1, std::max(sp.ntiles, gp.ntiles), true);
    const size_t off_mats = L.add(k * sizeof(MatDesc));
    const size_t off_gplan = L.add(4 * align_up((k + 1) * 8));
    const size_t off_splan = L.add(4 * kAlign);
    const size_t off_catoff = L.add((k + 1) * 8);
    const size_t off_lens = L.add(k * 8);
    const size_t off_total = L.add(8);
    ANS_TRY(ensure_scratch(c, L.size, st));
    char* m = (char*)c->scratch;
    UploadSet us;
    us.add(m + off_mats, md.data(), k * sizeof(MatDesc));
    SumPlan sump;
    ANS_TRY(sum_prepare(c, m, (uint32_t)k, caps, off_gplan, off_splan, off_lens, off_total, us, st, &sump));
    int rc = us.flush(c, st);
    if (rc) {
      block_discard(sump.blk, st);
      return rc;
    }
    rc = sum_launch(c, m, ps, at<MatDesc>(m, off_mats), (uint32_t)k, &sump, off_catoff, off_lens, off_total, st,
                    narrow && !any_neg, !any_neg, kHGroupGivenLinks);
    if (rc) {
      block_discard(sump.blk, st);
      return rc;
    }
    sblk = sump.blk;
    if (any_neg) {  // cancelled links are stored as zeros: compact them away
      Block* clean = nullptr;
      rc = drop_zeros(c, sblk, total_cap, narrow, st, &clean);
      block_discard(sblk, st);
      if (rc) return rc;
      sblk = clean;
    }
    rc = capture_err(c, sblk->status, st);
    if (rc == ANS_OK) rc = reset_err(c, st);
    if (rc) {
      block_discard(sblk, st);
      return rc;
    }
  }
  for (size_t i = 0; i < k; ++i) ANS_TRY(note_read(mats[i]->blk, st));
  ANS_CUDA(cudaEventRecord(sblk->done, st));
  sblk->refs = 1;
  *out = new ans_matrix{sblk, 0};
  return ANS_OK;
}

// Scratch given back before a batch that did not fit is tried again another
// way, which may need a little more: growing what is held would take a quarter
// more than that (ensure_scratch).
void drop_scratch(ans_ctx* c, cudaStream_t st) {
  dev_free(c, c->scratch, c->scratch_size, st);
  c->scratch = nullptr;
  c->scratch_size = 0;
}

bool page_locked(const void* p) {
  cudaPointerAttributes pa{};
  if (cudaPointerGetAttributes(&pa, p) == cudaSuccess) return pa.type == cudaMemoryTypeHost;
  cudaGetLastError();
  return false;
}

// Whether a batch's pairs are first copied to the device by a kernel: they lie
// in page-locked host memory, the offsets (offs null: on the device, at most
// `total` packets) are good, and the batch's sorts read the pairs more than
// once -- a packet sort reads them twice, and the batch's sum by re-sorting
// (sum_path 2) as often again -- which over the host link costs more than the
// copy's 8 bytes a packet written and read on the device (2^24 packets in 128
// windows: 1.27 ms against 1.95, with sum_path 2 2.98 against 4.84; 2^18 in one
// window 184 us against 204).  On-chip window sorts and the hash tables read
// them once, in place.
bool gather_pays(const ans_ctx* c, const uint32_t* src, const uint32_t* dst, const uint64_t* offs, uint64_t total,
                 size_t nwin, bool want_sum) {
  if (!src || !dst || !nwin || nwin > 0xFFFFFFF0ull) return false;
  bool big = !offs;  // (a batch planned on the device is never sorted on chip)
  for (size_t w = 0; offs && w < nwin; ++w) {
    if (offs[w + 1] < offs[w] || offs[w + 1] - offs[w] > kMaxWindow) return false;
    big = big || offs[w + 1] - offs[w] > kClusterWindowMax;
  }
  if (!total || (want_sum && total > kMaxWindow)) return false;
  const bool again = want_sum && (c->sum_path == 2 || c->agg_path == 3);
  const bool sorted = c->agg_path != 1 && (big || c->win_path != 0 || cluster_sort_clusters(c->device) <= 0);
  const uint64_t first = offs ? offs[0] : 0;
  return (again || sorted) && page_locked(src + first) && page_locked(dst + first);
}

// The pieces of windows in their own arrays to be copied to one pair of arrays:
// at most max(2^14, total / 4096) packets each, so that a few long windows are
// copied by as many CTAs as many short ones (a served batch of 100 windows of 2^12
// to 2^17 packets from page-locked memory: 848 us with a CTA per window, 824 so).
std::vector<GatherWin> gather_pieces(const uint32_t* const* srcs, const uint32_t* const* dsts, const uint64_t* lens,
                                     size_t nwin, uint64_t total) {
  const uint64_t most = std::max<uint64_t>(1u << 14, total >> 12);
  std::vector<GatherWin> table;
  table.reserve(nwin + (size_t)(total / most));
  uint64_t off = 0;
  for (size_t w = 0; w < nwin; ++w)
    for (uint64_t p = 0; p < lens[w]; p += most) {
      const uint64_t n = std::min(most, lens[w] - p);
      table.push_back(GatherWin{(uint64_t)(uintptr_t)(srcs[w] + p), (uint64_t)(uintptr_t)(dsts[w] + p), off, n});
      off += n;
    }
  return table;
}

// A batch of windows stored back to back, offsets on the host or (h_offsets
// null) on the device with at most `total` packets: analysed from where the
// pairs lie, or (gather_pays) from a copy made on the device, given back when
// the batch has been queued.  Where that copy or the batch beside it does not
// fit in memory, the pairs are read in place.
int run_pairs(ans_ctx* c, const uint32_t* src, const uint32_t* dst, const uint64_t* h_offsets,
              const uint64_t* d_offsets, uint64_t total, size_t nwin, uint32_t flags, ans_quantities* out,
              ans_matrix** per_window, ans_matrix** sum, ans_ticket* ticket, cudaStream_t st) {
  if (gather_pays(c, src, dst, h_offsets, total, nwin, (flags & ANS_BATCH_SUM) != 0)) {
    const size_t pairs = align_up((size_t)total * 4), bytes = 2 * pairs + (nwin + 3) * 8;
    void* mem = nullptr;
    int rc = dev_alloc(c, bytes, st, &mem);
    if (rc == ANS_OK) {
      uint32_t *gsrc = (uint32_t*)mem, *gdst = (uint32_t*)((char*)mem + pairs);
      uint64_t* span = (uint64_t*)((char*)mem + 2 * pairs);  // first packet, packets, offsets from the first
      std::vector<uint64_t> rel(h_offsets ? nwin + 1 : 0);
      for (size_t w = 0; w < rel.size(); ++w) rel[w] = h_offsets[w] - h_offsets[0];
      const auto feed = [&]() -> int {
        if (d_offsets) ANS_CUDA(launch_gather_offsets(d_offsets, nwin, total, span, st));
        ANS_CUDA(launch_gather_span(src, dst, h_offsets ? h_offsets[0] : 0, total, d_offsets ? span : nullptr, gsrc, gdst, st));
        return ANS_OK;
      };
      rc = run_windows(c, gsrc, gdst, h_offsets ? rel.data() : nullptr, nwin, flags, out, per_window, sum, ticket, st,
                       nullptr, nullptr, d_offsets ? span + 2 : nullptr, d_offsets ? total : 0, feed);
      dev_free(c, mem, bytes, st);
    }
    if (rc != ANS_ERR_OOM && rc != ANS_ERR_BUDGET) return rc;
    drop_scratch(c, st);
  }
  return run_windows(c, src, dst, h_offsets, nwin, flags, out, per_window, sum, ticket, st, nullptr, nullptr, d_offsets,
                     d_offsets ? total : 0);
}

}  // namespace

// =========================================================================
extern "C" {

const char* ans_status_string(int s) {
  switch (s) {
    case ANS_OK: return "ok";
    case ANS_ERR_INVALID_ARG: return "invalid argument";
    case ANS_ERR_BUDGET: return "memory budget exceeded";
    case ANS_ERR_OOM: return "out of device memory";
    case ANS_ERR_CUDA: return "CUDA error";
    case ANS_ERR_TIMEOUT: return "timed out";
    case ANS_ERR_INTERNAL: return "internal error";
    default: return "unknown status";
  }
}

const char* ans_last_error(ans_ctx*) { return t_last_error.c_str(); }

int ans_ctx_create(ans_ctx** out, int device, size_t mem_budget_bytes, ans_alloc_fn alloc, ans_free_fn free_fn,
                   void* user) {
  if (!out) return fail(ANS_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if ((alloc == nullptr) != (free_fn == nullptr))
    return fail(ANS_ERR_INVALID_ARG, "give both allocator hooks or neither");
  int ndev = 0;
  ANS_CUDA(cudaGetDeviceCount(&ndev));
  if (device < 0 || device >= ndev) return fail(ANS_ERR_INVALID_ARG, "no such device");
  DeviceGuard dg(device);
  ans_ctx* c = new ans_ctx();
  c->device = device;
  c->budget = mem_budget_bytes;
  c->alloc_fn = alloc;
  c->free_fn = free_fn;
  c->user = user;
  {
    const char* g = std::getenv("ANS_SCRATCH_GUARDS");
    c->guards = g && *g && std::strcmp(g, "0") != 0;
  }
  auto undo = [&](int rc) {
    for (auto& s : c->stage)
      if (s.ev) cudaEventDestroy(s.ev);
    if (c->h_err_slots) cudaFreeHost(c->h_err_slots);
    if (c->aux) cudaStreamDestroy(c->aux);
    delete c;
    return rc;
  };
  for (auto& s : c->stage) {
    if (cudaEventCreateWithFlags(&s.ev, cudaEventDisableTiming) != cudaSuccess)
      return undo(fail(ANS_ERR_CUDA, "cudaEventCreate failed"));
  }
  if (cudaHostAlloc((void**)&c->h_err_slots, kErrSlots * 4, cudaHostAllocDefault) != cudaSuccess)
    return undo(fail(ANS_ERR_CUDA, "cudaHostAlloc failed"));
  std::memset(c->h_err_slots, 0, kErrSlots * 4);
  if (cudaStreamCreateWithFlags(&c->aux, cudaStreamNonBlocking) != cudaSuccess)
    return undo(fail(ANS_ERR_CUDA, "cudaStreamCreate failed"));
  if (!alloc) {
    // Keep freed blocks in this process's stream-ordered pool instead of
    // returning them to the driver at every synchronisation.
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
      uint64_t keep = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    cudaGetLastError();
  }
  void* small = nullptr;
  int rc = dev_alloc(c, 256, c->aux, &small);
  if (rc != ANS_OK) return undo(rc);
  c->small_mem = small;
  c->d_err = (uint32_t*)small;
  if (cudaMemsetAsync(small, 0, 256, c->aux) != cudaSuccess || cudaStreamSynchronize(c->aux) != cudaSuccess)
    return undo(fail(ANS_ERR_CUDA, "initialising the error word failed"));
  *out = c;
  return ANS_OK;
}

int ans_ctx_destroy(ans_ctx* c) {
  if (!c) return ANS_OK;
  bool last = false;
  {
    std::lock_guard<std::mutex> g(c->mu);
    if (c->closed) return fail(ANS_ERR_INVALID_ARG, "context already destroyed");
    DeviceGuard dg(c->device);
    if (device_wait() == cudaErrorStreamCaptureUnsupported) {  // the caller's own capture
      cudaGetLastError();
      return fail(ANS_ERR_CUDA, "a stream is being captured: the context's work cannot be waited for");
    }
    for (auto& kv : c->tickets) cudaEventDestroy(kv.second.ev);
    c->tickets.clear();
    dev_free(c, c->scratch, c->scratch_size, c->aux);
    c->scratch = nullptr;
    c->scratch_size = 0;
    dev_free(c, c->small_mem, 256, c->aux);
    c->small_mem = nullptr;
    dev_free(c, c->hash_mem, c->hash_slots * 12, c->aux);
    c->hash_mem = nullptr;
    c->hash_slots = 0;
    dev_free(c, c->gather_mem, c->gather_bytes, c->aux);
    c->gather_mem = nullptr;
    c->gather_bytes = 0;
    for (auto& kv : c->graphs) cudaGraphExecDestroy(kv.second);
    c->graphs.clear();
    if (c->cap) cudaStreamDestroy(c->cap);
    c->cap = nullptr;
    if (c->side) cudaStreamDestroy(c->side);
    c->side = nullptr;
    if (c->ev_fork) cudaEventDestroy(c->ev_fork);
    if (c->ev_join) cudaEventDestroy(c->ev_join);
    c->ev_fork = c->ev_join = nullptr;
    for (auto& kv : c->prof.pending) {
      cudaEventDestroy(kv.a);
      cudaEventDestroy(kv.b);
    }
    c->prof.pending.clear();
    for (cudaEvent_t e : c->prof.spare) cudaEventDestroy(e);
    c->prof.spare.clear();
    c->closed = true;
    last = c->blocks == 0;
  }
  if (last) ctx_finalize(c);
  return ANS_OK;
}

int ans_build_window(ans_ctx* c, const uint32_t* d_src, const uint32_t* d_dst, uint64_t n, ans_matrix** out,
                     void* stream) {
  if (!c || !out) return fail(ANS_ERR_INVALID_ARG, "NULL context or output");
  if (n > kMaxWindow) return fail(ANS_ERR_INVALID_ARG, "a window is limited to 2^31 - 1 packets");
  *out = nullptr;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  const uint64_t offs[2] = {0, n};
  return run_windows(c, d_src, d_dst, offs, 1, ANS_BATCH_MATRICES, nullptr, out, nullptr, nullptr,
                     (cudaStream_t)stream);
}

int ans_batch_submit(ans_ctx* c, const uint32_t* d_src, const uint32_t* d_dst, const uint64_t* d_offsets,
                     size_t nwin, uint32_t flags, ans_quantities* out, ans_matrix** per_window, ans_matrix** sum,
                     ans_ticket* ticket, void* stream) {
  if (!c || !d_offsets) return fail(ANS_ERR_INVALID_ARG, "NULL context or offsets");
  if (flags & ~(ANS_BATCH_MATRICES | ANS_BATCH_SUM | ANS_BATCH_SYNC))
    return fail(ANS_ERR_INVALID_ARG, "unknown flag");
  if ((flags & ANS_BATCH_MATRICES) && !per_window) return fail(ANS_ERR_INVALID_ARG, "per_window is NULL");
  if ((flags & ANS_BATCH_SUM) && !sum) return fail(ANS_ERR_INVALID_ARG, "sum is NULL");
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  uint64_t cap = c->batch_cap;
  if (cap == 0 && nwin > 0) {  // no capacity set: size the batch by its first and last offsets
    uint64_t ends[2] = {0, 0};
    ANS_CUDA(cudaMemcpyAsync(&ends[0], d_offsets, 8, cudaMemcpyDeviceToHost, st));
    ANS_CUDA(cudaMemcpyAsync(&ends[1], d_offsets + nwin, 8, cudaMemcpyDeviceToHost, st));
    ANS_CUDA(cudaStreamSynchronize(st));
    if (ends[1] < ends[0]) return fail(ANS_ERR_INVALID_ARG, "offsets must be nondecreasing");
    cap = ends[1] - ends[0];
  }
  return run_pairs(c, d_src, d_dst, nullptr, d_offsets, cap, nwin, flags, out, per_window, sum, ticket, st);
}

int ans_batch_submit_host(ans_ctx* c, const uint32_t* d_src, const uint32_t* d_dst, const uint64_t* h_offsets,
                          size_t nwin, uint32_t flags, ans_quantities* out, ans_matrix** per_window, ans_matrix** sum,
                          ans_ticket* ticket, void* stream) {
  if (!c || !h_offsets) return fail(ANS_ERR_INVALID_ARG, "NULL context or offsets");
  if (flags & ~(ANS_BATCH_MATRICES | ANS_BATCH_SUM | ANS_BATCH_SYNC))
    return fail(ANS_ERR_INVALID_ARG, "unknown flag");
  if ((flags & ANS_BATCH_MATRICES) && !per_window) return fail(ANS_ERR_INVALID_ARG, "per_window is NULL");
  if ((flags & ANS_BATCH_SUM) && !sum) return fail(ANS_ERR_INVALID_ARG, "sum is NULL");
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  return run_pairs(c, d_src, d_dst, h_offsets, nullptr, h_offsets[nwin] - h_offsets[0], nwin, flags, out, per_window, sum,
                   ticket, (cudaStream_t)stream);
}

int ans_set_batch_capacity(ans_ctx* c, uint64_t max_packets) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  if (max_packets > ((uint64_t)0xFFFFFFF0ull - (1ull << 20)) * kTile)
    return fail(ANS_ERR_INVALID_ARG, "batch capacity too large");
  std::lock_guard<std::mutex> g(c->mu);
  c->batch_cap = max_packets;
  return ANS_OK;
}

int ans_batch_submit_windows(ans_ctx* c, const uint32_t* const* srcs, const uint32_t* const* dsts,
                             const uint64_t* lens, size_t nwin, uint32_t flags, ans_quantities* out,
                             ans_matrix** per_window, ans_matrix** sum, ans_ticket* ticket, void* stream) {
  if (!c || (nwin && (!srcs || !dsts || !lens))) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  if (flags & ~(ANS_BATCH_MATRICES | ANS_BATCH_SUM | ANS_BATCH_SYNC))
    return fail(ANS_ERR_INVALID_ARG, "unknown flag");
  if ((flags & ANS_BATCH_MATRICES) && !per_window) return fail(ANS_ERR_INVALID_ARG, "per_window is NULL");
  if ((flags & ANS_BATCH_SUM) && !sum) return fail(ANS_ERR_INVALID_ARG, "sum is NULL");
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  // Every nonempty window's arrays must be readable by the device: device or
  // page-locked host memory, or any host memory where the device reads
  // pageable memory.
  if (c->pageable < 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrPageableMemoryAccess, c->device) != cudaSuccess) {
      cudaGetLastError();
      v = 0;
    }
    c->pageable = v ? 1 : 0;
  }
  std::vector<uint64_t> offs(nwin + 1, 0);
  for (size_t w = 0; w < nwin; ++w) {
    offs[w + 1] = offs[w] + lens[w];
    if (!lens[w]) continue;
    if (!srcs[w] || !dsts[w]) return fail(ANS_ERR_INVALID_ARG, "NULL packet arrays of a nonempty window");
    if (!c->pageable) {
      for (const void* ptr : {(const void*)srcs[w], (const void*)dsts[w]}) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess || at.type == cudaMemoryTypeUnregistered) {
          cudaGetLastError();
          return fail(ANS_ERR_INVALID_ARG, "window " + std::to_string(w) +
                                               ": packet arrays in pageable host memory this device cannot read");
        }
      }
    }
  }
  // The paths that sort all of a batch's packets as one segment (the time sum
  // by re-sorting the packets) read the packets as one stream: the windows'
  // pairs are first gathered into one device buffer by a kernel (reading each
  // window in place), then analysed like contiguous windows.  If that buffer
  // cannot be had, the windows are analysed in place on the other paths.
  // Other packet sorts read the pairs twice; where the first window's lie in
  // page-locked host memory they are gathered too, into memory given back with
  // the batch (run_pairs; 100 windows of 2^12 to 2^17 packets served with
  // their sum: 708 us against 920 in place; one of 2^17: 212 against 220).
  const uint64_t total = offs[nwin];
  cudaStream_t st = (cudaStream_t)stream;
  const bool one_segment = c->agg_path == 2 || c->agg_path == 3 || c->sum_path == 2;
  bool fits = nwin <= 0xFFFFFFF0ull && !((flags & ANS_BATCH_SUM) && total > kMaxWindow);
  bool big = false;
  size_t first = nwin;
  for (size_t w = 0; w < nwin && fits; ++w) {
    fits = lens[w] <= kMaxWindow;
    big = big || lens[w] > kClusterWindowMax;
    if (lens[w] && first == nwin) first = w;
  }
  const bool twice = !one_segment && c->agg_path != 1 &&
                     (big || c->win_path != 0 || cluster_sort_clusters(c->device) <= 0) && first < nwin &&
                     page_locked(srcs[first]) && page_locked(dsts[first]);
  if ((one_segment || twice) && fits && total > 0) {  // (otherwise run_windows reports what does not fit)
    const std::vector<GatherWin> table = gather_pieces(srcs, dsts, lens, nwin, total);
    const size_t pairs = align_up((size_t)total * 4);
    const size_t need = 2 * pairs + table.size() * sizeof(GatherWin);
    void* mem = nullptr;
    if (twice) {
      const int rc = dev_alloc(c, need, st, &mem);
      if (rc != ANS_OK && rc != ANS_ERR_OOM && rc != ANS_ERR_BUDGET) return rc;
    } else if (need > c->gather_bytes) {
      const size_t want = std::max(need, c->gather_bytes + c->gather_bytes / 4);
      dev_free(c, c->gather_mem, c->gather_bytes, st);
      c->gather_mem = nullptr;
      c->gather_bytes = 0;
      void* p = nullptr;
      int rc = dev_alloc(c, want, st, &p);
      if (rc == ANS_OK) {
        c->gather_mem = p;
        c->gather_bytes = want;
      } else if (rc != ANS_ERR_OOM && rc != ANS_ERR_BUDGET) {
        return rc;
      }
    }
    if (char* gm = (char*)(twice ? mem : c->gather_mem)) {
      uint32_t* gsrc = (uint32_t*)gm;
      uint32_t* gdst = (uint32_t*)(gm + pairs);
      GatherWin* gw = (GatherWin*)(gm + 2 * pairs);
      const auto feed = [&]() -> int {
        UploadSet us;
        us.add(gw, table.data(), table.size() * sizeof(GatherWin));
        ANS_TRY(us.flush(c, st));
        ANS_CUDA(launch_gather_windows(gw, (uint32_t)table.size(), gsrc, gdst, st));
        return ANS_OK;
      };
      const int rc = run_windows(c, gsrc, gdst, offs.data(), nwin, flags, out, per_window, sum, ticket, st, nullptr,
                                 nullptr, nullptr, 0, feed);
      if (!twice) return rc;
      dev_free(c, mem, need, st);
      if (rc != ANS_ERR_OOM && rc != ANS_ERR_BUDGET) return rc;
      drop_scratch(c, st);  // (else in place)
    }
  }
  return run_windows(c, nullptr, nullptr, offs.data(), nwin, flags, out, per_window, sum, ticket, st, srcs, dsts);
}

int ans_sum_windows(ans_ctx* c, const ans_matrix* const* mats, size_t k, ans_matrix** out, void* stream) {
  return combine_matrices(c, mats, nullptr, k, out, (cudaStream_t)stream);
}

int ans_combine(ans_ctx* c, const ans_matrix* const* mats, const int* signs, size_t k, ans_matrix** out,
                void* stream) {
  if (k && !signs) return fail(ANS_ERR_INVALID_ARG, "NULL signs");
  for (size_t i = 0; i < k; ++i)
    if (signs[i] != 1 && signs[i] != -1) return fail(ANS_ERR_INVALID_ARG, "signs must be +1 or -1");
  return combine_matrices(c, mats, signs, k, out, (cudaStream_t)stream);
}

int ans_network_quantities(ans_ctx* c, const ans_matrix* x, ans_quantities* out, void* stream) {
  if (!c || !x || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  const Block* b = x->blk;
  if (b->ctx->device != c->device) return fail(ANS_ERR_INVALID_ARG, "matrix on another device");
  ANS_TRY(block_plan(const_cast<Block*>(b)));
  ANS_CUDA(cudaStreamWaitEvent(st, b->done, 0));
  ANS_TRY(matrix_stats(c, b, x->seg, out, st));
  ANS_CUDA(cudaMemsetAsync(c->d_err, 0, 4, st));
  ANS_TRY(note_read(const_cast<Block*>(b), st));
  return ANS_OK;
}

int ans_matrix_import(ans_ctx* c, uint64_t nrows, uint64_t nnz, const uint32_t* row_ids, const uint64_t* row_ptr,
                      const uint32_t* col_ids, const uint64_t* vals, ans_matrix** out, void* stream) {
  if (!c || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  if (nnz > kMaxWindow) return fail(ANS_ERR_INVALID_ARG, "an imported matrix is limited to 2^31 - 1 links");
  if (nrows > nnz) return fail(ANS_ERR_INVALID_ARG, "more rows than links (every stored row is nonempty)");
  if (!row_ptr || (nnz && (!row_ids || !col_ids || !vals))) return fail(ANS_ERR_INVALID_ARG, "NULL array");
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  Block* b = nullptr;
  const uint64_t pad = tiles_for(nnz) * kTile;
  ANS_TRY(make_block(c, pad, 1, std::vector<uint64_t>{0}, std::vector<uint64_t>{nnz}, st, &b));
  auto bail = [&](int rc) {
    block_discard(b, st);
    return rc;
  };
  auto cu = [&](cudaError_t e, const char* what) -> int {
    if (e == cudaSuccess) return ANS_OK;
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  int rc = ANS_OK;
  const uint64_t hdr[2] = {nrows, nnz};
  UploadSet us;
  us.add(b->hdr, hdr, 16);
  if ((rc = us.flush(c, st))) return bail(rc);
  if ((rc = cu(cudaMemcpyAsync(b->row_ptr, row_ptr, (nrows + 1) * 8, cudaMemcpyDefault, st), "copy row_ptr")))
    return bail(rc);
  if (nnz) {
    if ((rc = cu(cudaMemcpyAsync(b->row_ids, row_ids, nrows * 4, cudaMemcpyDefault, st), "copy row_ids")) ||
        (rc = cu(cudaMemcpyAsync(b->col_ids, col_ids, nnz * 4, cudaMemcpyDefault, st), "copy col_ids")) ||
        (rc = cu(cudaMemcpyAsync(b->vals, vals, nnz * 8, cudaMemcpyDefault, st), "copy vals")))
      return bail(rc);
  }
  // Canonical DCSR or nothing: the statistics kernels index by row_ptr.
  if ((rc = cu(cudaMemsetAsync(b->status, 0, 4, st), "memset"))) return bail(rc);
  if ((rc = cu(launch_check_dcsr(nrows, nnz, b->row_ids, b->row_ptr, b->col_ids, b->vals, b->status, st), "check")))
    return bail(rc);
  uint32_t bad = 0;
  if ((rc = cu(cudaMemcpyAsync(&bad, b->status, 4, cudaMemcpyDeviceToHost, st), "copy")) ||
      (rc = cu(cudaStreamSynchronize(st), "sync")))
    return bail(rc);
  if (bad) return bail(fail(ANS_ERR_INVALID_ARG, "not canonical DCSR (check code " + std::to_string(bad) + ")"));
  if ((rc = matrix_stats(c, b, 0, b->q, st))) return bail(rc);
  if ((rc = capture_err(c, b->status, st)) || (rc = reset_err(c, st))) return bail(rc);
  if ((rc = cu(cudaEventRecord(b->done, st), "record"))) return bail(rc);
  b->refs = 1;
  *out = new ans_matrix{b, 0};
  return ANS_OK;
}


int ans_wait(ans_ctx* c, ans_ticket t, uint64_t timeout_ns) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  cudaEvent_t ev;
  int slot;
  {
    std::lock_guard<std::mutex> g(c->mu);
    auto it = c->tickets.find(t);
    if (it == c->tickets.end()) return fail(ANS_ERR_INVALID_ARG, "unknown ticket");
    ev = it->second.ev;
    slot = it->second.slot;
  }
  DeviceGuard dg(c->device);
  const auto t0 = std::chrono::steady_clock::now();
  while (true) {
    cudaError_t e = cudaEventQuery(ev);
    if (e == cudaSuccess) break;
    if (e != cudaErrorNotReady) return fail(ANS_ERR_CUDA, std::string("cudaEventQuery: ") + cudaGetErrorString(e));
    const uint64_t el = (uint64_t)std::chrono::duration_cast<std::chrono::nanoseconds>(
                            std::chrono::steady_clock::now() - t0).count();
    if (el >= timeout_ns) return fail(ANS_ERR_TIMEOUT, "batch still running");
    // batches of up to 2 ms are polled (a sleep of 20 us lasts about 75)
    if (el < 2000000) std::this_thread::yield();
    else std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
  uint32_t err;
  {
    std::lock_guard<std::mutex> g(c->mu);
    err = c->h_err_slots[slot];
    cudaEventDestroy(ev);
    c->tickets.erase(t);
  }
  return status_of_err(err);
}

int ans_set_wait_limit(ans_ctx* c, uint32_t polls) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  if (polls > kSpinLimitMax) return fail(ANS_ERR_INVALID_ARG, "the poll limit is at most 2^24");
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  // the limit is read by kernels: change it only with nothing in flight
  ANS_CUDA(device_wait());
  ANS_CUDA(cudaMemcpy(c->d_err + 1, &polls, 4, cudaMemcpyHostToDevice));
  return ANS_OK;
}

int ans_probe_guards(ans_ctx* c, ans_ticket* ticket, void* stream) {
  if (!c || !ticket) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  // one 256-byte region of scratch and the guard after it
  ANS_TRY(ensure_scratch(c, kAlign + kGuardBytes, st));
  const std::vector<uint64_t> guard{(uint64_t)(uintptr_t)c->scratch + kAlign};
  ANS_CUDA(run_guards(guard, nullptr, st));
  ANS_CUDA(launch_guard_probe_write((uint64_t*)(uintptr_t)guard[0], st));
  ANS_CUDA(run_guards(guard, c->d_err, st));
  ANS_TRY(new_ticket(c, st, ticket));
  ANS_TRY(reset_err(c, st));
  return ANS_OK;
}

int ans_probe_wait_expiry(ans_ctx* c, ans_matrix** out, ans_ticket* ticket, void* stream) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  if (out) *out = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  // two status words beside the error word: tile 0 of the probed chain never
  // publishes, so tile 1's wait can only end at the poll limit
  uint64_t* words = (uint64_t*)((char*)c->small_mem + 64);
  ANS_CUDA(cudaMemsetAsync(words, 0, 16, st));
  ANS_CUDA(launch_wait_probe(words, c->d_err, st));
  Block* b = nullptr;
  if (out) {
    ANS_TRY(make_block(c, 0, 1, {0}, {0}, st, &b));
    auto cu = [&](cudaError_t e, const char* what) -> int {
      if (e == cudaSuccess) return ANS_OK;
      block_discard(b, st);
      return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
    };
    int rc;
    if ((rc = cu(cudaMemsetAsync(b->row_ptr, 0, 8, st), "memset")) || (rc = cu(cudaMemsetAsync(b->hdr, 0, 16, st), "memset")) ||
        (rc = cu(cudaMemsetAsync(b->q, 0, sizeof(ans_quantities), st), "memset")) ||
        (rc = cu(cudaMemcpyAsync(b->status, c->d_err, 4, cudaMemcpyDeviceToDevice, st), "copy")))
      return rc;
  }
  if (ticket) {
    const int rc = new_ticket(c, st, ticket);
    if (rc) {
      block_discard(b, st);
      return rc;
    }
  }
  ANS_TRY(reset_err(c, st));
  if (b) {
    ANS_CUDA(cudaEventRecord(b->done, st));
    b->refs = 1;
    *out = new ans_matrix{b, 0};
  }
  return ANS_OK;
}

int ans_matrix_view(const ans_matrix* x, uint64_t* nrows, uint64_t* nnz, const uint32_t** row_ids,
                    const uint64_t** row_ptr, const uint32_t** col_ids, const uint64_t** vals) {
  if (!x) return fail(ANS_ERR_INVALID_ARG, "NULL matrix");
  Block* b = x->blk;
  ANS_TRY(block_fill_cache(b));
  ANS_TRY(block_status(b));
  const uint64_t bs = b->base[x->seg];
  if (nrows) *nrows = b->h_hdr[2 * x->seg];
  if (nnz) *nnz = b->h_hdr[2 * x->seg + 1];
  if (row_ids) *row_ids = b->row_ids + bs;
  if (row_ptr) *row_ptr = b->row_ptr + bs + x->seg;
  if (col_ids) *col_ids = b->col_ids + bs;
  if (vals) *vals = b->vals + bs;
  return ANS_OK;
}

int ans_matrix_quantities(const ans_matrix* x, ans_quantities* out) {
  if (!x || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  Block* b = x->blk;
  ANS_TRY(block_fill_cache(b));
  ANS_TRY(block_status(b));
  *out = b->h_q[x->seg];
  return ANS_OK;
}

int ans_matrix_free(ans_matrix* x) {
  if (!x) return ANS_OK;
  block_release(x->blk);
  delete x;
  return ANS_OK;
}

int ans_matrix_split_rows(ans_ctx* c, const ans_matrix* x, uint32_t nparts, ans_matrix** out, void* stream) {
  if (!c || !x || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  if (nparts < 1 || nparts > kMaxSplitParts) return fail(ANS_ERR_INVALID_ARG, "nparts must be 1 .. 64");
  for (uint32_t o = 0; o < nparts; ++o) out[o] = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  Block* b = x->blk;
  if (b->ctx->device != c->device) return fail(ANS_ERR_INVALID_ARG, "matrix on another device");
  ANS_TRY(block_fill_cache(b));  // the matrix's size (waits for it)
  ANS_TRY(block_status(b));
  const uint64_t nrows = b->h_hdr[2 * (size_t)x->seg], nnz = b->h_hdr[2 * (size_t)x->seg + 1];
  const uint64_t bs = b->base[x->seg];
  const uint32_t* row_ids = b->row_ids + bs;
  const uint64_t* row_ptr = b->row_ptr + bs + x->seg;
  const uint32_t* col_ids = b->col_ids + bs;
  const uint64_t* vals = b->vals + bs;
  // scratch: per-tile counts, totals, per-row owner and first link
  const uint32_t nt = split_row_tiles(nrows);
  Layout L;
  const size_t o_trows = L.add((size_t)nt * nparts * 4);
  const size_t o_tlinks = L.add((size_t)nt * nparts * 8);
  const size_t o_tot = L.add((size_t)nparts * 16);
  const size_t o_rown = L.add(nrows * 4);
  const size_t o_rlink = L.add(nrows * 8);
  ANS_TRY(ensure_scratch(c, L.size, st));
  char* m = (char*)c->scratch;
  uint32_t* trows = at<uint32_t>(m, o_trows);
  uint64_t* tlinks = at<uint64_t>(m, o_tlinks);
  uint64_t* tot = at<uint64_t>(m, o_tot);
  ANS_CUDA(launch_split_count(nrows, row_ids, row_ptr, nparts, trows, tlinks, tot, st));
  std::vector<uint64_t> h_tot(2 * (size_t)nparts);
  ANS_CUDA(cudaMemcpyAsync(h_tot.data(), tot, h_tot.size() * 8, cudaMemcpyDeviceToHost, st));
  ANS_CUDA(cudaStreamSynchronize(st));
  // one block per owner
  std::vector<Block*> blks(nparts, nullptr);
  auto bail = [&](int rc) {
    for (Block* q : blks) block_discard(q, st);
    return rc;
  };
  SplitOut so{};
  for (uint32_t o = 0; o < nparts; ++o) {
    const uint64_t u = h_tot[2 * o + 1];
    int rc = make_block(c, tiles_for(u) * kTile, 1, {0}, {u}, st, &blks[o]);
    if (rc) return bail(rc);
    so.row_ids[o] = blks[o]->row_ids;
    so.row_ptr[o] = blks[o]->row_ptr;
    so.col_ids[o] = blks[o]->col_ids;
    so.vals[o] = blks[o]->vals;
    so.hdr[o] = blks[o]->hdr;
  }
  auto cu = [&](cudaError_t e, const char* what) -> int {
    if (e == cudaSuccess) return ANS_OK;
    return fail(ANS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  int rc = cu(launch_split_fill(nrows, nnz, row_ids, row_ptr, col_ids, vals, nparts, trows, tlinks, tot,
                                at<uint32_t>(m, o_rown), at<uint64_t>(m, o_rlink), so, st),
              "split");
  if (rc) return bail(rc);
  for (uint32_t o = 0; o < nparts && rc == ANS_OK; ++o) {
    if ((rc = cu(cudaMemsetAsync(blks[o]->status, 0, 4, st), "memset")) == ANS_OK &&
        (rc = matrix_stats(c, blks[o], 0, blks[o]->q, st)) == ANS_OK)
      rc = capture_err(c, blks[o]->status, st);
  }
  if (rc == ANS_OK) rc = reset_err(c, st);
  if (rc == ANS_OK) rc = note_read(b, st);
  if (rc) return bail(rc);
  for (uint32_t o = 0; o < nparts; ++o) {
    ANS_CUDA(cudaEventRecord(blks[o]->done, st));
    blks[o]->refs = 1;
    out[o] = new ans_matrix{blks[o], 0};
  }
  return ANS_OK;
}

int ans_matrix_retain(const ans_matrix* x, ans_matrix** out) {
  if (!x || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  ++x->blk->refs;
  *out = new ans_matrix{x->blk, x->seg};
  return ANS_OK;
}

int ans_profile_enable(ans_ctx* c, int enable) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  prof_collect(c);
  c->prof.acc.clear();
  c->prof.on = enable != 0;
  return ANS_OK;
}

int ans_profile_read(ans_ctx* c, char* buf, size_t buflen, size_t* needed) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  std::lock_guard<std::mutex> g(c->mu);
  DeviceGuard dg(c->device);
  prof_collect(c);
  std::string s;
  char line[256];
  for (const auto& kv : c->prof.acc) {
    std::snprintf(line, sizeof line, "%s %llu %.6f\n", kv.first.c_str(), (unsigned long long)kv.second.second,
                  kv.second.first);
    s += line;
  }
  if (needed) *needed = s.size() + 1;
  if (buf && buflen) {
    const size_t n = std::min(buflen - 1, s.size());
    std::memcpy(buf, s.data(), n);
    buf[n] = 0;
  }
  return ANS_OK;
}

int ans_ctx_memory(ans_ctx* c, size_t* live_bytes, size_t* budget_bytes) {
  if (!c) return fail(ANS_ERR_INVALID_ARG, "NULL context");
  std::lock_guard<std::mutex> g(c->mu);
  if (live_bytes) *live_bytes = c->live;
  if (budget_bytes) *budget_bytes = c->budget;
  return ANS_OK;
}

int ans_batch_bytes(ans_ctx* c, const uint64_t* h_offsets, size_t nwin, uint32_t flags, size_t* bytes) {
  if (!c || !h_offsets || !bytes) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  std::vector<uint64_t> lens(nwin);
  uint64_t total = 0, max_len = 0;
  for (size_t w = 0; w < nwin; ++w) {
    if (h_offsets[w + 1] < h_offsets[w]) return fail(ANS_ERR_INVALID_ARG, "offsets must be nondecreasing");
    lens[w] = h_offsets[w + 1] - h_offsets[w];
    total += lens[w];
    max_len = std::max(max_len, lens[w]);
  }
  HostPlan hp;
  hp.build(lens, nullptr);
  const bool want_mats = (flags & ANS_BATCH_MATRICES) != 0, want_sum = (flags & ANS_BATCH_SUM) != 0;
  std::lock_guard<std::mutex> g(c->mu);
  const bool hash = c->agg_path == 1 && nwin > 0;
  std::vector<size_t> guards;  // (debug mode: their bytes count too)
  GuardSink gs(c->guards ? &guards : nullptr);
  WinLayout wl;
  wl.reserve(hp, (uint32_t)nwin, want_mats, want_sum, total, max_len, hash);
  size_t need = 0;
  if (wl.size > c->scratch_size)  // the scratch is replaced by a larger one
    need += std::max(wl.size, c->scratch_size + c->scratch_size / 4) - c->scratch_size;
  if (hash) {
    std::vector<uint32_t> lg;
    HostPlan tab;
    plan_tables(lens, &lg, &tab);
    if (tab.pad > c->hash_slots) need += (tab.pad - c->hash_slots) * 12;  // the arena is replaced
  }
  if (want_mats && nwin) need += BlockLayout(hp.pad, (uint32_t)nwin).total;
  if (want_sum) need += BlockLayout((total + kTile - 1) / kTile * kTile, 1).total;
  *bytes = need;
  return ANS_OK;
}

int ans_get_tuning(ans_ctx* c, ans_tuning* out) {
  if (!c || !out) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  std::lock_guard<std::mutex> g(c->mu);
  out->key_threads = (uint32_t)c->cfg_keys.threads;
  out->key_rank = (uint32_t)c->cfg_keys.rank;
  out->key_blocks = (uint32_t)c->cfg_keys.blocks;
  out->kv_threads = (uint32_t)c->cfg_kv.threads;
  out->kv_rank = (uint32_t)c->cfg_kv.rank;
  out->kv_blocks = (uint32_t)c->cfg_kv.blocks;
  out->col_threads = (uint32_t)c->cfg_col.threads;
  out->col_rank = (uint32_t)c->cfg_col.rank;
  out->col_blocks = (uint32_t)c->cfg_col.blocks;
  out->win_path = (uint32_t)c->win_path;
  out->win_threads = (uint32_t)c->cfg_win.threads;
  out->win_rank = (uint32_t)c->cfg_win.rank;
  out->sum_path = (uint32_t)c->sum_path;
  out->agg_path = (uint32_t)c->agg_path;
  out->graph = (uint32_t)c->graph;
  out->col_hash = (uint32_t)c->col_hash;
  out->merge_tile = (uint32_t)c->merge_tile;
  return ANS_OK;
}

int ans_set_tuning(ans_ctx* c, const ans_tuning* t) {
  if (!c || !t) return fail(ANS_ERR_INVALID_ARG, "NULL argument");
  auto ok = [](uint32_t th, uint32_t rk, uint32_t bl) {
    return (th == 512 || th == 1024) && rk <= 2 && (bl == 1 || (bl == 2 && th == 512));
  };
  auto sub = [](uint32_t th, uint32_t rk, uint32_t bl) { return th == 256 && rk <= 2 && bl == 4; };
  if (!(sub(t->key_threads, t->key_rank, t->key_blocks) || ok(t->key_threads, t->key_rank, t->key_blocks)) ||
      !ok(t->kv_threads, t->kv_rank, t->kv_blocks) ||
      !(sub(t->col_threads, t->col_rank, t->col_blocks) || ok(t->col_threads, t->col_rank, t->col_blocks)))
    return fail(ANS_ERR_INVALID_ARG,
                "threads must be 512 or 1024, rank 0, 1 or 2, blocks 1 (or 2 with 512 threads); key and column "
                "passes also take 256 threads with blocks 4");
  if (t->win_path > 1 || t->win_rank > 1 || !ok(t->win_threads, t->win_rank, 1))
    return fail(ANS_ERR_INVALID_ARG, "win_path must be 0 or 1, win_threads 512 or 1024, win_rank 0 or 1");
  if (t->sum_path > 2) return fail(ANS_ERR_INVALID_ARG, "sum_path must be 0, 1 or 2");
  if (t->agg_path > 3) return fail(ANS_ERR_INVALID_ARG, "agg_path must be 0, 1, 2 or 3");
  if (t->graph > 1) return fail(ANS_ERR_INVALID_ARG, "graph must be 0 or 1");
  if (t->col_hash > 1) return fail(ANS_ERR_INVALID_ARG, "col_hash must be 0 or 1");
  if (t->merge_tile != 2048 && t->merge_tile != 4096) return fail(ANS_ERR_INVALID_ARG, "merge_tile must be 2048 or 4096");
  std::lock_guard<std::mutex> g(c->mu);
  c->win_path = (int)t->win_path;
  c->cfg_win = SortCfg{(int)t->win_threads, (int)t->win_rank, 1};
  c->sum_path = (int)t->sum_path;
  c->agg_path = (int)t->agg_path;
  c->graph = (int)t->graph;
  c->col_hash = (int)t->col_hash;
  c->merge_tile = (int)t->merge_tile;
  if (c->agg_path != 1 && c->hash_mem) {  // the hash tables are no longer needed
    DeviceGuard dg(c->device);
    ANS_CUDA(device_wait());
    dev_free(c, c->hash_mem, c->hash_slots * 12, c->aux);
    c->hash_mem = nullptr;
    c->hash_slots = 0;
  }
  c->cfg_keys = SortCfg{(int)t->key_threads, (int)t->key_rank, (int)t->key_blocks};
  c->cfg_kv = SortCfg{(int)t->kv_threads, (int)t->kv_rank, (int)t->kv_blocks};
  c->cfg_col = SortCfg{(int)t->col_threads, (int)t->col_rank, (int)t->col_blocks};
  return ANS_OK;
}

int ans_autotune(ans_ctx* c, const uint32_t* d_src, const uint32_t* d_dst, const uint64_t* h_offsets, size_t nwin,
                 uint32_t flags, ans_tuning* chosen, void* stream) {
  if (!c || !h_offsets || nwin == 0) return fail(ANS_ERR_INVALID_ARG, "NULL argument or empty batch");
  if (flags & ~(ANS_BATCH_MATRICES | ANS_BATCH_SUM | ANS_BATCH_SYNC)) return fail(ANS_ERR_INVALID_ARG, "unknown flag");
  flags &= ANS_BATCH_MATRICES | ANS_BATCH_SUM;
  // The last kColOnly shapes exist for the column passes only (not for the
  // kv passes).  Packets are sorted without digit passes: the key_* shape
  // stays as it is set.
  constexpr int kVariants = 12, kColOnly = 3;
  const SortCfg variants[kVariants] = {{512, kRankMatch, 1}, {512, kRankBallot, 1}, {512, kRankTable, 1},
                                       {512, kRankMatch, 2}, {512, kRankBallot, 2}, {512, kRankTable, 2},
                                       {1024, kRankMatch, 1}, {1024, kRankBallot, 1}, {1024, kRankTable, 1},
                                       {256, kRankMatch, 4}, {256, kRankBallot, 4}, {256, kRankTable, 4}};
  using Prof = std::map<std::string, double>;
  std::vector<ans_matrix*> per(nwin, nullptr);
  // The radix-pass shapes are timed with per-window matrices and the time
  // sum (every pass family runs); the paths by the caller's own flags.
  uint32_t run_flags = ANS_BATCH_MATRICES | ANS_BATCH_SUM;
  auto run_once = [&]() -> int {
    ans_matrix* sum = nullptr;
    int rc = ans_batch_submit_host(c, d_src, d_dst, h_offsets, nwin, run_flags | ANS_BATCH_SYNC, nullptr,
                                   per.data(), &sum, nullptr, stream);
    if (rc != ANS_OK) return rc;
    for (auto& m : per) {
      ans_matrix_free(m);
      m = nullptr;
    }
    ans_matrix_free(sum);
    return ANS_OK;
  };
  // One trial: apply `set` to the context, run the batch once untimed (module
  // load, shared-memory carve-out), then twice with per-kernel timing (the
  // kernel totals go to *out) and twice as the production path runs it (one
  // graph with its concurrent branches, no per-kernel events): the least
  // device time of those two, between CUDA events on `stream`, goes to
  // (*out)[kWall].  A trial that cannot get its memory (a path the device
  // cannot hold for this batch) reports false instead of failing.
  const std::string kWall = "(batch)";
  const char* log_env = std::getenv("ANS_AUTOTUNE_LOG");
  const bool log_trials = log_env && *log_env && std::strcmp(log_env, "0") != 0;
  auto trial = [&](auto&& set, Prof* out, bool* ran) -> int {
    {
      std::lock_guard<std::mutex> g(c->mu);
      set();
    }
    *ran = false;
    int rc = run_once();
    if (rc == ANS_OK) {
      ANS_TRY(ans_profile_enable(c, 1));
      for (int rep = 0; rep < 2 && rc == ANS_OK; ++rep) rc = run_once();
    }
    {
      std::lock_guard<std::mutex> g(c->mu);
      DeviceGuard dg(c->device);
      prof_collect(c);
      out->clear();
      for (const auto& kv : c->prof.acc) (*out)[kv.first] = kv.second.first;
      c->prof.acc.clear();
      c->prof.on = false;
    }
    double wall = 1e300;
    if (rc == ANS_OK) {
      DeviceGuard dg(c->device);
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return fail(ANS_ERR_CUDA, "cudaEventCreate failed");
      }
      for (int rep = 0; rep < 2 && rc == ANS_OK; ++rep) {
        cudaEventRecord(e0, (cudaStream_t)stream);
        ans_matrix* sum = nullptr;
        rc = ans_batch_submit_host(c, d_src, d_dst, h_offsets, nwin, run_flags, nullptr, per.data(), &sum, nullptr,
                                   stream);
        cudaEventRecord(e1, (cudaStream_t)stream);
        if (rc == ANS_OK) {
          float ms = 0;
          if (cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess)
            wall = std::min(wall, (double)ms);
          for (auto& m : per) {
            ans_matrix_free(m);
            m = nullptr;
          }
          ans_matrix_free(sum);
        }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
    }
    (*out)[kWall] = wall;
    if (log_trials) {
      std::string line = "ans_autotune: agg_path " + std::to_string(c->agg_path) + " sum_path " +
                         std::to_string(c->sum_path) + " win_path " + std::to_string(c->win_path) + " key " +
                         std::to_string(c->cfg_keys.threads) + "," + std::to_string(c->cfg_keys.rank) + "," +
                         std::to_string(c->cfg_keys.blocks) + " col " + std::to_string(c->cfg_col.threads) + "," +
                         std::to_string(c->cfg_col.rank) + "," + std::to_string(c->cfg_col.blocks) + ": " +
                         (rc == ANS_OK ? "batch " + std::to_string(wall) + " ms" : std::string("did not run"));
      for (const auto& kv : *out)
        if (kv.first != kWall) line += " " + kv.first + "=" + std::to_string(kv.second / 2);
      std::fprintf(stderr, "%s\n", line.c_str());
    }
    if (rc == ANS_ERR_OOM || rc == ANS_ERR_BUDGET) return ANS_OK;
    if (rc == ANS_OK) *ran = true;
    return rc;
  };

  auto get = [](const Prof& p, const char* k) {
    auto it = p.find(k);
    return it == p.end() ? 0.0 : it->second;
  };
  constexpr double kNever = 1e300;
  auto sort_time = [&](const Prof& p) {
    return get(p, "ss_sample") + get(p, "ss_count") + get(p, "ss_scatter") + get(p, "ss_plan") + get(p, "ss_local");
  };

  // Radix-pass launch shapes, per family, on the paths that use them all.
  double t_keys = kNever, t_kv[kVariants], t_col[kVariants];
  for (int v = 0; v < kVariants; ++v) {
    const bool col_only = v >= kVariants - kColOnly;
    Prof pr;
    bool ran = false;
    ANS_TRY(trial([&] {
      c->cfg_kv = variants[col_only ? 0 : v];
      c->cfg_col = variants[v];
      c->win_path = 1;  // the sample sort on every window
      c->sum_path = 1;  // the kv passes on the time sum
      c->agg_path = 0;
    }, &pr, &ran));
    if (!ran) return fail(ANS_ERR_OOM, "autotune: the batch does not fit the device with the default paths");
    t_keys = std::min(t_keys, sort_time(pr));
    t_kv[v] = col_only ? kNever : get(pr, "onesweep_sum") + get(pr, "gather");
    t_col[v] = get(pr, "onesweep_col");
  }
  auto best = [&](const double* t) {
    int b = 0;
    for (int v = 1; v < kVariants; ++v)
      if (t[v] < t[b]) b = v;
    return b;
  };
  const int bv_i = best(t_kv), bc_i = best(t_col);
  auto base = [&] {
    c->cfg_kv = variants[bv_i];
    c->cfg_col = variants[bc_i];
  };

  // The on-chip window sort (windows that fit a cluster) against the sample
  // sort.
  int win_path = 1;
  SortCfg win_cfg{1024, kRankMatch, 1};
  double best_win = t_keys;
  if (cluster_sort_clusters(c->device) > 0) {
    const SortCfg wv[3] = {{1024, kRankMatch, 1}, {1024, kRankBallot, 1}, {512, kRankMatch, 1}};
    for (const SortCfg& w : wv) {
      Prof pr;
      bool ran = false;
      ANS_TRY(trial([&] {
        base();
        c->win_path = 0;
        c->cfg_win = w;
        c->sum_path = 1;
        c->agg_path = 0;
      }, &pr, &ran));
      const double t = ran ? get(pr, "cluster_sort") + sort_time(pr) : kNever;
      if (t < best_win) {
        best_win = t;
        win_path = 0;
        win_cfg = w;
      }
    }
  }

  // Time sums (pairwise merges, whose ordering runs beside the window column
  // pass, against the kv passes and the packet re-sort) and then window
  // aggregation (sorting every packet, or hash counting of links): each by the
  // batch's device time as the production path runs it with the caller's
  // flags, everything else as chosen.
  run_flags = flags;
  int sum_path = 0;
  {
    double wall[3] = {kNever, kNever, kNever};
    for (int sp = 0; sp < 3; ++sp) {
      Prof pr;
      bool ran = false;
      ANS_TRY(trial([&] {
        base();
        c->win_path = win_path;
        c->cfg_win = win_cfg;
        c->sum_path = sp;
        c->agg_path = 0;
      }, &pr, &ran));
      if (ran) wall[sp] = pr[kWall];
    }
    for (int sp = 1; sp < 3; ++sp)
      if (wall[sp] < wall[sum_path]) sum_path = sp;
  }
  // Merge rounds: 4096 or 2048 output positions per CTA (the smaller tile
  // fits more CTAs per SM; the larger needs fewer merge-path searches).
  int merge_tile = 4096;
  if (sum_path == 0) {
    double wall[2] = {kNever, kNever};
    const int tiles[2] = {4096, 2048};
    for (int i = 0; i < 2; ++i) {
      Prof pr;
      bool ran = false;
      ANS_TRY(trial([&] {
        base();
        c->win_path = win_path;
        c->cfg_win = win_cfg;
        c->sum_path = 0;
        c->merge_tile = tiles[i];
        c->agg_path = 0;
      }, &pr, &ran));
      if (ran) wall[i] = pr[kWall];
    }
    merge_tile = wall[1] < wall[0] ? 2048 : 4096;
    c->merge_tile = merge_tile;
  }
  // (agg_path 2 is agg_path 0, and agg_path 3 is that with sum_path 2: both
  // have been timed)
  int agg_path = 0;
  {
    double wall[2] = {kNever, kNever};
    for (int a = 0; a < 2; ++a) {
      Prof pr;
      bool ran = false;
      ANS_TRY(trial([&] {
        base();
        c->win_path = win_path;
        c->cfg_win = win_cfg;
        c->sum_path = sum_path;
        c->agg_path = a;
      }, &pr, &ran));
      if (ran) wall[a] = pr[kWall];
    }
    if (wall[1] < wall[0]) agg_path = 1;
  }

  // With the paths chosen, the column passes' shape (on the large time sums
  // they order the summed links by destination hash) by the batch's device
  // time as the production path runs it.
  SortCfg bc = variants[bc_i];
  const SortCfg bv = variants[bv_i];
  {
    auto chosen_paths = [&] {
      base();
      c->cfg_col = bc;
      c->win_path = win_path;
      c->cfg_win = win_cfg;
      c->sum_path = sum_path;
      c->agg_path = agg_path;
      c->merge_tile = merge_tile;
    };
    Prof pr;
    bool ran = false;
    ANS_TRY(trial(chosen_paths, &pr, &ran));
    double best_wall = ran ? pr[kWall] : kNever;
    if (ran && get(pr, "onesweep_col") > 0) {
      const SortCfg cv[6] = {{512, kRankMatch, 1}, {512, kRankBallot, 1}, {512, kRankMatch, 2},
                             {512, kRankBallot, 2}, {256, kRankMatch, 4}, {256, kRankBallot, 4}};
      for (const SortCfg& v : cv) {
        if (v.threads == bc.threads && v.rank == bc.rank && v.blocks == bc.blocks) continue;
        ANS_TRY(trial([&] { chosen_paths(); c->cfg_col = v; }, &pr, &ran));
        if (ran && pr[kWall] < best_wall) {
          best_wall = pr[kWall];
          bc = v;
        }
      }
    }
  }

  ans_tuning res{};
  res.key_threads = (uint32_t)c->cfg_keys.threads;
  res.key_rank = (uint32_t)c->cfg_keys.rank;
  res.key_blocks = (uint32_t)c->cfg_keys.blocks;
  res.kv_threads = (uint32_t)bv.threads;
  res.kv_rank = (uint32_t)bv.rank;
  res.kv_blocks = (uint32_t)bv.blocks;
  res.col_threads = (uint32_t)bc.threads;
  res.col_rank = (uint32_t)bc.rank;
  res.col_blocks = (uint32_t)bc.blocks;
  res.win_path = (uint32_t)win_path;
  res.win_threads = (uint32_t)win_cfg.threads;
  res.win_rank = (uint32_t)win_cfg.rank;
  res.sum_path = (uint32_t)sum_path;
  res.agg_path = (uint32_t)agg_path;
  res.graph = (uint32_t)c->graph;
  res.col_hash = (uint32_t)c->col_hash;
  res.merge_tile = (uint32_t)merge_tile;
  ANS_TRY(ans_set_tuning(c, &res));
  if (chosen) *chosen = res;
  return ANS_OK;
}

}  // extern "C"
