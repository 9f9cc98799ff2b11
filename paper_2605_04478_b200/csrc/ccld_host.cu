// Host side of libccld: context, communicator registry, window upload, launch sequencing and result
// read-back. No analysis arithmetic lives here; every step of the hot path is a kernel in
// ccld_kernels.cuh.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <unordered_map>
#include <utility>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "ccld_kernels.cuh"
#include "ccld_verdict.cuh"
#include "ccld_rates.cuh"
#include "ccld_opset.cuh"

using namespace ccld;

namespace {

constexpr size_t ALIGN = 256;
inline size_t align_up(size_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }

struct Block { void* p = nullptr; size_t bytes = 0; };

struct CommHost {
  u32 id, seq0; std::vector<u32> ranks;
  u8 algo = 0;                      // 0 ring, 1 tree
  std::vector<u32> head;            // tree: lowest position of a member's layer (empty until the layers are set)
  const u32* d_head = nullptr;      // device copy inside the registry block
};

// What contexts that are gone leave to those that live: a process-wide store of pinned and device blocks. Allocating is what a
// context's first pass costs most (measured: cudaMallocHost 1 to 13 ms, cudaMalloc 0.36 ms whatever the size), and programs
// make a context per job or per device. The first pass over some 8 M records needs about 150 MB of the device; larger jobs
// allocate, and their memory is wanted elsewhere in the process. So the store holds at most 256 MB per device (with 64 MB the first
// pass over two windows of 4,096 ranks took 3.3 ms instead of 0.9) and 64 MB of pinned memory. Every access holds its lock, blocks enter it only once their stream has been waited for, and it is emptied when the
// last context goes or an allocation fails.
class BlockStore {
 public:
  static BlockStore& get() { static BlockStore* s = new BlockStore; return *s; }      // never destroyed: contexts may outlive static objects
  void enter() { std::lock_guard<std::mutex> g(m_); ++users_; }
  void leave() { std::lock_guard<std::mutex> g(m_); if (--users_ == 0) drain(); }
  bool take(int device, size_t bytes, Block* out) {       // device < 0: pinned
    std::lock_guard<std::mutex> g(m_);
    auto& l = lists_[device];
    int best = -1;
    for (size_t i = 0; i < l.size(); ++i) if (l[i].bytes >= bytes && l[i].bytes <= 2 * bytes + (1u << 20) && (best < 0 || l[i].bytes < l[best].bytes)) best = (int)i;
    if (best < 0) return false;
    *out = l[best]; l.erase(l.begin() + best); held_[device] -= out->bytes;
    return true;
  }
  void put(int device, Block b) {
    if (!b.p) return;
    std::lock_guard<std::mutex> g(m_);
    const size_t most = device < 0 ? PINNED_MOST : DEVICE_MOST;
    if (held_[device] + b.bytes > most) { free_block(device, b); return; }
    try { lists_[device].push_back(b); held_[device] += b.bytes; } catch (...) { free_block(device, b); }
  }
  void clear() { std::lock_guard<std::mutex> g(m_); drain(); }
  // Pinned blocks that callers keep (ccld_host_block): at most LENT_MOST bytes at a time.
  bool lend(size_t bytes) { std::lock_guard<std::mutex> g(m_); if (lent_ + bytes > LENT_MOST) return false; lent_ += bytes; return true; }
  void give_back(Block b, size_t lent) {
    bool used;
    { std::lock_guard<std::mutex> g(m_); lent_ -= lent; used = users_ > 0; }
    if (used) put(-1, b); else if (b.p) free_block(-1, b);
  }

 private:
  static constexpr size_t PINNED_MOST = 64u << 20, DEVICE_MOST = 256u << 20, LENT_MOST = 64u << 20;
  // Blocks are freed whenever the last array on one goes, also while the caller captures a graph: with this thread's own
  // captures set aside, freeing is no part of them and does not end them. (cudaFree takes any device's pointer.)
  static void free_block(int device, Block b) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (device < 0) cudaFreeHost(b.p); else cudaFree(b.p);
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
  void drain() { for (auto& kv : lists_) { for (Block& b : kv.second) free_block(kv.first, b); kv.second.clear(); held_[kv.first] = 0; } }
  std::mutex m_; int users_ = 0; size_t lent_ = 0;
  std::map<int, std::vector<Block>> lists_; std::map<int, size_t> held_;
};

// Device blocks are recycled through a free list so that steady-state analysis allocates nothing.
struct Pool {
  int device = 0;
  std::vector<Block> free_list;
  Block records;                                // space for a batch's records in their slots: see record_space
  Block get(size_t bytes, cudaError_t* err) {
    bytes = align_up(std::max<size_t>(bytes, ALIGN));
    int best = -1;
    for (size_t i = 0; i < free_list.size(); ++i)
      if (free_list[i].bytes >= bytes && free_list[i].bytes <= 2 * bytes + (1u << 20) && (best < 0 || free_list[i].bytes < free_list[best].bytes)) best = (int)i;
    if (best >= 0) { Block b = free_list[best]; free_list.erase(free_list.begin() + best); *err = cudaSuccess; return b; }
    Block b;
    if (BlockStore::get().take(device, bytes, &b)) { *err = cudaSuccess; return b; }
    b.bytes = bytes;
    *err = cudaMalloc(&b.p, bytes);
    if (*err != cudaSuccess) {                 // give cached blocks back to the driver and retry once
      cudaGetLastError();
      for (auto& f : free_list) cudaFree(f.p);
      free_list.clear();
      if (records.p) cudaFree(records.p);      // (waits for the kernels that use it; a batch asks for it last)
      records = Block{};
      BlockStore::get().clear();
      *err = cudaMalloc(&b.p, bytes);
      if (*err != cudaSuccess) { b.p = nullptr; b.bytes = 0; }
    }
    return b;
  }
  void put(Block b) { if (b.p) free_list.push_back(b); }
  void leave_all() { put(records); records = Block{}; for (auto& f : free_list) BlockStore::get().put(device, f); free_list.clear(); }      // the stream must be idle
};

struct Shared {                                 // a pooled block shared by the windows of one batch
  Pool* pool; Block b;
  Shared(Pool* p, Block blk) : pool(p), b(blk) {}
  ~Shared() { pool->put(b); }
};

struct WindowHost {
  u32 id = 0; u64 n_rec = 0; bool owns = false; Block own;
  WinDesc d;                                    // device pointers
  u32 n_frames = 0, n_channels = 0;
  const u32 *f_rank = nullptr, *f_comm = nullptr, *f_seq = nullptr, *progress = nullptr;
  const u8 *algo = nullptr, *proto = nullptr; bool owns_opset = false; Block opset_own;   // Operation Type Set columns
  bool analysed = false;
  std::shared_ptr<Shared> plan_blk, res_blk;
  WinDesc* d_desc = nullptr;                    // this window's descriptor on the device
  u64 totals[T_COUNT];
  WindowHost() { std::memset(&d, 0, sizeof d); std::memset(totals, 0, sizeof totals); }
};

// A batch that was enqueued on totals the host expected instead of waiting for the plan: its actual totals arrive in
// pinned memory behind the batch's kernels and are checked at the next call that synchronizes anyway.
// A batch that waited is listed only for its pinned block, which its last descriptor copy still reads.
struct PendingBatch { u32 first = 0, n = 0; i64 now = 0; Block pin; bool speculative = false, mixed = false; const u64* h_tot() const { return (const u64*)pin.p; } };
// Totals of the last batches that were planned with a wait, by shape (record count of every window).
struct ShapeEntry { std::vector<u64> n_rec; std::vector<u64> totals; bool no_record_space = false; };
constexpr size_t SHAPE_CACHE = 4;

// Pinned pieces that uploads of pageable memory pass through, with an event behind the last copy out of each.
struct UploadSlot { char* p = nullptr; cudaEvent_t done = nullptr; bool used = false; };
constexpr size_t UP_PIECE = 1u << 20;                      // a large upload goes piece by piece
constexpr u32 UP_WORKERS = 6, UP_SLOTS = 2 * UP_WORKERS;   // two pieces per worker: one being filled, one on its way
// Up to this size one kernel reads the pinned columns, beyond it they are copied one by one. Nine copies leave gaps of 2 us and more between
// them: 0.6 MB take 63 us with copies and 36 with the kernel, 2.3 MB 94 and 69, 6.9 MB 180 and 160, 23 MB 473 and 474, 32 MB 639 and 654; where
// others share the host's PCIe a pass over 23 MB took 723 to 1,169 us with copies, 563 to 641 with the kernel.
// One CTA per column with four words per thread on their way, because reads that wait for PCIe hold up what else runs on the GPU: a matrix
// product beside uploads takes 18 % longer, a copy of device memory 35 (beside copies 2 and 2; with 64 registers per thread instead of 32, which
// lets no other CTA onto the SM, 19 to 28 and 35 to 40). Twice the words: 30 and 55 % (no faster);
// half of them 16 and 34, a quarter 5 and 11 (23 MB 477 and 482 us); 32 CTAs of 256 threads and a word each per column: 68 and 60 %.
constexpr size_t UP_SMALL = 32u << 20;
constexpr int UP_AHEAD = 4, UP_THREADS = 1024;

constexpr u64 PACK_MOST = 8ull << 30;                      // space for records in their slots, at most (and at most half of what is free)

constexpr u32 TIMER_RING = 32;
constexpr int TIMER_PAIRS = CCLD_K_KINDS + 1;          // two launches of the plan per call
struct TimerSlot { cudaEvent_t a[TIMER_PAIRS], b[TIMER_PAIRS]; int kind[TIMER_PAIRS]; int n = 0; };

}  // namespace

struct ccld_ctx {
  ccld_params params; Params dp; int device = 0; cudaStream_t stream = nullptr;
  std::vector<CommHost> comms; std::unordered_map<u32, u32> comm_idx;
  bool finalized = false; u32 n_ranks = 0, max_n = 0, max_large_n[3] = {0, 0, 0}, max_mid_n[3] = {0, 0, 0};     // largest communicators of up to 2048, 4096, 8192 and of up to 256, 512, 1024 ranks 
  u64 sum_n = 0; u32 n_sms = 148;
  Block reg_blk, misc_blk; Registry reg; size_t stats_off = 0, stats_bytes = 0;
  const TreeRef* d_trees = nullptr; u32 n_trees = 0;     // tree communicators whose layers are known
  std::map<u32, WindowHost> windows;
  Pool pool; std::string err;
  cudaStream_t side[2] = {nullptr, nullptr}; cudaEvent_t fork = nullptr, join[2] = {nullptr, nullptr};     // see Chains
  Block h_verdict;                                       // pinned area of ccld_get_verdict (VerdictArea)
  Block h_io;                                            // pinned area small results pass through
  bool long_list = false;                                // the last suspect list was longer than VD_MERGE
  std::vector<char> long_suspects;                       // columns of a suspect list that outgrew the pinned area
  Block h_up; UploadSlot up[UP_SLOTS]; u32 up_next = 0;
  cudaStream_t up_stream = nullptr; cudaEvent_t up_event = nullptr;     // see UploadStream
  u64 batches_redone = 0;                                // batches settle() had to analyse again
  u64 unwaited = 0, packed = 0, filled_under_range = 0;  // batches that took these ways (ccld_get_route_counts)
  std::vector<PendingBatch> pending; std::vector<Block> pinned_free; std::vector<ShapeEntry> shapes;
  u32* d_poison = nullptr; int speculate = 1;
  // optional per-kernel timing: a ring of event pairs, harvested lazily
  bool timing = false; std::vector<TimerSlot> ring; u32 ring_next = 0;
  double t_ms[CCLD_K_KINDS]; u64 t_launches[CCLD_K_KINDS];
  ccld_ctx() { std::memset(&reg, 0, sizeof reg); std::memset(t_ms, 0, sizeof t_ms); std::memset(t_launches, 0, sizeof t_launches); }
};

namespace {

int fail(ccld_ctx* c, int code, const std::string& msg) { if (c) c->err = msg; return code; }

#define CK(call)                                                                                   \
  do { cudaError_t e_ = (call);                                                                    \
       if (e_ != cudaSuccess) return fail(ctx, e_ == cudaErrorMemoryAllocation ? CCLD_ERR_NOMEM : CCLD_ERR_CUDA, \
                                          std::string(#call) + ": " + cudaGetErrorString(e_)); } while (0)

// Host memory that runs out inside an entry point is a return code: nothing is thrown through the C boundary.
int caught(ccld_ctx* ctx) {
  try { return fail(ctx, CCLD_ERR_NOMEM, "out of host memory"); } catch (...) { return CCLD_ERR_NOMEM; }
}
#define CAUGHT catch (...) { return caught(ctx); }

// Adds the elapsed times of a slot's finished event pairs to the sums (waits for the last one).
void timer_harvest(ccld_ctx* ctx, TimerSlot& s) {
  for (int i = 0; i < s.n; ++i) {
    float ms = 0.f;
    if (cudaEventSynchronize(s.b[i]) == cudaSuccess && cudaEventElapsedTime(&ms, s.a[i], s.b[i]) == cudaSuccess) {
      ctx->t_ms[s.kind[i]] += ms; ctx->t_launches[s.kind[i]] += 1;
    }
  }
  s.n = 0;
}
TimerSlot* timer_begin(ccld_ctx* ctx) {
  if (!ctx->timing) return nullptr;
  TimerSlot& s = ctx->ring[ctx->ring_next++ % TIMER_RING];
  timer_harvest(ctx, s);
  return &s;
}
// A named range for timeline tools (a no-op unless one is attached).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete; NvtxRange& operator=(const NvtxRange&) = delete;
};
const char* const STAGE_NAMES[CCLD_K_KINDS] = {"ccld: op-counter ranges", "ccld: layout", "ccld: slot scatter", "ccld: reduce (up to 128 ranks)",
                                               "ccld: reduce (129 to 1024 ranks)", "ccld: reduce (more than 1024 ranks)", "ccld: window decision"};

struct TimedLaunch {                                     // a named range and, when timing is on, an event pair around one launch
  NvtxRange r; TimerSlot* s; cudaStream_t st; int i;
  TimedLaunch(TimerSlot* slot, int kind, cudaStream_t stream) : r(STAGE_NAMES[kind]), s(slot), st(stream), i(-1) {
    if (s && s->n < TIMER_PAIRS) { i = s->n++; s->kind[i] = kind; cudaEventRecord(s->a[i], st); }
  }
  ~TimedLaunch() { if (i >= 0) cudaEventRecord(s->b[i], st); }
};

// Every kernel of the library starts with begin_after(): it may be launched while the one before it in the stream still runs,
// waits there until that one is done, and lets the next one be launched. A launch then costs its latency beside the kernel
// before it instead of after it.
struct On {                                               // a stream; overlap = false: the launch follows a wait for another stream
  cudaStream_t stream; bool overlap;
  On(cudaStream_t s, bool o = true) : stream(s), overlap(o) {}
};
template <class... P, class... A>
void launch_cluster(On on, void (*kernel)(P...), u32 cluster, dim3 grid, dim3 block, size_t smem, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = on.stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[0].val.programmaticStreamSerializationAllowed = on.overlap ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension; at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);      // the caller looks at cudaGetLastError()
}

template <class... P, class... A>
void launch(On on, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, A&&... args) {
  launch_cluster(on, kernel, 1, grid, block, smem, std::forward<A>(args)...);
}

// The reductions of the three sizes of communicators do not depend on one another. Where a batch has more than one size, they
// run on streams of their own between the slot scatter and the window decision: the kernel of the largest communicators
// waits on barriers and round trips most of the time, that of 129 to 1,024 ranks may have no more than a few CTAs (a warp per
// group), and the kernel of the small ones, which keeps memory busy, fills the SMs beside both. The side streams have
// priority over the caller's: what has few CTAs, or long ones, gets its place first. With kernel timing on everything stays
// on the caller's stream, so that a time belongs to one kernel.
// A pass over a window of 16,384 ranks in groups of 8, 128, 1,024 and 2,048: 995 -> 872 us; over two windows of 4,128 ranks in
// groups of 4, 6 and 172: 536 -> 527 us.
struct Chains {
  ccld_ctx* ctx; int n; bool used[2] = {false, false};
  Chains(ccld_ctx* c, int sizes, bool timed) : ctx(c), n(timed ? 0 : sizes - 1) {
    if (n > 0 && !ready()) n = 0;                          // no stream to be had: one after the other
    if (n > 0) cudaEventRecord(ctx->fork, ctx->stream);
  }
  bool ready() {
    int low = 0, high = 0;
    if (ctx->join[1]) return true;
    cudaDeviceGetStreamPriorityRange(&low, &high);
    bool ok = ctx->fork || cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; i < 2 && ok; ++i)
      ok = (ctx->side[i] || cudaStreamCreateWithPriority(&ctx->side[i], cudaStreamNonBlocking, high) == cudaSuccess) &&
           (ctx->join[i] || cudaEventCreateWithFlags(&ctx->join[i], cudaEventDisableTiming) == cudaSuccess);
    if (!ok) cudaGetLastError();
    return ok;
  }
  On open(int i) {                                         // where chain i runs
    if (i >= n) return On(ctx->stream);
    used[i] = true;
    cudaStreamWaitEvent(ctx->side[i], ctx->fork, 0);
    return On(ctx->side[i], false);
  }
  On close() {                                             // the caller's stream, after all chains
    for (int i = 0; i < 2; ++i) if (used[i]) { cudaEventRecord(ctx->join[i], ctx->side[i]); cudaStreamWaitEvent(ctx->stream, ctx->join[i], 0); }
    return On(ctx->stream, n <= 0);
  }
  static void drop(ccld_ctx* c) {
    for (int i = 0; i < 2; ++i) { if (c->join[i]) cudaEventDestroy(c->join[i]); if (c->side[i]) cudaStreamDestroy(c->side[i]); }
    if (c->fork) cudaEventDestroy(c->fork);
  }
};

// Layout of the scratch block used by get_verdict and locate_hang.
struct MiscLayout { size_t sus, keys, counts, done, alerts, total; };
MiscLayout misc_layout(u32 n_ranks) {
  MiscLayout L; size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off = align_up(off + std::max<size_t>(b, 1)); return o; };
  const size_t pieces = (n_ranks + VD_THREADS - 1) / VD_THREADS;
  L.sus = take(2ull * n_ranks * sizeof(ccld_suspect)); L.keys = take(pieces * VD_KEYS * 8); L.counts = take(pieces * 4); L.done = take(4);
  L.alerts = take(CCLD_MAX_ALERTS_PER_WINDOW * sizeof(ccld_hang_alert));
  L.total = off;
  return L;
}

// Layout of the pinned area the verdict kernels write to.
struct VerdictArea { size_t rows, alerts, suspects, total; u32 sus_cap; };
VerdictArea verdict_area(u32 n_comms, u32 n_ranks) {
  VerdictArea L; size_t off = align_up(sizeof(VerdictHead));
  auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
  L.sus_cap = std::min<u32>(2 * n_ranks, VD_SUS_HOST);
  L.rows = take((size_t)n_comms * sizeof(ccld_comm_verdict)); L.alerts = take(CCLD_MAX_ALERTS_PER_WINDOW * sizeof(ccld_hang_alert));
  L.suspects = take((size_t)L.sus_cap * sizeof(ccld_suspect));
  L.total = off;
  return L;
}

// Builds the device tables of the communicator registry and the per-rank statistics.
int finalize_registry(ccld_ctx* ctx) {
  if (ctx->finalized) return CCLD_OK;
  const u32 nc = (u32)ctx->comms.size();
  if (nc == 0) return fail(ctx, CCLD_ERR_STATE, "no communicator registered");
  u32 max_rank = 0; u64 sum_n = 0; u32 max_n = 0;
  for (auto& c : ctx->comms) {
    for (u32 r : c.ranks) max_rank = std::max(max_rank, r);
    sum_n += c.ranks.size(); max_n = std::max<u32>(max_n, (u32)c.ranks.size());
    const u32 n = (u32)c.ranks.size(), cls = comm_class(n);
    if (cls == 3) { u32& m = ctx->max_large_n[n <= 2048 ? 0 : (n <= 4096 ? 1 : 2)]; m = std::max(m, n); }
    if (cls == 2) { u32& m = ctx->max_mid_n[n <= 256 ? 0 : (n <= 512 ? 1 : 2)]; m = std::max(m, n); }
  }
  const u32 nr = max_rank + 1;
  u32 hsize = 16; while (hsize < 2 * nc) hsize <<= 1;
  if (nc >= (1u << (32 - RANK_TAB_POS_BITS))) return fail(ctx, CCLD_ERR_CAPACITY, "too many communicators");
  std::vector<uint4> hash(hsize, make_uint4(0, NONE, 0, 0));
  std::vector<u32> comm_id(nc), comm_n(nc), comm_seq0(nc), members; std::vector<u64> moff(nc);
  std::vector<u32> rank_ptr(nr + 1, 0);
  members.reserve(sum_n);
  for (u32 i = 0; i < nc; ++i) {
    const CommHost& c = ctx->comms[i];
    comm_id[i] = c.id; comm_n[i] = (u32)c.ranks.size(); comm_seq0[i] = c.seq0; moff[i] = members.size();
    members.insert(members.end(), c.ranks.begin(), c.ranks.end());
    u32 h = (c.id * 2654435761u) & (hsize - 1);
    while (hash[h].y != NONE) h = (h + 1) & (hsize - 1);
    hash[h] = make_uint4(c.id, i, c.seq0, (u32)c.ranks.size());
    for (u32 r : c.ranks) ++rank_ptr[r + 1];
  }
  for (u32 r = 0; r < nr; ++r) rank_ptr[r + 1] += rank_ptr[r];
  std::vector<u32> ent_comm(sum_n), ent_pos(sum_n), fill(rank_ptr.begin(), rank_ptr.end() - 1);
  for (u32 i = 0; i < nc; ++i)
    for (u32 p = 0; p < ctx->comms[i].ranks.size(); ++p) { u32 r = ctx->comms[i].ranks[p]; ent_comm[fill[r]] = i; ent_pos[fill[r]] = p; ++fill[r]; }
  // inline (communicator id, index << 13 | position) pairs per rank, RANK_TAB_K of them in two uint4
  std::vector<u32> rank_tab((size_t)nr * 2 * RANK_TAB_K, NONE);
  for (u32 r = 0; r < nr; ++r) {
    const u32 cnt = rank_ptr[r + 1] - rank_ptr[r];
    const u32 inl = cnt <= (u32)RANK_TAB_K ? cnt : (u32)RANK_TAB_K - 1;
    for (u32 k = 0; k < inl; ++k) {
      const u32 ci = ent_comm[rank_ptr[r] + k];
      rank_tab[((size_t)r * RANK_TAB_K + k) * 2] = ctx->comms[ci].id;
      rank_tab[((size_t)r * RANK_TAB_K + k) * 2 + 1] = (ci << RANK_TAB_POS_BITS) | ent_pos[rank_ptr[r] + k];
    }
    if (cnt > (u32)RANK_TAB_K) rank_tab[((size_t)r * RANK_TAB_K + RANK_TAB_K - 1) * 2 + 1] = RANK_TAB_OVERFLOW;
  }

  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
  const size_t o_hash = take(hsize * sizeof(uint4)), o_rtab = take(rank_tab.size() * 4), o_id = take(nc * 4), o_n = take(nc * 4), o_s0 = take(nc * 4), o_moff = take(nc * 8),
               o_mem = take(sum_n * 4), o_ptr = take((nr + 1) * 4ull), o_ec = take(sum_n * 4), o_ep = take(sum_n * 4);
  std::vector<size_t> o_head(nc, 0);
  u32 n_trees = 0;
  for (u32 i = 0; i < nc; ++i) if (!ctx->comms[i].head.empty()) { o_head[i] = take(ctx->comms[i].head.size() * 4); ++n_trees; }
  const size_t o_trees = take(std::max<u32>(n_trees, 1) * sizeof(TreeRef)), o_chead = take(nc * sizeof(u32*));
  const size_t o_stats = off;
  const size_t o_state = take(nc * sizeof(CommState)), o_votes = take(nr * 16ull), o_ops = take(nr * 4ull), o_cnt = take(nr * 4ull), o_bw = take(nr * 8ull);
  const size_t stats_end = off, o_poison = take(256);
  cudaError_t e;
  ctx->reg_blk = ctx->pool.get(off, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "registry allocation failed");
  char* base = (char*)ctx->reg_blk.p;
  cudaStream_t st = ctx->stream;
  CK(cudaMemcpyAsync(base + o_hash, hash.data(), hsize * sizeof(uint4), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_rtab, rank_tab.data(), rank_tab.size() * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_id, comm_id.data(), nc * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_n, comm_n.data(), nc * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_s0, comm_seq0.data(), nc * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_moff, moff.data(), nc * 8, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_mem, members.data(), sum_n * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_ptr, rank_ptr.data(), (nr + 1) * 4ull, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_ec, ent_comm.data(), sum_n * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(base + o_ep, ent_pos.data(), sum_n * 4, cudaMemcpyHostToDevice, st));
  for (u32 i = 0; i < nc; ++i) {
    CommHost& c = ctx->comms[i];
    if (c.head.empty()) continue;
    CK(cudaMemcpyAsync(base + o_head[i], c.head.data(), c.head.size() * 4, cudaMemcpyHostToDevice, st));
    c.d_head = (const u32*)(base + o_head[i]);
  }
  std::vector<const u32*> comm_head(nc, nullptr);
  for (u32 i = 0; i < nc; ++i) if (ctx->comms[i].algo != 0) comm_head[i] = ctx->comms[i].d_head ? ctx->comms[i].d_head : REG_NO_LAYERS;
  CK(cudaMemcpyAsync(base + o_chead, comm_head.data(), nc * sizeof(u32*), cudaMemcpyHostToDevice, st));
  std::vector<TreeRef> trees;
  for (u32 i = 0; i < nc; ++i) if (ctx->comms[i].d_head) { TreeRef t; t.c = i; t.pad = 0; t.head = ctx->comms[i].d_head; trees.push_back(t); }
  if (n_trees) CK(cudaMemcpyAsync(base + o_trees, trees.data(), n_trees * sizeof(TreeRef), cudaMemcpyHostToDevice, st));
  ctx->d_trees = (const TreeRef*)(base + o_trees); ctx->n_trees = n_trees;
  CK(cudaMemsetAsync(base + o_stats, 0, off - o_stats, st));
  CK(cudaStreamSynchronize(st));              // the host vectors above go out of scope
  Registry& R = ctx->reg;
  R.n_comms = nc; R.hash_mask = hsize - 1; R.n_ranks = nr; R.pad = 0;
  R.hash = (const uint4*)(base + o_hash); R.rank_tab = (const uint4*)(base + o_rtab); R.comm_id = (const u32*)(base + o_id); R.comm_n = (const u32*)(base + o_n);
  R.comm_seq0 = (const u32*)(base + o_s0); R.comm_moff = (const u64*)(base + o_moff); R.members = (const u32*)(base + o_mem);
  R.rank_ptr = (const u32*)(base + o_ptr); R.ent_comm = (const u32*)(base + o_ec); R.ent_pos = (const u32*)(base + o_ep);
  R.comm_head = (const u32* const*)(base + o_chead);
  R.state = (CommState*)(base + o_state); R.votes = (u32*)(base + o_votes); R.ops = (u32*)(base + o_ops);
  R.bw_cnt = (u32*)(base + o_cnt); R.bw_sum = (double*)(base + o_bw);
  ctx->stats_off = o_stats; ctx->stats_bytes = stats_end - o_stats; ctx->d_poison = (u32*)(base + o_poison);
  ctx->n_ranks = nr; ctx->max_n = max_n; ctx->sum_n = sum_n;

  // scratch for suspects, alert ordering and hang location
  ctx->misc_blk = ctx->pool.get(misc_layout(nr).total, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "scratch allocation failed");
  CK(cudaMemsetAsync((char*)ctx->misc_blk.p + misc_layout(nr).done, 0, 4, st));

  CK(cudaFuncSetAttribute(k_reduce_mid<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mid_smem_bytes(256)));
  CK(cudaFuncSetAttribute(k_reduce_mid<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mid_smem_bytes(512)));
  CK(cudaFuncSetAttribute(k_reduce_mid<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mid_smem_bytes(MID_N)));
  CK(cudaFuncSetAttribute(k_reduce_large_deferred, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(16ull * CCLD_MAX_COMM_SIZE)));
  CK(cudaFuncSetAttribute(k_seq_range, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)range_smem_bytes(RANGE_DIRECT)));
  CK(cudaFuncSetAttribute(k_hang_locate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(HANG_SMEM_N * HANG_MEMBER_BYTES)));
  CK(cudaFuncSetAttribute(k_opset_check, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(CCLD_MAX_COMM_SIZE * OPSET_MEMBER_BYTES)));
  // The gathers of the small groups are held up by the cache lines an SM can have on their way: no more shared memory than the
  // CTAs need, the rest of the SM's 256 KB is L1. (The other kernels are best off with the driver's own choice.)
  CK(cudaFuncSetAttribute(k_reduce_fused<false>, cudaFuncAttributePreferredSharedMemoryCarveout, FUSED_CARVEOUT));
  CK(cudaFuncSetAttribute(k_reduce_fused<true>, cudaFuncAttributePreferredSharedMemoryCarveout, FUSED_CARVEOUT));
  CK(cudaFuncSetAttribute(k_reduce_large<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LargeTile<4>::BYTES));
  CK(cudaFuncSetAttribute(k_reduce_large<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LargeTile<8>::BYTES));
  CK(cudaFuncSetAttribute(k_reduce_large<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LargeTile<16>::BYTES));
  ctx->finalized = true;
  return CCLD_OK;
}

void drop_results(WindowHost& w) {
  w.analysed = false; w.plan_blk.reset(); w.res_blk.reset(); w.d_desc = nullptr;
  std::memset(w.totals, 0, sizeof w.totals);
}

int analyze_batch(ccld_ctx* ctx, u32 first_window, u32 n_windows, i64 now_ns, bool may_speculate);

Block pinned_get(ccld_ctx* ctx, size_t bytes) {
  for (size_t i = 0; i < ctx->pinned_free.size(); ++i)
    if (ctx->pinned_free[i].bytes >= bytes) { Block b = ctx->pinned_free[i]; ctx->pinned_free.erase(ctx->pinned_free.begin() + i); return b; }
  Block b;
  if (BlockStore::get().take(-1, bytes, &b)) return b;
  b.bytes = (bytes + 65535) / 65536 * 65536;              // whole 64 KB pieces, so that blocks fit other batches too
  if (cudaMallocHost(&b.p, b.bytes) != cudaSuccess) {
    cudaGetLastError();
    BlockStore::get().clear();
    if (cudaMallocHost(&b.p, b.bytes) != cudaSuccess) { cudaGetLastError(); b.p = nullptr; b.bytes = 0; }
  }
  return b;
}
// A pinned area of the context of at least `bytes` bytes. Nothing in flight may still use it.
int pinned_area(ccld_ctx* ctx, Block& area, size_t bytes) {
  if (area.bytes >= bytes) return CCLD_OK;
  BlockStore::get().put(-1, area);
  area = pinned_get(ctx, bytes);
  return area.p ? CCLD_OK : fail(ctx, CCLD_ERR_NOMEM, "pinned allocation failed");
}

// Copies device arrays to host memory, all with one wait. Up to FETCH_PINNED bytes in all pass through pinned memory, written
// there by one kernel: a copy each into pageable memory costs 15 to 20 us apiece, the kernel about 5 us for all. More than
// that is left to the driver's copies, whose fixed cost no longer counts.
struct Piece { const void* src; void* dst; size_t n; };
constexpr size_t FETCH_PINNED = 4u << 20;
// Lays pieces out behind `off` in the pinned area at `base` (each as far from a 16-byte boundary as its source is) and launches
// the kernel that copies them there; at[i] receives their offsets.
cudaError_t gather(ccld_ctx* ctx, const Piece* piece, u32 n_pieces, char* base, size_t off, size_t* at) {
  GatherArgs A; u32 k = 0; size_t most = 0;
  for (u32 i = 0; i < n_pieces; ++i) {
    at[i] = (off + 15) / 16 * 16 + ((uintptr_t)piece[i].src & 15);
    off = at[i] + piece[i].n; most = std::max(most, piece[i].n);
    if (piece[i].n) { A.piece[k].src = (const unsigned char*)piece[i].src; A.piece[k].dst = (unsigned char*)base + at[i]; A.piece[k].n = piece[i].n; ++k; }
  }
  if (k) launch(ctx->stream, k_gather<1, GATHER_THREADS>, dim3((u32)std::min<size_t>((most + 16 * GATHER_THREADS - 1) / (16 * GATHER_THREADS), 32), k), GATHER_THREADS, 0, A);
  return cudaGetLastError();
}
size_t gather_room(const Piece* piece, u32 n_pieces) { size_t t = 0; for (u32 i = 0; i < n_pieces; ++i) t += piece[i].n + 32; return t; }

int fetch(ccld_ctx* ctx, const Piece* piece, u32 n_pieces) {
  size_t total = 0;
  for (u32 i = 0; i < n_pieces; ++i) total += piece[i].n;
  if (total > FETCH_PINNED || n_pieces > GATHER_PIECES) {
    for (u32 i = 0; i < n_pieces; ++i) if (piece[i].n) CK(cudaMemcpyAsync(piece[i].dst, piece[i].src, piece[i].n, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return CCLD_OK;
  }
  { int rc = pinned_area(ctx, ctx->h_io, gather_room(piece, n_pieces)); if (rc != CCLD_OK) return rc; }
  size_t at[GATHER_PIECES];
  char* base = (char*)ctx->h_io.p;
  CK(gather(ctx, piece, n_pieces, base, 0, at));
  CK(cudaStreamSynchronize(ctx->stream));
  for (u32 i = 0; i < n_pieces; ++i) if (piece[i].n) std::memcpy(piece[i].dst, base + at[i], piece[i].n);
  return CCLD_OK;
}

// A pinned block for the caller to keep, if it is not too large and not too much is out already.
constexpr size_t TAKE_MOST = 16u << 20;
int take_block(ccld_ctx* ctx, size_t bytes, ccld_host_block* blk) {
  blk->p = nullptr; blk->bytes = 0;
  if (bytes > TAKE_MOST) return fail(ctx, CCLD_ERR_CAPACITY, "too large for a pinned block");
  Block b = pinned_get(ctx, bytes);
  if (!b.p) return fail(ctx, CCLD_ERR_NOMEM, "pinned allocation failed");
  if (!BlockStore::get().lend(b.bytes)) { ctx->pinned_free.push_back(b); return fail(ctx, CCLD_ERR_CAPACITY, "too many pinned blocks in use"); }
  blk->p = b.p; blk->bytes = b.bytes;
  return CCLD_OK;
}

// Host columns on their way into one device block.
struct UpCol { size_t off; const void* src; size_t n; };
constexpr u32 UP_COLS = 13;                                // columns of a trace and of its frames
static_assert(UP_COLS <= GATHER_PIECES, "a piece per column");
int upload_slots(ccld_ctx* ctx) {
  if (ctx->h_up.p) return CCLD_OK;
  for (UploadSlot& u : ctx->up) if (!u.done) CK(cudaEventCreateWithFlags(&u.done, cudaEventDisableTiming));
  ctx->h_up = pinned_get(ctx, UP_PIECE * UP_SLOTS);
  if (!ctx->h_up.p) return fail(ctx, CCLD_ERR_NOMEM, "pinned allocation failed");
  for (u32 i = 0; i < UP_SLOTS; ++i) { ctx->up[i].p = (char*)ctx->h_up.p + i * UP_PIECE; ctx->up[i].used = false; }
  return CCLD_OK;
}
// The stream that the threads of a large upload copy on. A thread resolves the handle cudaStreamPerThread to its own stream, so
// for a context on that handle it is a stream of the context's: behind what the caller's stream holds when the upload begins,
// before what it gets once the upload is through.
struct UploadStream {
  ccld_ctx* ctx; cudaStream_t stream;
  explicit UploadStream(ccld_ctx* c) : ctx(c), stream(c->stream) {}
  cudaError_t open() {
    if (ctx->stream != cudaStreamPerThread) return cudaSuccess;
    cudaError_t e = ctx->up_event ? cudaSuccess : cudaEventCreateWithFlags(&ctx->up_event, cudaEventDisableTiming);
    if (e == cudaSuccess && !ctx->up_stream) e = cudaStreamCreateWithFlags(&ctx->up_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventRecord(ctx->up_event, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->up_stream, ctx->up_event, 0);
    if (e == cudaSuccess) stream = ctx->up_stream;
    return e;
  }
  cudaError_t close() {                                    // whatever became of the copies
    if (stream == ctx->stream) return cudaSuccess;
    const cudaError_t e = cudaEventRecord(ctx->up_event, stream);
    return e == cudaSuccess ? cudaStreamWaitEvent(ctx->stream, ctx->up_event, 0) : e;
  }
  static void drop(ccld_ctx* c) { if (c->up_event) cudaEventDestroy(c->up_event); if (c->up_stream) cudaStreamDestroy(c->up_stream); }
};

// The pageable columns of an upload. (Where they share a piece with others, those are copied behind it.)
int upload_pageable(ccld_ctx* ctx, char* base, size_t total, const UpCol* col, u32 n_cols) {
  cudaStream_t st = ctx->stream;
  { int rc = upload_slots(ctx); if (rc != CCLD_OK) return rc; }
  if (total <= UP_PIECE) {
    UploadSlot& u = ctx->up[ctx->up_next++ % UP_SLOTS];
    if (u.used) CK(cudaEventSynchronize(u.done));
    for (u32 i = 0; i < n_cols; ++i) std::memcpy(u.p + col[i].off, col[i].src, col[i].n);
    CK(cudaMemcpyAsync(base, u.p, total, cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(u.done, st));
    u.used = true;
    return CCLD_OK;
  }
  std::vector<UpCol> piece;
  for (u32 i = 0; i < n_cols; ++i)
    for (size_t a = 0; a < col[i].n; a += UP_PIECE) piece.push_back(UpCol{col[i].off + a, (const char*)col[i].src + a, std::min(UP_PIECE, col[i].n - a)});
  std::atomic<u32> next{0}; std::atomic<int> err{(int)cudaSuccess};
  const int device = ctx->device;
  UploadStream us(ctx);
  CK(us.open());
  st = us.stream;
  auto work = [&](u32 me) {
    if (cudaSetDevice(device) != cudaSuccess) { err = (int)cudaErrorInvalidDevice; return; }
    for (u32 turn = 0; err == (int)cudaSuccess; turn ^= 1) {
      const u32 k = next.fetch_add(1);
      if (k >= piece.size()) break;
      UploadSlot& u = ctx->up[2 * me + turn];
      cudaError_t e = u.used ? cudaEventSynchronize(u.done) : cudaSuccess;
      if (e == cudaSuccess) { std::memcpy(u.p, piece[k].src, piece[k].n); e = cudaMemcpyAsync(base + piece[k].off, u.p, piece[k].n, cudaMemcpyHostToDevice, st); }
      if (e == cudaSuccess) e = cudaEventRecord(u.done, st);
      u.used = true;
      if (e != cudaSuccess) err = (int)e;
    }
  };
  const u32 workers = std::max(1u, std::min({UP_WORKERS, (u32)(piece.size() / 4), std::thread::hardware_concurrency() / 2}));
  std::vector<std::thread> crew;
  for (u32 i = 1; i < workers; ++i) {
    try { crew.emplace_back(work, i); } catch (...) { break; }      // no more threads to be had: fewer do the work
  }
  work(0);
  for (auto& t : crew) t.join();
  CK(us.close());
  CK((cudaError_t)err.load());
  return CCLD_OK;
}

// Copies the columns to `base` (device, `total` bytes with the columns at their offsets). The driver copies pageable memory
// column by column through its own buffers, one thread, 10 us and more per call. A small upload is put together in one
// pinned piece instead and crosses in one copy; a large one is cut into pieces that several threads fill while earlier ones
// cross. Pageable columns are read by the time the call returns. Any other column is read when its turn in the stream comes, so
// that what earlier work of the stream still writes there is what arrives: large ones go straight across, the others are
// read by one kernel.
int upload_columns(ccld_ctx* ctx, char* base, size_t total, const UpCol* cols, u32 n_cols) {
  cudaStream_t st = ctx->stream;
  UpCol col[UP_COLS]; u32 n_page = 0;                      // the pageable columns
  UpCol far[UP_COLS]; u32 n_far = 0;                       // those that are copied one by one
  GatherArgs G; u32 n_near = 0;                            // those that a kernel reads
  for (u32 i = 0; i < n_cols; ++i) {
    if (!cols[i].n) continue;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, cols[i].src) != cudaSuccess) { cudaGetLastError(); at.type = cudaMemoryTypeUnregistered; }
    if (at.type == cudaMemoryTypeUnregistered) col[n_page++] = cols[i];
    else if (total <= UP_SMALL && at.type == cudaMemoryTypeHost && at.devicePointer && ((uintptr_t)at.devicePointer & 15) == 0) {
      auto& g = G.piece[n_near++];
      g.src = (const unsigned char*)at.devicePointer; g.dst = (unsigned char*)base + cols[i].off; g.n = cols[i].n;
    } else far[n_far++] = cols[i];
  }
  if (n_page) { int rc = upload_pageable(ctx, base, total, col, n_page); if (rc != CCLD_OK) return rc; }
  for (u32 i = 0; i < n_far; ++i) CK(cudaMemcpyAsync(base + far[i].off, far[i].src, far[i].n, cudaMemcpyHostToDevice, st));
  if (n_near) {
    launch(On(st, false), k_gather<UP_AHEAD, UP_THREADS>, dim3(1, n_near), UP_THREADS, 0, G);
    CK(cudaGetLastError());
  }
  return CCLD_OK;
}

// Space for `bytes` bytes of records in their slots, or null. A batch's kernels may still use it when the call that enqueued them has
// returned, and the next batch's come after them in the stream: so it is one block that only batches use and that is not handed to
// anything else of the context (an upload on another thread's cudaStreamPerThread is not behind those kernels). Batches do without
// it as well: it takes no more than half of the memory that is free, nothing cached is given up for it, and a shape that was
// refused does not ask again.
void* record_space(ccld_ctx* ctx, size_t bytes, ShapeEntry& shape) {
  Block& have = ctx->pool.records;
  if (have.bytes >= bytes) return have.p;
  if (shape.no_record_space) return nullptr;
  size_t free_bytes = 0, total = 0;
  bool ok = cudaMemGetInfo(&free_bytes, &total) == cudaSuccess && bytes <= (free_bytes + have.bytes) / 2;
  if (ok) {
    if (have.p) cudaFree(have.p);                          // waits for the device
    have = Block{};
    if (!BlockStore::get().take(ctx->device, bytes, &have)) {
      ok = cudaMalloc(&have.p, align_up(bytes)) == cudaSuccess;
      if (ok) have.bytes = align_up(bytes); else have.p = nullptr;
    }
  }
  if (!ok) { cudaGetLastError(); shape.no_record_space = true; }
  return have.bytes >= bytes ? have.p : nullptr;
}

// Whether a batch that is through found another layout than it was sized for.
bool surprised(const PendingBatch& b) {
  for (u32 k = 0; k < b.n; ++k) if (b.h_tot()[(size_t)k * T_COUNT + T_FAILED] == FAILED_EXPECT) return true;
  return false;
}

// Takes over the order that a batch's records were in, for the next one of its shape.
void learn_order(ccld_ctx* ctx, const PendingBatch& b) {
  u64 mixed = 0, all = 0;
  for (u32 k = 0; k < b.n; ++k) { auto it = ctx->windows.find(b.first + k); if (it != ctx->windows.end()) { mixed += b.h_tot()[(size_t)k * T_COUNT + T_MIXED]; all += it->second.n_rec; } }
  if (mostly_mixed(mixed, all) == b.mixed) return;
  for (ShapeEntry& s : ctx->shapes) {
    bool same = s.n_rec.size() == b.n;
    for (u32 k = 0; k < b.n && same; ++k) { auto it = ctx->windows.find(b.first + k); same = it != ctx->windows.end() && it->second.n_rec == s.n_rec[k]; }
    for (u32 k = 0; k < b.n && same; ++k) s.totals[(size_t)k * T_COUNT + T_MIXED] = b.h_tot()[(size_t)k * T_COUNT + T_MIXED];
  }
}

// Brings the batches that were enqueued on expected totals to a definite state: waits for the stream, reads the totals
// their plans really found, and analyses again - this time waiting for the plan - every batch from the first one whose
// expectation failed (that batch and all later ones gave up on the device without touching any state, so the order of
// the windows is kept). Every call that hands out results or changes state goes through here first.
int settle(ccld_ctx* ctx) {
  if (ctx->pending.empty()) return CCLD_OK;
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  std::vector<PendingBatch> todo;
  for (PendingBatch& b : ctx->pending) { if (b.speculative) todo.push_back(b); else ctx->pinned_free.push_back(b.pin); }
  ctx->pending.clear();
  bool failed = false;
  int rc = CCLD_OK;
  for (PendingBatch& b : todo) {
    failed = failed || surprised(b);
    ctx->pinned_free.push_back(b.pin);
    if (!failed) {
      learn_order(ctx, b);
      // a window may still have been refused for its size, which the expectation cannot have foreseen: keep what the plan found,
      // which is then no groups and no slots
      for (u32 k = 0; k < b.n; ++k) {
        auto it = ctx->windows.find(b.first + k);
        if (it == ctx->windows.end() || !it->second.analysed) continue;
        WindowHost& w = it->second;
        std::memcpy(w.totals, b.h_tot() + (size_t)k * T_COUNT, sizeof w.totals);
        w.d.n_groups = w.totals[T_GROUPS]; w.d.n_slots = w.totals[T_SLOTS];
      }
      continue;
    }
  }
  if (!failed) return CCLD_OK;
  CK(cudaMemsetAsync(ctx->d_poison, 0, 4, ctx->stream));
  failed = false;
  for (PendingBatch& b : todo) {
    failed = failed || surprised(b);
    if (!failed) continue;
    bool present = true;
    for (u32 k = 0; k < b.n; ++k) {
      auto it = ctx->windows.find(b.first + k);
      if (it == ctx->windows.end()) { present = false; continue; }
      drop_results(it->second);
    }
    ++ctx->batches_redone;
    if (!present) continue;                                // released in the meantime: nothing to analyse
    const int r = analyze_batch(ctx, b.first, b.n, b.now, false);
    if (r != CCLD_OK && rc == CCLD_OK) rc = r;
  }
  return rc;
}

int find_analysed(ccld_ctx* ctx, u32 wid, WindowHost** out) {
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  auto it = ctx->windows.find(wid);
  if (it == ctx->windows.end()) return fail(ctx, CCLD_ERR_NO_WINDOW, "unknown window id");
  if (!it->second.analysed) return fail(ctx, CCLD_ERR_NO_WINDOW, "window not analysed");
  *out = &it->second;
  return CCLD_OK;
}

}  // namespace

extern "C" {

void ccld_params_default(ccld_params* p) {
  if (!p) return;
  p->tbase_init_ns = 2000000; p->theta_slow_milli = 3000; p->alpha_milli = 400; p->beta_milli = 600;
  p->m_max_rounds = 100; p->m_max_ns = 120000000000ll; p->hang_ns = 300000000000ll; p->barrier_bytes = 4;
  p->slow_rep_threshold = 1; p->k_milli = 5189; p->min_group = 4; p->vote_rep_milli = 100;
}

int ccld_create(ccld_ctx** out, const ccld_params* params, int device, void* cuda_stream) {
  if (!out || !params) return CCLD_ERR_ARG;
  *out = nullptr;
  if (params->tbase_init_ns <= 0 || params->m_max_rounds == 0 || params->m_max_ns <= 0 || params->min_group == 0) return CCLD_ERR_ARG;
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device < 0 || device >= n_dev) return CCLD_ERR_CUDA;
  if (cudaSetDevice(device) != cudaSuccess) return CCLD_ERR_CUDA;
  ccld_ctx* ctx = new (std::nothrow) ccld_ctx();
  if (!ctx) return CCLD_ERR_NOMEM;
  ctx->params = *params; ctx->device = device; ctx->pool.device = device; ctx->stream = (cudaStream_t)cuda_stream;
  BlockStore::get().enter();
  { int sms = 0; if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) == cudaSuccess && sms > 0) ctx->n_sms = (u32)sms; }
  Params& d = ctx->dp;
  d.tbase_init_ns = params->tbase_init_ns; d.m_max_ns = params->m_max_ns; d.hang_ns = params->hang_ns; d.barrier_bytes = params->barrier_bytes;
  d.theta_slow_milli = params->theta_slow_milli; d.alpha_milli = params->alpha_milli; d.beta_milli = params->beta_milli;
  d.m_max_rounds = params->m_max_rounds; d.slow_rep_threshold = params->slow_rep_threshold; d.k_milli = params->k_milli;
  d.min_group = params->min_group; d.vote_rep_milli = params->vote_rep_milli;
  *out = ctx;
  return CCLD_OK;
}

int ccld_destroy(ccld_ctx* ctx) {
  if (!ctx) return CCLD_ERR_ARG;
  cudaSetDevice(ctx->device);
  if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) { cudaGetLastError(); cudaDeviceSynchronize(); }      // (the caller's stream may be gone)
  for (auto& kv : ctx->windows) { drop_results(kv.second); if (kv.second.owns) ctx->pool.put(kv.second.own); if (kv.second.owns_opset) ctx->pool.put(kv.second.opset_own); }
  ctx->windows.clear();
  ctx->pool.put(ctx->reg_blk); ctx->pool.put(ctx->misc_blk);
  ctx->pool.leave_all();
  for (auto& b : ctx->pending) ctx->pinned_free.push_back(b.pin);
  ctx->pinned_free.push_back(ctx->h_verdict); ctx->pinned_free.push_back(ctx->h_io); ctx->pinned_free.push_back(ctx->h_up);
  for (UploadSlot& u : ctx->up) if (u.done) cudaEventDestroy(u.done);
  Chains::drop(ctx); UploadStream::drop(ctx);
  for (auto& f : ctx->pinned_free) BlockStore::get().put(-1, f);
  BlockStore::get().leave();
  for (auto& sl : ctx->ring) for (int i = 0; i < TIMER_PAIRS; ++i) { cudaEventDestroy(sl.a[i]); cudaEventDestroy(sl.b[i]); }
  delete ctx;
  return CCLD_OK;
}

const char* ccld_last_error(ccld_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

int ccld_comm_register(ccld_ctx* ctx, uint32_t comm, const uint32_t* ranks, uint32_t n, uint8_t algo, uint32_t seq0) try {
  if (!ctx) return CCLD_ERR_ARG;
  if (ctx->finalized) return fail(ctx, CCLD_ERR_STATE, "communicators must be registered before the first analysis");
  if (!ranks || n == 0) return fail(ctx, CCLD_ERR_ARG, "empty communicator");
  if (algo > 1) return fail(ctx, CCLD_ERR_ARG, "algo must be 0 (ring) or 1 (tree)");
  if (n > CCLD_MAX_COMM_SIZE) return fail(ctx, CCLD_ERR_CAPACITY, "communicator larger than CCLD_MAX_COMM_SIZE");
  if (ctx->comm_idx.count(comm)) return fail(ctx, CCLD_ERR_ARG, "communicator id registered twice");
  CommHost c; c.id = comm; c.seq0 = seq0; c.algo = algo; c.ranks.assign(ranks, ranks + n);
  std::vector<u32> sorted(c.ranks); std::sort(sorted.begin(), sorted.end());
  if (std::adjacent_find(sorted.begin(), sorted.end()) != sorted.end()) return fail(ctx, CCLD_ERR_ARG, "rank listed twice in a communicator");
  if (sorted.back() >= CCLD_MAX_RANK_ID) return fail(ctx, CCLD_ERR_CAPACITY, "rank id not below CCLD_MAX_RANK_ID");
  const auto at = ctx->comm_idx.emplace(comm, (u32)ctx->comms.size()).first;
  try { ctx->comms.push_back(std::move(c)); } catch (...) { ctx->comm_idx.erase(at); throw; }
  return CCLD_OK;
} CAUGHT

int ccld_comm_set_layers(ccld_ctx* ctx, uint32_t comm, const uint32_t* layer) try {
  if (!ctx) return CCLD_ERR_ARG;
  if (ctx->finalized) return fail(ctx, CCLD_ERR_STATE, "layers must be set before the first analysis");
  if (!layer) return fail(ctx, CCLD_ERR_ARG, "layer is null");
  auto ci = ctx->comm_idx.find(comm);
  if (ci == ctx->comm_idx.end()) return fail(ctx, CCLD_ERR_UNKNOWN_COMM, "unknown communicator");
  CommHost& c = ctx->comms[ci->second];
  if (c.algo != 1) return fail(ctx, CCLD_ERR_ARG, "layers belong to tree communicators (algo 1)");
  const u32 n = (u32)c.ranks.size();
  std::unordered_map<u32, u32> first;       // layer id -> lowest position that carries it
  c.head.resize(n);
  for (u32 p = 0; p < n; ++p) c.head[p] = first.emplace(layer[p], p).first->second;
  return CCLD_OK;
} CAUGHT

int ccld_trace_upload(ccld_ctx* ctx, uint32_t window_id, uint64_t n_rec, int mem_kind,
                      const uint32_t* rank, const uint32_t* comm, const uint32_t* seq, const uint8_t* op,
                      const uint64_t* bytes, const int64_t* t_enter_ns, const int64_t* t_exit_ns,
                      const uint32_t* send_chg, const uint32_t* recv_chg,
                      uint32_t n_frames, const uint32_t* f_rank, const uint32_t* f_comm, const uint32_t* f_seq,
                      uint32_t n_channels, const uint32_t* progress) try {
  NvtxRange nvtx_range("ccld_trace_upload");
  if (!ctx) return CCLD_ERR_ARG;
  if (mem_kind != 0 && mem_kind != 1) return fail(ctx, CCLD_ERR_ARG, "mem_kind must be 0 (host) or 1 (device)");
  if (n_rec >= 0xFFFFFFFFull) return fail(ctx, CCLD_ERR_CAPACITY, "window of 2^32 - 1 or more records");
  if (n_rec > 0 && (!rank || !comm || !seq || !op || !bytes || !t_enter_ns || !t_exit_ns)) return fail(ctx, CCLD_ERR_ARG, "null column");
  if ((send_chg == nullptr) != (recv_chg == nullptr)) return fail(ctx, CCLD_ERR_ARG, "send_chg and recv_chg must both be given or both be null");
  if (n_frames > 0 && (!f_rank || !f_comm || !f_seq || !progress || n_channels == 0)) return fail(ctx, CCLD_ERR_ARG, "incomplete progress frames");
  if (ctx->windows.count(window_id)) return fail(ctx, CCLD_ERR_STATE, "window id already uploaded");
  CK(cudaSetDevice(ctx->device));
  WindowHost w; w.id = window_id; w.n_rec = n_rec; w.n_frames = n_frames; w.n_channels = n_channels;
  WinDesc& d = w.d;
  d.n_rec = n_rec;
  if (mem_kind == 1) {
    d.rank = rank; d.comm = comm; d.seq = seq; d.op = op; d.bytes = bytes; d.t_enter = t_enter_ns; d.t_exit = t_exit_ns;
    d.send_chg = send_chg; d.recv_chg = recv_chg;
    w.f_rank = f_rank; w.f_comm = f_comm; w.f_seq = f_seq; w.progress = progress;
  } else {
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
    const size_t o_rank = take(n_rec * 4), o_comm = take(n_rec * 4), o_seq = take(n_rec * 4), o_op = take(n_rec), o_bytes = take(n_rec * 8),
                 o_te = take(n_rec * 8), o_tx = take(n_rec * 8), o_sc = take(send_chg ? n_rec * 4 : 0), o_rc = take(recv_chg ? n_rec * 4 : 0),
                 o_fr = take(n_frames * 4ull), o_fc = take(n_frames * 4ull), o_fs = take(n_frames * 4ull), o_pr = take((size_t)n_frames * n_channels * 8);
    cudaError_t e;
    w.own = ctx->pool.get(off, &e);
    if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "window allocation failed");
    w.owns = true;
    char* b = (char*)w.own.p;
    const size_t chg = send_chg ? n_rec * 4 : 0, fr = n_frames * 4ull;
    const UpCol col[] = {{o_rank, rank, n_rec * 4}, {o_comm, comm, n_rec * 4}, {o_seq, seq, n_rec * 4}, {o_op, op, n_rec}, {o_bytes, bytes, n_rec * 8},
                         {o_te, t_enter_ns, n_rec * 8}, {o_tx, t_exit_ns, n_rec * 8}, {o_sc, send_chg, chg}, {o_rc, recv_chg, chg},
                         {o_fr, f_rank, fr}, {o_fc, f_comm, fr}, {o_fs, f_seq, fr}, {o_pr, progress, (size_t)n_frames * n_channels * 8}};
    static_assert(sizeof col / sizeof col[0] == UP_COLS, "all of them");
    { int rc; try { rc = upload_columns(ctx, b, off, col, sizeof col / sizeof col[0]); } catch (...) { rc = caught(ctx); } if (rc != CCLD_OK) { cudaStreamSynchronize(ctx->stream); ctx->pool.put(w.own); return rc; } }
    d.rank = (const u32*)(b + o_rank); d.comm = (const u32*)(b + o_comm); d.seq = (const u32*)(b + o_seq); d.op = (const u8*)(b + o_op);
    d.bytes = (const u64*)(b + o_bytes); d.t_enter = (const i64*)(b + o_te); d.t_exit = (const i64*)(b + o_tx);
    d.send_chg = send_chg ? (const u32*)(b + o_sc) : nullptr; d.recv_chg = recv_chg ? (const u32*)(b + o_rc) : nullptr;
    if (n_frames) { w.f_rank = (const u32*)(b + o_fr); w.f_comm = (const u32*)(b + o_fc); w.f_seq = (const u32*)(b + o_fs); w.progress = (const u32*)(b + o_pr); }
  }
  ctx->windows.emplace(window_id, std::move(w));
  return CCLD_OK;
} CAUGHT

int ccld_window_release(ccld_ctx* ctx, uint32_t window_id) try {
  if (!ctx) return CCLD_ERR_ARG;
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  auto it = ctx->windows.find(window_id);
  if (it == ctx->windows.end()) return fail(ctx, CCLD_ERR_NO_WINDOW, "unknown window id");
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));     // nothing in flight may still read the blocks we recycle
  drop_results(it->second);
  if (it->second.owns) ctx->pool.put(it->second.own);
  if (it->second.owns_opset) ctx->pool.put(it->second.opset_own);
  ctx->windows.erase(it);
  return CCLD_OK;
} CAUGHT

int ccld_reset(ccld_ctx* ctx) try {
  if (!ctx) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  // batches still in doubt need no second analysis: their results are dropped with all the others
  bool failed = false;
  for (auto& b : ctx->pending) {
    failed = failed || (b.speculative && surprised(b));
    if (b.speculative && !failed) learn_order(ctx, b);
    ctx->pinned_free.push_back(b.pin);
  }
  ctx->pending.clear();
  for (auto& kv : ctx->windows) drop_results(kv.second);
  if (ctx->finalized) {
    char* const from = (char*)ctx->reg_blk.p + ctx->stats_off;          // the statistics and, behind them, the flag
    CK(cudaMemsetAsync(from, 0, (char*)(ctx->d_poison + 1) - from, ctx->stream));
  }
  return CCLD_OK;
} CAUGHT

int ccld_analyze_window(ccld_ctx* ctx, uint32_t first_window, uint32_t n_windows, int64_t now_ns) try {
  NvtxRange nvtx_range("ccld_analyze_window");
  if (!ctx) return CCLD_ERR_ARG;
  if (n_windows == 0) return fail(ctx, CCLD_ERR_ARG, "n_windows is zero");
  if (n_windows > 65535) return fail(ctx, CCLD_ERR_CAPACITY, "more than 65,535 windows in one batch");
  return analyze_batch(ctx, first_window, n_windows, now_ns, ctx->speculate != 0);
} CAUGHT

int ccld_set_speculation(ccld_ctx* ctx, int on) try {
  if (!ctx) return CCLD_ERR_ARG;
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  ctx->speculate = on != 0;
  return CCLD_OK;
} CAUGHT

}  // extern "C"

namespace {

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) != cudaSuccess) { cudaGetLastError(); return true; }
  return s != cudaStreamCaptureStatusNone;
}

int analyze_batch(ccld_ctx* ctx, u32 first_window, u32 n_windows, i64 now_ns, bool may_speculate) {
  CK(cudaSetDevice(ctx->device));
  std::vector<WindowHost*> ws(n_windows);
  for (u32 k = 0; k < n_windows; ++k) {
    auto it = ctx->windows.find(first_window + k);
    if (it == ctx->windows.end()) return fail(ctx, CCLD_ERR_NO_WINDOW, "window not uploaded");
    if (it->second.analysed) return fail(ctx, CCLD_ERR_STATE, "window already analysed");
    ws[k] = &it->second;
  }
  { int rc = finalize_registry(ctx); if (rc != CCLD_OK) return rc; }
  const u32 B = n_windows, nc = ctx->reg.n_comms;
  cudaStream_t st = ctx->stream;

  // A batch of a shape seen before (the same record count in every window) is enqueued without waiting for its plan:
  // the results are sized from the totals that shape had last time, and the plan checks them on the device.
  ShapeEntry* expect = nullptr;
  if (may_speculate) {
    for (ShapeEntry& e : ctx->shapes) {
      if (e.n_rec.size() != B) continue;
      bool same = true;
      for (u32 k = 0; k < B && same; ++k) same = e.n_rec[k] == ws[k]->n_rec;
      if (same) { expect = &e; break; }
    }
  }
  if (!expect) { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }    // the waiting path runs with nothing in doubt before it

  // ---- plan block: descriptors, op-counter ranges, layout rows, totals, counters ----
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
  const size_t tot_bytes = (size_t)B * T_COUNT * 8;
  const size_t o_desc = take(B * sizeof(WinDesc)), o_exp = take(expect ? tot_bytes : 0), up_bytes = off,      // what comes from the host
               o_zero = off, o_rmax = take((size_t)B * nc * 4), o_cnt = take((size_t)B * C_COUNT * 8), o_defn = take(16), o_zero_end = off,
               o_rmin = take((size_t)B * nc * 4), o_rng = take((size_t)B * nc * sizeof(RangeRow)), o_srow = take((size_t)B * nc * sizeof(uint4)),
               o_tot = take(tot_bytes), o_chunk = take((size_t)B * (CHUNK_MAX + 1) * sizeof(uint2));
  cudaError_t e;
  Block pb = ctx->pool.get(off, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "plan allocation failed");
  auto plan_blk = std::make_shared<Shared>(&ctx->pool, pb);
  char* pbase = (char*)pb.p;
  // pinned: the totals the layout finds, then the descriptors and expected totals on their way to the device. It belongs to
  // the batch until the next call that synchronizes.
  PendingBatch pbatch; pbatch.first = first_window; pbatch.n = B; pbatch.now = now_ns; pbatch.speculative = expect != nullptr;
  pbatch.pin = pinned_get(ctx, align_up(tot_bytes) + up_bytes);
  if (!pbatch.pin.p) return fail(ctx, CCLD_ERR_NOMEM, "pinned allocation failed");
  struct Guard {                                           // whatever way the call ends, the batch's pinned block is accounted for
    ccld_ctx* ctx; PendingBatch& b; bool queued = false;
    ~Guard() { if (!queued) { cudaStreamSynchronize(ctx->stream); ctx->pinned_free.push_back(b.pin); } }
  } guard{ctx, pbatch};
  char* const h_up = (char*)pbatch.pin.p + align_up(tot_bytes);
  WinDesc* const hd = (WinDesc*)h_up;
  u64 cta = 0;
  for (u32 k = 0; k < B; ++k) {
    WinDesc d = ws[k]->d;
    d.slot_cap = 2 * d.n_rec + ctx->sum_n;
    cta = std::max<u64>(cta, (d.n_rec + REC_PER_CTA - 1) / REC_PER_CTA);
    d.rmin = (u32*)(pbase + o_rmin) + (size_t)k * nc; d.rmax = (u32*)(pbase + o_rmax) + (size_t)k * nc;
    d.ranges = (RangeRow*)(pbase + o_rng) + (size_t)k * nc; d.srow = (uint4*)(pbase + o_srow) + (size_t)k * nc;
    d.totals = (u64*)(pbase + o_tot) + (size_t)k * T_COUNT; d.counters = (u64*)(pbase + o_cnt) + (size_t)k * C_COUNT;
    d.chunks = (uint2*)(pbase + o_chunk) + (size_t)k * (CHUNK_MAX + 1); d.totals_host = (u64*)pbatch.pin.p + (size_t)k * T_COUNT;
    d.expect = expect ? (const u64*)(pbase + o_exp) + (size_t)k * T_COUNT : nullptr; d.poison = ctx->d_poison;
    d.n_groups = d.n_slots = 0; d.perm = nullptr; d.flags = nullptr; d.gi64 = nullptr; d.gu32 = nullptr; d.gbw = nullptr;
    d.comm_rows = nullptr; d.alerts = nullptr; d.packed = nullptr;
    for (int q = 0; q < B_COUNT; ++q) d.base[q] = 0;
    d.pad = 0; d.tsum[0] = d.tsum[1] = d.tsum[2] = nullptr;
    hd[k] = d;
  }
  if (expect) std::memcpy(h_up + o_exp, expect->totals.data(), tot_bytes);
  if (cta > 0x7FFFFFFFull) return fail(ctx, CCLD_ERR_CAPACITY, "batch too large for one launch");
  WinDesc* d_desc = (WinDesc*)(pbase + o_desc);
  TimerSlot* ts = timer_begin(ctx);
  const u32 layout_threads = nc <= 128 ? 128 : (nc <= 256 ? 256 : (nc <= 512 ? 512 : LAYOUT_THREADS));
  auto start_plan = [&](bool fill, u32 fill_ctas) -> cudaError_t {        // uploads the descriptors, sets the start values, runs the range pass and the layout
    BeginArgs ba;
    ba.desc_host = (const u32*)h_up; ba.desc = (u32*)(pbase + o_desc); ba.desc_words = up_bytes / 4;
    ba.rmin = (u32*)(pbase + o_rmin); ba.n_rmin = (u64)B * nc; ba.zero = (u32*)(pbase + o_zero); ba.n_zero = (o_zero_end - o_zero) / 4;
    const u64 most = std::max<u64>(std::max<u64>(ba.desc_words, ba.n_rmin), ba.n_zero);
    { TimedLaunch tl(ts, 1, st); launch(st, k_begin, (u32)std::min<u64>((most + BEGIN_THREADS - 1) / BEGIN_THREADS, 2ull * ctx->n_sms), BEGIN_THREADS, 0, ba); }
    if (cta > 0) {
      // enough CTAs to fill the device several times over, then as many blocks per CTA as that leaves
      const u64 want = 32ull * ctx->n_sms;
      const u32 per = (u32)std::min<u64>(RANGE_BLOCKS_MAX, std::max<u64>(1, cta * B / want));
      TimedLaunch tl(ts, 0, st);
      launch(st, k_seq_range, dim3((u32)((cta + per - 1) / per), B), REC_THREADS, range_smem_bytes(nc), d_desc, ctx->reg, per, fill);
    }
    { TimedLaunch tl(ts, 1, st); launch(st, k_layout, dim3(1 + fill_ctas, B), layout_threads, 0, d_desc, ctx->reg, ctx->n_sms * CCLD_FUSED_MIN_CTAS * (SMALL_SEQS / 32)); }
    return cudaGetLastError();
  };
  const u64* tot = nullptr;                                // [B][T_COUNT] totals the results are sized from
  std::vector<u64> found;
  if (!expect) {
    CK(start_plan(false, 0));
    CK(cudaStreamSynchronize(st));
    found.assign(pbatch.h_tot(), pbatch.h_tot() + (size_t)B * T_COUNT);
    tot = found.data();
  } else tot = expect->totals.data();

  // ---- result block: sized from the totals ----
  off = 0;
  u64 total_slots = 0, max_slots = 0, n_list[B_COUNT] = {0, 0, 0, 0, 0};       // batch-wide list lengths (B_*)
  u32 chunk_ctas = 1;
  const int t_of[B_COUNT] = {T_FCTA, T_FWT, T_FSUM, T_TILES2, T_TILES3};
  for (u32 k = 0; k < B; ++k) { const u64* t = tot + (size_t)k * T_COUNT; total_slots += t[T_SLOTS]; max_slots = std::max(max_slots, t[T_SLOTS]); chunk_ctas = std::max(chunk_ctas, (u32)t[T_CHUNKS]); }
  const size_t o_perm = take(total_slots * 4 + ALIGN);
  std::vector<size_t> o_flags(B), o_gi(B), o_gu(B), o_gb(B), o_rows(B), o_al(B), perm_off(B);
  { size_t po = 0;
    for (u32 k = 0; k < B; ++k) {
      const u64* t = tot + (size_t)k * T_COUNT;
      perm_off[k] = po; po += t[T_SLOTS] * 4;
      o_flags[k] = take(t[T_SLOTS]); o_gi[k] = take(t[T_GROUPS] * 8 * GI_COUNT); o_gu[k] = take(t[T_GROUPS] * 4 * GU_COUNT);
      o_gb[k] = take(t[T_GROUPS] * 8); o_rows[k] = take(t[T_ROWS] * sizeof(ccld_comm_verdict));
      o_al[k] = take(CCLD_MAX_ALERTS_PER_WINDOW * sizeof(ccld_hang_alert));
      for (int q = 0; q < B_COUNT; ++q) { hd[k].base[q] = (u32)n_list[q]; n_list[q] += t[t_of[q]]; }
    } }
  for (int q = 0; q < B_COUNT; ++q) if (n_list[q] > 0x7FFFFFFFull) return fail(ctx, CCLD_ERR_CAPACITY, "too many tiles in one batch");
  const size_t o_fcta = take(n_list[B_FCTA] * sizeof(FusedCta)), o_fwt = take(n_list[B_FWT] * sizeof(WarpTile)),
               o_fsum = take(n_list[B_FSUM] * sizeof(TileSum)), o_t2 = take(n_list[B_T2] * sizeof(Tile)), o_s2 = take(n_list[B_T2] * sizeof(TileSum)),
               o_t3 = take(n_list[B_T3] * sizeof(Tile)), o_s3 = take(n_list[B_T3] * sizeof(TileSum));
  // groups the fused kernel may set aside for the deferred kernel: at most every group of the batch
  u64 total_groups = 0;
  for (u32 k = 0; k < B; ++k) total_groups += tot[(size_t)k * T_COUNT + T_GROUPS];
  const size_t o_def = take(n_list[B_FCTA] ? total_groups * 8 : 0),
               o_def3 = take((n_list[B_T2] + n_list[B_T3]) * (size_t)LARGE_SEQS * 8);          // likewise for the kernels of larger communicators
  Block rb = ctx->pool.get(off, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "result allocation failed");
  auto res_blk = std::make_shared<Shared>(&ctx->pool, rb);
  char* rbase = (char*)rb.p;
  // Records in another order than their ranks' (as this shape had them last; both ways are right whatever the order): the fused
  // kernel's records go to their slots. Where the space is not to be had, and in a graph, whose launches would share it, the kernel gathers.
  // From half of the slots on, because the larger communicators' kernels read through the table anyway (4.1 M records, groups of 8 with a tenth of the
  // slots beside rings of 256: 399 us for the batch with and 350 without; half 344 and 372, three quarters 289 and 299; groups of 4 with a quarter beside
  // rings of 172 364 and 338, half 353 and 334), and not for records in their ranks' order (nine communicators in turn per rank: 297 and 271).
  void* records = nullptr;
  if (expect) {
    u64 mixed = 0, all = 0, fused = 0;
    for (u32 k = 0; k < B; ++k) { const u64* t = tot + (size_t)k * T_COUNT; mixed += t[T_MIXED]; fused += t[T_FUSED]; all += ws[k]->n_rec; }
    pbatch.mixed = mostly_mixed(mixed, all);
    if (pbatch.mixed && n_list[B_FCTA] && fused * 32 * 2 >= total_slots && total_slots * sizeof(PackedRecord) <= PACK_MOST && !capturing(st))
      records = record_space(ctx, total_slots * sizeof(PackedRecord), *expect);
  }
  const bool pack = records != nullptr;
  if (pack) ++ctx->packed;
  for (u32 k = 0; k < B; ++k) {
    const u64* t = tot + (size_t)k * T_COUNT;
    WinDesc& d = hd[k];
    d.n_groups = t[T_GROUPS]; d.n_slots = t[T_SLOTS];
    if (pack) d.packed = (uint4*)records + perm_off[k] / 2;                // 32 bytes where perm has 4
    d.perm = (u32*)(rbase + o_perm + perm_off[k]); d.flags = (u8*)(rbase + o_flags[k]);
    d.gi64 = (i64*)(rbase + o_gi[k]); d.gu32 = (u32*)(rbase + o_gu[k]); d.gbw = (double*)(rbase + o_gb[k]);
    d.comm_rows = (ccld_comm_verdict*)(rbase + o_rows[k]); d.alerts = (ccld_hang_alert*)(rbase + o_al[k]);
    d.tsum[0] = (TileSum*)(rbase + o_fsum) + d.base[B_FSUM]; d.tsum[1] = (TileSum*)(rbase + o_s2) + d.base[B_T2]; d.tsum[2] = (TileSum*)(rbase + o_s3) + d.base[B_T3];
  }
  if (expect) {
    // Descriptors already complete: nothing was waited for. What fills in the time of the layout's one CTA per window is filled
    // beside it, two CTAs per SM together; a larger table under the range pass, which has issue slots and not memory for
    // its limit (twelve windows of 4,096 ranks, 49 M slots: 141 us for both kernels instead of 151; one window of 16.4 M: 70 instead of 65).
    const bool under_range = cta > 0 && total_slots > FILL_BESIDE;
    ++ctx->unwaited; if (under_range) ++ctx->filled_under_range;
    const u64 want = (max_slots + 16ull * layout_threads - 1) / (16ull * layout_threads);
    CK(start_plan(under_range, under_range ? 0u : (u32)std::max<u64>(1, std::min<u64>(want, 2ull * (LAYOUT_THREADS / layout_threads) * ctx->n_sms / B))));
  } else {
    CK(cudaMemcpyAsync(d_desc, hd, B * sizeof(WinDesc), cudaMemcpyHostToDevice, st));
    if (total_slots) CK(cudaMemsetAsync(rbase + o_perm, 0xFF, total_slots * 4, st));
  }
  PlanLists pl; pl.fcta = (FusedCta*)(rbase + o_fcta); pl.fwt = (WarpTile*)(rbase + o_fwt); pl.t2 = (Tile*)(rbase + o_t2); pl.t3 = (Tile*)(rbase + o_t3);
  {
    // the CTAs that write the work lists come first in the scatter's launch
    const u32 comm_blocks = (nc + EMIT_THREADS - 1) / EMIT_THREADS, per_slice = (comm_blocks + EMIT_SLICES - 1) / EMIT_SLICES,
              slices = (comm_blocks + per_slice - 1) / per_slice, emit_ctas = chunk_ctas * slices;
    const u64 blocks = (cta * REC_PER_CTA + SCAT_PER_CTA - 1) / SCAT_PER_CTA;      // of the largest window
    // Two blocks per CTA as soon as that leaves each SM eight: a CTA's first block waits for the chain to its ranks' rows, the next
    // one does not (two windows of one communicator of 4,096: 38.2 us with one, 35.3 with two, 37.6 with four; 1,088 communicators
    // of 8 and 100: 41.9, 38.3, 41.6; 16,384 ranks: 68.1, 68.6, 74.9).
    const u32 per = (u32)std::min<u64>(SCAT_BLOCKS_MAX, std::max<u64>(1, blocks * B / (8ull * ctx->n_sms)));
    TimedLaunch tl(ts, 2, st);
    if (pack) launch(st, k_slot_pack, dim3(emit_ctas + (u32)((cta * REC_PER_CTA + PACK_PER_CTA - 1) / PACK_PER_CTA), B), SCAT_THREADS, 0, d_desc, ctx->reg, pl, emit_ctas, slices, per_slice);
    else launch(st, k_slot_scatter, dim3(emit_ctas + (u32)((blocks + per - 1) / per), B), SCAT_THREADS, 0, d_desc, ctx->reg, pl, emit_ctas, slices, per_slice, per);
  }
  const DeferList dl_big{(u64*)(rbase + o_def3), (u32*)(pbase + o_defn) + 2};
  static_assert(MID_SEQS == LARGE_SEQS, "one list for the groups of both classes");
  Chains chains(ctx, (n_list[B_FCTA] ? 1 : 0) + (n_list[B_T2] ? 1 : 0) + (n_list[B_T3] ? 1 : 0), ts != nullptr);
  auto deferred_big = [&](On on) {
    u32 n = 0;
    for (int q = 0; q < 3; ++q) n = std::max(n, std::max(ctx->max_mid_n[q], ctx->max_large_n[q]));
    launch(on, k_reduce_large_deferred, LARGE_DEF_GRID, LARGE_DEF_THREADS, 16ull * n, d_desc, dl_big, ctx->reg, ctx->dp, now_ns);
  };
  if (n_list[B_T2]) {
    On on = chains.open(0);
    TimedLaunch tl(ts, 4, st);
    const u32 grid = (u32)n_list[B_T2]; TileSum* sums = (TileSum*)(rbase + o_s2);
    // one launch per padded size the registry has; a tile of another size ends at once
    const u32* m = ctx->max_mid_n;
    if (m[0]) launch(on, k_reduce_mid<8>, grid, MID_THREADS, mid_smem_bytes(m[0]), d_desc, pl.t2, sums, ctx->reg, ctx->dp, dl_big);
    if (m[1]) launch(on, k_reduce_mid<16>, grid, MID_THREADS, mid_smem_bytes(m[1]), d_desc, pl.t2, sums, ctx->reg, ctx->dp, dl_big);
    if (m[2]) launch(on, k_reduce_mid<32>, grid, MID_THREADS, mid_smem_bytes(m[2]), d_desc, pl.t2, sums, ctx->reg, ctx->dp, dl_big);
    if (chains.n <= 0 && !n_list[B_T3]) deferred_big(on);
  }
  if (n_list[B_T3]) {
    On on = chains.open(n_list[B_T2] ? 1 : 0);
    TimedLaunch tl(ts, 5, st);
    const u32 grid = (u32)(n_list[B_T3] * LARGE_SEQS); TileSum* sums = (TileSum*)(rbase + o_s3);
    const u32* m = ctx->max_large_n;
    if (m[0]) launch_cluster(on, k_reduce_large<4>, LARGE_SEQS, grid, LQ_THREADS, LargeTile<4>::BYTES, d_desc, pl.t3, sums, ctx->reg, ctx->dp, dl_big);
    if (m[1]) launch_cluster(on, k_reduce_large<8>, LARGE_SEQS, grid, LQ_THREADS, LargeTile<8>::BYTES, d_desc, pl.t3, sums, ctx->reg, ctx->dp, dl_big);
    if (m[2]) launch_cluster(on, k_reduce_large<16>, LARGE_SEQS, grid, LQ_THREADS, LargeTile<16>::BYTES, d_desc, pl.t3, sums, ctx->reg, ctx->dp, dl_big);
    if (chains.n <= 0) deferred_big(on);
  }
  if (n_list[B_FCTA]) {
    const DeferList dl{(u64*)(rbase + o_def), (u32*)(pbase + o_defn)};
    TimedLaunch tl(ts, 3, st);
    launch(st, pack ? k_reduce_fused<true> : k_reduce_fused<false>, (u32)n_list[B_FCTA], SMALL_SEQS, 0, d_desc, pl.fcta, pl.fwt, (TileSum*)(rbase + o_fsum), ctx->reg, ctx->dp, dl);
    launch(st, k_reduce_deferred, DEF_GRID, DEF_WARPS * 32, 0, d_desc, dl, ctx->reg, ctx->dp, now_ns);
  }
  On joined = chains.close();
  if (chains.n > 0) deferred_big(joined);                  // its list is filled by two chains
  {
    TimedLaunch tl(ts, 6, st);
    const u32 ctas = (nc + WD_THREADS / 32 - 1) / (WD_THREADS / 32);
    if (B > 1) launch(st, k_window_rounds, dim3(ctas, B), WD_THREADS, 0, d_desc, ctx->reg);
    if (B > 1) launch(st, k_window_decide<false>, ctas, WD_THREADS, 0, d_desc, B, ctx->reg, ctx->dp);
    else launch(st, k_window_decide<true>, ctas, WD_THREADS, 0, d_desc, B, ctx->reg, ctx->dp);      // one window: both stages in one launch
    if (ctx->n_trees) launch(st, k_tree_root_comm, dim3(ctx->n_trees, B), TREE_THREADS, 0, d_desc, ctx->d_trees, ctx->reg);
  }
  CK(cudaGetLastError());
  for (u32 k = 0; k < B; ++k) {
    WindowHost& w = *ws[k];
    w.analysed = true; w.plan_blk = plan_blk; w.res_blk = res_blk; w.d_desc = d_desc + k; w.d = hd[k]; w.d.packed = nullptr;      // (the batch's, not the window's)
    std::memcpy(w.totals, tot + (size_t)k * T_COUNT, sizeof w.totals);
  }
  // what the layout really found is in pinned memory once the stream has passed it; settle() reads it
  ctx->pending.push_back(pbatch); guard.queued = true;
  if (!expect) {
    // remember the totals of this shape, unless a window was refused
    bool clean = true;
    for (u32 k = 0; k < B && clean; ++k) clean = tot[(size_t)k * T_COUNT + T_FAILED] == 0;
    if (clean) {
      ShapeEntry se; se.n_rec.resize(B); se.totals.assign(tot, tot + (size_t)B * T_COUNT);
      for (u32 k = 0; k < B; ++k) se.n_rec[k] = ws[k]->n_rec;
      for (size_t i = 0; i < ctx->shapes.size(); ++i) if (ctx->shapes[i].n_rec == se.n_rec) { ctx->shapes.erase(ctx->shapes.begin() + i); break; }
      if (ctx->shapes.size() >= SHAPE_CACHE) ctx->shapes.erase(ctx->shapes.begin());
      ctx->shapes.push_back(std::move(se));
    }
  }
  return CCLD_OK;
}

}  // namespace

extern "C" {

// Fills out's counts and, unless `columns` is given, its lists; with `columns` the lists stay in pinned memory, column by column.
static int verdict(ccld_ctx* ctx, uint32_t window_id, ccld_verdict* out, ccld_verdict_columns* columns) {
  WindowHost* w = nullptr;
  CK(cudaSetDevice(ctx->device));
  // The kernels that gather the verdict are enqueued before batches still in doubt are settled: one wait serves both. In
  // the rare case that a batch has to be analysed again (settle() counts those) what was gathered is gathered once more.
  const VerdictHead* head = nullptr; VerdictArea area{}; char* hv = nullptr;
  u32 n_rows = 0;
  char* m = (char*)ctx->misc_blk.p;
  MiscLayout L{};
  for (int attempt = 0; ; ++attempt) {
    auto it = ctx->windows.find(window_id);
    if (it == ctx->windows.end() || !it->second.analysed) { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
    else w = &it->second;
    area = verdict_area(ctx->reg.n_comms, ctx->n_ranks);
    L = misc_layout(ctx->n_ranks);
    { int rc = pinned_area(ctx, ctx->h_verdict, area.total); if (rc != CCLD_OK) return rc; }
    hv = (char*)ctx->h_verdict.p;
    head = (const VerdictHead*)hv;
    n_rows = columns ? (u32)w->totals[T_ROWS] : std::min<u32>((u32)w->totals[T_ROWS], out->comm_rows ? out->comm_rows_cap : 0);
    VerdictArgs A;
    A.counters = w->d.counters; A.rows = w->d.comm_rows; A.n_rows = n_rows; A.alerts = w->d.alerts; A.columns = columns != nullptr;
    A.keys = (u64*)(m + L.keys); A.counts = (u32*)(m + L.counts); A.done = (u32*)(m + L.done);
    A.head = (VerdictHead*)hv; A.rows_out = (ccld_comm_verdict*)(hv + area.rows);
    A.alerts_out = (ccld_hang_alert*)(hv + area.alerts);
    A.sus_host = (ccld_suspect*)(hv + area.suspects); A.sus_host_cap = area.sus_cap; A.sus_dev = (ccld_suspect*)(m + L.sus);
    const u32 pieces = (ctx->n_ranks + VD_THREADS - 1) / VD_THREADS;
    launch(ctx->stream, k_verdict_collect, pieces + 1 + n_rows / VD_THREADS, VD_THREADS, 0, A, ctx->reg, ctx->dp, pieces);
    // suspect lists keep their length from call to call, roughly: where the last one was long, the merge goes along at once
    if (pieces > 1 && ctx->long_list) launch(ctx->stream, k_verdict_merge, pieces, VD_THREADS, 0, A, ctx->reg);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(ctx->stream));
    if (!head->listed) {
      launch(ctx->stream, k_verdict_merge, pieces, VD_THREADS, 0, A, ctx->reg);
      CK(cudaGetLastError());
      CK(cudaStreamSynchronize(ctx->stream));
    }
    ctx->long_list = head->n_suspects > (u32)VD_MERGE;
    const u64 redone = ctx->batches_redone;
    { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
    if (ctx->batches_redone == redone) break;
    if (attempt > 2) return fail(ctx, CCLD_ERR_CUDA, "internal: a settled batch changed again");
  }
  n_rows = std::min<u32>(n_rows, (u32)w->totals[T_ROWS]);      // (fewer than were gathered only where the window was refused: none)
  const u64* cnt = head->counters;
  out->n_records = w->n_rec; out->n_groups = w->totals[T_GROUPS]; out->n_slots = w->totals[T_SLOTS];
  out->n_rejected = w->n_rec - cnt[C_PRESENT]; out->n_complete = cnt[C_COMPLETE]; out->n_incomplete = cnt[C_INCOMPLETE];
  out->n_barrier = cnt[C_BARRIER]; out->n_analysed = cnt[C_ANALYSED]; out->n_flag_skew = cnt[C_FLAG_SKEW]; out->n_flag_dur = cnt[C_FLAG_DUR];
  out->n_opset_mismatch = cnt[C_MISMATCH];
  u32 err = (u32)cnt[C_ERR];
  if (!w->totals[T_FAILED] && w->n_rec - cnt[C_PRESENT] != cnt[C_REJECTED]) err |= CCLD_E_DUPLICATE;   // a slot was written twice
  out->error_bits = err;
  out->n_comm_rows_total = (u32)w->totals[T_ROWS];
  if (columns) {
    const u32 n_al = (u32)std::min<u64>(cnt[C_ALERTS], CCLD_MAX_ALERTS_PER_WINDOW), n_sus = head->n_suspects;
    columns->n_rows = n_rows; columns->n_alerts = n_al; columns->n_suspects = n_sus;
    columns->rows = hv + area.rows; columns->alerts = hv + area.alerts; columns->suspects = hv + area.suspects;
    if (n_sus > area.sus_cap) {                                 // a list this long was left in device memory, as structs
      std::vector<ccld_suspect> list(n_sus);
      { const Piece pc{m + L.sus, list.data(), n_sus * sizeof(ccld_suspect)}; int rc = fetch(ctx, &pc, 1); if (rc != CCLD_OK) return rc; }
      ctx->long_suspects.resize((size_t)n_sus * sizeof(ccld_suspect));
      double* d = (double*)ctx->long_suspects.data(); u32* u = (u32*)(d + n_sus);
      for (size_t i = 0; i < n_sus; ++i) { d[i] = list[i].mean_busbw; u[i] = list[i].kind; u[n_sus + i] = list[i].rank; u[2ull * n_sus + i] = list[i].votes; u[3ull * n_sus + i] = list[i].ops; }
      columns->suspects = ctx->long_suspects.data();
    }
  }
  if (!columns && n_rows) std::memcpy(out->comm_rows, hv + area.rows, n_rows * sizeof(ccld_comm_verdict));
  // hang alerts, ordered by (communicator, seq)
  out->n_alerts_total = (u32)std::min<u64>(cnt[C_ALERTS], 0xFFFFFFFFull);
  const u32 n_al = columns ? 0 : std::min<u32>(std::min<u32>(out->n_alerts_total, CCLD_MAX_ALERTS_PER_WINDOW), out->alerts ? out->alerts_cap : 0);
  if (n_al) std::memcpy(out->alerts, hv + area.alerts, n_al * sizeof(ccld_hang_alert));
  // cumulative suspects
  out->n_suspects_total = head->n_suspects;
  const u32 n_out = columns ? 0 : std::min<u32>(head->n_suspects, out->suspects ? out->suspects_cap : 0);
  if (n_out && head->n_suspects <= area.sus_cap) std::memcpy(out->suspects, hv + area.suspects, n_out * sizeof(ccld_suspect));
  else if (n_out) {
    CK(cudaMemcpyAsync(out->suspects, m + L.sus, n_out * sizeof(ccld_suspect), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
  }
  if (cnt[C_INTERNAL]) return fail(ctx, CCLD_ERR_CUDA, "internal: slot index out of range");
  if (err & CCLD_E_UNKNOWN_COMM) return fail(ctx, CCLD_ERR_UNKNOWN_COMM, "record of an unregistered communicator");
  if (err & CCLD_E_NOT_MEMBER) return fail(ctx, CCLD_ERR_NOT_MEMBER, "record of a rank that is not a member of its communicator");
  if (err & CCLD_E_SEQ_RANGE) return fail(ctx, CCLD_ERR_SEQ_RANGE, "record with an op counter below the communicator's first");
  if (err & CCLD_E_DUPLICATE) return fail(ctx, CCLD_ERR_DUPLICATE, "duplicate (communicator, op counter, rank) record");
  if (err & CCLD_E_CAPACITY) return fail(ctx, CCLD_ERR_CAPACITY, "op counters of the window span too many slots");
  return CCLD_OK;
}

int ccld_get_verdict(ccld_ctx* ctx, uint32_t window_id, ccld_verdict* out) try {
  NvtxRange nvtx_range("ccld_get_verdict");
  if (!ctx || !out) return CCLD_ERR_ARG;
  return verdict(ctx, window_id, out, nullptr);
} CAUGHT

int ccld_get_verdict_columns(ccld_ctx* ctx, uint32_t window_id, ccld_verdict* out, ccld_verdict_columns* columns) try {
  NvtxRange nvtx_range("ccld_get_verdict_columns");
  if (!ctx || !out || !columns) return CCLD_ERR_ARG;
  return verdict(ctx, window_id, out, columns);
} CAUGHT

// Launches the hang kernel over one op or over the window's alerts (A.alerts set) and waits; results are in pinned memory.
static int hang_run(ccld_ctx* ctx, const WindowHost* w, HangArgs& A, u32 ctas) {
  A.n_frames = w->n_frames; A.n_channels = w->n_channels;
  A.f_rank = w->f_rank; A.f_comm = w->f_comm; A.f_seq = w->f_seq; A.progress = w->progress;
  A.scratch_stride = (u64)align_up((size_t)ctx->max_n * HANG_MEMBER_BYTES); A.scratch = nullptr;
  Block blk;
  if (ctx->max_n > HANG_SMEM_N) {
    cudaError_t e;
    blk = ctx->pool.get(A.scratch_stride * ctas, &e);
    if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "scratch allocation failed");
    A.scratch = (unsigned char*)blk.p;
  }
  launch(ctx->stream, k_hang_locate, ctas, HANG_THREADS, hang_smem(std::min<u32>(ctx->max_n, HANG_SMEM_N)), w->d_desc, ctx->reg, A);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  ctx->pool.put(blk);
  return e == cudaSuccess ? CCLD_OK : fail(ctx, CCLD_ERR_CUDA, std::string("hang location: ") + cudaGetErrorString(e));
}

int ccld_locate_hang(ccld_ctx* ctx, uint32_t window_id, uint32_t comm, uint32_t seq, ccld_hang_verdict* out) try {
  NvtxRange nvtx_range("ccld_locate_hang");
  if (!ctx || !out) return CCLD_ERR_ARG;
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  auto ci = ctx->comm_idx.find(comm);
  if (ci == ctx->comm_idx.end()) return fail(ctx, CCLD_ERR_UNKNOWN_COMM, "unknown communicator");
  CK(cudaSetDevice(ctx->device));
  const u32 n = (u32)ctx->comms[ci->second].ranks.size();
  if (ctx->comms[ci->second].algo != 0 && !ctx->comms[ci->second].d_head) return fail(ctx, CCLD_ERR_STATE, "tree communicator without layers (ccld_comm_set_layers)");
  u32* roots = out->roots; const u32 cap = roots ? out->roots_cap : 0, keep = std::min(cap, n);
  const size_t o_roots = align_up(sizeof(ccld_hang_verdict));
  { int rc = pinned_area(ctx, ctx->h_io, o_roots + keep * 4ull); if (rc != CCLD_OK) return rc; }
  char* h = (char*)ctx->h_io.p;
  HangArgs A; std::memset(&A, 0, sizeof A);
  A.c = ci->second; A.seq = seq; A.roots = (u32*)(h + o_roots); A.roots_cap = keep; A.out = (ccld_hang_verdict*)h;
  { int rc = hang_run(ctx, w, A, 1); if (rc != CCLD_OK) return rc; }
  std::memcpy(out, h, sizeof *out); out->roots = roots; out->roots_cap = cap;
  const u32 n_copy = std::min(out->n_roots_total, keep);
  if (n_copy) std::memcpy(roots, h + o_roots, n_copy * 4ull);
  return CCLD_OK;
} CAUGHT

int ccld_locate_hangs(ccld_ctx* ctx, uint32_t window_id, ccld_hang_alert* alerts, ccld_hang_verdict* out, uint32_t cap,
                      uint32_t* roots, uint32_t roots_stride, uint32_t* n_total) try {
  NvtxRange nvtx_range("ccld_locate_hangs");
  if (!ctx || !n_total) return CCLD_ERR_ARG;
  if (cap && !out) return fail(ctx, CCLD_ERR_ARG, "out is null");
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  u32 most = std::min<u32>(cap, CCLD_MAX_ALERTS_PER_WINDOW);
  const u32 keep = roots ? std::min(roots_stride, ctx->max_n) : 0;                 // roots kept per alert
  if ((size_t)most * keep * 4 > FETCH_PINNED) {
    // a pinned area for every alert there could be would be large: ask how many there are
    u64 n_al64 = 0; const Piece pc{w->d.counters + C_ALERTS, &n_al64, 8};
    { int rc = fetch(ctx, &pc, 1); if (rc != CCLD_OK) return rc; }
    most = (u32)std::min<u64>(most, n_al64);
  }
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
  const size_t o_n = take(8), o_al = take(most * sizeof(ccld_hang_alert)), o_out = take(most * sizeof(ccld_hang_verdict)), o_roots = take((size_t)most * keep * 4);
  { int rc = pinned_area(ctx, ctx->h_io, off); if (rc != CCLD_OK) return rc; }
  char* h = (char*)ctx->h_io.p;
  ccld_hang_alert* al = (ccld_hang_alert*)((char*)ctx->misc_blk.p + misc_layout(ctx->n_ranks).alerts);
  launch(st, k_order_alerts, 1, VD_THREADS, 0, w->d.counters, w->d.alerts, al, ctx->reg);
  HangArgs A; std::memset(&A, 0, sizeof A);
  A.alerts = al; A.counters = w->d.counters; A.cap = most; A.roots = (u32*)(h + o_roots); A.roots_cap = keep;
  A.out = (ccld_hang_verdict*)(h + o_out); A.alerts_out = (ccld_hang_alert*)(h + o_al); A.n_alerts_out = (u64*)(h + o_n);
  { int rc = hang_run(ctx, w, A, std::max(1u, std::min(most, ctx->n_sms))); if (rc != CCLD_OK) return rc; }
  const u64 found = *(const u64*)(h + o_n);
  *n_total = (u32)std::min<u64>(found, 0xFFFFFFFFull);
  const u32 n = (u32)std::min<u64>(found, most);
  const ccld_hang_verdict* hv = (const ccld_hang_verdict*)(h + o_out);
  for (u32 i = 0; i < n; ++i) if (hv[i].cls == HANG_NO_LAYERS) return fail(ctx, CCLD_ERR_STATE, "tree communicator without layers (ccld_comm_set_layers)");
  for (u32 i = 0; i < n; ++i) {
    ccld_hang_verdict v = hv[i];
    v.roots = roots ? roots + (size_t)i * roots_stride : nullptr; v.roots_cap = roots ? roots_stride : 0;
    const u32 n_copy = std::min(v.n_roots_total, keep);
    if (n_copy) std::memcpy(v.roots, h + o_roots + (size_t)i * keep * 4, n_copy * 4ull);
    out[i] = v;
  }
  if (alerts && n) std::memcpy(alerts, h + o_al, n * sizeof(ccld_hang_alert));
  return CCLD_OK;
} CAUGHT

int ccld_get_optable(ccld_ctx* ctx, uint32_t window_id, ccld_optable* out) try {
  if (!ctx || !out) return CCLD_ERR_ARG;
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  const WinDesc& d = w->d; const u64 G = d.n_groups;
  out->n_groups = G; out->n_slots = d.n_slots;
  const i64* gi = d.gi64; const u32* gu = d.gu32;
  out->e_min = gi + GI_E_MIN * G; out->arrival_skew = gi + GI_ARRIVAL_SKEW * G; out->t_max = gi + GI_T_MAX * G; out->t_min = gi + GI_T_MIN * G;
  out->span = gi + GI_SPAN * G; out->med_skew = gi + GI_MED_SKEW * G; out->mad_skew = gi + GI_MAD_SKEW * G;
  out->med_dur = gi + GI_MED_DUR * G; out->mad_dur = gi + GI_MAD_DUR * G;
  out->rank_tmin = gu + GU_RANK_TMIN * G; out->rank_tmax = gu + GU_RANK_TMAX * G; out->max_chg = gu + GU_MAX_CHG * G;
  out->rank_max_chg = gu + GU_RANK_MAX_CHG * G; out->n_present = gu + GU_N_PRESENT * G; out->gflags = gu + GU_GFLAGS * G;
  out->busbw = d.gbw; out->flags = d.flags; out->perm = d.perm;
  return CCLD_OK;
} CAUGHT

int ccld_get_ranges(ccld_ctx* ctx, uint32_t window_id, ccld_comm_range* rows, uint32_t cap, uint32_t* n_total) try {
  if (!ctx || !n_total) return CCLD_ERR_ARG;
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  CK(cudaSetDevice(ctx->device));
  const u32 nc = ctx->reg.n_comms;
  std::vector<RangeRow> rr(nc);
  { const Piece pc{w->d.ranges, rr.data(), nc * sizeof(RangeRow)}; int rc = fetch(ctx, &pc, 1); if (rc != CCLD_OK) return rc; }
  u32 k = 0;
  for (u32 c = 0; c < nc; ++c) {
    if (rr[c].n_seq == 0) continue;
    if (rows && k < cap) { rows[k].comm = ctx->comms[c].id; rows[k].n = rr[c].n; rows[k].seq_lo = rr[c].seq_lo; rows[k].n_seq = rr[c].n_seq;
                           rows[k].group0 = rr[c].group0; rows[k].slot0 = rr[c].slot0; }
    ++k;
  }
  *n_total = k;
  return CCLD_OK;
} CAUGHT

void ccld_host_release(ccld_host_block* blk) {
  if (!blk || !blk->p) return;
  Block b; b.p = blk->p; b.bytes = blk->bytes;
  BlockStore::get().give_back(b, b.bytes);
  blk->p = nullptr; blk->bytes = 0;
}

int ccld_take_optable(ccld_ctx* ctx, uint32_t window_id, ccld_host_optable* out) try {
  NvtxRange nvtx_range("ccld_take_optable");
  if (!ctx || !out) return CCLD_ERR_ARG;
  std::memset(out, 0, sizeof *out);
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  CK(cudaSetDevice(ctx->device));
  const WinDesc& d = w->d; const u64 G = d.n_groups, S = d.n_slots;
  // the table's columns follow each other on the device, so five pieces make it up; the key columns are written beside them
  const Piece pc[5] = {{d.gi64, nullptr, G * 8 * GI_COUNT}, {d.gu32, nullptr, G * 4 * GU_COUNT}, {d.gbw, nullptr, G * 8}, {d.flags, nullptr, S}, {d.perm, nullptr, S * 4}};
  const size_t keys = G * 16;
  if (S > TAKE_MOST || G > TAKE_MOST) return fail(ctx, CCLD_ERR_CAPACITY, "too large for a pinned block");
  { int rc = take_block(ctx, align_up(keys) + gather_room(pc, 5), &out->block); if (rc != CCLD_OK) return rc; }
  char* base = (char*)out->block.p; size_t at[5];
  u64* slot0 = (u64*)base; u32* comm = (u32*)(slot0 + G); u32* seq = comm + G;
  cudaError_t e = cudaSuccess;
  if (G) { launch(ctx->stream, k_op_keys, (u32)((G + 255) / 256), 256, 0, d.ranges, ctx->reg, G, comm, seq, slot0); e = cudaGetLastError(); }
  if (e == cudaSuccess) e = gather(ctx, pc, 5, base, align_up(keys), at);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) { cudaStreamSynchronize(ctx->stream); ccld_host_release(&out->block); return fail(ctx, CCLD_ERR_CUDA, std::string("table copy: ") + cudaGetErrorString(e)); }
  ccld_optable& t = out->t;
  const i64* gi = (const i64*)(base + at[0]); const u32* gu = (const u32*)(base + at[1]);
  t.n_groups = G; t.n_slots = S;
  t.e_min = gi + GI_E_MIN * G; t.arrival_skew = gi + GI_ARRIVAL_SKEW * G; t.t_max = gi + GI_T_MAX * G; t.t_min = gi + GI_T_MIN * G; t.span = gi + GI_SPAN * G;
  t.med_skew = gi + GI_MED_SKEW * G; t.mad_skew = gi + GI_MAD_SKEW * G; t.med_dur = gi + GI_MED_DUR * G; t.mad_dur = gi + GI_MAD_DUR * G;
  t.rank_tmin = gu + GU_RANK_TMIN * G; t.rank_tmax = gu + GU_RANK_TMAX * G; t.max_chg = gu + GU_MAX_CHG * G;
  t.rank_max_chg = gu + GU_RANK_MAX_CHG * G; t.n_present = gu + GU_N_PRESENT * G; t.gflags = gu + GU_GFLAGS * G;
  t.busbw = (const double*)(base + at[2]); t.flags = (const u8*)(base + at[3]); t.perm = (const u32*)(base + at[4]);
  out->comm = comm; out->seq = seq; out->slot0 = slot0;
  return CCLD_OK;
} CAUGHT

int ccld_take_rank_stats(ccld_ctx* ctx, uint32_t n_ranks, ccld_host_rank_stats* out) try {
  if (!ctx || !out) return CCLD_ERR_ARG;
  std::memset(out, 0, sizeof *out);
  if (!ctx->finalized) return fail(ctx, CCLD_ERR_STATE, "nothing analysed yet");
  if (n_ranks > ctx->reg.n_ranks) return fail(ctx, CCLD_ERR_CAPACITY, "more ranks than the registry knows");
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  CK(cudaSetDevice(ctx->device));
  const size_t n = n_ranks;
  const Piece pc[4] = {{ctx->reg.votes, nullptr, n * 16}, {ctx->reg.ops, nullptr, n * 4}, {ctx->reg.bw_cnt, nullptr, n * 4}, {ctx->reg.bw_sum, nullptr, n * 8}};
  { int rc = take_block(ctx, gather_room(pc, 4), &out->block); if (rc != CCLD_OK) return rc; }
  char* base = (char*)out->block.p; size_t at[4];
  cudaError_t e = gather(ctx, pc, 4, base, 0, at);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) { cudaStreamSynchronize(ctx->stream); ccld_host_release(&out->block); return fail(ctx, CCLD_ERR_CUDA, std::string("statistics copy: ") + cudaGetErrorString(e)); }
  out->votes = (const u32*)(base + at[0]); out->ops = (const u32*)(base + at[1]); out->bw_cnt = (const u32*)(base + at[2]); out->bw_sum = (const double*)(base + at[3]);
  return CCLD_OK;
} CAUGHT

int ccld_get_rank_stats(ccld_ctx* ctx, uint32_t n_ranks, uint32_t* votes, uint32_t* ops, uint32_t* bw_cnt, double* bw_sum) try {
  if (!ctx || !votes || !ops || !bw_cnt || !bw_sum) return CCLD_ERR_ARG;
  if (!ctx->finalized) return fail(ctx, CCLD_ERR_STATE, "nothing analysed yet");
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  CK(cudaSetDevice(ctx->device));
  const size_t n = std::min(n_ranks, ctx->reg.n_ranks), rest = n_ranks - n;      // ranks the registry does not know: zeros
  std::memset(votes + n * 4, 0, rest * 16); std::memset(ops + n, 0, rest * 4); std::memset(bw_cnt + n, 0, rest * 4); std::memset(bw_sum + n, 0, rest * 8);
  const Piece pc[4] = {{ctx->reg.votes, votes, n * 16}, {ctx->reg.ops, ops, n * 4}, {ctx->reg.bw_cnt, bw_cnt, n * 4}, {ctx->reg.bw_sum, bw_sum, n * 8}};
  return fetch(ctx, pc, 4);
} CAUGHT

int ccld_trace_attach_opset(ccld_ctx* ctx, uint32_t window_id, int mem_kind, const uint8_t* algo, const uint8_t* proto) try {
  if (!ctx) return CCLD_ERR_ARG;
  if (mem_kind != 0 && mem_kind != 1) return fail(ctx, CCLD_ERR_ARG, "mem_kind must be 0 (host) or 1 (device)");
  auto it = ctx->windows.find(window_id);
  if (it == ctx->windows.end()) return fail(ctx, CCLD_ERR_NO_WINDOW, "unknown window id");
  WindowHost& w = it->second;
  if (w.n_rec > 0 && (!algo || !proto)) return fail(ctx, CCLD_ERR_ARG, "null column");
  CK(cudaSetDevice(ctx->device));
  if (w.owns_opset) { CK(cudaStreamSynchronize(ctx->stream)); ctx->pool.put(w.opset_own); w.owns_opset = false; }
  if (mem_kind == 1 || w.n_rec == 0) { w.algo = algo; w.proto = proto; return CCLD_OK; }
  cudaError_t e;
  const size_t half = align_up(w.n_rec);
  w.opset_own = ctx->pool.get(2 * half, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "window allocation failed");
  w.owns_opset = true;
  char* b = (char*)w.opset_own.p;
  CK(cudaMemcpyAsync(b, algo, w.n_rec, cudaMemcpyHostToDevice, ctx->stream));
  CK(cudaMemcpyAsync(b + half, proto, w.n_rec, cudaMemcpyHostToDevice, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));       // the caller's host arrays are free again
  w.algo = (const u8*)b; w.proto = (const u8*)(b + half);
  return CCLD_OK;
} CAUGHT

int ccld_opset_check(ccld_ctx* ctx, uint32_t window_id, uint32_t comm, uint32_t seq, ccld_opset_verdict* out) try {
  if (!ctx || !out) return CCLD_ERR_ARG;
  WindowHost* w;
  { int rc = find_analysed(ctx, window_id, &w); if (rc != CCLD_OK) return rc; }
  auto ci = ctx->comm_idx.find(comm);
  if (ci == ctx->comm_idx.end()) return fail(ctx, CCLD_ERR_UNKNOWN_COMM, "unknown communicator");
  CK(cudaSetDevice(ctx->device));
  const u32 n = (u32)ctx->comms[ci->second].ranks.size();
  u32* ranks = out->ranks; const u32 cap = ranks ? out->ranks_cap : 0, keep = std::min(cap, n);
  const size_t o_rk = align_up(sizeof(ccld_opset_verdict));
  { int rc = pinned_area(ctx, ctx->h_io, o_rk + keep * 4ull); if (rc != CCLD_OK) return rc; }
  char* h = (char*)ctx->h_io.p;
  OpsetArgs A; A.c = ci->second; A.seq = seq; A.algo = w->algo; A.proto = w->proto;
  A.ranks = (u32*)(h + o_rk); A.ranks_cap = keep; A.out = (ccld_opset_verdict*)h;
  launch(ctx->stream, k_opset_check, 1, OPSET_THREADS, (size_t)n * OPSET_MEMBER_BYTES, w->d_desc, ctx->reg, A);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(ctx->stream));
  std::memcpy(out, h, sizeof *out); out->ranks = ranks; out->ranks_cap = cap;
  const u32 n_copy = std::min(out->n_deviating_total, keep);
  if (n_copy) std::memcpy(ranks, h + o_rk, n_copy * 4ull);
  return CCLD_OK;
} CAUGHT

namespace {
struct StateHeader { u64 magic; u32 version, n_comms, n_ranks, pad; u64 stats_bytes; };
constexpr u64 STATE_MAGIC = 0x3130545344434343ull;    // "CCCDST01"
}  // namespace

int ccld_state_export(ccld_ctx* ctx, void* buf, uint64_t cap, uint64_t* n_bytes) try {
  if (!ctx || !n_bytes) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  { int rc = finalize_registry(ctx); if (rc != CCLD_OK) return rc; }
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  const u32 nc = ctx->reg.n_comms;
  const u64 need = sizeof(StateHeader) + (u64)nc * 12 + ctx->stats_bytes;
  *n_bytes = need;
  if (!buf || cap < need) return buf ? fail(ctx, CCLD_ERR_CAPACITY, "state buffer too small") : CCLD_OK;
  char* p = (char*)buf;
  StateHeader h{STATE_MAGIC, 1u, nc, ctx->n_ranks, 0u, (u64)ctx->stats_bytes};
  std::memcpy(p, &h, sizeof h); p += sizeof h;
  for (u32 c = 0; c < nc; ++c) { const u32 row[3] = {ctx->comms[c].id, (u32)ctx->comms[c].ranks.size(), ctx->comms[c].seq0}; std::memcpy(p, row, 12); p += 12; }
  CK(cudaMemcpyAsync(p, (char*)ctx->reg_blk.p + ctx->stats_off, ctx->stats_bytes, cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CCLD_OK;
} CAUGHT

int ccld_state_import(ccld_ctx* ctx, const void* buf, uint64_t n_bytes) try {
  if (!ctx || !buf) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  { int rc = finalize_registry(ctx); if (rc != CCLD_OK) return rc; }
  { int rc = settle(ctx); if (rc != CCLD_OK) return rc; }
  const u32 nc = ctx->reg.n_comms;
  StateHeader h;
  if (n_bytes < sizeof h) return fail(ctx, CCLD_ERR_ARG, "state blob too short");
  std::memcpy(&h, buf, sizeof h);
  if (h.magic != STATE_MAGIC || h.version != 1) return fail(ctx, CCLD_ERR_ARG, "not a state blob of this library version");
  if (h.n_comms != nc || h.n_ranks != ctx->n_ranks || h.stats_bytes != ctx->stats_bytes || n_bytes != sizeof h + (u64)nc * 12 + h.stats_bytes)
    return fail(ctx, CCLD_ERR_ARG, "state blob belongs to another set of communicators");
  const char* p = (const char*)buf + sizeof h;
  for (u32 c = 0; c < nc; ++c) {
    u32 row[3]; std::memcpy(row, p, 12); p += 12;
    if (row[0] != ctx->comms[c].id || row[1] != (u32)ctx->comms[c].ranks.size() || row[2] != ctx->comms[c].seq0)
      return fail(ctx, CCLD_ERR_ARG, "state blob belongs to another set of communicators");
  }
  CK(cudaStreamSynchronize(ctx->stream));
  CK(cudaMemcpyAsync((char*)ctx->reg_blk.p + ctx->stats_off, p, ctx->stats_bytes, cudaMemcpyHostToDevice, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CCLD_OK;
} CAUGHT

int ccld_derive_rates(ccld_ctx* ctx, uint64_t n_rec, const uint32_t* rank, const int64_t* t_enter_ns, const int64_t* t_exit_ns,
                      uint32_t n_ranks, uint64_t n_ticks, const uint64_t* tick_off, const int64_t* tick_ns,
                      const uint32_t* send_count, const uint32_t* recv_count, uint32_t* send_chg, uint32_t* recv_chg) try {
  if (!ctx) return CCLD_ERR_ARG;
  if (n_rec && (!rank || !t_enter_ns || !t_exit_ns || !send_chg || !recv_chg)) return fail(ctx, CCLD_ERR_ARG, "null record column");
  if (n_ranks == 0 || !tick_off) return fail(ctx, CCLD_ERR_ARG, "tick_off is required (n_ranks + 1 entries)");
  if (n_ticks && (!tick_ns || !send_count || !recv_count)) return fail(ctx, CCLD_ERR_ARG, "null tick column");
  if (n_ticks >= 0xFFFFFFFFull) return fail(ctx, CCLD_ERR_CAPACITY, "too many ticks for 32-bit change counts");
  if ((n_rec + RT_THREADS - 1) / RT_THREADS > 0x7FFFFFFFull) return fail(ctx, CCLD_ERR_CAPACITY, "too many records for one launch");
  CK(cudaSetDevice(ctx->device));
  if (n_rec == 0) return CCLD_OK;
  cudaStream_t st = ctx->stream;
  const u64 n_tiles = (n_ticks + RT_TILE - 1) / RT_TILE;
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
  const size_t o_blk = take(n_tiles * (RT_TILE / 32) * sizeof(TickBlock)), o_tile = take(n_tiles * sizeof(uint2)), o_rank = take(n_ranks * sizeof(RankTicks)),
               o_far = take((((u64)n_ranks + RT_THREADS - 1) / RT_THREADS + 1) * 4);
  cudaError_t e;
  Block blk = ctx->pool.get(off, &e);
  if (e != cudaSuccess) return fail(ctx, CCLD_ERR_NOMEM, "scratch allocation failed");
  TickArgs A; A.n_ticks = n_ticks; A.n_ranks = n_ranks; A.n_tiles = (u32)n_tiles;
  A.tick_off = tick_off; A.tick_ns = tick_ns; A.send = send_count; A.recv = recv_count;
  A.blk = (TickBlock*)((char*)blk.p + o_blk); A.tile = (uint2*)((char*)blk.p + o_tile); A.ranks = (RankTicks*)((char*)blk.p + o_rank);
  A.vec = (((uintptr_t)send_count | (uintptr_t)recv_count) & 15) == 0;
  const u32 rank_ctas = (u32)(((u64)n_ranks + RT_THREADS - 1) / RT_THREADS);
  const bool long_ranks = n_tiles > (u64)RT_NEAR * n_ranks;      // on average
  A.far = (u32*)((char*)blk.p + o_far); A.scanned = n_tiles > (long_ranks ? RT_SCAN : RT_LOOK) ? A.far + rank_ctas : nullptr;
  launch(st, k_tick_blocks, (u32)n_tiles + rank_ctas, RT_THREADS, 0, A);
  if (A.scanned) launch(st, k_tile_scan, 1, TS_THREADS, 0, A.tile, A.n_tiles, long_ranks ? nullptr : A.far, rank_ctas, A.scanned);
  launch(st, k_record_rates, (u32)((n_rec + RT_THREADS - 1) / RT_THREADS), RT_THREADS, 0, A, n_rec, rank, t_enter_ns, t_exit_ns, send_chg, recv_chg);
  const cudaError_t le = cudaGetLastError();
  ctx->pool.put(blk);           // later work on this stream runs after these kernels: the block can be handed out again
  if (le != cudaSuccess) return fail(ctx, CCLD_ERR_CUDA, std::string("rate kernels: ") + cudaGetErrorString(le));
  return CCLD_OK;
} CAUGHT

int ccld_timing_enable(ccld_ctx* ctx, int on) try {
  if (!ctx) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  if (on && ctx->ring.empty()) {
    ctx->ring.resize(TIMER_RING);
    for (auto& sl : ctx->ring) for (int i = 0; i < TIMER_PAIRS; ++i) { CK(cudaEventCreate(&sl.a[i])); CK(cudaEventCreate(&sl.b[i])); }
  }
  for (auto& sl : ctx->ring) sl.n = 0;
  std::memset(ctx->t_ms, 0, sizeof ctx->t_ms); std::memset(ctx->t_launches, 0, sizeof ctx->t_launches);
  ctx->timing = on != 0;
  return CCLD_OK;
} CAUGHT

int ccld_get_kernel_times(ccld_ctx* ctx, double* ms, uint64_t* launches) {
  if (!ctx || !ms || !launches) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  for (auto& sl : ctx->ring) timer_harvest(ctx, sl);
  for (int k = 0; k < CCLD_K_KINDS; ++k) { ms[k] = ctx->t_ms[k]; launches[k] = ctx->t_launches[k]; }
  return CCLD_OK;
}

int ccld_get_route_counts(ccld_ctx* ctx, uint64_t* counts) {
  if (!ctx || !counts) return CCLD_ERR_ARG;
  counts[0] = ctx->unwaited; counts[1] = ctx->batches_redone; counts[2] = ctx->packed; counts[3] = ctx->filled_under_range;
  return CCLD_OK;
}

int ccld_copy_many_to_host(ccld_ctx* ctx, uint32_t n, void* const* dst_host, const void* const* src_device, const uint64_t* bytes) try {
  if (!ctx || (n && (!dst_host || !src_device || !bytes))) return CCLD_ERR_ARG;
  for (u32 i = 0; i < n; ++i) if (bytes[i] && (!dst_host[i] || !src_device[i])) return fail(ctx, CCLD_ERR_ARG, "null array");
  CK(cudaSetDevice(ctx->device));
  if (n <= GATHER_PIECES) {
    Piece pc[GATHER_PIECES];
    for (u32 i = 0; i < n; ++i) pc[i] = Piece{src_device[i], dst_host[i], bytes[i]};
    return fetch(ctx, pc, n);
  }
  for (u32 i = 0; i < n; ++i) if (bytes[i]) CK(cudaMemcpyAsync(dst_host[i], src_device[i], bytes[i], cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CCLD_OK;
} CAUGHT

int ccld_copy_to_host(ccld_ctx* ctx, void* dst_host, const void* src_device, uint64_t bytes) try {
  if (!ctx || (bytes && (!dst_host || !src_device))) return CCLD_ERR_ARG;
  CK(cudaSetDevice(ctx->device));
  if (bytes) CK(cudaMemcpyAsync(dst_host, src_device, bytes, cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CCLD_OK;
} CAUGHT

}  // extern "C"
