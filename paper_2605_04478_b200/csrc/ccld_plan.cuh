// Group-by, part 2: the closed-form layout of every window and the work lists of the reduction kernels (sm_100a).
//   slot(comm, seq, pos) = slot0[comm] + (seq - seq_lo[comm]) * n[comm] + pos
//
//   k_begin   the batch's descriptors move from pinned host memory to the device and its op-counter ranges, counters and list
//             lengths get their start values
//   k_layout  one CTA per window: prefix sums over the communicators (groups, slots, rows, work units) and the start of every
//             chunk of the work lists; the other CTAs of the launch, if any, fill the slot table of a batch that does not wait
//   emit_lists  a CTA per (window, chunk, 256 communicators) writes their part of the chunk's work lists, beside the scatter
//             pass and in its launch (ccld_kernels.cuh)
//
// All are bound by latency: little data, a chain of dependent reads and barriers. What a chunk holds follows from the communicators' unit
// counts alone, so the chunks' starts come from a histogram along the chunks, and the lists are written by as many CTAs as there
// are chunks. (One CTA per window for all of it took 155 us for the 2,185 communicators of 16,384 ranks, k_layout takes 18.)
#pragma once
#include "ccld_device.cuh"

namespace ccld {

constexpr int BEGIN_THREADS = 256;
constexpr u32 LAYOUT_THREADS = 1024;                   // at most: as many as there are communicators do for a small registry
constexpr u32 LAYOUT_CACHED = 4;                       // communicators per thread whose ranges wait in registers (4,096 per window)
constexpr int EMIT_THREADS = 256;
constexpr u32 EMIT_SLICES = 32;

struct BeginArgs {
  const u32* desc_host; u32* desc; u64 desc_words;     // pinned source, device copy: descriptors (and expected totals behind them)
  u32* rmin; u64 n_rmin;                               // set to NONE
  u32* zero; u64 n_zero;                               // set to 0: rmax, counters, list lengths
};

__global__ void __launch_bounds__(BEGIN_THREADS) k_begin(BeginArgs A) {
  begin_after();
  const u64 i0 = (u64)blockIdx.x * BEGIN_THREADS + threadIdx.x, st = (u64)gridDim.x * BEGIN_THREADS;
  for (u64 i = i0; i < A.desc_words; i += st) A.desc[i] = A.desc_host[i];
  for (u64 i = i0; i < A.n_rmin; i += st) A.rmin[i] = NONE;
  for (u64 i = i0; i < A.n_zero; i += st) A.zero[i] = 0;
}

// op counters a communicator covers in the window (0 if none; clamped to 2^32 - 1)
__device__ __forceinline__ u32 range_len(u32 lo, u32 hi) {
  if (!(lo <= hi && lo != NONE)) return 0;
  const u64 ns = (u64)hi - lo + 1;
  return ns > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)ns;
}
__device__ __forceinline__ u32 plan_nseq(const WinDesc& D, u32 c) { return range_len(D.rmin[c], D.rmax[c]); }

// Work units (warp-tiles of class 0, CTA tiles of class 1) of a communicator; 0 for other classes.
__device__ __forceinline__ u32 fused_units(u32 ns, u32 n) { return comm_class(n) > 1 ? 0u : ceil_div(ns, tile_seqs(n)); }

// CTA `cta` of `ctas` sets its part of the slot table to NONE.
constexpr u64 FILL_BESIDE = 24ull << 20;                // slots of a batch that are filled beside the layout, at most
__device__ __forceinline__ void fill_slots(u32* perm, u64 n, u32 cta, u32 ctas) {
  const u64 head = min(n, (u64)((16 - ((uintptr_t)perm & 15)) & 15) / 4), n4 = (n - head) / 4, per = (n4 + ctas - 1) / ctas;
  uint4* p4 = reinterpret_cast<uint4*>(perm + head);
  for (u64 i = cta * per + threadIdx.x, end = min(n4, (cta + 1) * per); i < end; i += blockDim.x) p4[i] = make_uint4(NONE, NONE, NONE, NONE);
  if (cta != 0) return;
  if (threadIdx.x < head) perm[threadIdx.x] = NONE;
  if (threadIdx.x < n - head - n4 * 4) perm[head + n4 * 4 + threadIdx.x] = NONE;
}

struct PlanAcc { u64 groups, slots; u32 rows, units, t2, t3; };
__device__ __forceinline__ PlanAcc plan_add(const PlanAcc& a, const PlanAcc& b) {
  PlanAcc r; r.groups = a.groups + b.groups; r.slots = a.slots + b.slots; r.rows = a.rows + b.rows; r.units = a.units + b.units;
  r.t2 = a.t2 + b.t2; r.t3 = a.t3 + b.t3; return r;
}
__device__ __forceinline__ PlanAcc plan_shfl_up(const PlanAcc& a, int d) {
  PlanAcc r;
  r.groups = __shfl_up_sync(0xFFFFFFFFu, a.groups, d); r.slots = __shfl_up_sync(0xFFFFFFFFu, a.slots, d);
  r.rows = __shfl_up_sync(0xFFFFFFFFu, a.rows, d); r.units = __shfl_up_sync(0xFFFFFFFFu, a.units, d);
  r.t2 = __shfl_up_sync(0xFFFFFFFFu, a.t2, d); r.t3 = __shfl_up_sync(0xFFFFFFFFu, a.t3, d);
  return r;
}
__device__ __forceinline__ PlanAcc plan_item(u32 ns, u32 n) {
  PlanAcc a = {0, 0, 0, 0, 0, 0};
  if (ns == 0) return a;
  const u32 cls = comm_class(n);
  a.groups = ns; a.slots = (u64)ns * n; a.rows = 1;
  if (cls <= 1) a.units = fused_units(ns, n);
  else { const u32 t = ceil_div(ns, tile_seqs(n)); a.t2 = cls == 2 ? t : 0; a.t3 = cls == 3 ? t : 0; }
  return a;
}

// Work lists of the batch.
struct PlanLists { FusedCta* fcta; WarpTile* fwt; Tile* t2; Tile* t3; };

// When the host sized the results from totals it expected (D.expect) instead of waiting for these, a window whose totals
// differ gives up and raises the poison flag; so does every window planned after the flag went up - in the same batch
// (seen by emit_lists) or in a later one - so that windows are never analysed out of order.
// Grid: (1 + filling CTAs, windows). fused_warps: warps of k_reduce_fused that run at a time.
__global__ void __launch_bounds__(LAYOUT_THREADS) k_layout(const WinDesc* wd, Registry R, u32 fused_warps) {
  begin_after();
  __shared__ PlanAcc s_warp[33];
  __shared__ u32 s_red[32];
  __shared__ u32 s_hist[2][CHUNK_MAX], s_fused;                // units per chunk: warp-tiles of class 0, tiles of class 1; slots / 32 of both
  __shared__ bool s_turns;                                     // records in their ranks' order, only that ranks take turns over many communicators
  const WinDesc& D = wd[blockIdx.y];
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (blockIdx.x > 0) { fill_slots(D.perm, D.n_slots, blockIdx.x - 1, gridDim.x - 1); return; }
  // what warp 0 compares its findings with; poisoned: an earlier batch's layout was not the expected one
  const u64 slot_cap = D.slot_cap; const bool expects = D.expect != nullptr;
  u64 expected = 0; bool poisoned = false;
  const u64 mixed = D.counters[C_MIXED];
  if (wid == 0 && expects) { expected = lane < T_COUNT ? D.expect[lane] : 0; poisoned = *(volatile u32*)D.poison != 0; }
  if (wid == 1) {
    // Stretches that did not fold: another order than the ranks', unless sixteen records on the rank is mostly the same. Looked at in eight
    // places of such a window, and not by k_seq_range: there it cost every upload 1 us, in the loop 4 % of the pass.
    u32 pairs = 0, changes = 0;
    const u64 n_rec = D.n_rec;
    if (mostly_mixed(mixed, n_rec)) {
      u32 rk[8]; bool in[8];
#pragma unroll
      for (u32 q = 0; q < 8; ++q) { const u64 at = n_rec / 8 * q + lane * REC_PER_THREAD; in[q] = at < n_rec; rk[q] = in[q] ? D.rank[at] : NONE; }
#pragma unroll
      for (u32 q = 0; q < 8; ++q) {
        const u32 before = __shfl_up_sync(0xFFFFFFFFu, rk[q], 1);
        in[q] = in[q] && lane != 0;
        pairs += __popc(__ballot_sync(0xFFFFFFFFu, in[q])); changes += __popc(__ballot_sync(0xFFFFFFFFu, in[q] && rk[q] != before));
      }
    }
    if (lane == 0) s_turns = changes * 2 < pairs;
  }
  const u32 per = ceil_div(R.n_comms, blockDim.x), c_lo = threadIdx.x * per, c_hi = min(R.n_comms, c_lo + per);   // my communicators
  // counters covered and members of my first few communicators stay in registers, all loads issued at once
  u32 c_ns[LAYOUT_CACHED], c_n[LAYOUT_CACHED];
  {
    u32 lo[LAYOUT_CACHED], hi[LAYOUT_CACHED];
#pragma unroll
    for (u32 k = 0; k < LAYOUT_CACHED; ++k) {
      const bool in = c_lo + k < c_hi;
      lo[k] = in ? D.rmin[c_lo + k] : NONE; hi[k] = in ? D.rmax[c_lo + k] : 0; c_n[k] = in ? R.comm_n[c_lo + k] : 1u;
    }
#pragma unroll
    for (u32 k = 0; k < LAYOUT_CACHED; ++k) c_ns[k] = range_len(lo[k], hi[k]);
  }
  const auto each = [&](auto&& f) {                            // f(k, counters covered, members), the same number of steps in every thread
#pragma unroll
    for (u32 k = 0; k < LAYOUT_CACHED; ++k) if (k < per) f(k, c_ns[k], c_n[k]);
    for (u32 k = LAYOUT_CACHED; k < per; ++k) { const bool in = c_lo + k < c_hi; f(k, in ? plan_nseq(D, c_lo + k) : 0u, in ? R.comm_n[c_lo + k] : 1u); }
  };
  // the busiest communicator of the fused classes decides how many chunks there are
  u32 mx = 0;
  each([&](u32, u32 ns, u32 n) { if (comm_class(n) <= 1) mx = max(mx, ns); });
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  const u32 n_warps = blockDim.x / 32;
  if (lane == 0) s_red[wid] = mx;
  for (u32 i = threadIdx.x; i < 2 * CHUNK_MAX; i += blockDim.x) (&s_hist[0][0])[i] = 0;
  if (threadIdx.x == 0) s_fused = 0;
  __syncthreads();
  mx = __reduce_max_sync(0xFFFFFFFFu, lane < n_warps ? s_red[lane] : 0u);
  u32 T = mx ? ceil_div(mx, CHUNK_REF) : 1u;
  T = T > CHUNK_MAX ? CHUNK_MAX : T;
  // sums over my communicators, and their units along the chunks
  PlanAcc mine = {0, 0, 0, 0, 0, 0}; u32 fused = 0;
  each([&](u32, u32 ns, u32 n) {
    mine = plan_add(mine, plan_item(ns, n));
    fused += comm_class(n) <= 1 ? (u32)(((u64)ns * n + 31) / 32) : 0u;
    // communicators of one family have as many units: the lanes that agree are counted, then the lanes run along the chunks
    const u32 units = fused_units(ns, n), key = units * 2 + comm_class(n);
    u32 pend = __ballot_sync(0xFFFFFFFFu, units != 0);
    while (pend) {
      const u32 lead = __shfl_sync(0xFFFFFFFFu, key, (u32)__ffs(pend) - 1u), same = __ballot_sync(0xFFFFFFFFu, units != 0 && key == lead);
      const u32 times = (u32)__popc(same), u = lead >> 1;
      for (u32 tau = lane; tau < T; tau += 32) atomicAdd(&s_hist[lead & 1][tau], times * (units_before(u, T, tau + 1) - units_before(u, T, tau)));
      pend &= ~same;
    }
  });
  fused = __reduce_add_sync(0xFFFFFFFFu, fused);
  if (lane == 0 && fused) atomicAdd(&s_fused, fused);
  // exclusive prefix over the threads
  PlanAcc inc = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) { PlanAcc o = plan_shfl_up(inc, d); if (lane >= (u32)d) inc = plan_add(inc, o); }
  if (lane == 31) s_warp[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    PlanAcc xi = lane < n_warps ? s_warp[lane] : PlanAcc{0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { PlanAcc o = plan_shfl_up(xi, d); if (lane >= (u32)d) xi = plan_add(xi, o); }
    PlanAcc ex = plan_shfl_up(xi, 1);
    if (lane == 0) ex = PlanAcc{0, 0, 0, 0, 0, 0};
    s_warp[lane] = ex;
    if (lane == 31) s_warp[32] = xi;
  }
  __syncthreads();
  PlanAcc run = plan_shfl_up(inc, 1);
  if (lane == 0) run = PlanAcc{0, 0, 0, 0, 0, 0};
  run = plan_add(s_warp[wid], run);
  const PlanAcc all = s_warp[32];
  // first CTA and first warp-tile of every chunk, in warp 0; two chunks per lane
  if (wid == 0) {
    u32 wt[2], c1[2], wt_per_cta;
#pragma unroll
    for (int q = 0; q < 2; ++q) { wt[q] = s_hist[0][2 * lane + q]; c1[q] = s_hist[1][2 * lane + q]; }
    // (gridDim.y: windows of the batch, which are mostly alike)
    const u32 wt_all = __reduce_add_sync(0xFFFFFFFFu, wt[0] + wt[1]);
    wt_per_cta = (u64)wt_all * gridDim.y <= fused_warps ? FUSED_WT_PER_CTA / 2 : FUSED_WT_PER_CTA;
    const u32 a0 = ceil_div(wt[0], wt_per_cta) + c1[0], a1 = ceil_div(wt[1], wt_per_cta) + c1[1];
    u32 pc = a0 + a1, pw = wt[0] + wt[1];                      // CTAs and warp-tiles of my two chunks
    const u32 oc_ = pc, ow_ = pw;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 oc = __shfl_up_sync(0xFFFFFFFFu, pc, d), ow = __shfl_up_sync(0xFFFFFFFFu, pw, d);
      if (lane >= (u32)d) { pc += oc; pw += ow; }
    }
    D.chunks[2 * lane] = make_uint2(pc - oc_, pw - ow_);
    D.chunks[2 * lane + 1] = make_uint2(pc - oc_ + a0, pw - ow_ + wt[0]);
    const u64 n_cta = __shfl_sync(0xFFFFFFFFu, pc, 31), n_wt = __shfl_sync(0xFFFFFFFFu, pw, 31);
    static_assert(CHUNK_MAX == 64, "two chunks per lane");
    if (lane == 31) D.chunks[CHUNK_MAX] = make_uint2(pc, pw);
    // the totals, one per lane
    u64 t = 0;
    t = lane == T_GROUPS ? all.groups : t; t = lane == T_SLOTS ? all.slots : t; t = lane == T_FCTA ? n_cta : t; t = lane == T_FWT ? n_wt : t;
    t = lane == T_FSUM ? all.units : t; t = lane == T_TILES2 ? all.t2 : t; t = lane == T_TILES3 ? all.t3 : t; t = lane == T_ROWS ? all.rows : t;
    t = lane == T_CHUNKS ? T : t; t = lane == T_WT_PER_CTA ? wt_per_cta : t;
    t = lane == T_MIXED ? (s_turns ? 0 : mixed) : t; t = lane == T_FUSED ? s_fused : t;
    // op counters further apart than 2^31, or more slots than the cap: refuse the window
    u64 failed = (all.slots > slot_cap || all.groups > 0x7FFFFFFFull) ? FAILED_CAPACITY : 0;
    if (!failed && expects) {
      const bool same = lane == T_FAILED || lane == T_MIXED || lane >= T_COUNT || t == expected;      // (any order of the records is as good)
      if (!__all_sync(0xFFFFFFFFu, same) || poisoned) { failed = FAILED_EXPECT; if (lane == 0) atomicExch(D.poison, 1u); }
    }
    if (failed) t = lane == T_CHUNKS || lane == T_WT_PER_CTA ? 1 : 0;
    if (lane == T_FAILED) t = failed;
    if (lane < T_COUNT) { D.totals[lane] = t; D.totals_host[lane] = t; }
    if (lane == 0) {
      if (failed == FAILED_CAPACITY) atomicOr((unsigned*)&D.counters[C_ERR], (unsigned)CCLD_E_CAPACITY);
      s_red[0] = failed != 0;
    }
  }
  __syncthreads();
  const bool failed = s_red[0] != 0;                           // a window that is given up leaves no work behind: empty rows
  RangeRow* const ranges = D.ranges; uint4* const srow = D.srow; const u32* const rmin = D.rmin;
  each([&](u32 k, u32 ns, u32 n) {
    const u32 c = c_lo + k;
    if (c >= c_hi) return;
    const PlanAcc it = plan_item(ns, n);
    RangeRow r = {0, 0, 0, n, 0, 0, 0, 0};
    if (!failed) {
      const u32 cls = comm_class(n);
      r.seq_lo = ns ? rmin[c] : 0; r.n_seq = ns; r.row_idx = run.rows; r.group0 = run.groups; r.slot0 = run.slots;
      r.tile0 = cls <= 1 ? run.units : (cls == 2 ? run.t2 : run.t3); r.n_units = it.units + it.t2 + it.t3;
    }
    ranges[c] = r;
    srow[c] = make_uint4((u32)r.slot0, (u32)(r.slot0 >> 32), r.n_seq, r.seq_lo);
    run = plan_add(run, it);
  });
}

// The work lists, written by the first `ctas` CTAs of k_slot_scatter's launch for every window: CTA x takes slice x % slices of
// chunk x / slices, `blocks` times EMIT_THREADS communicators (one time, unless a registry has more than EMIT_SLICES times as
// many). There are enough of them for every chunk of any window of the batch. base[] of the descriptors is filled. A window that
// gave up fills its stretch of the lists with entries that hold no work, because the kernels that follow are launched over the
// expected lengths. Neither the lists nor the scatter reads what the other writes; a launch of its own in between took 4.5
// (one communicator) to 17 us (twelve windows of 1,088 communicators) of every pass.
__device__ __forceinline__ bool gives_up(const WinDesc& D) {
  // the flag can only go up while k_layout runs, so every CTA of the launch sees the same value
  return D.totals[T_FAILED] != 0 || (D.expect != nullptr && *(volatile u32*)D.poison != 0);
}
__device__ __forceinline__ void emit_lists(const WinDesc& D, const Registry& R, const PlanLists& L, u32 ctas, u32 slices, u32 blocks, uint4* s_pair /* a warp's */) {
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (gives_up(D)) {
    if (D.expect == nullptr) return;                           // the host knows: it sized nothing for this window
    const u32 i0 = blockIdx.x * EMIT_THREADS + threadIdx.x, st = ctas * EMIT_THREADS;
    if (D.totals[T_FAILED] == 0) {                             // another window's layout was the surprise: this one's rows go too
      for (u32 c = i0; c < R.n_comms; c += st) { D.ranges[c] = RangeRow{0, 0, 0, R.comm_n[c], 0, 0, 0, 0}; D.srow[c] = make_uint4(0, 0, 0, 0); }
      if (i0 == 0) for (int q = 0; q < T_COUNT; ++q) { const u64 v = q == T_FAILED ? FAILED_EXPECT : 0; D.totals_host[q] = v; }
    }
    const u64 n_cta = D.expect[T_FCTA], n2 = D.expect[T_TILES2], n3 = D.expect[T_TILES3];
    for (u64 j = i0; j < n_cta; j += st) {
      FusedCta x; x.w = blockIdx.y; x.cls = 0; x.c = 0; x.seq_off = 0; x.count = 0; x.sum_idx = 0; x.wt_first = 0; x.wt_count = 0; x.moff = 0;
      x.row = RangeRow{0, 0, 0, 0, 0, 0, 0, 0};
      L.fcta[D.base[B_FCTA] + j] = x;
    }
    const Tile none = {blockIdx.y, 0, 0, 0, RangeRow{0, 0, 0, 0, 0, 0, 0, 0}, 0, 0};
    for (u64 j = i0; j < n2; j += st) L.t2[D.base[B_T2] + j] = none;
    for (u64 j = i0; j < n3; j += st) L.t3[D.base[B_T3] + j] = none;
    return;
  }
  const u32 T = (u32)D.totals[T_CHUNKS], tau = blockIdx.x / slices, slice = blockIdx.x % slices;
  if (tau >= T) return;
  // tiles of classes 2 and 3: a warp per communicator, lanes along its tiles
  for (u32 c = blockIdx.x * (EMIT_THREADS / 32) + wid; c < R.n_comms; c += T * slices * (EMIT_THREADS / 32)) {
    const u32 n = R.comm_n[c], cls = comm_class(n);
    if (cls < 2) continue;
    const RangeRow row = D.ranges[c];
    const u32 S = tile_seqs(n), first = D.base[cls == 2 ? B_T2 : B_T3] + row.tile0;
    Tile* dst = cls == 2 ? L.t2 : L.t3;
    const u64 moff = R.comm_moff[c];
    for (u32 k = lane; k < row.n_units; k += 32) {
      Tile t; t.w = blockIdx.y; t.c = c; t.seq_off = k * S; t.row = row; t.moff = moff; t.pad = 0;
      const u32 left = row.n_seq - k * S; t.count = left < S ? left : S;
      dst[first + k] = t;
    }
  }
  // fused classes: the units of this chunk that earlier slices hold, those of my communicator, then where they go
  const auto units_of = [&](u32 c, u32& wt, u32& c1) {
    const u32 n = R.comm_n[c], cls = comm_class(n), all = cls <= 1 ? fused_units(D.srow[c].z, n) : 0u;
    const u32 u = units_before(all, T, tau + 1) - units_before(all, T, tau);
    if (cls == 0) wt += u; else c1 += u;
  };
  const uint2 here = D.chunks[tau], next = D.chunks[tau + 1];
  const u32 wt_base = D.base[B_FWT] + here.y, wt_total = next.y - here.y, cta_base = D.base[B_FCTA] + here.x, per_cta = (u32)D.totals[T_WT_PER_CTA], n0 = ceil_div(wt_total, per_cta);
  u32 ew = 0, ec = 0;                                          // this thread's share of what lies before
#pragma unroll 4
  for (u32 k = 0; k < slice * blocks; ++k) units_of(k * EMIT_THREADS + threadIdx.x, ew, ec);
  for (u32 m = 0; m < blocks; ++m) {
    const u32 c = (slice * blocks + m) * EMIT_THREADS + threadIdx.x;
    u32 wt = 0, c1 = 0;
    if (c < R.n_comms) units_of(c, wt, c1);
    u32 iw = wt, ic = c1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 ow = __shfl_up_sync(0xFFFFFFFFu, iw, d), oc = __shfl_up_sync(0xFFFFFFFFu, ic, d);
      if (lane >= (u32)d) { iw += ow; ic += oc; }
    }
    const u32 rw = __reduce_add_sync(0xFFFFFFFFu, ew), rc = __reduce_add_sync(0xFFFFFFFFu, ec);
    if (lane == 31) s_pair[wid] = make_uint4(iw, ic, rw, rc);
    __syncthreads();
    u32 bw = 0, bc = 0;                                        // before my warp: all that came earlier, and the warps before mine
#pragma unroll
    for (u32 q = 0; q < EMIT_THREADS / 32; ++q) { const uint4 x = s_pair[q]; bw += x.z; bc += x.w; if (q < wid) { bw += x.x; bc += x.y; } }
    u32 at_w = wt_base + bw + iw - wt, at_c = cta_base + n0 + bc + ic - c1;      // class-1 CTAs come after the chunk's class-0 CTAs
    if (wt + c1 != 0) {
      const u32 n = R.comm_n[c], cls = comm_class(n);
      const RangeRow row = D.ranges[c];
      const u64 moff = R.comm_moff[c];
      const u32 U = tile_seqs(n), first = units_before(fused_units(row.n_seq, n), T, tau);
      const u32 sum0 = D.base[B_FSUM] + row.tile0 + first;
      for (u32 k = 0; k < wt + c1; ++k) {
        const u32 off = (first + k) * U, len = min(U, row.n_seq - off);
        if (cls == 0) { WarpTile x; x.c = c; x.seq_off = off; x.count = len; x.sum_idx = sum0 + k; x.row = row; x.moff = moff; L.fwt[at_w++] = x; }
        else { FusedCta x; x.w = blockIdx.y; x.cls = 1; x.c = c; x.seq_off = off; x.count = len; x.sum_idx = sum0 + k; x.wt_first = 0; x.wt_count = 0;
               x.row = row; x.moff = moff; L.fcta[at_c++] = x; }
      }
    }
    ew += wt; ec += c1;
    __syncthreads();
  }
  for (u32 j = slice * EMIT_THREADS + threadIdx.x; j < n0; j += slices * EMIT_THREADS) {
    FusedCta x; x.w = blockIdx.y; x.cls = 0; x.c = 0; x.seq_off = 0; x.count = 0; x.sum_idx = 0; x.moff = 0;
    x.row = RangeRow{0, 0, 0, 0, 0, 0, 0, 0};
    x.wt_first = wt_base + per_cta * j; x.wt_count = min(per_cta, wt_total - per_cta * j);
    L.fcta[cta_base + j] = x;
  }
}

}  // namespace ccld
