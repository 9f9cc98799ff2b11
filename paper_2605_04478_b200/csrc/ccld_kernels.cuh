// Kernels of the CCL-D analyzer hot path for sm_100a. Everything the analysis computes runs here;
// the host side only sizes buffers and launches.
//
//   k_seq_range     group-by, part 1: op-counter range per (window, communicator)
//   k_layout        group-by, part 2: closed-form slot layout (prefix sums over communicators; ccld_plan.cuh)
//   k_slot_scatter  group-by, part 3: perm[slot] = record index; beside it the work lists of the reduction kernels
//   k_slot_pack     the same for uploads whose records are not in their ranks' order: the record itself goes along
//   k_reduce_fused  per-op reductions + median/MAD + flags + votes for n <= 128, chunk-major work list:
//                   n <= 8 one thread per group (warp-tiles), 9 <= n <= 128 n_pad / 8 lanes per group (register /
//                   shuffle bitonic network); complete groups whose times fit 32-bit offsets
//   k_reduce_deferred  the groups k_reduce_fused sets aside (incomplete, in flight, 64-bit spreads)
//   k_reduce_mid    same, 129 <= n <= 1024 (ccld_mid.cuh: tiles of 8 op counters staged in shared memory, a warp per group)
//   k_reduce_large  same, n > 1024 (ccld_large.cuh: a cluster of eight CTAs per tile of 8 op counters)
//   k_reduce_large_deferred  the groups k_reduce_mid and k_reduce_large set aside
//   k_window_rounds Eq. 2 per (communicator, window): round counts, selected round, location candidates
//   k_window_decide Eq. 1, 3, 4 per communicator, windows in order: baseline state, class, slow location
//   k_hang_locate   hang decision tree over presence / completion / progress counters (ccld_hang.cuh)
// The suspect list and the ordered output lists are in ccld_verdict.cuh.
#pragma once
#include "ccld_device.cuh"
#include "ccld_plan.cuh"

namespace ccld {

// ------------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ u32 hash_home(const Registry& R, u32 id) { return (id * 2654435761u) & R.hash_mask; }

// Continues a probe sequence whose first entry (at the home slot) the caller already holds.
__device__ __forceinline__ uint4 comm_find(const Registry& R, u32 id, uint4 e) {
  u32 h = hash_home(R, id);
  for (u32 probe = 0; probe <= R.hash_mask; ++probe) {
    if (e.y == NONE || e.x == id) return e;
    h = (h + 1) & R.hash_mask;
    e = R.hash[h];
  }
  return make_uint4(0, NONE, 0, 0);
}

__device__ __forceinline__ u32 comm_lookup(const Registry& R, u32 id) { return comm_find(R, id, R.hash[hash_home(R, id)]).y; }

__device__ __forceinline__ u32 pos_lookup(const Registry& R, u32 rank, u32 c) {
  if (rank >= R.n_ranks) return NONE;
  u32 b = R.rank_ptr[rank], e = R.rank_ptr[rank + 1];
  for (u32 i = b; i < e; ++i)
    if (R.ent_comm[i] == c) return R.ent_pos[i];
  return NONE;
}

// a * ka > b * kb in exact 128-bit arithmetic
__device__ __forceinline__ bool mul_gt(u64 a, u32 ka, u64 b, u32 kb) {
  u64 alo = a * ka, ahi = __umul64hi(a, (u64)ka);
  u64 blo = b * kb, bhi = __umul64hi(b, (u64)kb);
  return ahi > bhi || (ahi == bhi && alo > blo);
}
__device__ __forceinline__ bool mul_lt(u64 a, u32 ka, u64 b, u32 kb) { return mul_gt(b, kb, a, ka); }

// bus-bandwidth factor num/den of an op over n ranks
__device__ __forceinline__ void bus_factor(u32 op, u32 n, double* num, double* den) {
  if (op == CCLD_OP_ALLREDUCE) { *num = 2.0 * (double)(n - 1); *den = (double)n; }
  else if (op == CCLD_OP_ALLGATHER || op == CCLD_OP_REDUCESCATTER || op == CCLD_OP_ALLTOALL) { *num = (double)(n - 1); *den = (double)n; }
  else { *num = 1.0; *den = 1.0; }
}
__device__ __forceinline__ double busbw(double bytes_num, double den, i64 t) {
  return t > 0 ? bytes_num / ((double)t * den) : 0.0;
}

__device__ __forceinline__ u64 absdiff(u64 a, u64 b) { return a >= b ? a - b : b - a; }

// Where the record index of (communicator row, op-counter offset, ring position) sits in `perm`. The permutation
// is member-major inside a communicator - [position][op counter] - so that consecutive records of one rank, which
// carry consecutive op counters, scatter to consecutive entries, and so that a warp reading 32 consecutive op
// counters of one member reads 128 contiguous bytes. Flags and per-op rows stay group-major.
__device__ __forceinline__ u64 perm_at(const RangeRow& row, u32 seq_off, u32 pos) { return row.slot0 + (u64)pos * row.n_seq + seq_off; }

__device__ __forceinline__ u64 shfl_xor64(u64 v, int m) { return __shfl_xor_sync(0xFFFFFFFFu, v, m); }

__device__ __forceinline__ void count_add(u64* counters, int which, u32 v) {
  if (v) atomicAdd((ull*)&counters[which], (ull)v);
}

__device__ __forceinline__ void raise_alert(const WinDesc& D, u32 comm_id, u32 seq, i64 age) {
  ull k = atomicAdd((ull*)&D.counters[C_ALERTS], 1ull);
  if (k < CCLD_MAX_ALERTS_PER_WINDOW) { ccld_hang_alert a; a.comm = comm_id; a.seq = seq; a.age_ns = age; D.alerts[k] = a; }
}

// Eq. 2 candidate merge: larger range wins, then the earlier op counter (k = NONE means "no round")
__device__ __forceinline__ void best_merge(u64& rng, u32& k, u64 o_rng, u32 o_k) {
  if (o_k != NONE && (k == NONE || o_rng > rng || (o_rng == rng && o_k < k))) { rng = o_rng; k = o_k; }
}
__device__ __forceinline__ void best_warp_reduce(u64& rng, u32& k) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const u64 o_rng = shfl_xor64(rng, d); const u32 o_k = __shfl_xor_sync(0xFFFFFFFFu, k, d);
    best_merge(rng, k, o_rng, o_k);
  }
}

// ------------------------------------------------------------------------------------------------
// record-streaming kernels (group-by parts 1 and 3)
// ------------------------------------------------------------------------------------------------
constexpr int REC_RUN = REC_PER_CTA / REC_THREADS;       // consecutive records per thread

__device__ __forceinline__ void range_widen(const WinDesc& D, u32 c, u32 mn, u32 mx) {
  if (mn < __ldcg(&D.rmin[c])) atomicMin(&D.rmin[c], mn);
  if (mx > __ldcg(&D.rmax[c])) atomicMax(&D.rmax[c], mx);
}

// A CTA keeps the op-counter extremes of every communicator it meets in a shared-memory table indexed by the
// communicator's registry index (registries of up to RANGE_DIRECT communicators; beyond that updates go to global
// memory, checked before each atomic) and merges the entries it touched into the window's global ranges at the end.
constexpr u32 RANGE_DIRECT = 4096;
inline size_t range_smem_bytes(u32 n_comms) { return n_comms <= RANGE_DIRECT ? (size_t)8 * n_comms : 0; }

__device__ __forceinline__ void range_put(const WinDesc& D, u32* s_mn, u32* s_mx, u32 c, u32 mn, u32 mx) {
  if (s_mn != nullptr) { atomicMin(&s_mn[c], mn); atomicMax(&s_mx[c], mx); }
  else range_widen(D, c, mn, mx);
}

// ---- group-by, part 1: which op counters does every communicator cover in every window ----
// A thread takes a run of REC_RUN consecutive records. A rank's stream alternates between a handful of communicators, so
// the thread folds its run in registers, one distinct communicator at a time (up to RANGE_FOLDS of them), and the warp
// then merges what its lanes found - in a rank-major upload all lanes meet the same few communicators - so that one lane
// updates the CTA's table per communicator. Records left over after the folds (an upload in arrival or random order)
// look their communicator up and update the table themselves: one registry lookup and two shared-memory atomics per
// record at worst.
constexpr int RANGE_FOLDS = 4;
constexpr int RANGE_WARP_FOLDS = 8;
constexpr u32 RANGE_BLOCKS_MAX = 16;                  // blocks of REC_PER_CTA records a CTA takes at most (the host takes fewer for small batches)

// cid[i] for the lowest i with bit i of `left` set (any element if left is 0)
__device__ __forceinline__ u32 first_left(const u32 (&cid)[REC_RUN], u32 left) {
  static_assert(REC_RUN == 16, "selection tree over a run of 16");
  const u32 b = (u32)__ffs(left) - 1u;
  u32 x8[8], x4[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) x8[i] = (b & 8u) ? cid[8 + i] : cid[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) x4[i] = (b & 4u) ? x8[4 + i] : x8[i];
  const u32 y0 = (b & 2u) ? x4[2] : x4[0], y1 = (b & 2u) ? x4[3] : x4[1];
  return (b & 1u) ? y1 : y0;
}

// fill: whether the slot table, sized from what the host expects, is to be set to NONE as well. The stores run under the pass,
// which issues instructions most of the time (FILL_BESIDE).
__global__ void __launch_bounds__(REC_THREADS) k_seq_range(const WinDesc* wd, Registry R, u32 blocks_per_cta, int fill) {
  begin_after();
  extern __shared__ u32 s_dyn[];
  u32* const s_mn = R.n_comms <= RANGE_DIRECT ? s_dyn : nullptr;
  u32* const s_mx = R.n_comms <= RANGE_DIRECT ? s_dyn + R.n_comms : nullptr;
  const WinDesc& D = wd[blockIdx.y];                          // grid: (CTAs of the largest window, windows)
  const u64 n_rec = D.n_rec; const u32* const c_comm = D.comm; const u32* const c_seq = D.seq;
  if ((u64)blockIdx.x * blocks_per_cta * REC_PER_CTA >= n_rec) return;
  const u32 lane = threadIdx.x & 31;
  if (fill) fill_slots(D.perm, D.n_slots, blockIdx.x, (u32)((n_rec + blocks_per_cta * REC_PER_CTA - 1) / (blocks_per_cta * REC_PER_CTA)));
  if (s_mn != nullptr) {
    for (u32 c = threadIdx.x; c < R.n_comms; c += REC_THREADS) { s_mn[c] = NONE; s_mx[c] = 0; }
    __syncthreads();
  }
  u32 mixed = 0;                                             // stretches of 32 runs that the warp could not fold
  // a CTA takes blocks_per_cta consecutive blocks of the window, one after the other, and keeps one table for them: the
  // table's set-up, its barriers and its merge into the window's ranges are paid once
  for (u32 blk = 0; blk < blocks_per_cta; ++blk) {
    const u64 first = ((u64)blockIdx.x * blocks_per_cta + blk) * REC_PER_CTA;
    if (first >= n_rec) break;
    const u32 n_valid = n_rec - first < REC_PER_CTA ? (u32)(n_rec - first) : (u32)REC_PER_CTA;
    const u32 r0 = threadIdx.x * REC_RUN;
    const u32 len = r0 >= n_valid ? 0u : (n_valid - r0 < REC_RUN ? n_valid - r0 : (u32)REC_RUN);
    // the run goes straight into registers: four 128-bit loads per column where the column allows it
    u32 cid[REC_RUN], sq[REC_RUN];
    {
      const u32* __restrict__ pc = c_comm + first + r0; const u32* __restrict__ ps = c_seq + first + r0;
      if (len == REC_RUN && ((reinterpret_cast<uintptr_t>(pc) | reinterpret_cast<uintptr_t>(ps)) & 15) == 0) {
  #pragma unroll
        for (int q = 0; q < REC_RUN / 4; ++q) {
          const uint4 a = __ldg(reinterpret_cast<const uint4*>(pc) + q), b = __ldg(reinterpret_cast<const uint4*>(ps) + q);
          cid[4 * q] = a.x; cid[4 * q + 1] = a.y; cid[4 * q + 2] = a.z; cid[4 * q + 3] = a.w;
          sq[4 * q] = b.x; sq[4 * q + 1] = b.y; sq[4 * q + 2] = b.z; sq[4 * q + 3] = b.w;
        }
      } else {
  #pragma unroll
        for (int k = 0; k < REC_RUN; ++k) { cid[k] = (u32)k < len ? pc[k] : NONE; sq[k] = (u32)k < len ? ps[k] : 0u; }
      }
    }
    // records of the run not yet accounted for; a run cut short by the end of the window skips the folds (its padding
    // would match a record that names communicator 0xFFFFFFFF) and goes record by record
    const u32 tail = len < REC_RUN ? (1u << len) - 1u : 0u;
    u32 left = len < REC_RUN ? 0u : (1u << REC_RUN) - 1u;
    // warp folds: in a rank-major upload the 32 runs of a warp belong to one or two ranks, so all lanes meet the same few
    // communicators. One of them at a time - the communicator of the first record left in the lowest lane that has one -
    // is folded by every lane and reduced over the warp, and lane 0 updates the table once. The stage ends as soon as a
    // fold clears less than an eighth of what was left (an upload in another order): the lanes then fold on their own.
    {
      u32 remaining = __reduce_add_sync(0xFFFFFFFFu, (u32)__popc(left));
      for (int f = 0; f < RANGE_WARP_FOLDS && remaining != 0; ++f) {
        const u32 have = __ballot_sync(0xFFFFFFFFu, left != 0);
        const u32 id = __shfl_sync(0xFFFFFFFFu, first_left(cid, left), (u32)__ffs(have) - 1u);
        const uint4 h = comm_find(R, id, R.hash[hash_home(R, id)]);        // the same in every lane
        u32 m = 0, mn = NONE, mx = 0;
  #pragma unroll
        for (int k = 0; k < REC_RUN; ++k) {
          if (cid[k] == id) { m |= 1u << k; mn = min(mn, sq[k]); mx = max(mx, sq[k]); }
        }
        m &= left;                                             // a run cut short holds padding and takes no part
        u32 a = __reduce_min_sync(0xFFFFFFFFu, m ? mn : NONE), b = __reduce_max_sync(0xFFFFFFFFu, m ? mx : 0u);
        if (h.y != NONE && a < h.z) {
          // counters below the communicator's first name no operation: fold again without them
          mn = NONE; mx = 0;
  #pragma unroll
          for (int k = 0; k < REC_RUN; ++k) if (((m >> k) & 1u) && sq[k] >= h.z) { mn = min(mn, sq[k]); mx = max(mx, sq[k]); }
          a = __reduce_min_sync(0xFFFFFFFFu, mn); b = __reduce_max_sync(0xFFFFFFFFu, mx);
        }
        if (lane == 0 && h.y != NONE && a <= b) range_put(D, s_mn, s_mx, h.y, a, b);
        left &= ~m;
        const u32 cleared = __reduce_add_sync(0xFFFFFFFFu, (u32)__popc(m));
        const bool worth = cleared * 8u >= remaining;
        remaining -= cleared;
        if (!worth) break;
      }
      mixed += remaining > 32 * REC_RUN / 2 ? 1u : 0u;
    }
    // folds: the communicator of the first record still left takes every record of the run that names it
    for (int f = 0; f < RANGE_FOLDS && __any_sync(0xFFFFFFFFu, left != 0); ++f) {
      const bool act = left != 0;
      u32 id = NONE;
  #pragma unroll
      for (int k = REC_RUN - 1; k >= 0; --k) id = (left >> k) & 1u ? cid[k] : id;
      uint4 h = make_uint4(0, NONE, 0, 0);                      // (id, index, first counter, members); index NONE: unregistered
      if (act) h = comm_find(R, id, R.hash[hash_home(R, id)]);
      // a record folded earlier carries another id, so matching the id is enough (the run is complete: no padding)
      u32 m = 0, mn = NONE, mx = 0;
  #pragma unroll
      for (int k = 0; k < REC_RUN; ++k) {
        if (cid[k] == id) { m |= 1u << k; mn = min(mn, sq[k]); mx = max(mx, sq[k]); }
      }
      m &= left;
      if (h.y != NONE && m != 0 && mn < h.z) {
        // counters below the communicator's first name no operation: fold again without them
        mn = NONE; mx = 0;
  #pragma unroll
        for (int k = 0; k < REC_RUN; ++k) if (((m >> k) & 1u) && sq[k] >= h.z) { mn = min(mn, sq[k]); mx = max(mx, sq[k]); }
      }
      if (m == 0) { mn = NONE; mx = 0; }
      left &= ~m;
      // lanes that hold the same communicator merge: a few rounds, each led by the lowest lane still waiting
      bool mine = act && h.y != NONE && mn <= mx;
      u32 pend = __ballot_sync(0xFFFFFFFFu, mine);
      for (int it = 0; it < RANGE_FOLDS && pend; ++it) {
        const u32 leader = (u32)__ffs(pend) - 1u;
        const u32 lid = __shfl_sync(0xFFFFFFFFu, h.y, leader);
        const bool same = mine && h.y == lid;
        const u32 a = __reduce_min_sync(0xFFFFFFFFu, same ? mn : NONE), b = __reduce_max_sync(0xFFFFFFFFu, same ? mx : 0u);
        if (lane == leader) range_put(D, s_mn, s_mx, lid, a, b);
        if (same) mine = false;
        pend &= ~__ballot_sync(0xFFFFFFFFu, same);
      }
      if (mine) range_put(D, s_mn, s_mx, h.y, mn, mx);
    }
    // every record still left: one lookup each, four in flight
    left |= tail;
    if (left != 0) {
  #pragma unroll
      for (int k0 = 0; k0 < REC_RUN; k0 += 4) {
        uint4 h[4]; bool need[4];
  #pragma unroll
        for (int q = 0; q < 4; ++q) {
          need[q] = ((left >> (k0 + q)) & 1u) != 0;
          h[q] = need[q] ? R.hash[hash_home(R, cid[k0 + q])] : make_uint4(0, NONE, 0, 0);
        }
  #pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (!need[q]) continue;
          const uint4 e = comm_find(R, cid[k0 + q], h[q]);
          if (e.y != NONE && sq[k0 + q] >= e.z) range_put(D, s_mn, s_mx, e.y, sq[k0 + q], sq[k0 + q]);
        }
      }
    }
  }
  if (lane == 0) count_add(D.counters, C_MIXED, mixed);
  if (s_mn == nullptr) return;
  __syncthreads();
  u32* const rmin = D.rmin; u32* const rmax = D.rmax;
  for (u32 c = threadIdx.x; c < R.n_comms; c += REC_THREADS) {
    const u32 mn = s_mn[c];
    if (mn != NONE) { atomicMin(&rmin[c], mn); atomicMax(&rmax[c], s_mx[c]); }      // nothing waits for these
  }
}

// ------------------------------------------------------------------------------------------------
// group-by, part 3: every accepted record drops its index into its slot.
// ------------------------------------------------------------------------------------------------
// Registry walk for a record whose (rank, communicator) pair is not inline: returns index << 13 | position in the
// low word, or NONE there with the rejecting CCLD_E_* bit in the high word.
constexpr int SCAT_THREADS = 256;     // lanes on consecutive records: the stores of a warp land close together
constexpr int SCAT_PER_THREAD = 12;    // records per thread: enough to spread the two dependent table reads a warp starts with
constexpr int SCAT_PER_CTA = SCAT_THREADS * SCAT_PER_THREAD;
constexpr u32 SCAT_BLOCKS_MAX = 8;    // blocks of SCAT_PER_CTA records a CTA takes at most

__device__ __noinline__ u64 resolve_slow(const Registry& R, u32 rank, u32 cid) {
  const u32 c = comm_lookup(R, cid);
  if (c == NONE) return ((u64)CCLD_E_UNKNOWN_COMM << 32) | NONE;
  const u32 pos = pos_lookup(R, rank, c);
  if (pos == NONE) return ((u64)CCLD_E_NOT_MEMBER << 32) | NONE;
  return (c << RANK_TAB_POS_BITS) | pos;
}

// Where the record (rank, communicator id, op counter) goes, given the communicator's index c, the member's position
// and the scatter row of c. Returns false if nothing is stored; *err / *rej / *internal collect what went wrong.
__device__ __forceinline__ bool scatter_slot(const Registry& R, u32 c, u32 ns, u32 lo, u64 base_pos, u32 sq, u64 n_slots, u64* slot,
                                             u32* err, u32* rej, u32* internal) {
  if (ns == 0 || sq < lo) {
    if (sq < R.comm_seq0[c]) { *err |= CCLD_E_SEQ_RANGE; ++*rej; }
    else if (ns != 0) *internal = 1;
    return false;
  }
  *slot = base_pos + (sq - lo);
  if (sq - lo >= ns || *slot >= n_slots) { *internal = 1; return false; }
  return true;
}

// What the lanes of a warp found wrong with their records.
__device__ __forceinline__ void count_rejects(const WinDesc& D, u32 err, u32 rej, u32 internal) {
  err = __reduce_or_sync(0xFFFFFFFFu, err);
  rej = __reduce_add_sync(0xFFFFFFFFu, rej);
  internal = __reduce_or_sync(0xFFFFFFFFu, internal);
  if ((threadIdx.x & 31) == 0) {
    if (err) atomicOr((unsigned*)&D.counters[C_ERR], err);
    count_add(D.counters, C_REJECTED, rej);
    if (internal) atomicOr((unsigned*)&D.counters[C_INTERNAL], 1u);
  }
}

constexpr u32 SCAT_LOCAL = 8;     // ranks, counted from the rank of the CTA's first record, whose table rows a CTA resolves once
static_assert(SCAT_THREADS == EMIT_THREADS, "CTAs of both kinds in one launch");

// A CTA's records mostly belong to a few neighbouring ranks (a rank-major upload: one or two), so each warp first resolves
// the inline pairs of SCAT_LOCAL ranks - communicator id -> (counters covered, first counter, slot of the member's
// first counter) - against the window's scatter rows into shared memory; a record of those ranks then needs no global table at all and, in windows of
// fewer than 2^32 slots, only 32-bit arithmetic. Any other record (another rank, a communicator beyond the inline pairs,
// a counter outside the range, a rejected record) takes the two dependent table loads and the full checks.
// Grid: (emitting CTAs + CTAs of the largest window, windows).
__global__ void __launch_bounds__(SCAT_THREADS, 4) k_slot_scatter(const WinDesc* wd, Registry R, PlanLists L, u32 emit_ctas, u32 slices, u32 slice_blocks, u32 blocks_per_cta) {
  begin_after();
  // (communicator id, counters covered, first counter, first slot) per resolved pair; counters covered 0: unused. Every
  // warp keeps its own copy, so no warp waits for another; two copies, because the entries of the next block are written
  // while lanes may still read those of the current one.
  __shared__ uint4 s_ent_all[2][SCAT_THREADS / 32][SCAT_LOCAL * RANK_TAB_K];
  static_assert(SCAT_LOCAL * RANK_TAB_K == 32, "one resolved pair per lane");
  const WinDesc& D = wd[blockIdx.y];
  if (blockIdx.x < emit_ctas) { emit_lists(D, R, L, emit_ctas, slices, slice_blocks, &s_ent_all[0][0][0]); return; }
  const u64 base0 = (u64)(blockIdx.x - emit_ctas) * blocks_per_cta * SCAT_PER_CTA;
  if (base0 >= D.n_rec) return;
  // a window that was refused has empty scatter rows: nothing is stored, and what it rejects is counted. The rows of one that gives up
  // because of another window are being cleared: it is left alone and will be analysed again. (Read here, looked at when the first
  // records have arrived.)
  const u64 failed = D.totals[T_FAILED]; const u32 poisoned = *(volatile u32*)D.poison; const bool expects = D.expect != nullptr;
  u32 err = 0, rej = 0, internal = 0;
  // descriptor fields in registers: the stores below could alias the descriptor as far as the compiler knows
  u32* const perm = D.perm; const u64 n_slots = D.n_slots; const uint4* const srow = D.srow; const u64 n_rec = D.n_rec;
  const u32 *c_rank = D.rank, *c_comm = D.comm, *c_seq = D.seq;
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // lane's inline pair (communicator id, index and position) of the SCAT_LOCAL ranks that start at rank r0, and the scatter row it names
  auto pair_of = [&](u32 r0) {
    const u32 r = r0 + lane / RANK_TAB_K;
    return r0 < R.n_ranks && r < R.n_ranks ? reinterpret_cast<const uint2*>(R.rank_tab)[(u64)r * RANK_TAB_K + lane % RANK_TAB_K] : make_uint2(NONE, NONE);
  };
  auto row_of = [&](uint2 p) { return p.x != NONE && p.y < RANK_TAB_OVERFLOW ? srow[p.y >> RANK_TAB_POS_BITS] : make_uint4(0, 0, 0, 0); };
  // The member's column starts at the communicator's first slot + position * counters covered. Only where slots fit 32 bits and the
  // whole column lies inside the table; other pairs stay unused, and so that they match no record they carry no communicator's id.
  auto resolve = [&](uint2 p, uint4 sr) {
    const u64 b = ((u64)sr.x | ((u64)sr.y << 32)) + (u64)(p.y & ((1u << RANK_TAB_POS_BITS) - 1)) * sr.z;
    return sr.z != 0 && n_slots <= 0xFFFFFFFFull && b + sr.z <= n_slots ? make_uint4(p.x, sr.z, sr.w, (u32)b) : make_uint4(NONE, 0, 0, 0);
  };
  // A CTA takes blocks_per_cta consecutive blocks. The chain "first record's rank -> that rank's pairs -> their rows" of a
  // block is started one block ahead, so a block waits for its records only.
  u32 r_first = c_rank[base0];
  uint2 p_mine = pair_of(r_first);
  uint4 row_mine = row_of(p_mine);
  for (u32 blk = 0; blk < blocks_per_cta; ++blk) {
    const u64 base = base0 + (u64)blk * SCAT_PER_CTA;
    if (base >= n_rec) break;
    u32 rk[SCAT_PER_THREAD], cid[SCAT_PER_THREAD], sq[SCAT_PER_THREAD];
    u32 todo = 0;                                             // records that still need placing
#pragma unroll
    for (int k = 0; k < SCAT_PER_THREAD; ++k) {
      const u64 i = base + (u64)k * SCAT_THREADS + threadIdx.x;
      const bool in = i < n_rec;
      rk[k] = in ? c_rank[i] : 0u; cid[k] = in ? c_comm[i] : 0u; sq[k] = in ? c_seq[i] : 0u;
      if (in) todo |= 1u << k;
    }
    const u64 base_next = base + SCAT_PER_CTA;
    const bool has_next = blk + 1 < blocks_per_cta && base_next < n_rec;
    const u32 r_next = has_next ? c_rank[base_next] : NONE;   // in flight with the records
    uint4* const s_ent = s_ent_all[blk & 1][wid];
    s_ent[lane] = resolve(p_mine, row_mine);
    __syncwarp();
    if (failed == 0 && expects && poisoned) return;           // the same in the whole launch
    p_mine = pair_of(r_next);                                 // the next block's pairs: its first rank has arrived with this block's records
#pragma unroll
    for (int k = 0; k < SCAT_PER_THREAD; ++k) {
      const u32 dr = rk[k] - r_first;
      if (dr < SCAT_LOCAL) {
        const uint4* ent = s_ent + dr * RANK_TAB_K;
        uint4 e = ent[0];
#pragma unroll
        for (int q = 1; q < RANK_TAB_K; ++q) { const uint4 x = ent[q]; if (x.x == cid[k]) e = x; }
        const u32 off = sq[k] - e.z;                          // below the first counter: wraps to a huge value
        if (e.x == cid[k] && off < e.y && ((todo >> k) & 1u)) {
          perm[e.w + off] = (u32)base + (u32)k * SCAT_THREADS + threadIdx.x;
          todo &= ~(1u << k);
        }
      }
    }
    row_mine = row_of(p_mine);
    if (__any_sync(0xFFFFFFFFu, todo != 0)) {
#pragma unroll
      for (int k = 0; k < SCAT_PER_THREAD; ++k) {
        if (!((todo >> k) & 1u)) continue;
        u32 v = NONE;
        if (rk[k] < R.n_ranks) {
          const uint4 ta = R.rank_tab[(u64)rk[k] * 2], tb = R.rank_tab[(u64)rk[k] * 2 + 1];
          v = ta.x == cid[k] ? ta.y : v; v = ta.z == cid[k] ? ta.w : v;
          v = tb.x == cid[k] ? tb.y : v; v = tb.z == cid[k] ? tb.w : v;
        }
        if (v == NONE || v == RANK_TAB_OVERFLOW || cid[k] == NONE) {
          const u64 rs = resolve_slow(R, rk[k], cid[k]);
          v = (u32)rs;
          if (rs >> 32) { err |= (u32)(rs >> 32); ++rej; }
        }
        if (v == NONE) continue;
        const u32 c = v >> RANK_TAB_POS_BITS;
        const uint4 sr = srow[c];
        u64 slot;
        if (scatter_slot(R, c, sr.z, sr.w, ((u64)sr.x | ((u64)sr.y << 32)) + (u64)(v & ((1u << RANK_TAB_POS_BITS) - 1)) * sr.z, sq[k], n_slots, &slot, &err, &rej, &internal))
          perm[slot] = (u32)(base + (u64)k * SCAT_THREADS + threadIdx.x);
      }
    }
    r_first = r_next;
  }
  count_rejects(D, err, rej, internal);
}


// The same where the upload has its records in another order (see PackedRecord): few of them belong to the ranks a CTA would resolve,
// so every record takes the two table loads, and its values, which the reading of the columns brings along whole, go to the slot
// with its index. Two windows of 4,096 ranks in arrival order, 8.2 M records: 232 us, and the fused kernel 98 (48 bytes of tables per record from
// L1 or L2, 36 bytes to random sectors), where indices alone take 129 and the gathers 252; 0.5 M records each of 512 ranks 35 and 19, 24 and 36. In
// rank-major order it is the other way round (a record read and written twice, 109 instead of 79 bytes).
// Two records per thread with their values asked for together with the keys; four with the values asked for last took 219, one 283.
constexpr int PACK_PER_THREAD = 2;
constexpr int PACK_PER_CTA = SCAT_THREADS * PACK_PER_THREAD;
// Read once: these leave L1 to the tables.
__device__ __forceinline__ u32 load_once(const u32* p) { u32 v; asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ u64 load_once(const u64* p) { u64 v; asm volatile("ld.global.L1::no_allocate.u64 %0, [%1];" : "=l"(v) : "l"(p)); return v; }
__device__ __forceinline__ u32 load_once(const u8* p) { u32 v; asm volatile("ld.global.L1::no_allocate.u8 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__global__ void __launch_bounds__(SCAT_THREADS, 4) k_slot_pack(const WinDesc* wd, Registry R, PlanLists L, u32 emit_ctas, u32 slices, u32 slice_blocks) {
  begin_after();
  __shared__ uint4 s_pair[EMIT_THREADS / 32];
  const WinDesc& D = wd[blockIdx.y];
  if (blockIdx.x < emit_ctas) { emit_lists(D, R, L, emit_ctas, slices, slice_blocks, s_pair); return; }
  const u64 base = (u64)(blockIdx.x - emit_ctas) * PACK_PER_CTA + threadIdx.x, n_rec = D.n_rec, n_slots = D.n_slots;
  if (base - threadIdx.x >= n_rec) return;
  const u64 failed = D.totals[T_FAILED]; const u32 poisoned = *(volatile u32*)D.poison; const bool expects = D.expect != nullptr;
  u32* const perm = D.perm; uint4* const packed = D.packed; const uint4* const srow = D.srow;
  u32 err = 0, rej = 0, internal = 0, rk[PACK_PER_THREAD], cid[PACK_PER_THREAD], sq[PACK_PER_THREAD], v[PACK_PER_THREAD];
  PackedRecord r[PACK_PER_THREAD];
  {
    const u32 *c_rank = D.rank, *c_comm = D.comm, *c_seq = D.seq, *c_sc = D.send_chg, *c_rc = D.recv_chg;
    const u64 *c_te = (const u64*)D.t_enter, *c_tx = (const u64*)D.t_exit, *c_by = D.bytes; const u8* c_op = D.op;
#pragma unroll
    for (int k = 0; k < PACK_PER_THREAD; ++k) {
      const u64 i = min(base + (u64)k * SCAT_THREADS, n_rec - 1);          // beyond the end: not looked at
      rk[k] = load_once(c_rank + i); cid[k] = load_once(c_comm + i); sq[k] = load_once(c_seq + i);
    }
#pragma unroll
    for (int k = 0; k < PACK_PER_THREAD; ++k) {
      const u64 i = min(base + (u64)k * SCAT_THREADS, n_rec - 1);
      r[k].te = load_once(c_te + i); r[k].tx = load_once(c_tx + i); r[k].by = load_once(c_by + i); r[k].op = load_once(c_op + i); r[k].ch = 0;
      if (c_sc != nullptr) { const u32 sc = load_once(c_sc + i), rc = load_once(c_rc + i); r[k].ch = max(sc, rc); }
    }
  }
#pragma unroll
  for (int k = 0; k < PACK_PER_THREAD; ++k) {
    v[k] = NONE;
    if (rk[k] < R.n_ranks) {
      u32 t[8];
      asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7]) : "l"(R.rank_tab + (u64)rk[k] * 2));
#pragma unroll
      for (int q = 0; q < RANK_TAB_K; ++q) v[k] = t[2 * q] == cid[k] ? t[2 * q + 1] : v[k];
    }
  }
  if (failed == 0 && expects && poisoned) return;             // as in k_slot_scatter
  uint4 sr[PACK_PER_THREAD];
#pragma unroll
  for (int k = 0; k < PACK_PER_THREAD; ++k) {
    if (base + (u64)k * SCAT_THREADS >= n_rec) v[k] = NONE;
    else if (v[k] == NONE || v[k] == RANK_TAB_OVERFLOW || cid[k] == NONE) {
      const u64 rs = resolve_slow(R, rk[k], cid[k]);
      v[k] = (u32)rs;
      if (rs >> 32) { err |= (u32)(rs >> 32); ++rej; }
    }
    sr[k] = v[k] != NONE ? srow[v[k] >> RANK_TAB_POS_BITS] : make_uint4(0, 0, 0, 0);
  }
  // Of two copies of a record the first one here has the slot to itself: index and sector are separate stores, and a sector that two wrote was
  // seen half and half. The answer that is waited for costs a tenth (232 us, 211 with plain stores; an index in each half, to be compared with
  // the table's, needs two stores instead of one: 268).
  u64 slot[PACK_PER_THREAD]; u32 before[PACK_PER_THREAD];
#pragma unroll
  for (int k = 0; k < PACK_PER_THREAD; ++k) {
    before[k] = 0;
    if (v[k] == NONE) continue;
    if (!scatter_slot(R, v[k] >> RANK_TAB_POS_BITS, sr[k].z, sr[k].w, ((u64)sr[k].x | ((u64)sr[k].y << 32)) + (u64)(v[k] & ((1u << RANK_TAB_POS_BITS) - 1)) * sr[k].z, sq[k],
                      n_slots, &slot[k], &err, &rej, &internal)) continue;
    before[k] = atomicCAS(perm + slot[k], NONE, (u32)(base + (u64)k * SCAT_THREADS));
  }
#pragma unroll
  for (int k = 0; k < PACK_PER_THREAD; ++k) if (before[k] == NONE) store_packed(packed + slot[k] * 2, r[k]);
  count_rejects(D, err, rej, internal);
}

}  // namespace ccld

#include "ccld_fused.cuh"
#include "ccld_mid.cuh"
#include "ccld_large.cuh"

namespace ccld {

// ------------------------------------------------------------------------------------------------
// window decision per communicator (Sec. 4.2.1 Eq. 1-3, Sec. 4.2.2 Eq. 4): a warp per communicator.
// Bound by latency: chains of dependent reads over little data.
// ------------------------------------------------------------------------------------------------
constexpr int WD_THREADS = 128;

// What of a window's decision does not depend on the state carried from window to window: the round counts, the round Eq. 2
// selects with its T_max / T_min and the ranks the location step would name.
struct RoundPart { u32 n_rounds, sel_seq, root_comp, root_comm, rate_source; i64 t_max, t_min; };

__device__ __forceinline__ RoundPart rounds_of(const WinDesc& D, const RangeRow& row, u32 lane, u32* n_analysed) {
  RoundPart x = {0, NONE, NONE, NONE, 0, 0, 0};
  *n_analysed = 0;
  if (row.n_seq == 0) return x;
  const u32 cls = comm_class(row.n);
  const u64 G = D.n_groups;
  const i64* t_max = D.gi64 + (u64)GI_T_MAX * G + row.group0;
  const i64* t_min = D.gi64 + (u64)GI_T_MIN * G + row.group0;
  // round counts and the Eq. 2 candidate come from the tile summaries the reduce kernels left behind
  const TileSum* ts = D.tsum[cls <= 1 ? 0 : cls - 1] + row.tile0;   // both relative to the window
  u32 n_rounds = 0, n_an = 0;
  u64 best_rng = 0; u32 best_k = NONE;
  bool redo = false;                                     // a unit left groups to the deferred kernel: its summary is partial
  for (u32 q = lane; q < row.n_units; q += 32) {
    const TileSum s = ts[q];
    n_rounds += s.n_rounds; n_an += s.n_an;
    best_merge(best_rng, best_k, s.best_rng, s.best_k);
    redo = redo || s.pad != 0;
  }
  if (__any_sync(0xFFFFFFFFu, redo)) {
    // recount the communicator's window from the per-op rows
    const u32* gfl = D.gu32 + (u64)GU_GFLAGS * G + row.group0;
    n_rounds = 0; n_an = 0; best_rng = 0; best_k = NONE;
    constexpr u32 AHEAD = 8;                             // ops per lane whose rows are asked for at once
    for (u32 k0 = lane; k0 < row.n_seq; k0 += 32 * AHEAD) {
      u32 f[AHEAD]; u64 rng[AHEAD];
#pragma unroll
      for (u32 u = 0; u < AHEAD; ++u) {
        const u32 k = min(k0 + 32 * u, row.n_seq - 1);
        f[u] = gfl[k]; rng[u] = (u64)(t_max[k] - t_min[k]);
      }
#pragma unroll
      for (u32 u = 0; u < AHEAD; ++u) {
        const u32 k = k0 + 32 * u;
        if (k >= row.n_seq) break;
        if ((f[u] & CCLD_G_COMPLETE) && !(f[u] & CCLD_G_BARRIER)) { ++n_rounds; best_merge(best_rng, best_k, rng[u], k); }
        if (f[u] & CCLD_G_ANALYSED) ++n_an;
      }
    }
  }
  x.n_rounds = __reduce_add_sync(0xFFFFFFFFu, n_rounds); *n_analysed = __reduce_add_sync(0xFFFFFFFFu, n_an);
  best_warp_reduce(best_rng, best_k);
  if (best_k != NONE) {
    const u64 gq = row.group0 + best_k;
    const u32 mc = D.gu32[(u64)GU_MAX_CHG * G + gq], by_rate = D.gu32[(u64)GU_RANK_MAX_CHG * G + gq], by_time = D.gu32[(u64)GU_RANK_TMAX * G + gq];
    x.sel_seq = row.seq_lo + best_k; x.t_max = t_max[best_k]; x.t_min = t_min[best_k];
    x.root_comp = D.gu32[(u64)GU_RANK_TMIN * G + gq];
    x.root_comm = mc > 0 ? by_rate : by_time; x.rate_source = mc > 0 ? 0u : 1u;
  }
  return x;
}

// Analysed ops of a window count towards every member's denominator. A warp goes along the members of its communicator; one
// of more than OPS_WARP is left to all warps of the CTA, when they have met (a warp alone took 20 us over a communicator of
// 4,096). Bound by latency: sixteen members per thread are looked up at a time, and what the lookups need was left in shared
// memory (four at a time, behind three more loads: the whole kernel took 45.6 us instead of 21.0 on a window of 16,384 ranks with
// communicators of up to 2,048, and 23.5 instead of 18.9 on two windows of one communicator of 4,096).
constexpr u32 OPS_WARP = 512;
struct OpsShared { u32 n_an[WD_THREADS / 32], n[WD_THREADS / 32]; u64 moff[WD_THREADS / 32]; };
template <u32 THREADS> __device__ __forceinline__ void add_ops(const Registry& R, u64 moff, u32 n, u32 n_an, u32 first) {
  constexpr u32 AHEAD = 16;
  const u32* __restrict__ mem = R.members + moff;
  for (u32 p0 = first; p0 < n; p0 += THREADS * AHEAD) {
    u32 r[AHEAD];
#pragma unroll
    for (u32 u = 0; u < AHEAD; ++u) r[u] = p0 + u * THREADS < n ? __ldg(mem + p0 + u * THREADS) : NONE;
#pragma unroll
    for (u32 u = 0; u < AHEAD; ++u) if (r[u] != NONE) atomicAdd(&R.ops[r[u]], n_an);
  }
}
// All threads of the CTA; a warp brings its communicator's analysed ops, members and their place.
__device__ __forceinline__ void count_ops(const Registry& R, OpsShared& sh, u32 n_an, u32 n, u64 moff) {
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool all = n_an != 0 && n > OPS_WARP;
  if (lane == 0) { sh.n_an[wid] = all ? n_an : 0u; sh.n[wid] = n; sh.moff[wid] = moff; }
  if (n_an != 0 && !all) add_ops<32>(R, moff, n, n_an, lane);
  if (!__syncthreads_or(all)) return;
  for (u32 q = 0; q < WD_THREADS / 32; ++q) if (sh.n_an[q] != 0) add_ops<WD_THREADS>(R, sh.moff[q], sh.n[q], sh.n_an[q], threadIdx.x);
}

// Stage 1 of a batch of several windows, all at once: leaves the part above in the communicator's verdict row.
// (Twelve CTAs per SM: with the registers that eight ops per lane in the recount would like it took 14.8 instead of 11.9 us on twelve windows
// of 1,088 communicators; recounting 1,000 op counters takes 9.4 us with eight, 12.1 with four at a time.)
__global__ void __launch_bounds__(WD_THREADS, 12) k_window_rounds(const WinDesc* wd, Registry R) {
  begin_after();
  __shared__ OpsShared s_ops;
  const u32 c = blockIdx.x * (WD_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const WinDesc& D = wd[blockIdx.y];
  u32 n_an = 0, n = 0; u64 moff = 0;
  if (c < R.n_comms) {
    const RangeRow row = D.ranges[c];
    n = row.n; moff = R.comm_moff[c];
    const RoundPart x = rounds_of(D, row, lane, &n_an);
    if (lane == 0 && row.n_seq) {
      ccld_comm_verdict* v = D.comm_rows + row.row_idx;
      v->n_rounds = x.n_rounds; v->sel_seq = x.sel_seq; v->root_comp = x.root_comp; v->root_comm = x.root_comm; v->rate_source = x.rate_source;
      v->t_max = x.t_max; v->t_min = x.t_min;
    }
  }
  count_ops(R, s_ops, n_an, n, moff);
}

// Stage 2, windows in order: the recurrences - Eq. 1's baseline, which reads the per-op rows until m is fixed, and the
// repetition counter - and with them Eq. 3, Eq. 4 and the location rule, which complete the row. What a window needs is
// fetched ahead (range rows two windows, the stage-1 row and the result pointers one window), so the walk waits for
// arithmetic only. SINGLE: a batch of one window, stage 1 is done here too.
template <bool SINGLE>
__global__ void __launch_bounds__(WD_THREADS) k_window_decide(const WinDesc* wd, u32 nw, Registry R, Params P) {
  begin_after();
  __shared__ OpsShared s_ops;
  const u32 c = blockIdx.x * (WD_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  u32 n_an = 0, n = 0; u64 moff = 0;
  if (c < R.n_comms) {
    CommState st = R.state[c];
    if (SINGLE) moff = R.comm_moff[c];
    struct Res { const RangeRow* ranges; u64 n_groups; const i64* gi64; const u32* gu32; ccld_comm_verdict* comm_rows; };   // pointers of a window
    // three steps, each on values fetched during an earlier window: descriptor -> range row -> stage-1 row
    auto load_res = [&](u32 w) {
      Res r = {nullptr, 0, nullptr, nullptr, nullptr};
      if (w < nw) { r.ranges = wd[w].ranges; r.n_groups = wd[w].n_groups; r.gi64 = wd[w].gi64; r.gu32 = wd[w].gu32; r.comm_rows = wd[w].comm_rows; }
      return r;
    };
    auto load_row = [&](const Res& r) { RangeRow x = {0, 0, 0, 0, 0, 0, 0, 0}; if (r.ranges != nullptr) x = r.ranges[c]; return x; };
    auto load_part = [&](const Res& r, const RangeRow& row) {
      RoundPart x = {0, NONE, NONE, NONE, 0, 0, 0};
      if (r.comm_rows != nullptr && row.n_seq != 0) {
        const ccld_comm_verdict* v = r.comm_rows + row.row_idx;
        x.n_rounds = v->n_rounds; x.sel_seq = v->sel_seq; x.root_comp = v->root_comp; x.root_comm = v->root_comm;
        x.rate_source = v->rate_source; x.t_max = v->t_max; x.t_min = v->t_min;
      }
      return x;
    };
    Res res_a = load_res(0), res_b = load_res(1), res_c = load_res(2);
    RangeRow row_a = load_row(res_a), row_b = load_row(res_b);
    RoundPart part_a;
    if (SINGLE) { n = row_a.n; part_a = rounds_of(wd[0], row_a, lane, &n_an); } else part_a = load_part(res_a, row_a);
    for (u32 w = 0; w < nw; ++w) {
      const RangeRow row = row_a; const Res D = res_a; const RoundPart pt = part_a;
      if (!SINGLE) {
        part_a = load_part(res_b, row_b);                    // window w + 1
        row_a = row_b; row_b = load_row(res_c);              // window w + 2
        res_a = res_b; res_b = res_c; res_c = load_res(w + 3);
      }
      if (row.n_seq == 0) continue;
      const u64 G = D.n_groups;
      const u32 n_rounds = pt.n_rounds;
      // Eq. 1: rounds feed the baseline, in op-counter order, until m is fixed: by the first round that comes after
      // m_max_rounds others or m_max_ns after the first. 32 ops at a time; a lane knows from the vote how many rounds
      // precede its own.
      u32 walked = 0;
      if (st.m == 0 && n_rounds > 0) {
        const u32* gfl = D.gu32 + (u64)GU_GFLAGS * G + row.group0;
        const i64* e_min = D.gi64 + (u64)GI_E_MIN * G + row.group0;
        const i64* t_max = D.gi64 + (u64)GI_T_MAX * G + row.group0;
        constexpr u32 AHEAD = 4;                             // steps of 32 ops whose rows are asked for at once
        u32 f_[AHEAD]; i64 em_[AHEAD], tM_[AHEAD];
        for (u32 k0 = 0, u = 0; k0 < row.n_seq && st.m == 0; k0 += 32, u = (u + 1) % AHEAD) {
          if (u == 0) {
#pragma unroll
            for (u32 q = 0; q < AHEAD; ++q) {
              const u32 k = k0 + 32 * q + lane;
              f_[q] = 0; em_[q] = tM_[q] = 0;
              if (k < row.n_seq) { f_[q] = gfl[k]; em_[q] = e_min[k]; tM_[q] = t_max[k]; }
            }
          }
          u32 f = f_[0]; i64 em = em_[0], tM = tM_[0];
#pragma unroll
          for (u32 q = 0; q + 1 < AHEAD; ++q) { f_[q] = f_[q + 1]; em_[q] = em_[q + 1]; tM_[q] = tM_[q + 1]; }
          const bool round = (f & CCLD_G_COMPLETE) && !(f & CCLD_G_BARRIER);
          const u32 bal = __ballot_sync(0xFFFFFFFFu, round);
          if (bal == 0) continue;
          if (st.rounds == 0) st.t_first = __shfl_sync(0xFFFFFFFFu, em, __ffs(bal) - 1);
          const u64 before = st.rounds + (u32)__popc(bal & ((1u << lane) - 1u));
          const u32 stop = __ballot_sync(0xFFFFFFFFu, round && (before == (u64)P.m_max_rounds || (before > 0 && em - st.t_first >= P.m_max_ns)));
          const u32 take = stop ? bal & ((1u << (__ffs(stop) - 1)) - 1u) : bal;      // rounds that still feed the baseline
          i64 sum = (take >> lane) & 1u ? tM : 0;
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) sum += (i64)shfl_xor64((u64)sum, d);
          st.sum_m += sum;
          u32 seen = (u32)__popc(take);
          if (stop) { st.m = st.rounds + seen; ++seen; }
          st.rounds += seen; walked += seen;
        }
      }
      st.rounds += n_rounds - walked;
      if (lane == 0) {
        ccld_comm_verdict v;
        v.comm = R.comm_id[c]; v.n_rounds = n_rounds; v.sel_seq = pt.sel_seq; v.cls = 0; v.slow_detected = 0; v.located = 0;
        v.baseline_static = st.m == 0; v.rate_source = 0; v.root_comp = NONE; v.root_comm = NONE;
        v.t_max = pt.t_max; v.t_min = pt.t_min; v.R = 0.0; v.P = 0.0;
        v.t_base = st.m > 0 ? st.sum_m / (i64)st.m : P.tbase_init_ns;
        v.rounds_total = st.rounds; v.m = st.m;
        if (pt.sel_seq != NONE) {
          v.R = (double)(v.t_max - v.t_base) / (double)v.t_base;                                     // Eq. 3
          const bool slow = v.t_max > v.t_base && mul_gt((u64)(v.t_max - v.t_base), 1000u, (u64)v.t_base, P.theta_slow_milli);
          v.slow_detected = slow;
          if (slow) {
            ++st.slow_count;
            v.located = st.slow_count > (u64)P.slow_rep_threshold;
            const u64 num = (u64)(v.t_max - v.t_min), den = (u64)(v.t_max - v.t_base);
            v.P = (double)num / (double)den;                                                         // Eq. 4
            v.cls = mul_gt(num, 1000u, den, P.beta_milli) ? 1u : (mul_lt(num, 1000u, den, P.alpha_milli) ? 2u : 3u);
            v.root_comp = pt.root_comp; v.root_comm = pt.root_comm; v.rate_source = pt.rate_source;
          }
        }
        v.slow_count = st.slow_count;
        D.comm_rows[row.row_idx] = v;
      }
      st.slow_count = __shfl_sync(0xFFFFFFFFu, st.slow_count, 0);
    }
    if (lane == 0) R.state[c] = st;
  }
  if (!SINGLE) return;
  count_ops(R, s_ops, n_an, n, moff);
}

}  // namespace ccld
#include "ccld_hang.cuh"
#include "ccld_tree.cuh"
