// Hang location (Sec. 4.2.2, Fig. 6) for one op, or for every alert of a window, one CTA per op (sm_100a). Included by
// ccld_kernels.cuh.
//
// Bound by latency: a ring's presence bits, frames and counters are a few hundred KB at most, and what takes time is the
// number of dependent steps. Per-member state lives in shared memory (global scratch beyond HANG_SMEM_N members); a member
// is looked up at the op itself first, and only one that did not report it is searched for at later counters, a warp along
// its contiguous column of the slot table; the layers of a tree get their extremes by atomics on the layer's entry instead
// of one thread walking the layer; verdicts and roots go straight to pinned memory. A tree of 1,024: 52 -> 12 us.
#pragma once

namespace ccld {

constexpr int HANG_THREADS = 1024;
constexpr u32 HANG_SMEM_N = 2048;
constexpr u32 HANG_MEMBER_BYTES = 8 + 8 + 8 + 4 + 4;       // counter total, layer minimum and maximum, frame, state and layer candidate
inline size_t hang_smem(u32 max_n) { return max_n <= HANG_SMEM_N ? (size_t)max_n * HANG_MEMBER_BYTES : 0; }
constexpr u32 HANG_NO_LAYERS = 0xFFFFFFFFu;                // verdict class of a tree communicator whose layers are not known

struct HangArgs {
  u32 c, seq;                          // the op, unless `alerts` is given
  const ccld_hang_alert* alerts; const u64* counters;      // ordered alerts of the window and its counters: CTA i takes alerts i, i + grid, ...
  u32 cap;                             //   of the first `cap`
  u32 n_frames, n_channels;
  const u32 *f_rank, *f_comm, *f_seq, *progress;
  unsigned char* scratch; u64 scratch_stride;              // per CTA, for communicators beyond HANG_SMEM_N
  u32* roots; u32 roots_cap;           // list i starts at roots + i * roots_cap
  ccld_hang_verdict* out;              // verdict i (pointer fields unused)
  ccld_hang_alert* alerts_out;         // alert i once more, for the host
  u64* n_alerts_out;
};

// Sums and extremes of a CTA's threads, met in shared memory with one barrier.
struct HangSums { u32 n_ne, n_ok, n_missing, root; u64 mn, lag; };

__device__ __forceinline__ void hang_locate_cta(const WinDesc& D, const Registry& R, const HangArgs& A, u32 c, u32 seq, u32 slot) {
  extern __shared__ __align__(16) unsigned char hang_smem_raw[];
  __shared__ HangSums s;
  __shared__ u32 s_n_late, s_red32[32];
  const u32 n = R.comm_n[c], cid = R.comm_id[c];
  const u32* mem = R.members + R.comm_moff[c];
  const u32* const head = R.comm_head[c];
  if (head == REG_NO_LAYERS) {
    if (threadIdx.x == 0) { ccld_hang_verdict v; memset(&v, 0, sizeof v); v.cls = HANG_NO_LAYERS; A.out[slot] = v; }
    return;
  }
  const RangeRow row = D.ranges[c];
  unsigned char* const base = n <= HANG_SMEM_N ? hang_smem_raw : A.scratch + (u64)blockIdx.x * A.scratch_stride;
  u64* const tot = (u64*)base; u64* const lmin = tot + n; u64* const lmax = lmin + n;
  u32* const frame = (u32*)(lmax + n); u32* const state = frame + n;                  // state: 1 entered, 2 done; later a layer's candidate
  u32* const late = (u32*)lmax;                                                       // members to be looked for at later counters (lmax is not used yet)
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) { s.n_ne = s.n_ok = s.n_missing = 0; s.root = NONE; s.mn = U64_MAX_; s.lag = 0; s_n_late = 0; }
  __syncthreads();
  // a member has entered if it reported this or a later op counter
  const bool covered = row.n_seq > 0 && seq <= row.seq_lo + (row.n_seq - 1);
  const u32 s_first = covered && seq > row.seq_lo ? seq - row.seq_lo : 0;
  const u32* const perm = D.perm; const i64* const t_exit = D.t_exit;
  for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) {
    u32 st = 0;
    if (covered) {
      const u32 idx = perm[perm_at(row, s_first, p)];
      if (idx != NONE) st = 1u | (row.seq_lo + s_first == seq && t_exit[idx] != -1 ? 2u : 0u);
      else if (s_first + 1 < row.n_seq) late[atomicAdd(&s_n_late, 1u)] = p;
    }
    state[p] = st; frame[p] = NONE;
  }
  __syncthreads();
  for (u32 q = wid; q < s_n_late; q += HANG_THREADS / 32) {
    const u32 p = late[q];
    const u32* col = perm + perm_at(row, 0, p);
    bool found = false;
    for (u32 k0 = s_first + 1; k0 < row.n_seq && !found; k0 += 32) found = __any_sync(0xFFFFFFFFu, k0 + lane < row.n_seq && col[k0 + lane] != NONE);
    if (found && lane == 0) state[p] = 1;
  }
  // progress frames of this op: the first frame uploaded for a member counts
  for (u32 f = threadIdx.x; f < A.n_frames; f += HANG_THREADS) {
    if (A.f_comm[f] != cid || A.f_seq[f] != seq) continue;
    const u32 p = pos_lookup(R, A.f_rank[f], c);
    if (p != NONE) atomicMin(&frame[p], f);
  }
  __syncthreads();
  {
    u32 n_ne = 0, n_ok = 0, n_missing = 0; u64 mn = U64_MAX_;
    for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) {
      const u32 st = state[p], f = frame[p];
      n_ne += !(st & 1); n_ok += st >> 1;
      u64 t = 0;
      if (f == NONE) ++n_missing;
      else {
        const u32* pr = A.progress + (u64)f * A.n_channels * 2;
        if (((uintptr_t)A.progress & 7) == 0) {
#pragma unroll 4
          for (u32 ch = 0; ch < A.n_channels; ++ch) { const uint2 x = reinterpret_cast<const uint2*>(pr)[ch]; t += (u64)x.x + x.y; }
        } else {
          for (u32 ch = 0; ch < A.n_channels; ++ch) t += (u64)pr[2 * ch] + pr[2 * ch + 1];
        }
      }
      tot[p] = t; lmin[p] = U64_MAX_; lmax[p] = 0; mn = t < mn ? t : mn;
    }
    n_ne = __reduce_add_sync(0xFFFFFFFFu, n_ne); n_ok = __reduce_add_sync(0xFFFFFFFFu, n_ok); n_missing = __reduce_add_sync(0xFFFFFFFFu, n_missing);
    mn = warp_min64(mn);
    if (lane == 0) { if (n_ne) atomicAdd(&s.n_ne, n_ne); if (n_ok) atomicAdd(&s.n_ok, n_ok); if (n_missing) atomicAdd(&s.n_missing, n_missing); atomicMin((ull*)&s.mn, (ull)mn); }
  }
  __syncthreads();
  const u32 n_ne = s.n_ne, n_ok = s.n_ok, n_missing = s.n_missing;
  const u64 mn = s.mn;
  const u32 cls = n_ne > 0 ? 1u : (n_ok > 0 ? 2u : 3u);
  u32 n_roots = 0, root = NONE;
  if (cls == 3 && head != nullptr) {
    // tree (Sec. 4.2.1): counters are comparable inside a layer only. A layer's entry, at its lowest position, collects the
    // layer's minimum, maximum and the lowest position that holds the minimum. The layer whose minimum is furthest behind
    // its maximum names the root; equal gaps: the lowest position; no gap anywhere: nobody.
    for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) { const u32 h = head[p]; atomicMin((ull*)&lmin[h], (ull)tot[p]); atomicMax((ull*)&lmax[h], (ull)tot[p]); state[p] = NONE; }
    __syncthreads();
    u64 lag = 0;
    for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) {
      const u32 h = head[p];
      if (tot[p] == lmin[h]) atomicMin(&state[h], p);
      if (h == p) { const u64 g = lmax[p] - lmin[p]; lag = g > lag ? g : lag; }
    }
    lag = warp_max64(lag);
    if (lane == 0 && lag) atomicMax((ull*)&s.lag, (ull)lag);
    __syncthreads();
    const u64 best = s.lag;
    if (best) for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) if (head[p] == p && lmax[p] - lmin[p] == best) atomicMin(&s.root, state[p]);
    __syncthreads();
    root = s.root;
    n_roots = root != NONE ? 1u : 0u;
  } else if (cls == 3) {
    // fewest counters; among equals the most upstream of a run (predecessor ahead), then the lowest position. Members
    // without such a predecessor rank behind all that have one.
    u32 cand = NONE;
    for (u32 p = threadIdx.x; p < n; p += HANG_THREADS) {
      if (tot[p] != mn) continue;
      const u32 k = p | (tot[p ? p - 1 : n - 1] > mn ? 0u : 0x80000000u);
      cand = k < cand ? k : cand;
    }
    cand = __reduce_min_sync(0xFFFFFFFFu, cand);
    if (lane == 0) atomicMin(&s.root, cand);
    __syncthreads();
    root = s.root & 0x7FFFFFFFu;
    n_roots = 1;
  } else {
    // ordered compaction of the not-entered (H1) or not-hung (H2) members
    for (u32 p0 = 0; p0 < n; p0 += HANG_THREADS) {
      const u32 p = p0 + threadIdx.x;
      const bool sel = p < n && (cls == 1 ? !(state[p] & 1) : (state[p] & 2) != 0);
      const u32 bal = __ballot_sync(0xFFFFFFFFu, sel);
      if (lane == 0) s_red32[wid] = __popc(bal);
      __syncthreads();
      const u32 mine = s_red32[lane];                                                 // 32 warps
      const u32 before = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? mine : 0u), all = __reduce_add_sync(0xFFFFFFFFu, mine);
      const u32 off = n_roots + before + __popc(bal & ((1u << lane) - 1));
      if (sel && off < A.roots_cap) A.roots[(u64)slot * A.roots_cap + off] = mem[p];
      n_roots += all;                                                                 // the same in every thread
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    ccld_hang_verdict v;
    v.cls = cls; v.n_roots_total = n_roots; v.n_not_entered = n_ne; v.n_hung = n - n_ok; v.n_not_hung = n_ok;
    v.n_missing_frames = cls == 3 ? n_missing : 0; v.stuck_step = 0; v.n_members = n; v.min_total = 0;
    v.roots = nullptr; v.roots_cap = 0;
    if (cls == 3 && root != NONE) {
      v.min_total = tot[root];
      if (A.roots_cap > 0) A.roots[(u64)slot * A.roots_cap] = mem[root];
      const u32 f = frame[root];
      if (f != NONE && A.n_channels > 0) {
        u32 least = NONE;
        for (u32 ch = 0; ch < A.n_channels; ++ch) { const u32 r = A.progress[((u64)f * A.n_channels + ch) * 2 + 1]; least = r < least ? r : least; }
        v.stuck_step = least;
      }
    }
    A.out[slot] = v;
  }
}

__global__ void __launch_bounds__(HANG_THREADS) k_hang_locate(const WinDesc* wd, Registry R, HangArgs A) {
  begin_after();
  const WinDesc& D = wd[0];
  if (A.alerts == nullptr) { hang_locate_cta(D, R, A, A.c, A.seq, 0); return; }
  // every alert of the window
  const u64 total = A.counters[C_ALERTS];
  if (blockIdx.x == 0 && threadIdx.x == 0) *A.n_alerts_out = total;
  const u32 n = (u32)min(total, (u64)min(A.cap, CCLD_MAX_ALERTS_PER_WINDOW));
  for (u32 i = blockIdx.x; i < n; i += gridDim.x) {
    const ccld_hang_alert a = A.alerts[i];
    if (threadIdx.x == 0) A.alerts_out[i] = a;
    hang_locate_cta(D, R, A, comm_lookup(R, a.comm), a.seq, i);
    __syncthreads();                                       // the shared state is set up anew
  }
}

}  // namespace ccld
