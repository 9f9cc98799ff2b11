// What ccld_get_verdict hands out, gathered on the device and written straight into pinned host memory (sm_100a).
//
//   k_verdict_collect  a CTA per 1,024 ranks: which of its ranks are suspects (vote shares against the threshold), as one
//                      64-bit key each that orders like the list - kind, votes descending, rank -, sorted in shared
//                      memory; the last of them to finish puts the pieces of a list of up to 1,024 together. Further CTAs
//                      copy the window's communicator rows and counters and order the hang alerts (apart, so that the fence
//                      before "finished" does not wait for their writes across PCIe).
//   k_verdict_merge    longer lists: the sorted pieces become one list. A key's place is its place in its own
//                      piece plus, for every other piece, the number of keys before it (a binary search).
//
// Bound by latency: the inputs are a few hundred KB at most. One launch (two for long lists), no copy and one wait of the
// host per verdict, where a copy of the counters, a launch, a copy of the count, a launch and two more copies with three
// waits used to be; the rank-by-counting sort of an 8,000-suspect list over global memory took 243 us, the sorted pieces
// with the merge take under 10 (communicators of four ranks, whose MAD rests on two values, name that many).
#pragma once
#include <cstddef>
#include "ccld_kernels.cuh"

namespace ccld {

constexpr int VD_THREADS = 1024;             // ranks per CTA
constexpr int VD_KEYS = 2 * VD_THREADS;      // a rank is on the list at most twice
constexpr u32 VD_SUS_HOST = 65536;           // suspects the pinned area holds at most; longer lists stay in device memory

constexpr int VD_MERGE = 1024;               // lists up to this long are put together by the last CTA of k_verdict_collect

struct VerdictHead { u64 counters[C_COUNT]; u32 n_suspects, listed; };     // listed: the suspects are in place
struct VerdictArgs {
  const u64* counters;                       // the window's
  const ccld_comm_verdict* rows; u32 n_rows; // (null, 0): nothing to copy
  const ccld_hang_alert* alerts;
  u64* keys; u32* counts;                    // device scratch: [CTAs][VD_KEYS] sorted keys, [CTAs] how many
  u32* done;                                 // device: CTAs finished so far (0 between launches)
  VerdictHead* head;                         // pinned: counters and number of suspects
  int columns;                               // 1: the pinned lists column by column, 64-bit fields first, each column as long as the list
  ccld_comm_verdict* rows_out;               // pinned [n_rows]
  ccld_hang_alert* alerts_out;               // pinned [CCLD_MAX_ALERTS_PER_WINDOW]
  ccld_suspect* sus_host; u32 sus_host_cap;  // pinned; lists longer than that go to sus_dev (as structs)
  ccld_suspect* sus_dev;
};

__device__ __forceinline__ u64 suspect_key(u32 kind, u32 votes, u32 rank) { return ((u64)(kind - 1) << 54) | ((u64)(~votes) << 22) | rank; }
static_assert(CCLD_MAX_RANK_ID <= (1u << 22), "a rank id fits its field of the key");
__device__ __forceinline__ ccld_suspect suspect_of(const Registry& R, u64 key) {
  ccld_suspect s;
  s.kind = (u32)(key >> 54) + 1; s.votes = ~(u32)(key >> 22); s.rank = (u32)key & ((1u << 22) - 1);
  s.ops = R.ops[s.rank];
  const u32 cnt = R.bw_cnt[s.rank];
  s.mean_busbw = cnt ? R.bw_sum[s.rank] / (double)cnt : 0.0;
  return s;
}

// Entry i of n into a list of structs, or into its columns.
__device__ __forceinline__ void put_suspect(ccld_suspect* out, u32 i, u32 n, bool columns, const ccld_suspect& s) {
  if (!columns) { out[i] = s; return; }
  double* d = (double*)out; u32* u = (u32*)(d + n);
  d[i] = s.mean_busbw; u[i] = s.kind; u[n + i] = s.rank; u[2 * n + i] = s.votes; u[3 * n + i] = s.ops;
}
__device__ __forceinline__ void put_alert(ccld_hang_alert* out, u32 i, u32 n, bool columns, const ccld_hang_alert& a) {
  if (!columns) { out[i] = a; return; }
  i64* t = (i64*)out; u32* u = (u32*)(t + n);
  t[i] = a.age_ns; u[i] = a.comm; u[n + i] = a.seq;
}

// The alerts of a window in the order they are listed: registration order of the communicator, then op counter (then the
// place in the unordered list: an op raises one alert). One CTA; s_key holds CCLD_MAX_ALERTS_PER_WINDOW keys.
__device__ __forceinline__ void order_alerts(const Registry& R, const ccld_hang_alert* in, u32 n, ccld_hang_alert* out, bool columns, u64* s_key) {
  for (u32 i = threadIdx.x; i < n; i += blockDim.x) s_key[i] = ((u64)comm_lookup(R, in[i].comm) << 32) | in[i].seq;
  __syncthreads();
  for (u32 i = threadIdx.x; i < n; i += blockDim.x) {
    const u64 k = s_key[i];
    u32 before = 0;
    for (u32 j = 0; j < n; ++j) before += (s_key[j] < k || (s_key[j] == k && j < i)) ? 1u : 0u;
    put_alert(out, before, n, columns, in[i]);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(VD_THREADS) k_verdict_collect(VerdictArgs A, Registry R, Params P, u32 pieces) {
  begin_after();
  __shared__ u64 s_key[VD_KEYS];
  __shared__ u32 s_n;
  const u32 lane = threadIdx.x & 31;
  if (blockIdx.x >= pieces) {
    // communicator rows: whole 8-byte words, or the struct's ten 32-bit and eight 64-bit fields as columns
    static_assert(sizeof(ccld_comm_verdict) == 13 * 8 && offsetof(ccld_comm_verdict, slow_count) == 40, "ten 32-bit fields, then eight of 64");
    const u64 t0 = (u64)(blockIdx.x - pieces) * VD_THREADS + threadIdx.x, st = (u64)(gridDim.x - pieces) * VD_THREADS;
    const u64* src = (const u64*)A.rows; u64* dst = (u64*)A.rows_out;
    if (!A.columns) for (u64 i = t0; i < (u64)A.n_rows * 13; i += st) dst[i] = src[i];
    else {
      u32* dst32 = (u32*)(dst + (u64)A.n_rows * 8);
      for (u64 r = t0; r < A.n_rows; r += st) {                // a thread per row: lanes write along the columns
        u64 x[13];
#pragma unroll
        for (int k = 0; k < 13; ++k) x[k] = src[r * 13 + k];
#pragma unroll
        for (int f = 0; f < 8; ++f) dst[(u64)f * A.n_rows + r] = x[5 + f];
#pragma unroll
        for (int f = 0; f < 5; ++f) { dst32[(u64)(2 * f) * A.n_rows + r] = (u32)x[f]; dst32[(u64)(2 * f + 1) * A.n_rows + r] = (u32)(x[f] >> 32); }
      }
    }
    if (blockIdx.x == pieces) {
      if (threadIdx.x < C_COUNT) A.head->counters[threadIdx.x] = A.counters[threadIdx.x];
      const u64 n_al = A.counters[C_ALERTS];
      if (n_al) order_alerts(R, A.alerts, n_al < CCLD_MAX_ALERTS_PER_WINDOW ? (u32)n_al : CCLD_MAX_ALERTS_PER_WINDOW, A.alerts_out, A.columns != 0, s_key);
    }
    return;
  }
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  const u32 r = blockIdx.x * VD_THREADS + threadIdx.x;
  u32 ops = 0; uint4 v = make_uint4(0, 0, 0, 0);
  if (r < R.n_ranks) { ops = R.ops[r]; v = *reinterpret_cast<const uint4*>(R.votes + (u64)r * 4); }
#pragma unroll
  for (u32 kind = 1; kind <= 2; ++kind) {
    const u32 votes = kind == 1 ? v.x : v.z;
    const bool is = ops != 0 && (u64)votes * 1000u >= (u64)P.vote_rep_milli * ops;
    const u32 bal = __ballot_sync(0xFFFFFFFFu, is);
    u32 base = 0;
    if (lane == 0 && bal) base = atomicAdd(&s_n, (u32)__popc(bal));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (is) s_key[base + __popc(bal & ((1u << lane) - 1u))] = suspect_key(kind, votes, r);
  }
  __syncthreads();
  // bitonic sort over the next power of two
  const u32 n = s_n;
  u32 n_pad = 1; while (n_pad < n) n_pad <<= 1;
  for (u32 i = n + threadIdx.x; i < n_pad; i += VD_THREADS) s_key[i] = U64_MAX_;
  __syncthreads();
  for (u32 k = 2; k <= n_pad; k <<= 1) {
    for (u32 j = k >> 1; j > 0; j >>= 1) {
      const u32 q = threadIdx.x;                                // VD_KEYS / 2 pairs at most: one per thread
      if (q < n_pad >> 1) {
        const u32 i = ((q & ~(j - 1)) << 1) | (q & (j - 1)), l = i | j;
        const u64 a = s_key[i], b = s_key[l];
        if ((a > b) == ((i & k) == 0)) { s_key[i] = b; s_key[l] = a; }
      }
      __syncthreads();
    }
  }
  if (pieces == 1) {
    const bool host = n <= A.sus_host_cap;
    for (u32 i = threadIdx.x; i < n; i += VD_THREADS) put_suspect(host ? A.sus_host : A.sus_dev, i, n, host && A.columns, suspect_of(R, s_key[i]));
    if (threadIdx.x == 0) { A.head->n_suspects = n; A.head->listed = 1; }
    return;
  }
  for (u32 i = threadIdx.x; i < n; i += VD_THREADS) A.keys[(u64)blockIdx.x * VD_KEYS + i] = s_key[i];
  if (threadIdx.x == 0) A.counts[blockIdx.x] = n;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_n = atomicAdd(A.done, 1u);
  __syncthreads();
  if (s_n != pieces - 1) return;
  // the last CTA: short lists are put together here, longer ones are left to k_verdict_merge
  __threadfence();
  __shared__ u32 s_tot;
  if (threadIdx.x == 0) { s_tot = 0; *A.done = 0; }
  __syncthreads();
  u32 t = 0;
  for (u32 o = threadIdx.x; o < pieces; o += VD_THREADS) t += __ldcg(&A.counts[o]);
  t = __reduce_add_sync(0xFFFFFFFFu, t);
  if (lane == 0 && t) atomicAdd(&s_tot, t);
  __syncthreads();
  const u32 total = s_tot;
  if (threadIdx.x == 0) { A.head->n_suspects = total; A.head->listed = total <= VD_MERGE; s_n = 0; }
  if (total > VD_MERGE) return;
  __syncthreads();
  for (u32 o = threadIdx.x >> 5; o < pieces; o += VD_THREADS / 32) {                // a warp per piece, in any order
    const u32 k = __ldcg(&A.counts[o]);
    u32 at = 0;
    if (lane == 0 && k) at = atomicAdd(&s_n, k);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    for (u32 i = lane; i < k; i += 32) s_key[at + i] = __ldcg(&A.keys[(u64)o * VD_KEYS + i]);
  }
  __syncthreads();
  if (threadIdx.x < total) {
    const u64 key = s_key[threadIdx.x];
    u32 pos = 0;
    for (u32 i = 0; i < total; ++i) pos += s_key[i] < key ? 1u : 0u;                 // keys are unique
    put_suspect(A.sus_host, pos, total, A.columns, suspect_of(R, key));
  }
}

__global__ void __launch_bounds__(VD_THREADS) k_verdict_merge(VerdictArgs A, Registry R) {
  begin_after();
  __shared__ u32 s_tot;
  if (threadIdx.x == 0) s_tot = 0;
  __syncthreads();
  u32 t = 0;
  for (u32 o = threadIdx.x; o < gridDim.x; o += VD_THREADS) t += A.counts[o];
  t = __reduce_add_sync(0xFFFFFFFFu, t);
  if ((threadIdx.x & 31) == 0 && t) atomicAdd(&s_tot, t);
  __syncthreads();
  const u32 total = s_tot, n = A.counts[blockIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) { A.head->n_suspects = total; A.head->listed = 1; }
  const bool host = total <= A.sus_host_cap;
  const u64* mine = A.keys + (u64)blockIdx.x * VD_KEYS;
  for (u32 i = threadIdx.x; i < n; i += VD_THREADS) {
    const u64 key = mine[i];
    u32 pos = i;
    for (u32 o = 0; o < gridDim.x; ++o) {
      if (o == blockIdx.x) continue;
      const u64* other = A.keys + (u64)o * VD_KEYS;
      u32 lo = 0, hi = A.counts[o];                             // keys are unique: how many of the other piece are smaller
      while (lo < hi) { const u32 mid = (lo + hi) >> 1; if (other[mid] < key) lo = mid + 1; else hi = mid; }
      pos += lo;
    }
    put_suspect(host ? A.sus_host : A.sus_dev, pos, total, host && A.columns, suspect_of(R, key));
  }
}

// Several device arrays into one pinned area, one launch: a row of CTAs per piece. Source and destination agree modulo 16, so
// whole 16-byte words cross PCIe and only a piece's ends go byte by byte. AHEAD: words a thread asks for at once. (32 registers
// for large CTAs, so that one leaves room for others on its SM.)
constexpr int GATHER_THREADS = 256;
constexpr u32 GATHER_PIECES = 24;
struct GatherArgs { struct { const unsigned char* src; unsigned char* dst; u64 n; } piece[GATHER_PIECES]; };
template <int AHEAD, int THREADS> __global__ void __launch_bounds__(THREADS, THREADS == 1024 ? 2 : 1) k_gather(GatherArgs A) {
  begin_after();
  const unsigned char* src = A.piece[blockIdx.y].src; unsigned char* __restrict__ dst = A.piece[blockIdx.y].dst;
  const u64 n = A.piece[blockIdx.y].n;
  const u64 head = min(n, (u64)((16 - ((uintptr_t)src & 15)) & 15)), n16 = (n - head) / 16, tail = head + n16 * 16;
  const u64 i0 = (u64)blockIdx.x * THREADS + threadIdx.x, st = (u64)gridDim.x * THREADS;
  const uint4* s16 = reinterpret_cast<const uint4*>(src + head); uint4* d16 = reinterpret_cast<uint4*>(dst + head);
  u64 i = i0;
  if constexpr (AHEAD > 1) {
    for (; i + (AHEAD - 1) * st < n16; i += AHEAD * st) {
      uint4 v[AHEAD];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) v[k] = s16[i + k * st];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) d16[i + k * st] = v[k];
    }
  }
  for (; i < n16; i += st) d16[i] = s16[i];
  if (i0 < head) dst[i0] = src[i0];
  if (i0 < n - tail) dst[tail + i0] = src[tail + i0];
}

// communicator id, op counter and first slot of every group of a window
__global__ void __launch_bounds__(256) k_op_keys(const RangeRow* ranges, Registry R, u64 n_groups, u32* __restrict__ comm, u32* __restrict__ seq, u64* __restrict__ slot0) {
  begin_after();
  const u64 g = (u64)blockIdx.x * 256 + threadIdx.x;
  if (g >= n_groups) return;
  u32 lo = 0, hi = R.n_comms - 1;                              // owner: the last communicator whose first group is <= g
  while (lo < hi) { const u32 mid = (lo + hi + 1) >> 1; if (ranges[mid].group0 <= g) lo = mid; else hi = mid - 1; }
  const RangeRow row = ranges[lo];
  const u32 k = (u32)(g - row.group0);
  comm[g] = R.comm_id[lo]; seq[g] = row.seq_lo + k; slot0[g] = row.slot0 + (u64)k * row.n;
}

// the ordered alerts alone, for the hang sweep
__global__ void __launch_bounds__(VD_THREADS) k_order_alerts(const u64* counters, const ccld_hang_alert* in, ccld_hang_alert* out, Registry R) {
  begin_after();
  __shared__ u64 s_key[CCLD_MAX_ALERTS_PER_WINDOW];
  const u64 n = counters[C_ALERTS];
  order_alerts(R, in, n < CCLD_MAX_ALERTS_PER_WINDOW ? (u32)n : CCLD_MAX_ALERTS_PER_WINDOW, out, false, s_key);
}

}  // namespace ccld
