// Operation Type Set consistency of one op (Sec. 4.1.2: algorithm, protocol, data size and operation name are constant
// during a communication; Sec. 4.2.2: inconsistent operations are what leaf H2 of the hang tree points at). One CTA:
// the most frequent (op, bytes, algo, proto) among the members that reported the op - ties go to the tuple whose first
// holder stands earliest in the ring - and the members that carry another tuple, in ring order.
//
// Bound by latency. The members' tuples sit in shared memory; one tuple at a time is counted over all members - the one
// of the lowest position not counted yet - and the search ends once the members left could not outnumber the best. An op
// has one or two tuples, so that takes one or two passes where every member used to count its own tuple over all others
// (1,024 members: 67 -> 6 us). Should OPSET_PASSES tuples not decide it, every member left counts its own.
#pragma once
#include "ccld_kernels.cuh"

namespace ccld {

constexpr int OPSET_THREADS = 1024;
constexpr u32 OPSET_MEMBER_BYTES = 12;       // bytes, and op | algo << 8 | proto << 16 | counted << 30 | present << 31
constexpr u32 OPSET_PASSES = 48;

struct OpsetArgs {
  u32 c, seq;
  const u8 *algo, *proto;        // per record, may both be null (then 0)
  u32* ranks; u32 ranks_cap;     // pinned list of the deviating ranks
  ccld_opset_verdict* out;       // pinned (pointer fields unused)
};

__global__ void __launch_bounds__(OPSET_THREADS) k_opset_check(const WinDesc* wd, Registry R, OpsetArgs A) {
  begin_after();
  extern __shared__ __align__(16) unsigned char opset_smem[];
  constexpr u32 PRESENT = 0x80000000u, COUNTED = 0x40000000u, TUPLE = 0xFFFFFFu;
  __shared__ u32 s_cnt[3], s_next[3], s_red32[32], s_present;
  __shared__ u64 s_best;
  const WinDesc& D = wd[0];
  const u32 c = A.c, n = R.comm_n[c];
  const u32* mem = R.members + R.comm_moff[c];
  const RangeRow row = D.ranges[c];
  u64* const hi = (u64*)opset_smem; u32* const lo = (u32*)(hi + n);
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x < 3) { s_cnt[threadIdx.x] = 0; s_next[threadIdx.x] = NONE; }
  if (threadIdx.x == 0) { s_present = 0; s_best = 0; }
  __syncthreads();
  const bool in_range = row.n_seq > 0 && A.seq >= row.seq_lo && A.seq - row.seq_lo < row.n_seq;
  u32 n_present = 0, first = NONE;
  const u32* const perm = D.perm; const u64* const c_by = D.bytes; const u8* const c_op = D.op;
  for (u32 p = threadIdx.x; p < n; p += OPSET_THREADS) {
    const u32 idx = in_range ? perm[perm_at(row, A.seq - row.seq_lo, p)] : NONE;
    u64 h = 0; u32 l = 0;
    if (idx != NONE) {
      h = c_by[idx];
      l = (u32)c_op[idx] | (A.algo ? (u32)A.algo[idx] << 8 : 0u) | (A.proto ? (u32)A.proto[idx] << 16 : 0u) | PRESENT;
      ++n_present; first = min(first, p);
    }
    hi[p] = h; lo[p] = l;
  }
  n_present = __reduce_add_sync(0xFFFFFFFFu, n_present); first = __reduce_min_sync(0xFFFFFFFFu, first);
  if (lane == 0 && n_present) { atomicAdd(&s_present, n_present); atomicMin(&s_next[2], first); }
  __syncthreads();
  n_present = s_present;
  u32 cand = s_next[2], left = n_present, maj_cnt = 0, maj_p = 0;
  // pass k counts the tuple of position `cand` and finds the lowest position with another tuple not counted yet; three sets
  // of accumulators, so that the one of the pass before last is cleared while nobody uses it
  u32 pass = 0;
  for (; pass < OPSET_PASSES && left > maj_cnt; ++pass) {
    const u64 h = hi[cand]; const u32 l = lo[cand] & TUPLE;
    u32 cnt = 0, nxt = NONE;
    for (u32 p = threadIdx.x; p < n; p += OPSET_THREADS) {
      const u32 x = lo[p];
      if (!(x & PRESENT) || (x & COUNTED)) continue;
      if ((x & TUPLE) == l && hi[p] == h) { ++cnt; if (p != cand) lo[p] = x | COUNTED; }     // (every thread still reads cand's own word)
      else nxt = min(nxt, p);
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt); nxt = __reduce_min_sync(0xFFFFFFFFu, nxt);
    const u32 b = pass % 3;
    if (lane == 0) { if (cnt) atomicAdd(&s_cnt[b], cnt); if (nxt != NONE) atomicMin(&s_next[b], nxt); }
    __syncthreads();
    cnt = s_cnt[b]; nxt = s_next[b];
    if (threadIdx.x == 0) { lo[cand] |= COUNTED; const u32 z = (pass + 2) % 3; s_cnt[z] = 0; s_next[z] = NONE; }
    if (cnt > maj_cnt) { maj_cnt = cnt; maj_p = cand; }                                      // candidates come in ring order: ties stay
    left -= cnt; cand = nxt;
    __syncthreads();
  }
  if (left > maj_cnt) {
    // many different tuples: every member left counts its own; the largest count wins, then the lowest position
    u64 best = 0;
    for (u32 p = threadIdx.x; p < n; p += OPSET_THREADS) {
      const u64 h = hi[p]; const u32 x = lo[p];
      if (!(x & PRESENT) || (x & COUNTED)) continue;
      u32 cnt = 0;
      for (u32 q = 0; q < n; ++q) cnt += ((lo[q] & (PRESENT | TUPLE)) == (x & (PRESENT | TUPLE)) && hi[q] == h) ? 1u : 0u;
      const u64 k = ((u64)cnt << 32) | (u64)(NONE - p);
      best = k > best ? k : best;
    }
    best = warp_max64(best);
    if (lane == 0 && best) atomicMax((ull*)&s_best, (ull)best);
    __syncthreads();
    best = s_best;
    if ((u32)(best >> 32) > maj_cnt) { maj_cnt = (u32)(best >> 32); maj_p = NONE - (u32)best; }      // positions counted before stand earlier: ties stay
  }
  const u64 m_hi = maj_cnt ? hi[maj_p] : 0; const u32 m_lo = maj_cnt ? lo[maj_p] & TUPLE : 0;
  // ordered compaction of the deviating members
  u32 n_dev = 0;
  for (u32 p0 = 0; p0 < n; p0 += OPSET_THREADS) {
    const u32 p = p0 + threadIdx.x;
    const bool sel = p < n && (lo[p] & PRESENT) && ((lo[p] & TUPLE) != m_lo || hi[p] != m_hi);
    const u32 bal = __ballot_sync(0xFFFFFFFFu, sel);
    if (lane == 0) s_red32[wid] = __popc(bal);
    __syncthreads();
    const u32 mine = s_red32[lane];                            // 32 warps
    const u32 before = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? mine : 0u), all = __reduce_add_sync(0xFFFFFFFFu, mine);
    const u32 off = n_dev + before + __popc(bal & ((1u << lane) - 1));
    if (sel && off < A.ranks_cap) A.ranks[off] = mem[p];
    n_dev += all;                                              // the same in every thread
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ccld_opset_verdict v;
    v.n_members = n; v.n_present = n_present; v.n_deviating_total = n_dev; v.majority_count = maj_cnt;
    v.op = (u8)(m_lo & 0xFF); v.algo = (u8)((m_lo >> 8) & 0xFF); v.proto = (u8)((m_lo >> 16) & 0xFF); v.pad = 0;
    v.bytes = m_hi; v.ranks = nullptr; v.ranks_cap = 0;
    *A.out = v;
  }
}

}  // namespace ccld
