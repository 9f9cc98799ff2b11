// Counter changes per op from raw probe samples (Sec. 4.1.2: SendRate / RecvRate are reciprocals of the number of
// changes of SendCount / RecvCount seen by a probe that samples at a fixed period; Sec. 5.2 step 2 does this on the
// host's diagnostic thread). For sm_100a, streaming and HBM-bound.
//
//   k_tick_blocks   per block of 32 ticks: which ticks carry another SendCount / RecvCount than the tick before, as two
//                   32-bit masks with the number of changes before the block inside its tile of 2,048 ticks; per tile the
//                   number of changes. Further CTAs note per rank where its ticks lie in the table and in time, and
//                   whether a rank's ticks cover more than RT_NEAR tiles.
//   k_tile_scan     only for long segments: exclusive prefix over the tiles' numbers (one CTA). Where the host cannot tell from
//                   the average that there are any, the kernel is launched and looks.
//   k_record_rates  per record: the two ticks around its enter time and the two around its exit time, at the places even
//                   spacing gives (checked; a search where the samples are not even), then a difference of prefixes
//
// A rank's first tick is compared with another rank's last one; that bit is never counted, because a record counts the ticks
// after one of its own rank's. So the samples are read as one stream, without a look at the ranks.
//
// Measured on 4,096 ranks x 5,600 ticks and 4.1 M records (467 MB to move, 71 us at the measured copy rate): the version
// before searched the rank of every warp's ticks, loaded 4 bytes per lane and ran two more kernels for a global prefix
// (k_tick_blocks 61 us, prefix 21 us, k_record_rates 74 us with two dependent searches: 160 us); now 33 + 50 us, 82 us for the call.
// No kernel waits on another CTA.
#pragma once
#include "ccld_device.cuh"

namespace ccld {

constexpr int RT_THREADS = 256;
constexpr int RT_TILE = RT_THREADS * 8;            // ticks per CTA of k_tick_blocks, eight consecutive ones per lane
// A record adds up the tiles its op spans. Ops of one rank hardly overlap, so that is a read or two per record while no rank's
// samples cover more than this many tiles (8 tiles = 16 s at a sample per millisecond). With longer segments an op in flight
// since their beginning would add up many, and the scan pays: 20,000 tiles of one rank among 4,096, 50,000 records: 1,067 -> 99 us.
// (4,096 equal ranks of 5,600 ticks, whose scan is launched to find out that there are none: 80.1 -> 81.5 us.)
constexpr u32 RT_NEAR = 8;
// Up to RT_SCAN tiles in all a record adds up what it spans whatever the segments are. Up to RT_LOOK the scan is launched only
// where the ranks' average is beyond RT_NEAR: calls of that size are bound by the host, and a launch in order to look makes them
// 2 us longer (11.6 us without it at 2,000 tiles of 4,096 equal ranks, 13.8 with it at 2,100). Without it 2,000 tiles of one rank among
// 4,096 and 20,000 records, a third in flight, take 59 us instead of 20.
constexpr u64 RT_SCAN = 256, RT_LOOK = 2048;

// before: changes before the block inside the tile (send in the low half, recv in the high half); the ticks' change bits
struct alignas(16) TickBlock { u32 before, send, recv, pad; };
// A rank's ticks: [lo, lo + n) of the table, from t0 to t1; scale = ticks per nanosecond if they were evenly spaced
struct alignas(32) RankTicks { i64 t0, t1; u32 lo, n; float scale; u32 pad; };

struct TickArgs {
  u64 n_ticks; u32 n_ranks, n_tiles;
  const u64* tick_off;                             // [n_ranks + 1]
  const i64* tick_ns; const u32 *send, *recv;      // [n_ticks], a rank's ticks contiguous and in time order
  TickBlock* blk;                                  // [n_tiles * RT_TILE / 32]
  uint2* tile;                                     // [n_tiles] changes inside the tile, or before it once scanned
  RankTicks* ranks;                                // [n_ranks]
  u32* far;                                        // [CTAs of ranks] 1: one of the CTA's ranks covers more than RT_NEAR tiles
  u32* scanned;                                    // 1: k_tile_scan made prefixes of the tiles' sums; null: it does not run
  u32 vec;                                         // send and recv may be read 16 bytes at a time
};

// the eight counters from tick i on (past the end: the last one there is, so that nothing changes)
__device__ __forceinline__ void eight_ticks(const u32* c, u64 i, u64 n, bool vec, u32 (&v)[8]) {
  if (vec && i + 8 <= n) {
    const uint4 a = reinterpret_cast<const uint4*>(c + i)[0], b = reinterpret_cast<const uint4*>(c + i)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = c[i + k < n ? i + k : n - 1];
  }
}
__device__ __forceinline__ u32 change_bits(const u32 (&v)[8], u32 before) {
  u32 m = v[0] != before ? 1u : 0u;
#pragma unroll
  for (int k = 1; k < 8; ++k) m |= v[k] != v[k - 1] ? 1u << k : 0u;
  return m;
}

// Grid: n_tiles CTAs for the ticks, then one per RT_THREADS ranks.
__global__ void __launch_bounds__(RT_THREADS) k_tick_blocks(TickArgs A) {
  begin_after();
  __shared__ u32 s_cnt[RT_THREADS / 32];
  if (blockIdx.x >= A.n_tiles) {
    const u64 r = (u64)(blockIdx.x - A.n_tiles) * RT_THREADS + threadIdx.x;
    bool far = false;
    if (r < A.n_ranks) {
      const u64 lo = min(A.tick_off[r], A.n_ticks), hi = min(A.tick_off[r + 1], A.n_ticks);      // (every rank is looked at, also one without records)
      RankTicks x; x.t0 = 0; x.t1 = 0; x.lo = (u32)lo; x.n = hi > lo ? (u32)(hi - lo) : 0u; x.scale = 0.f; x.pad = 0;
      if (x.n) {
        x.t0 = A.tick_ns[lo]; x.t1 = A.tick_ns[hi - 1];
        if (x.t1 > x.t0) x.scale = (float)(x.n - 1) / (float)(x.t1 - x.t0);
        far = (hi - 1) / RT_TILE - lo / RT_TILE > RT_NEAR;
      }
      A.ranks[r] = x;
    }
    far = __syncthreads_or(far);
    if (threadIdx.x == 0) A.far[blockIdx.x - A.n_tiles] = far;
    return;
  }
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const u64 i = (u64)blockIdx.x * RT_TILE + (u64)threadIdx.x * 8;
  u32 sv[8], rv[8];
  eight_ticks(A.send, i, A.n_ticks, A.vec != 0, sv);
  eight_ticks(A.recv, i, A.n_ticks, A.vec != 0, rv);
  u32 ps = __shfl_up_sync(0xFFFFFFFFu, sv[7], 1), pr = __shfl_up_sync(0xFFFFFFFFu, rv[7], 1);
  if (lane == 0) {
    const u64 b = i ? (i - 1 < A.n_ticks ? i - 1 : A.n_ticks - 1) : 0;
    ps = A.send[b]; pr = A.recv[b];
  }
  u32 ms = change_bits(sv, ps), mr = change_bits(rv, pr);
  const u32 cnt = (u32)__popc(ms) | ((u32)__popc(mr) << 16);          // a tile has 2,048 ticks: sixteen bits are enough
  u32 inc = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) { const u32 o = __shfl_up_sync(0xFFFFFFFFu, inc, d); if (lane >= (u32)d) inc += o; }
  if (lane == 31) s_cnt[wid] = inc;
  // four lanes make a block
  ms <<= 8 * (lane & 3); mr <<= 8 * (lane & 3);
  ms |= __shfl_xor_sync(0xFFFFFFFFu, ms, 1); mr |= __shfl_xor_sync(0xFFFFFFFFu, mr, 1);
  ms |= __shfl_xor_sync(0xFFFFFFFFu, ms, 2); mr |= __shfl_xor_sync(0xFFFFFFFFu, mr, 2);
  __syncthreads();
  u32 before = 0, all = 0;
#pragma unroll
  for (u32 w = 0; w < RT_THREADS / 32; ++w) { const u32 x = s_cnt[w]; if (w < wid) before += x; all += x; }
  if ((lane & 3) == 0) A.blk[i >> 5] = TickBlock{before + inc - cnt, ms, mr, 0};
  if (threadIdx.x == 0) A.tile[blockIdx.x] = make_uint2(all & 0xFFFFu, all >> 16);
}

// One CTA of 1,024 threads; a round covers 16,384 tiles (33.5 M ticks). A warp owns 512 consecutive tiles of the round and
// reads them 32 at a time, lanes on consecutive ones, scans each 32 with shuffles and carries its running total from step
// to step; the warps' totals are scanned by every warp.
constexpr int TS_THREADS = 1024;
constexpr int TS_PER = 16;
__global__ void __launch_bounds__(TS_THREADS) k_tile_scan(uint2* tile, u32 n_tiles, const u32* far, u32 n_far, u32* scanned) {
  begin_after();
  __shared__ u64 s_warp[TS_THREADS / 32];
  bool any = far == nullptr;                          // null: the host knows that the scan pays
  for (u32 k = threadIdx.x; k < n_far && !any; k += TS_THREADS) any = far[k] != 0;
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) *scanned = any;
  if (!any) return;
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const auto pack = [](uint2 x) { return (u64)x.x | ((u64)x.y << 32); };          // fewer than 2^32 ticks: no carry into the upper half
  u64 carry = 0;
  for (u64 base = 0; base < n_tiles; base += (u64)TS_THREADS * TS_PER) {
    const u64 i0 = base + (u64)wid * (32 * TS_PER) + lane;
    u64 v[TS_PER];
#pragma unroll
    for (int k = 0; k < TS_PER; ++k) v[k] = i0 + 32 * k < n_tiles ? pack(tile[i0 + 32 * k]) : 0;
    u64 run = 0;                                      // the warp's sums before step k
#pragma unroll
    for (int k = 0; k < TS_PER; ++k) {
      u64 inc = v[k];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) { const u64 o = __shfl_up_sync(0xFFFFFFFFu, inc, d); if (lane >= (u32)d) inc += o; }
      v[k] = run + inc - v[k];                        // exclusive inside the warp's span
      run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) s_warp[wid] = run;
    __syncthreads();
    u64 w = s_warp[lane], winc = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const u64 o = __shfl_up_sync(0xFFFFFFFFu, winc, d); if (lane >= (u32)d) winc += o; }
    const u64 before = carry + __shfl_sync(0xFFFFFFFFu, winc - w, wid);
    carry += __shfl_sync(0xFFFFFFFFu, winc, 31);
#pragma unroll
    for (int k = 0; k < TS_PER; ++k) if (i0 + 32 * k < n_tiles) { const u64 x = before + v[k]; tile[i0 + 32 * k] = make_uint2((u32)x, (u32)(x >> 32)); }
    __syncthreads();                                  // s_warp is written again in the next round
  }
}

// changes inside its tile up to and including tick i (send in the low half, recv in the high half)
__device__ __forceinline__ u32 changes_upto(const TickBlock& e, u32 i) {
  const u32 keep = 0xFFFFFFFFu >> (31 - (i & 31));
  return e.before + ((u32)__popc(e.send & keep) | ((u32)__popc(e.recv & keep) << 16));
}

// Where even spacing puts time t, t0 <= t < t1, among n >= 2 ticks: tick g at or before t, tick g + 1 after it.
__device__ __forceinline__ u32 even_guess(const RankTicks& r, i64 t) {
  const u32 g = (u32)((float)(t - r.t0) * r.scale);
  return g > r.n - 2 ? r.n - 2 : g;
}
// Number of ticks at or before t (t0 <= t < t1), searched from tick g: doubling steps up or down, then bisection.
__device__ __noinline__ u32 search_from(const i64* __restrict__ tn, u32 n, u32 g, i64 t) {
  u32 a, b;                                        // the first tick after t lies in [a, b]
  if (__ldg(tn + g) <= t) {
    u32 pos = g, step = 1;                         // tn[pos] <= t
    for (int it = 0; it < 32 && pos + step < n && __ldg(tn + pos + step) <= t; ++it) { pos += step; step <<= 1; }
    a = pos + 1; b = pos + step < n - 1 ? pos + step : n - 1;
  } else {
    u32 pos = g, step = 1;                         // tn[pos] > t
    for (int it = 0; it < 32 && pos >= step && __ldg(tn + pos - step) > t; ++it) { pos -= step; step <<= 1; }
    a = (pos >= step ? pos - step : 0) + 1; b = pos;
  }
  for (int it = 0; it < 32 && a < b; ++it) { const u32 mid = a + ((b - a) >> 1); if (__ldg(tn + mid) <= t) a = mid + 1; else b = mid; }
  return a;
}

// A record per thread and four dependent steps: record columns -> the rank's entry -> four ticks -> two blocks. Latency is
// covered by warps alone: 32 registers, 64 warps per SM, measured 51 us (283 MB to move: 5.5 TB/s); two records per thread,
// every step issued for both before the next, took 58.7 us (58 registers), four 72.9.
__global__ void __launch_bounds__(RT_THREADS) k_record_rates(TickArgs A, u64 n_rec, const u32* __restrict__ rank, const i64* __restrict__ t_enter,
                                                           const i64* __restrict__ t_exit, u32* __restrict__ send_chg, u32* __restrict__ recv_chg) {
  begin_after();
  const u64 i = (u64)blockIdx.x * RT_THREADS + threadIdx.x;
  if (i >= n_rec) return;
  const u32 rk = __ldg(rank + i);
  const i64 a = __ldg(t_enter + i), b = __ldg(t_exit + i);
  u32 s = 0, q = 0;
  RankTicks r; r.t0 = r.t1 = 0; r.lo = r.n = 0; r.scale = 0.f;
  if (rk < A.n_ranks) {
    const uint4* e = reinterpret_cast<const uint4*>(A.ranks + rk);
    const uint4 x = e[0], y = e[1];
    r.t0 = (i64)((u64)x.x | ((u64)x.y << 32)); r.t1 = (i64)((u64)x.z | ((u64)x.w << 32));
    r.lo = y.x; r.n = y.y; r.scale = __uint_as_float(y.z);
  }
  const bool some = r.n != 0, fly = b == -1;
  const bool la = some && a >= r.t0 && a < r.t1;                     // inside the rank's ticks: there are at least two
  const bool lb = some && !fly && b >= a && b >= r.t0 && b < r.t1;
  const i64* __restrict__ tn = A.tick_ns + r.lo;
  const u32 ga = la ? even_guess(r, a) : 0u, gb = lb ? even_guess(r, b) : 0u;
  i64 x0 = 0, x1 = 0, y0 = 0, y1 = 0;
  if (la) { x0 = __ldg(tn + ga); x1 = __ldg(tn + ga + 1); }
  if (lb) { y0 = __ldg(tn + gb); y1 = __ldg(tn + gb + 1); }
  u32 ca = some && a >= r.t1 ? r.n : 0u;                             // ticks at or before the enter time
  u32 cb = some && (fly || (b >= a && b >= r.t1)) ? r.n : 0u;        // at or before the exit time
  if (la) ca = x0 <= a && x1 > a ? ga + 1 : search_from(tn, r.n, ga, a);
  if (lb) cb = y0 <= b && y1 > b ? gb + 1 : search_from(tn, r.n, gb, b);
  // ticks (ia, ib] count; before the rank's first tick counts as at it, since a first tick is no change
  const u32 ia = r.lo + (ca ? ca - 1 : 0u), ib = r.lo + (cb ? cb - 1 : 0u);
  if (ib > ia) {
    const uint4* t = reinterpret_cast<const uint4*>(A.blk);
    const uint4 ea = t[ia >> 5], eb = t[ib >> 5];
    const u32 pa = changes_upto(TickBlock{ea.x, ea.y, ea.z, 0}, ia), pb = changes_upto(TickBlock{eb.x, eb.y, eb.z, 0}, ib);
    s = (pb & 0xFFFFu) - (pa & 0xFFFFu); q = (pb >> 16) - (pa >> 16);
    const u32 ta = ia / RT_TILE, tb = ib / RT_TILE;
    if (ta != tb) {
      if (A.scanned != nullptr && *A.scanned != 0) { const uint2 x = A.tile[ta], y = A.tile[tb]; s += y.x - x.x; q += y.y - x.y; }
      else for (u32 k = ta; k < tb; ++k) { const uint2 x = A.tile[k]; s += x.x; q += x.y; }
    }
  }
  send_chg[i] = s; recv_chg[i] = q;
}

}  // namespace ccld
