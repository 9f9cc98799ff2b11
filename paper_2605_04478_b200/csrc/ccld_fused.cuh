// Per-op reductions, median / MAD, flags and votes for communicators of up to 128 ranks (sm_100a).
//
//   k_reduce_fused     the common case: every member reported, nothing in flight, all times of the group within
//                      2^31 ns of its first member's enter time (or with equal upper words). n <= 8: one thread per group
//                      with everything in its registers, lanes along consecutive op counters so that the gathers of one
//                      member coalesce. Larger: a tile of op counters is gathered by the whole CTA, lanes along the op
//                      counter, and parked in shared memory as 32-bit keys; then a group sits in L = n_pad / 8 lanes of a
//                      warp, eight ring positions per lane. Three CTAs of 256 threads fit an SM. Any other group is
//                      appended to a list.
//   k_reduce_deferred  the listed groups, one warp each, in full 64-bit generality: missing members, records in
//                      flight (hang alerts), invalid times, spreads beyond 32 bits.
//
// Windows whose records do not lie in their ranks' order have them in the slots (PackedRecord); the second instance of the kernel
// reads them there, coalesced, with the presence of a member still taken from its index.
//
// The work list of k_reduce_fused is chunk-major (see emit_lists), so CTAs that run together gather from the same stretch
// of every rank's records and share the fetched sectors in L2.
#pragma once
#include "ccld_device.cuh"

namespace ccld {

constexpr u32 FULLM = 0xFFFFFFFFu;
#ifndef CCLD_FUSED_MIN_CTAS
#define CCLD_FUSED_MIN_CTAS 3
#endif

template <class K> __device__ __forceinline__ void cswap(K& a, K& b) { const K lo = min(a, b), hi = max(a, b); a = lo; b = hi; }
__device__ __forceinline__ u32 key_absdiff(u32 a, u32 b) { return __usad(a, b, 0u); }
__device__ __forceinline__ u64 key_absdiff(u64 a, u64 b) { return a >= b ? a - b : b - a; }

// 19-exchange sorting network for 8 keys
template <class K> __device__ __forceinline__ void sort8(K (&v)[8]) {
  cswap(v[0], v[2]); cswap(v[1], v[3]); cswap(v[4], v[6]); cswap(v[5], v[7]);
  cswap(v[0], v[4]); cswap(v[1], v[5]); cswap(v[2], v[6]); cswap(v[3], v[7]);
  cswap(v[0], v[1]); cswap(v[2], v[3]); cswap(v[4], v[5]); cswap(v[6], v[7]);
  cswap(v[2], v[4]); cswap(v[3], v[5]);
  cswap(v[1], v[4]); cswap(v[3], v[6]);
  cswap(v[1], v[2]); cswap(v[3], v[4]); cswap(v[5], v[6]);
}
// bitonic merge: sorts 8 keys that first fall and then rise
template <class K> __device__ __forceinline__ void merge8(K (&v)[8]) {
  cswap(v[0], v[4]); cswap(v[1], v[5]); cswap(v[2], v[6]); cswap(v[3], v[7]);
  cswap(v[0], v[2]); cswap(v[1], v[3]); cswap(v[4], v[6]); cswap(v[5], v[7]);
  cswap(v[0], v[1]); cswap(v[2], v[3]); cswap(v[4], v[5]); cswap(v[6], v[7]);
}
template <class K> __device__ __forceinline__ K pick4(const K (&v)[8], u32 k) {
  K r = v[0];
  r = k == 1 ? v[1] : r; r = k == 2 ? v[2] : r; r = k == 3 ? v[3] : r;
  return r;
}

template <class K> struct KeyMax;
template <> struct KeyMax<u32> { static __device__ __forceinline__ u32 v() { return 0xFFFFFFFFu; } };
template <> struct KeyMax<u64> { static __device__ __forceinline__ u64 v() { return U64_MAX_; } };

// lower median and lower-median absolute deviation of x[0..n), n <= 8 (x[p] = maximum key for p >= n)
template <class K> __device__ __forceinline__ void median_mad8(const K (&x)[8], u32 n, K* med, K* mad) {
  K s[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) s[p] = x[p];
  sort8(s);
  const u32 k = (n - 1) >> 1;
  const K m = pick4(s, k);
#pragma unroll
  for (int p = 0; p < 8; ++p) s[p] = (u32)p < n ? key_absdiff(s[p], m) : KeyMax<K>::v();   // falls to 0 at k, then rises
  merge8(s);
  *med = m; *mad = pick4(s, k);
}

// The same for n <= 4. Of three or four members the median is the second smallest, and its neighbour that is nearer is the
// second smallest deviation after its own; of one or two it is the smallest, whose own deviation is 0.
__device__ __forceinline__ void median_mad4(const u32 (&x)[4], u32 n, u32* med, u32* mad) {
  u32 v0 = x[0], v1 = x[1], v2 = x[2], v3 = x[3];
  cswap(v0, v1); cswap(v2, v3); cswap(v0, v2); cswap(v1, v3); cswap(v1, v2);
  *med = n > 2 ? v1 : v0; *mad = n > 2 ? min(v1 - v0, v2 - v1) : 0u;
}

// 1 / x, 1 <= x < 2^64, rounded: Newton's method on the approximate single-precision reciprocal. That is good to about 2^-22
// with the rounding of its argument, and a step squares the relative error (always towards smaller values): two steps leave
// the rounding of the last one.
__device__ __forceinline__ double rcp_newton(double x) {
  float s; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"((float)x));
  double r = (double)s;
  double e = fma(-x, r, 1.0); r = fma(r, e, r);
  e = fma(-x, r, 1.0); r = fma(r, e, r);
  return r;
}
// The same from a whole number >= 1, whose single-precision form needs no detour over fp64, with one step: at most 2^-44 (6e-14)
// too small; the sums of members' bandwidths it serves are 0.7 to 1.6e-15 (rms) below extended precision's.
__device__ __forceinline__ double rcp_u32(u32 x) {
  float s; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint2float_rn(x)));
  const double r = (double)s;
  return fma(r, fma(-(double)x, r, 1.0), r);
}
__device__ __forceinline__ double busbw_fast(double bytes_num, double den, i64 t) {
  return t > 0 ? bytes_num * rcp_newton((double)t * den) : 0.0;
}

// Sums v[m] over the warp for m = 0..P-1; lane l ends up with the total of member l / 4 % P. P = 8: 9 shuffles.
template <int P> __device__ __forceinline__ double warp_sum(double (&v)[P], u32 lane) {
#pragma unroll
  for (int w = P / 2, bit = P * 2; w >= 1; w >>= 1, bit >>= 1) {
    const bool hi = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const double send = hi ? v[i] : v[i + w], keep = hi ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, bit);
    }
  }
  if (P == 4) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 16);
  v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 2);
  v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
  return v[0];
}

template <class K> __device__ __forceinline__ K pick8(const K (&v)[8], u32 r) {
  K x = v[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) x = r == (u32)i ? v[i] : x;
  return x;
}

// One cross-lane step of a merge network: element r of this lane against element r (MIRROR: 7 - r) of lane ^ mask;
// the lane with keep_low set keeps the smaller key of each pair.
template <class K, bool MIRROR>
__device__ __forceinline__ void sub_exchange(K (&v)[8], int mask, bool keep_low) {
  K o[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) o[r] = __shfl_xor_sync(0xFFFFFFFFu, v[MIRROR ? 7 - r : r], mask);
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = keep_low ? min(v[r], o[r]) : max(v[r], o[r]);
}

// Sorts the 8 L keys of a group ascending; element i lives in lane i / 8 (of the group), register i % 8.
template <int L, class K>
__device__ __forceinline__ void sub_sort(K (&v)[8], u32 s) {
  sort8(v);
#pragma unroll
  for (int m = 1; m < L; m <<= 1) {
    // two ascending runs of m lanes each: the mirror step leaves every key of the low run <= every key of the high
    // run and both runs bitonic; half-cleaners across lanes and then inside the lane finish the merge
    sub_exchange<K, true>(v, 2 * m - 1, (s & m) == 0);
#pragma unroll
    for (int h = m >> 1; h >= 1; h >>= 1) sub_exchange<K, false>(v, h, (s & h) == 0);
    merge8(v);
  }
}
// Sorts 8 L keys that fall and then rise.
template <int L, class K>
__device__ __forceinline__ void sub_merge(K (&v)[8], u32 s) {
#pragma unroll
  for (int h = L >> 1; h >= 1; h >>= 1) sub_exchange<K, false>(v, h, (s & h) == 0);
  merge8(v);
}

// Smallest and largest key, lower median and lower-median absolute deviation of a group's keys (v[q] = largest key where no
// member exists; any order). Every lane of the warp must call it.
template <int L, bool FULL>
__device__ __forceinline__ void sub_stats(u32 (&v)[8], u32 n, u32 s, u32 lane, u32* mn, u32* mx, u32* med, u32* mad) {
  const u32 first = lane & ~(u32)(L - 1), k = (n - 1) >> 1;
  sub_sort<L, u32>(v, s);
  *mn = __shfl_sync(0xFFFFFFFFu, v[0], first);
  *mx = __shfl_sync(0xFFFFFFFFu, FULL ? v[7] : pick8(v, (n - 1) & 7), first | ((n - 1) >> 3));
  const u32 m = __shfl_sync(0xFFFFFFFFu, FULL ? v[7] : pick8(v, k & 7), first | (k >> 3));         // full: k = 4 L - 1
  *med = m;
  if constexpr (FULL) {
    // Below the median (element k) the deviations grow downwards, above it upwards. The k + 1 smallest are those of some p .. p + k, p <= k, so
    // the largest of them is the least of max(med - key[p], key[p + k] - med): no second merge. Element p + k = p + 4 L - 1 is one register
    // down in lane s + L / 2, and the last one of the lane before it for register 0.
    u32 best = 0xFFFFFFFFu;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const u32 o = r ? __shfl_xor_sync(0xFFFFFFFFu, v[r ? r - 1 : 0], L / 2) : __shfl_sync(0xFFFFFFFFu, v[7], first + ((s + L / 2 - 1) & (L - 1)));
      best = min(best, max(m - v[r], o - m));
    }
    if (s >= L / 2) best = 0xFFFFFFFFu;
#pragma unroll
    for (int h = 1; h < L; h <<= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, h));
    *mad = best;
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = s * 8 + r < n ? key_absdiff(v[r], m) : 0xFFFFFFFFu;   // falls to 0 at k, then rises
    sub_merge<L, u32>(v, s);
    *mad = __shfl_sync(0xFFFFFFFFu, pick8(v, k & 7), first | (k >> 3));
  }
}

enum { SC_COMP = 0, SC_INC, SC_BAR, SC_AN, SC_MIS, SC_PRES, SC_FS, SC_FD, SC_COUNT };

struct DeferList { u64* entries; u32* count; };    // entry: window index in the batch << 32 | group index in the window

// Where a window's outputs go; kept in shared memory and read when a group stores, so that the pointers do not occupy
// registers across the gathers.
struct OutPtrs { u8* flags; i64* gi64; u32* gu32; double* gbw; u64 G; };
struct InPtrs { const uint4* packed; const u32* perm; const i64 *te, *tx; const u64* by; const u8* op; const u32 *sc, *rc; };
template <class T> __device__ __forceinline__ T ld_volatile(const T& x) { return *(const volatile T*)&x; }

constexpr u32 TILE_KEYS = 8 * SMALL_SEQS;                     // keys of a metric of a staged tile
constexpr u32 TILE_OPS = 64;                                  // op counters of a staged tile at most
struct FusedShared {
  u32 cnt[SC_COUNT];
  OutPtrs out; InPtrs in;
  // n <= 8: eight warps' slots for the record indices of a tile. Larger: a tile's keys as [metric][member][op counter].
  u32 stage[2 * TILE_KEYS];
  // staged tiles, per op counter: why the group is set aside (1) or its op set differs (2), latest exit, first member's
  u32 t_bits[TILE_OPS], t_xmax[TILE_OPS], t_gop[TILE_OPS];    //   op code,
  u64 t_base[TILE_OPS], t_gby[TILE_OPS];                      //   time base and size
  u64 t_ck[TILE_OPS];                                         //   most changes, then the lowest position
  double t_bd[TILE_OPS];                                      //   bytes * factor where the group adds bandwidth, else 0
  u32 mem[WARP_N];                                            // the communicator's ranks
  u32 brng[SMALL_SEQS / 32], bk[SMALL_SEQS / 32], rounds[SMALL_SEQS / 32], n_an[SMALL_SEQS / 32], n_def[SMALL_SEQS / 32];
};

// Three CTAs fit 64 KB of shared memory, which leaves 192 KB of an SM to its L1. How many lines L1 holds is how many gathers can
// be on their way: on twelve windows of 4,096 ranks in groups of 8 and 64 the kernel took 1,071 us with 28 KB of L1, 598 with
// 121, 587 with 156 and 577 with 192 (541 now, with full units in short chunks).
static_assert(CCLD_FUSED_MIN_CTAS * (sizeof(FusedShared) + 1024) <= 64 * 1024, "fits the 64 KB split (a CTA's first KB is the system's)");
constexpr int FUSED_CARVEOUT = (int)((100 * CCLD_FUSED_MIN_CTAS * (sizeof(FusedShared) + 1024) + 228 * 1024 - 1) / (228 * 1024));     // percent

__device__ __forceinline__ void flush_counters(const WinDesc& D, const FusedShared& sh) {
  u64* const counters = D.counters;
  count_add(counters, C_COMPLETE, sh.cnt[SC_COMP]); count_add(counters, C_BARRIER, sh.cnt[SC_BAR]); count_add(counters, C_ANALYSED, sh.cnt[SC_AN]);
  count_add(counters, C_MISMATCH, sh.cnt[SC_MIS]); count_add(counters, C_PRESENT, sh.cnt[SC_PRES]);
  count_add(counters, C_FLAG_SKEW, sh.cnt[SC_FS]); count_add(counters, C_FLAG_DUR, sh.cnt[SC_FD]);
}

// ------------------------------------------------------------------------------------------------
// n <= 8: a warp per tile of up to 32 consecutive op counters, one group per lane
// ------------------------------------------------------------------------------------------------
// What a warp carries from tile to tile.
struct SmallAcc { u32 complete = 0, barrier = 0, analysed = 0, mismatch = 0, present = 0, flagged = 0; };   // flagged: this lane's kind of vote (lane % 4)

// Up to four ranks a lane holds four positions: with eight, half of them empty, two windows of groups of 4, 4 and 128 took 86 us
// instead of 75, of 2 and 3 134 instead of 119. (Five to seven of eight are used above.)
constexpr u32 HALF_N = 4;

// A tile's list entry as one word per lane (16 words), so that the next tile's can wait in a single register.
static_assert(sizeof(WarpTile) == 64, "an entry is sixteen words");
__device__ __forceinline__ u32 entry_word(u32 e, u32 w) { return __shfl_sync(FULLM, e, w); }
__device__ __forceinline__ u64 entry_pair(u32 e, u32 w) { return (u64)entry_word(e, w) | ((u64)entry_word(e, w + 1) << 32); }

// The record indices of the tile behind entry e, asked into the warp's slots; lane l reads back what lane l asked for.
__device__ __forceinline__ void ask_indices(const FusedShared& sh, u32 e, u32 lane, u32* __restrict__ slots /* [8][32] */) {
  const u32 count = entry_word(e, 2), n_seq = entry_word(e, 5), n = entry_word(e, 7);
  const u32* pm = ld_volatile(sh.in.perm) + entry_pair(e, 10) + entry_word(e, 1) + (lane < count ? lane : 0u);
  const u32 dst = (u32)__cvta_generic_to_shared(slots + lane);
#pragma unroll
  for (u32 q = 0; q < 8; ++q) {
    if (q >= HALF_N && n <= HALF_N) break;
    // positions beyond the communicator repeat its first member, which changes no extreme and no comparison
    const u32* src = pm + (u64)(q < n ? q : 0u) * n_seq;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst + q * 128u), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// P: positions a lane holds, eight or, for communicators of up to four ranks, four. FULL: as many members. PACKED: the records lie in their slots. e: the tile's entry, its indices asked for earlier; e_next: the entry of the warp's next tile, if it has
// one. One exposed round trip to memory per tile: times, sizes and op codes are asked for together as soon as the indices
// are there, the rate columns while the order statistics are worked out, the next tile's indices before any of it.
template <int P, bool FULL, bool PACKED>
__device__ __forceinline__ void small_tile(u32 w_idx, u32 e, u32 e_next, bool has_next, TileSum* __restrict__ sums, const Registry& R, const Params& Pm,
                                           const DeferList& DL, FusedShared& sh, u32* __restrict__ slots, u32 lane, SmallAcc& acc) {
  static_assert(P == 8 || (P == 4 && !FULL), "positions");
  const u32 n = FULL ? 8u : entry_word(e, 7), count = entry_word(e, 2);
  const bool active = lane < count;
  const u32* __restrict__ mem = R.members + entry_pair(e, 14);
  const u32 mem_l = lane < n ? __ldg(mem + lane) : 0u;        // lane m holds the rank of position m
  if (!PACKED) asm volatile("cp.async.wait_group 0;" ::: "memory");
  u32 a[P], d[P];                                             // enter time against base, duration
  u64 base, gby; u32 gop, idx[P], xmax, ch[P];
  bool ok, mm;
  {
    i64 ta[P], tb[P]; u64 by[P]; u32 op[P];
    if (PACKED) {
      const u32 n_seq = entry_word(e, 5);
      const uint4* at = ld_volatile(sh.in.packed) + 2 * (entry_pair(e, 10) + entry_word(e, 1) + (active ? lane : 0u));
#pragma unroll
      for (int q = 0; q < P; ++q) {
        const PackedRecord r = load_packed(at + 2 * (u64)((u32)q < n ? q : 0) * n_seq);
        ta[q] = (i64)r.te; tb[q] = (i64)r.tx; by[q] = r.by; op[q] = r.op; ch[q] = r.ch;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    u32 top = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) { idx[q] = slots[q * 32 + lane]; top = max(top, idx[q]); }
    const bool present = top != NONE;                         // a missing member: the group is deferred
#pragma unroll
    for (int q = 0; q < P; ++q) idx[q] = present ? idx[q] : 0u;
    if (has_next) ask_indices(sh, e_next, lane, slots);
    if (!PACKED) {
      const i64* __restrict__ c_te = ld_volatile(sh.in.te); const i64* __restrict__ c_tx = ld_volatile(sh.in.tx);
      const u64* __restrict__ c_by = ld_volatile(sh.in.by); const u8* __restrict__ c_op = ld_volatile(sh.in.op);
#pragma unroll
      for (int q = 0; q < P; ++q) { ta[q] = __ldg(c_te + idx[q]); tb[q] = __ldg(c_tx + idx[q]); }
#pragma unroll
      for (int q = 0; q < P; ++q) { by[q] = __ldg(c_by + idx[q]); op[q] = __ldg(c_op + idx[q]); }
    }
    // The upper words of a group's times are nearly always the same (they change every 4.3 s): the lower words are the keys
    // then. Otherwise, and for anything irregular, offsets from the first member's enter time - 2^31 decide.
    const u32 h0 = (u32)((u64)ta[0] >> 32);
    u32 x = 0; bool back = false;
    xmax = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      x |= ((u32)((u64)ta[q] >> 32) ^ h0) | ((u32)((u64)tb[q] >> 32) ^ h0);
      a[q] = (u32)ta[q]; d[q] = (u32)tb[q] - (u32)ta[q];
      back = back || (u32)tb[q] < (u32)ta[q];
      xmax = max(xmax, (u32)tb[q]);
    }
    base = (u64)h0 << 32;
    ok = x == 0 && (int)h0 >= 0 && !back;
    if (!ok) {
      base = (u64)ta[0] - 0x80000000ull;
      u32 hx = 0, neg = 0;
      back = false; xmax = 0;
#pragma unroll
      for (int q = 0; q < P; ++q) {
        const u64 ra = (u64)ta[q] - base, rb = (u64)tb[q] - base;
        a[q] = (u32)ra; d[q] = (u32)rb - (u32)ra; xmax = max(xmax, (u32)rb);
        hx |= (u32)(ra >> 32) | (u32)(rb >> 32);
        neg |= (u32)((u64)ta[q] >> 32) | (u32)((u64)tb[q] >> 32);
        back = back || (u32)rb < (u32)ra;
      }
      ok = hx == 0 && (int)neg >= 0 && !back;                 // within 32 bits, not negative, not in flight (t_exit = -1), exit after enter
    }
    ok = ok && present;
    gby = by[0]; gop = op[0];
    u32 y = 0;
#pragma unroll
    for (int q = 1; q < P; ++q) y |= ((u32)by[q] ^ (u32)gby) | ((u32)(by[q] >> 32) ^ (u32)(gby >> 32)) | (op[q] ^ gop);
    mm = y != 0;
  }
  // the rate columns, read only after the order statistics
  if (!PACKED) {
    const u32* __restrict__ c_sc = ld_volatile(sh.in.sc); const u32* __restrict__ c_rc = ld_volatile(sh.in.rc);
    if (c_sc != nullptr) {
      u32 rc[P];
#pragma unroll
      for (int q = 0; q < P; ++q) { ch[q] = __ldg(c_sc + idx[q]); rc[q] = __ldg(c_rc + idx[q]); }
#pragma unroll
      for (int q = 0; q < P; ++q) ch[q] = max(ch[q], rc[q]);
    } else {
#pragma unroll
      for (int q = 0; q < P; ++q) ch[q] = 0;
    }
  }
  const u32 sum_idx = entry_word(e, 3), seq_off = entry_word(e, 1);      // (every lane takes part in these)
  const u64 group0 = entry_pair(e, 8), slot0 = entry_pair(e, 10);
  const bool gok = active && ok;
  if (active && !ok) {
    const u32 at = atomicAdd(DL.count, 1u);
    DL.entries[at] = ((u64)w_idx << 32) | (u64)(group0 + seq_off + lane);
  }
  const u32 b_ok = __ballot_sync(FULLM, gok);
  const bool barrier = gop == CCLD_OP_ALLREDUCE && gby < Pm.barrier_bytes;
  const bool round = gok && !barrier, analysed = round && n >= Pm.min_group;
  const u32 b_an = __ballot_sync(FULLM, analysed), b_round = __ballot_sync(FULLM, round), b_mm = __ballot_sync(FULLM, gok && mm);
  // ---- extremes and order statistics ----
  u32 emin, emax, tmx, tmn, ms = 0, ds = 0, md = 0, dm = 0;
  if constexpr (FULL) {
    // the sorted keys give the extremes and the median (element 3). Below it the deviations L grow downwards, above it R
    // upwards; the lower-median deviation is the third smallest of the two rows, and that is the least of max(L_i, R_j)
    // over i + j = 3: no second sort.
    u32 v[8];
#pragma unroll
    for (int q = 0; q < P; ++q) v[q] = a[q];
    sort8(v);
    emin = v[0]; emax = v[7]; ms = v[3] - emin;
    ds = min(min(v[3] - v[0], v[6] - v[3]), min(max(v[3] - v[2], v[5] - v[3]), max(v[3] - v[1], v[4] - v[3])));
#pragma unroll
    for (int q = 0; q < P; ++q) v[q] = d[q];
    sort8(v);
    tmn = v[0]; tmx = v[7]; md = v[3] - tmn;
    dm = min(min(v[3] - v[0], v[6] - v[3]), min(max(v[3] - v[2], v[5] - v[3]), max(v[3] - v[1], v[4] - v[3])));
  } else {
    emin = a[0]; emax = a[0]; tmx = d[0]; tmn = d[0];
#pragma unroll
    for (int q = 1; q < P; ++q) { emin = min(emin, a[q]); emax = max(emax, a[q]); tmx = max(tmx, d[q]); tmn = min(tmn, d[q]); }
    if (b_an != 0) {
      u32 v[P];
#pragma unroll
      for (int q = 0; q < P; ++q) v[q] = q < (int)n ? a[q] - emin : 0xFFFFFFFFu;
      if constexpr (P == 8) median_mad8<u32>(v, n, &ms, &ds); else median_mad4(v, n, &ms, &ds);
#pragma unroll
      for (int q = 0; q < P; ++q) v[q] = q < (int)n ? d[q] - tmn : 0xFFFFFFFFu;
      if constexpr (P == 8) median_mad8<u32>(v, n, &md, &dm); else median_mad4(v, n, &md, &dm);
    }
  }
  if (!analysed) { ms = ds = md = dm = 0; }
  // ---- flags ----
  u32 f_lo = 0, f_hi = 0;
  {
    // |x - med| * 1000 > k * MAD in whole numbers: |x - med| > T = floor(k * MAD / 1000), which holds outside
    // [med - T, med + T]; a quotient of 2^32 - 1 or more is never exceeded. One subtraction and one comparison per value.
    const u64 qs = (u64)ds * Pm.k_milli / 1000u, qd = (u64)dm * Pm.k_milli / 1000u;
    const u32 ts = qs > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qs, td = qd > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qd;
    const u32 los = ms > ts ? ms - ts : 0u, lod = md > td ? md - td : 0u;
    const u32 ws = (ms + ts < ms ? 0xFFFFFFFFu : ms + ts) - los, wd = (md + td < md ? 0xFFFFFFFFu : md + td) - lod;
    const u32 s0 = emin + los, d0 = tmn + lod, sm = emin + ms, dmd = tmn + md;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      u32& f = q < 4 ? f_lo : f_hi;
      const int at = 8 * (q & 3);
      if (a[q] - s0 > ws) f |= (u32)CCLD_F_SKEW_OUT << at;
      if (d[q] - d0 > wd) f |= (u32)CCLD_F_DUR_OUT << at;
      if (a[q] > sm) f |= (u32)CCLD_F_SKEW_HI << at;
      if (d[q] > dmd) f |= (u32)CCLD_F_DUR_HI << at;
    }
    if (!FULL) {                                              // positions that do not exist
      f_lo &= n >= 4 ? 0xFFFFFFFFu : (1u << (8 * n)) - 1u;
      if (P == 8) f_hi &= n > 4 ? (n >= 8 ? 0xFFFFFFFFu : (1u << (8 * (n - 4))) - 1u) : 0u;
    }
    if (!analysed) { f_lo = 0x80808080u; f_hi = 0x80808080u; }
  }
  if (gok) {
    u8* __restrict__ fp = ld_volatile(sh.out.flags) + slot0 + (u64)(seq_off + lane) * n;
    if (FULL && (reinterpret_cast<uintptr_t>(fp) & 7) == 0) *reinterpret_cast<uint2*>(fp) = make_uint2(f_lo, f_hi);
    else if (P == 4 && n == 4 && (reinterpret_cast<uintptr_t>(fp) & 3) == 0) *reinterpret_cast<u32*>(fp) = f_lo;
    else {
#pragma unroll
      for (int q = 0; q < P; ++q) if (FULL || q < (int)n) fp[q] = (u8)((q < 4 ? f_lo >> (8 * q) : f_hi >> (8 * (q - 4))) & 0xFFu);
    }
  }
  // ---- votes: the four kinds of outlier as one bit per member's byte, summed over the warp four members at a time (a sum
  // fits its byte); lane 4 m + kind then holds member m's count of its kind and adds it with the warp's one atomic ----
  static_assert(CCLD_F_SKEW_OUT == 1 && CCLD_F_DUR_OUT == 2 && CCLD_F_SKEW_HI == 4 && CCLD_F_DUR_HI == 8, "flag bit layout");
  const u32 m = lane / 4 % P, rank_m = __shfl_sync(FULLM, mem_l, m);
  {
    const u32 one = 0x01010101u;
    u32 mine = 0;
#pragma unroll
    for (int half = 0; half < P / 4; ++half) {
      const u32 f = gok ? (half ? f_hi : f_lo) : 0u;
      const u32 so = f & one, dq = (f >> 1) & one, sh_ = so & (f >> 2), dh = dq & (f >> 3);
      const u32 v0 = __reduce_add_sync(FULLM, sh_), v1 = __reduce_add_sync(FULLM, so ^ sh_), v2 = __reduce_add_sync(FULLM, dh), v3 = __reduce_add_sync(FULLM, dq ^ dh);
      const u32 v01 = lane & 1 ? v1 : v0, v23 = lane & 1 ? v3 : v2, v = lane & 2 ? v23 : v01;
      if ((lane >> 4) == (u32)half) mine = v;
    }
    mine = (mine >> (8 * (m & 3))) & 0xFFu;
    if (mine) atomicAdd(&R.votes[(u64)rank_m * 4 + (lane & 3)], mine);
    acc.flagged += mine;
  }
  // ---- positions of the extremes (lowest among equals), ranks the row names ----
  u32 cmx = ch[0];
#pragma unroll
  for (int q = 1; q < P; ++q) cmx = max(cmx, ch[q]);
  u32 pmax = 0, pmin = 0, pchg = 0;
#pragma unroll
  for (int q = P - 1; q >= 0; --q) { pmax = d[q] == tmx ? (u32)q : pmax; pmin = d[q] == tmn ? (u32)q : pmin; pchg = ch[q] == cmx ? (u32)q : pchg; }
  const u32 r_tmin = __shfl_sync(FULLM, mem_l, pmin), r_tmax = __shfl_sync(FULLM, mem_l, pmax), r_chg = __shfl_sync(FULLM, mem_l, pchg);
  // bytes * num / den: for eight members the factors 14/8 and 7/8 are exact; for others one rounding, and the row's value, which
  // is a single quotient, is taken from the product before it
  double bn, bnum = 0.0, den = 1.0;
  if (FULL) bn = (double)gby * (gop == CCLD_OP_ALLREDUCE ? 1.75 : ((gop == CCLD_OP_ALLGATHER || gop == CCLD_OP_REDUCESCATTER || gop == CCLD_OP_ALLTOALL) ? 0.875 : 1.0));
  else { double num; bus_factor(gop, n, &num, &den); bnum = (double)gby * num; bn = bnum / den; }
  if (gok) {
    const u64 g = group0 + seq_off + lane, G = ld_volatile(sh.out.G);
    i64* __restrict__ gi = ld_volatile(sh.out.gi64) + g; u32* __restrict__ gu = ld_volatile(sh.out.gu32) + g;
    const u32 span = xmax - emin;
    gi[(u64)GI_E_MIN * G] = (i64)(base + emin); gi[(u64)GI_ARRIVAL_SKEW * G] = (i64)(u64)(emax - emin);
    gi[(u64)GI_T_MAX * G] = (i64)(u64)tmx; gi[(u64)GI_T_MIN * G] = (i64)(u64)tmn; gi[(u64)GI_SPAN * G] = (i64)(u64)span;
    gi[(u64)GI_MED_SKEW * G] = (i64)(u64)ms; gi[(u64)GI_MAD_SKEW * G] = (i64)(u64)ds;
    gi[(u64)GI_MED_DUR * G] = analysed ? (i64)((u64)tmn + md) : 0; gi[(u64)GI_MAD_DUR * G] = (i64)(u64)dm;
    gu[(u64)GU_RANK_TMIN * G] = r_tmin; gu[(u64)GU_RANK_TMAX * G] = r_tmax;
    gu[(u64)GU_MAX_CHG * G] = cmx; gu[(u64)GU_RANK_MAX_CHG * G] = r_chg;
    gu[(u64)GU_N_PRESENT * G] = n;
    gu[(u64)GU_GFLAGS * G] = CCLD_G_COMPLETE | (barrier ? CCLD_G_BARRIER : 0) | (mm ? CCLD_G_OPSET_MISMATCH : 0) | (analysed ? CCLD_G_ANALYSED : 0);
    ld_volatile(sh.out.gbw)[g] = !span ? 0.0 : (FULL ? bn * rcp_newton((double)span) : bnum * rcp_newton((double)span * den));
  }
  // ---- per-member bandwidth, summed over the warp; the Eq. 2 candidate; counts ----
  double bw[P];
  const double bd = round ? bn : 0.0;
  if (!__any_sync(FULLM, tmn == 0)) {
#pragma unroll
    for (int q = 0; q < P; ++q) bw[q] = bd * rcp_u32(d[q]);
  } else {                                                    // an op of no duration adds nothing
#pragma unroll
    for (int q = 0; q < P; ++q) bw[q] = d[q] != 0 ? bd * rcp_u32(d[q]) : 0.0;
  }
  const double tot = warp_sum<P>(bw, lane);                   // lane l holds member m
  const u32 rounds = (u32)__popc(b_round);
  if ((lane & 3) == 0 && lane < 4 * n && rounds) { atomicAdd(&R.bw_sum[rank_m], tot); atomicAdd(&R.bw_cnt[rank_m], rounds); }
  const u32 rng = round ? tmx - tmn : 0u, best = __reduce_max_sync(FULLM, rng);
  const u32 b_best = __ballot_sync(FULLM, round && rng == best);            // ties: the lowest op counter
  const u32 n_ok = (u32)__popc(b_ok), n_an = (u32)__popc(b_an);
  if (lane == 0) {
    TileSum ts; ts.best_rng = b_best ? best : 0u; ts.best_k = b_best ? seq_off + (u32)__ffs(b_best) - 1u : NONE; ts.n_rounds = rounds; ts.n_an = n_an;
    ts.pad = count - n_ok;
    sums[sum_idx] = ts;
  }
  acc.complete += n_ok; acc.barrier += n_ok - rounds; acc.analysed += n_an; acc.mismatch += (u32)__popc(b_mm); acc.present += n_ok * n;
}

// Class-0 CTA: up to FUSED_WT_PER_CTA warp-tiles of one window and one time chunk, each up to 32 consecutive op counters of
// one communicator with its own summary entry. A warp takes every eighth tile and meets the other warps only at the end, so
// the warps of a CTA drift apart and one warp's gathers overlap another's arithmetic.
template <bool PACKED> __device__ __forceinline__ void fused_small_cta(const WinDesc& D, const FusedCta& t, const WarpTile* wts, TileSum* __restrict__ sums,
                                                const Registry& R, const Params& P, const DeferList& DL, FusedShared& sh) {
  const u32 wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr u32 NW = SMALL_SEQS / 32;
  u32* const slots = sh.stage + wid * 256;
  const u32* list = reinterpret_cast<const u32*>(wts + t.wt_first);
  const auto entry = [&](u32 i) { return i < t.wt_count ? list[(u64)i * 16 + (lane & 15)] : 0u; };
  u32 e = entry(wid);
  __syncthreads();                                          // the CTA's counters and pointers are set
  if (wid < t.wt_count) ask_indices(sh, e, lane, slots);
  u32 e_next = entry(wid + NW);
  SmallAcc acc;
  for (u32 i = wid; i < t.wt_count; i += NW) {
    const u32 e_after = entry(i + 2 * NW);
    const bool has_next = i + NW < t.wt_count;
    const u32 n = entry_word(e, 7);
    if (n == SMALL_N) small_tile<8, true, PACKED>(t.w, e, e_next, has_next, sums, R, P, DL, sh, slots, lane, acc);
    else if (n > HALF_N) small_tile<8, false, PACKED>(t.w, e, e_next, has_next, sums, R, P, DL, sh, slots, lane, acc);
    else small_tile<4, false, PACKED>(t.w, e, e_next, has_next, sums, R, P, DL, sh, slots, lane, acc);
    e = e_next; e_next = e_after;
  }
  const u32 f_skew = __reduce_add_sync(FULLM, lane & 2 ? 0u : acc.flagged), f_dur = __reduce_add_sync(FULLM, lane & 2 ? acc.flagged : 0u);
  if (lane == 0) {
    atomicAdd(&sh.cnt[SC_COMP], acc.complete); atomicAdd(&sh.cnt[SC_BAR], acc.barrier); atomicAdd(&sh.cnt[SC_AN], acc.analysed);
    atomicAdd(&sh.cnt[SC_MIS], acc.mismatch); atomicAdd(&sh.cnt[SC_PRES], acc.present); atomicAdd(&sh.cnt[SC_FS], f_skew); atomicAdd(&sh.cnt[SC_FD], f_dur);
  }
  __syncthreads();
  if (threadIdx.x == 0) flush_counters(D, sh);
}

// Class-1 CTA (9 <= n <= 128, L = n_pad / 8): one tile of S = 256 / L consecutive op counters of one communicator, eight
// records per thread. A thread gathers op counter t % S of members t / S, t / S + L, ... - lanes along the op counter, so the
// record indices of a warp are contiguous and, in a rank-major upload, its records lie in one short stretch of a rank's
// stream - with one exposed round trip for times, sizes and op codes; the rate columns are on their way while the groups
// are sorted. Keys meet in shared memory; then L lanes take a group, eight members each (position q L + s in lane s). Last, a thread sums eight op counters of one member's
// bandwidth.
template <int L, bool FULL, bool PACKED>
__device__ __forceinline__ void fused_sub_cta(const WinDesc& D, const FusedCta& t, TileSum* __restrict__ sums, const Registry& R, const Params& P,
                                              const DeferList& DL, FusedShared& sh) {
  constexpr u32 S = SMALL_SEQS / L, GW = 32 / L, NW = SMALL_SEQS / 32;
  // Member p's key of op counter j lies at p S + (j ^ turn(p)): the lanes of an access, GW op counters of L members (or S of
  // 32 / S), meet 32 different banks.
  const auto turn = [](u32 p) { return L == 4 ? (p & 3u) << 3 : (L == 8 ? (p & 7u) << 2 : (p >> 1 & 7u) << 1); };
  static_assert(8 * L * S == TILE_KEYS && S <= TILE_OPS, "tile fits");
  const u32 wid = threadIdx.x >> 5, lane = threadIdx.x & 31, n = FULL ? (u32)(8 * L) : t.row.n, count = t.count;
  u32* __restrict__ k_a = sh.stage; u32* __restrict__ k_d = sh.stage + TILE_KEYS;
  if (threadIdx.x < S) { sh.t_bits[threadIdx.x] = 0; sh.t_xmax[threadIdx.x] = 0; sh.t_ck[threadIdx.x] = 0; }
  if (threadIdx.x < n) sh.mem[threadIdx.x] = __ldg(R.members + t.moff + threadIdx.x);
  __syncthreads();                                            // counters and pointers are set, the arrays above clear
  // ---- gather ----
  const u32 sq = threadIdx.x % S, mr = threadIdx.x / S;
  u32 sc[8], rc[8];
  {
    const u32* pm = ld_volatile(sh.in.perm) + t.row.slot0 + t.seq_off + (sq < count ? sq : 0u);
    u32 idx[8], top = 0;
    const u32 i0 = *pm;
#pragma unroll
    for (int q = 0; q < 8; ++q) { const u32 p = mr + (u32)q * L; idx[q] = pm[(u64)(FULL || p < n ? p : mr) * t.row.n_seq]; top = max(top, idx[q]); }
    u32 bits = top == NONE || i0 == NONE ? 1u : 0u;           // a missing member: the group is set aside
#pragma unroll
    for (int q = 0; q < 8; ++q) idx[q] = idx[q] == NONE ? 0u : idx[q];
    i64 ta[8], tb[8], te0; u64 by[8], by0; u32 op[8], op0;
    if (PACKED) {
      const uint4* at = ld_volatile(sh.in.packed) + 2 * (t.row.slot0 + t.seq_off + (sq < count ? sq : 0u));
      { const PackedRecord r = load_packed(at); te0 = (i64)r.te; by0 = r.by; op0 = r.op; }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const u32 p = mr + (u32)q * L;
        const PackedRecord r = load_packed(at + 2 * (u64)(FULL || p < n ? p : mr) * t.row.n_seq);
        ta[q] = (i64)r.te; tb[q] = (i64)r.tx; by[q] = r.by; op[q] = r.op; sc[q] = r.ch; rc[q] = 0;
      }
    } else {
      const i64* __restrict__ c_te = ld_volatile(sh.in.te); const i64* __restrict__ c_tx = ld_volatile(sh.in.tx);
      const u64* __restrict__ c_by = ld_volatile(sh.in.by); const u8* __restrict__ c_op = ld_volatile(sh.in.op);
      const u32 j0 = i0 == NONE ? 0u : i0;
      te0 = __ldg(c_te + j0); by0 = __ldg(c_by + j0); op0 = __ldg(c_op + j0);
#pragma unroll
      for (int q = 0; q < 8; ++q) { ta[q] = __ldg(c_te + idx[q]); tb[q] = __ldg(c_tx + idx[q]); }
#pragma unroll
      for (int q = 0; q < 8; ++q) { by[q] = __ldg(c_by + idx[q]); op[q] = __ldg(c_op + idx[q]); }
    }
    const u64 base = (u64)te0 - 0x80000000ull;
    u32 hx = 0, neg = 0, xmax = 0; bool back = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const u32 p = mr + (u32)q * L;
      const u64 ra = (u64)ta[q] - base, rb = (u64)tb[q] - base;
      const u32 a = (u32)ra, b = (u32)rb;
      hx |= (u32)(ra >> 32) | (u32)(rb >> 32);
      neg |= (u32)((u64)ta[q] >> 32) | (u32)((u64)tb[q] >> 32);
      back = back || b < a; xmax = max(xmax, b);
      const u32 k = p * S + (sq ^ turn(p));
      k_a[k] = FULL || p < n ? a : 0xFFFFFFFFu; k_d[k] = FULL || p < n ? b - a : 0xFFFFFFFFu;
    }
    if (hx != 0 || (int)neg < 0 || back) bits |= 1;           // beyond 32 bits, negative or in flight, exit before enter
    u32 y = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) y |= ((u32)by[q] ^ (u32)by0) | ((u32)(by[q] >> 32) ^ (u32)(by0 >> 32)) | (op[q] ^ op0);
    if (y) bits |= 2;
    if (bits) atomicOr(&sh.t_bits[sq], bits);
    atomicMax(&sh.t_xmax[sq], xmax);
    if (mr == 0) { sh.t_base[sq] = base; sh.t_gby[sq] = by0; sh.t_gop[sq] = op0; }
    if (!PACKED) {
      const u32* __restrict__ c_sc = ld_volatile(sh.in.sc); const u32* __restrict__ c_rc = ld_volatile(sh.in.rc);
      if (c_sc != nullptr) {
#pragma unroll
        for (int q = 0; q < 8; ++q) { sc[q] = __ldg(c_sc + idx[q]); rc[q] = __ldg(c_rc + idx[q]); }
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) sc[q] = rc[q] = 0;
      }
    }
  }
  __syncthreads();
  // ---- a group in L lanes ----
  {
    const u32 s = lane % L, jt = wid * GW + lane / L;         // my group's op counter inside the tile
    const bool lead = s == 0, active = jt < count;
    const u32 bits = sh.t_bits[jt], gop = sh.t_gop[jt]; const u64 gby = sh.t_gby[jt];
    const bool gok = active && !(bits & 1), mm = (bits & 2) != 0;
    const bool barrier = gop == CCLD_OP_ALLREDUCE && gby < P.barrier_bytes;
    const bool round = gok && !barrier, analysed = round && n >= P.min_group;
    const u32 mine = s * S + (jt ^ turn(s));                  // member q L + s: 256 q further
    const u32* __restrict__ ka = k_a + mine; const u32* __restrict__ kd = k_d + mine;
    u32 emin, emax, ms, ds, tmn, tmx, md, dm;
    {
      u32 v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = ka[q * SMALL_SEQS];
      sub_stats<L, FULL>(v, n, s, lane, &emin, &emax, &ms, &ds);
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = kd[q * SMALL_SEQS];
      sub_stats<L, FULL>(v, n, s, lane, &tmn, &tmx, &md, &dm);
    }
    ms -= emin; md -= tmn;
    if (!analysed) { ms = ds = md = dm = 0; }
    // lowest position that holds the longest / shortest duration; flags, votes
    u32 pmax = NONE, pmin = NONE, n_fs = 0, n_fd = 0;
    {
      const u64 qs = (u64)ds * P.k_milli / 1000u, qd = (u64)dm * P.k_milli / 1000u;     // outside [med - T, med + T], T = floor(k * MAD / 1000)
      const u32 ts = qs > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qs, td = qd > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qd;
      const u32 los = ms > ts ? ms - ts : 0u, lod = md > td ? md - td : 0u;
      const u32 ws = (ms + ts < ms ? 0xFFFFFFFFu : ms + ts) - los, wd = (md + td < md ? 0xFFFFFFFFu : md + td) - lod;
      const u32 s0 = emin + los, d0 = tmn + lod, sm = emin + ms, dmd = tmn + md;
      u8* __restrict__ fp = ld_volatile(sh.out.flags) + t.row.slot0 + (u64)(t.seq_off + (active ? jt : 0u)) * n + s;
      u32 out = 0;                                            // outlier bits of my eight members, four apiece
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        if (!FULL && q * L + s >= n) continue;
        const u32 a = ka[q * SMALL_SEQS], d = kd[q * SMALL_SEQS];
        u32 f = a - s0 > ws ? (u32)CCLD_F_SKEW_OUT : 0u;
        if (d - d0 > wd) f |= CCLD_F_DUR_OUT;
        if (a > sm) f |= CCLD_F_SKEW_HI;
        if (d > dmd) f |= CCLD_F_DUR_HI;
        if (d == tmx) pmax = q * L + s;
        if (d == tmn) pmin = q * L + s;
        out |= f << (4 * q);
        if (gok) fp[q * L] = analysed ? (u8)f : (u8)CCLD_F_NOT_ANALYSED;
      }
      // votes: outliers are rare, so they are taken off the flag bits one at a time
      if (analysed) {
        n_fs = (u32)__popc(out & 0x11111111u); n_fd = (u32)__popc(out & 0x22222222u);
        for (u32 o = out & 0x33333333u; o; o &= o - 1u) {
          const u32 b = (u32)__ffs(o) - 1u, dur = b & 1u, hi = (out >> (b + 2u)) & 1u;
          atomicAdd(&R.votes[(u64)sh.mem[(b >> 2) * L + s] * 4 + 2u * dur + (hi ? 0u : 1u)], 1u);
        }
      }
    }
#pragma unroll
    for (int h = 1; h < L; h <<= 1) { pmax = min(pmax, __shfl_xor_sync(FULLM, pmax, h)); pmin = min(pmin, __shfl_xor_sync(FULLM, pmin, h)); }
    double num, den; bus_factor(gop, n, &num, &den);
    const double bnum = (double)gby * num, bd = bnum / den;   // (a full group's den is a power of two: exact)
    if (lead && active) {
      sh.t_bd[jt] = round ? bd : 0.0;
      if (gok) {
        const u64 g = t.row.group0 + t.seq_off + jt, G = ld_volatile(sh.out.G);
        i64* __restrict__ gi = ld_volatile(sh.out.gi64) + g; u32* __restrict__ gu = ld_volatile(sh.out.gu32) + g;
        const u32 span = sh.t_xmax[jt] - emin;
        gi[(u64)GI_E_MIN * G] = (i64)(sh.t_base[jt] + emin); gi[(u64)GI_ARRIVAL_SKEW * G] = (i64)(u64)(emax - emin);
        gi[(u64)GI_T_MAX * G] = (i64)(u64)tmx; gi[(u64)GI_T_MIN * G] = (i64)(u64)tmn; gi[(u64)GI_SPAN * G] = (i64)(u64)span;
        gi[(u64)GI_MED_SKEW * G] = (i64)(u64)ms; gi[(u64)GI_MAD_SKEW * G] = (i64)(u64)ds;
        gi[(u64)GI_MED_DUR * G] = analysed ? (i64)((u64)tmn + md) : 0; gi[(u64)GI_MAD_DUR * G] = (i64)(u64)dm;
        gu[(u64)GU_RANK_TMIN * G] = sh.mem[pmin]; gu[(u64)GU_RANK_TMAX * G] = sh.mem[pmax];
        gu[(u64)GU_N_PRESENT * G] = n;
        gu[(u64)GU_GFLAGS * G] = CCLD_G_COMPLETE | (barrier ? CCLD_G_BARRIER : 0) | (mm ? CCLD_G_OPSET_MISMATCH : 0) | (analysed ? CCLD_G_ANALYSED : 0);
        ld_volatile(sh.out.gbw)[g] = !span ? 0.0 : (FULL ? bd * rcp_newton((double)span) : bnum * rcp_newton((double)span * den));
      } else {
        const u32 e = atomicAdd(DL.count, 1u);
        DL.entries[e] = ((u64)t.w << 32) | (u64)(t.row.group0 + t.seq_off + jt);
      }
    }
    // the warp's counts and Eq. 2 candidate (ties: the lowest op counter)
    const u32 rng = round ? tmx - tmn : 0u, best = __reduce_max_sync(FULLM, rng);
    const u32 b_best = __ballot_sync(FULLM, round && rng == best), b_ok = __ballot_sync(FULLM, gok && lead), b_round = __ballot_sync(FULLM, round && lead),
              b_an = __ballot_sync(FULLM, analysed && lead), b_mm = __ballot_sync(FULLM, gok && mm && lead), b_act = __ballot_sync(FULLM, active && lead);
    n_fs = __reduce_add_sync(FULLM, n_fs); n_fd = __reduce_add_sync(FULLM, n_fd);
    if (lane == 0) {
      const u32 n_ok = (u32)__popc(b_ok), n_round = (u32)__popc(b_round);
      sh.brng[wid] = best; sh.bk[wid] = b_best ? t.seq_off + wid * GW + ((u32)__ffs(b_best) - 1u) / L : NONE;
      sh.rounds[wid] = n_round; sh.n_an[wid] = (u32)__popc(b_an); sh.n_def[wid] = (u32)__popc(b_act) - n_ok;
      if (n_ok) { atomicAdd(&sh.cnt[SC_COMP], n_ok); atomicAdd(&sh.cnt[SC_PRES], n_ok * n); }
      if (n_ok != n_round) atomicAdd(&sh.cnt[SC_BAR], n_ok - n_round);
      if (b_an) atomicAdd(&sh.cnt[SC_AN], (u32)__popc(b_an));
      if (b_mm) atomicAdd(&sh.cnt[SC_MIS], (u32)__popc(b_mm));
      if (n_fs) atomicAdd(&sh.cnt[SC_FS], n_fs);
      if (n_fd) atomicAdd(&sh.cnt[SC_FD], n_fd);
    }
  }
  // ---- most changes, then the lowest position: my members, the lanes that share my op counter, later the warps ----
  {
    u64 ck = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const u32 p = mr + (u32)q * L;
      const u64 k = ((u64)max(sc[q], rc[q]) << 32) | (u64)(NONE - p);
      if (FULL || p < n) ck = k > ck ? k : ck;
    }
#pragma unroll
    for (u32 h = S; h < 32; h <<= 1) { const u64 o = shfl_xor64(ck, h); ck = o > ck ? o : ck; }
    if (S >= 32 || lane < S) atomicMax((unsigned long long*)&sh.t_ck[sq], (unsigned long long)ck);
  }
  __syncthreads();
  u32 rounds = 0;
#pragma unroll
  for (u32 q = 0; q < NW; ++q) rounds += sh.rounds[q];
  if (threadIdx.x < count && !(sh.t_bits[threadIdx.x] & 1)) {
    const u64 ck = sh.t_ck[threadIdx.x];
    const u64 g = t.row.group0 + t.seq_off + threadIdx.x, G = ld_volatile(sh.out.G);
    u32* __restrict__ gu = ld_volatile(sh.out.gu32) + g;
    gu[(u64)GU_MAX_CHG * G] = (u32)(ck >> 32); gu[(u64)GU_RANK_MAX_CHG * G] = sh.mem[NONE - (u32)ck];
  }
  if (rounds) {
    constexpr u32 TPM = GW;                                   // threads per member, eight op counters each
    const u32 p = threadIdx.x / TPM, part = threadIdx.x % TPM;
    double v = 0.0;
    if (FULL || p < n) {
#pragma unroll
      for (u32 i = 0; i < 8; ++i) {
        const u32 o = part + TPM * i, d = k_d[p * S + (o ^ turn(p))];
        const double bd = o < count ? sh.t_bd[o] : 0.0;
        if (bd != 0.0 && d != 0) v += bd * rcp_u32(d);
      }
    }
#pragma unroll
    for (u32 h = 1; h < TPM; h <<= 1) v += __shfl_xor_sync(FULLM, v, h);
    if (part == 0 && (FULL || p < n)) { atomicAdd(&R.bw_sum[sh.mem[p]], v); atomicAdd(&R.bw_cnt[sh.mem[p]], rounds); }
  }
  if (threadIdx.x == 0) {
    u64 brng = 0; u32 bk = NONE, n_an = 0, n_def = 0;
    for (u32 q = 0; q < NW; ++q) { best_merge(brng, bk, sh.brng[q], sh.bk[q]); n_an += sh.n_an[q]; n_def += sh.n_def[q]; }
    TileSum ts; ts.best_rng = brng; ts.best_k = bk; ts.n_rounds = rounds; ts.n_an = n_an; ts.pad = n_def;
    sums[t.sum_idx] = ts;
    flush_counters(D, sh);
  }
}

template <bool PACKED>
__global__ void __launch_bounds__(SMALL_SEQS, CCLD_FUSED_MIN_CTAS) k_reduce_fused(const WinDesc* wd, const FusedCta* ctas,
    const WarpTile* wts, TileSum* __restrict__ sums, Registry R, Params P, DeferList DL) {
  begin_after();
  __shared__ FusedShared sh;
  const FusedCta t = ctas[blockIdx.x];
  const WinDesc& D = wd[t.w];
  if (threadIdx.x < SC_COUNT) sh.cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) { sh.out.flags = D.flags; sh.out.gi64 = D.gi64; sh.out.gu32 = D.gu32; sh.out.gbw = D.gbw; sh.out.G = D.n_groups; }
  if (threadIdx.x == 32) { sh.in.packed = D.packed; sh.in.perm = D.perm; sh.in.te = D.t_enter; sh.in.tx = D.t_exit; sh.in.by = D.bytes; sh.in.op = D.op; sh.in.sc = D.send_chg; sh.in.rc = D.recv_chg; }
  if (t.cls == 0) { fused_small_cta<PACKED>(D, t, wts, sums, R, P, DL, sh); return; }
  const u32 n = t.row.n;
  if (n <= 32) { if (n == 32) fused_sub_cta<4, true, PACKED>(D, t, sums, R, P, DL, sh); else fused_sub_cta<4, false, PACKED>(D, t, sums, R, P, DL, sh); }
  else if (n <= 64) { if (n == 64) fused_sub_cta<8, true, PACKED>(D, t, sums, R, P, DL, sh); else fused_sub_cta<8, false, PACKED>(D, t, sums, R, P, DL, sh); }
  else { if (n == 128) fused_sub_cta<16, true, PACKED>(D, t, sums, R, P, DL, sh); else fused_sub_cta<16, false, PACKED>(D, t, sums, R, P, DL, sh); }
}

// ------------------------------------------------------------------------------------------------
// the groups k_reduce_fused set aside: one warp per group, ring position p in lane p % 32; 64-bit
// throughout, order statistics by counting ranks (a group has at most 128 members)
// ------------------------------------------------------------------------------------------------
constexpr int DEF_WARPS = 4;
constexpr int DEF_GRID = 148 * 4;   // grid-stride over the list: four CTAs per SM of a B200
constexpr int DEF_Q = WARP_N / 32;

__device__ __forceinline__ u64 warp_max64(u64 v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) { const u64 o = shfl_xor64(v, d); v = o > v ? o : v; }
  return v;
}
__device__ __forceinline__ u64 warp_min64(u64 v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) { const u64 o = shfl_xor64(v, d); v = o < v ? o : v; }
  return v;
}
// k-th smallest (0-based) of x over positions < n: the element that k others precede in (value, position) order
__device__ __forceinline__ u64 rank_select(const u64 (&x)[DEF_Q], u32 n, u32 k, u64* key, u32 lane) {
  __syncwarp();
#pragma unroll
  for (int i = 0; i < DEF_Q; ++i) { const u32 p = lane + 32u * i; if (p < n) key[p] = x[i]; }
  __syncwarp();
  u64 res = 0; bool mine = false;
#pragma unroll
  for (int i = 0; i < DEF_Q; ++i) {
    const u32 p = lane + 32u * i;
    if (p < n) {
      u32 r = 0;
      for (u32 q = 0; q < n; ++q) { const u64 kq = key[q]; r += (kq < x[i] || (kq == x[i] && q < p)) ? 1u : 0u; }
      if (r == k) { mine = true; res = x[i]; }
    }
  }
  const u32 src = (u32)__ffs(__ballot_sync(FULLM, mine)) - 1u;
  return __shfl_sync(FULLM, res, src & 31);
}

// The communicator of group g: the last one whose first group is <= g (communicators without groups share their successor's start).
// A warp looks at 32 places at a time: three reads one after the other for 2,185 communicators where halving took eleven.
__device__ __forceinline__ u32 owner_of(const RangeRow* ranges, u32 n_comms, u64 g, u32 lane) {
  u32 lo = 0, len = n_comms;                                  // it is one of the len communicators from lo on
  while (len > 1) {
    const u32 step = (len + 31) / 32, at = lane * step;
    const u32 b = __ballot_sync(FULLM, at < len && ranges[lo + at].group0 <= g), k = b ? 31u - (u32)__clz(b) : 0u;
    lo += k * step; len = min(step, len - k * step);
  }
  return lo;
}

// A group set aside is a chain of dependent reads - count, entry, owner, row, record indices, values - on little data.
__global__ void __launch_bounds__(DEF_WARPS * 32) k_reduce_deferred(const WinDesc* wd, DeferList DL, Registry R, Params P, i64 now) {
  begin_after();
  __shared__ u64 s_key[DEF_WARPS][WARP_N];
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  u64* key = s_key[wid];
  const u32 total = *DL.count;
  for (u32 e = blockIdx.x * DEF_WARPS + wid; e < total; e += gridDim.x * DEF_WARPS) {
    const u64 ent = DL.entries[e];
    const WinDesc& D = wd[(u32)(ent >> 32)];
    const u64 g = (u32)ent;
    const u32 c = owner_of(D.ranges, R.n_comms, g, lane);
    const RangeRow row = D.ranges[c];
    const u32 n = row.n, so = (u32)(g - row.group0);
    const u32* mem = R.members + R.comm_moff[c];

    bool pres[DEF_Q]; i64 ta[DEF_Q], tb[DEF_Q]; u64 by[DEF_Q]; u32 op[DEF_Q], ch[DEF_Q];
    u32 npres = 0, first_p = NONE; bool miss = false, inflight = false, bad = false;
    i64 age = -1, x_max = INT64_MIN; u64 ck = 0;
    // all indices, then all values: two round trips, not two per 32 members
    u32 idx[DEF_Q];
    {
      const u32* perm = D.perm; const i64 *c_te = D.t_enter, *c_tx = D.t_exit; const u64* c_by = D.bytes; const u8* c_op = D.op; const u32 *c_sc = D.send_chg, *c_rc = D.recv_chg;
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) { const u32 p = lane + 32u * i; idx[i] = p < n ? perm[perm_at(row, so, p)] : NONE; }
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) {
        pres[i] = idx[i] != NONE;
        const u32 ix = pres[i] ? idx[i] : 0u;                // (a window with a group has a record)
        ta[i] = c_te[ix]; tb[i] = c_tx[ix]; by[i] = c_by[ix]; op[i] = c_op[ix]; ch[i] = 0;
        if (c_sc != nullptr) { const u32 sc = c_sc[ix], rc = c_rc[ix]; ch[i] = sc > rc ? sc : rc; }
      }
    }
#pragma unroll
    for (int i = 0; i < DEF_Q; ++i) {
      const u32 p = lane + 32u * i;
      if (!pres[i]) { ta[i] = 0; tb[i] = 0; by[i] = 0; op[i] = 0; ch[i] = 0; }
      if (p < n) {
        if (!pres[i]) miss = true;
        else {
          ++npres; if (first_p == NONE) first_p = p;
          if (tb[i] == -1) { inflight = true; const i64 ag = now - ta[i]; age = ag > age ? ag : age; }
          else if (ta[i] < 0 || tb[i] < ta[i]) bad = true;
          x_max = tb[i] > x_max ? tb[i] : x_max;
          const u64 k2 = ((u64)ch[i] << 32) | (u64)(NONE - p);          // most changes, then the lowest position
          ck = k2 > ck ? k2 : ck;
        }
      }
    }
    npres = __reduce_add_sync(FULLM, npres); first_p = __reduce_min_sync(FULLM, first_p);
    miss = __any_sync(FULLM, miss); inflight = __any_sync(FULLM, inflight); bad = __any_sync(FULLM, bad);
    age = (i64)(warp_max64((u64)age ^ 0x8000000000000000ull) ^ 0x8000000000000000ull);
    x_max = (i64)(warp_max64((u64)x_max ^ 0x8000000000000000ull) ^ 0x8000000000000000ull);
    ck = warp_max64(ck);
    const bool complete = !miss && !inflight && !bad;
    // op set: the first present member's op and size
    const bool have_first = first_p != NONE;
    u64 gbytes = 0; u32 gop = 0;
    if (have_first) {
      u64 fby = 0; u32 fop = 0;
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) if ((first_p >> 5) == (u32)i) { fby = by[i]; fop = op[i]; }
      gbytes = __shfl_sync(FULLM, fby, first_p & 31); gop = __shfl_sync(FULLM, fop, first_p & 31);
    }
    bool mm = false;
#pragma unroll
    for (int i = 0; i < DEF_Q; ++i) if (pres[i] && (op[i] != gop || by[i] != gbytes)) mm = true;
    const bool mismatch = __any_sync(FULLM, mm);
    const bool barrier = have_first && gop == CCLD_OP_ALLREDUCE && gbytes < P.barrier_bytes;
    const bool analysed = complete && !barrier && n >= P.min_group;
    const bool hang = !complete && inflight && age > P.hang_ns && !barrier;
    const u32 gfl = (mismatch ? CCLD_G_OPSET_MISMATCH : 0) | (barrier ? CCLD_G_BARRIER : 0) | (inflight ? CCLD_G_INFLIGHT : 0) |
                    (bad ? CCLD_G_BAD_TIME : 0) | (complete ? CCLD_G_COMPLETE : CCLD_G_INCOMPLETE) | (analysed ? CCLD_G_ANALYSED : 0) |
                    (hang ? CCLD_G_HANG_ALERT : 0);

    u64 e_min = 0, e_max = 0, tmax = 0, tmin = 0, med_s = 0, mad_s = 0, med_d = 0, mad_d = 0; u32 pmax = 0, pmin = 0;
    u32 n_fs = 0, n_fd = 0;
    u32 fl[DEF_Q];
#pragma unroll
    for (int i = 0; i < DEF_Q; ++i) fl[i] = CCLD_F_NOT_ANALYSED | (pres[i] ? 0 : CCLD_F_MISSING);
    double num = 1.0, den = 1.0; bus_factor(gop, n, &num, &den);
    const double bn = (double)gbytes * num;
    if (complete) {
      u64 sk[DEF_Q], du[DEF_Q];
      u64 l_emin = U64_MAX_, l_emax = 0, l_tmax = 0, l_tmin = U64_MAX_;
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) {
        du[i] = (u64)(tb[i] - ta[i]);
        if (pres[i]) {
          const u64 te = (u64)ta[i];
          l_emin = te < l_emin ? te : l_emin; l_emax = te > l_emax ? te : l_emax;
          l_tmax = du[i] > l_tmax ? du[i] : l_tmax; l_tmin = du[i] < l_tmin ? du[i] : l_tmin;
        }
      }
      e_min = warp_min64(l_emin); e_max = warp_max64(l_emax); tmax = warp_max64(l_tmax); tmin = warp_min64(l_tmin);
      u32 c_mx = NONE, c_mn = NONE;                          // ties: the lowest position
#pragma unroll
      for (int i = DEF_Q - 1; i >= 0; --i) if (pres[i]) { const u32 p = lane + 32u * i; if (du[i] == tmax) c_mx = p; if (du[i] == tmin) c_mn = p; }
      pmax = __reduce_min_sync(FULLM, c_mx); pmin = __reduce_min_sync(FULLM, c_mn);
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) sk[i] = (u64)ta[i] - e_min;
      if (!barrier) {
#pragma unroll
        for (int i = 0; i < DEF_Q; ++i) if (pres[i]) { const u32 p = lane + 32u * i; atomicAdd(&R.bw_sum[mem[p]], busbw_fast(bn, den, (i64)du[i])); atomicAdd(&R.bw_cnt[mem[p]], 1u); }
      }
      if (analysed) {
        const u32 k = (n - 1) >> 1;
        u64 dv[DEF_Q];
        med_s = rank_select(sk, n, k, key, lane);
#pragma unroll
        for (int i = 0; i < DEF_Q; ++i) dv[i] = absdiff(sk[i], med_s);
        mad_s = rank_select(dv, n, k, key, lane);
        med_d = rank_select(du, n, k, key, lane);
#pragma unroll
        for (int i = 0; i < DEF_Q; ++i) dv[i] = absdiff(du[i], med_d);
        mad_d = rank_select(dv, n, k, key, lane);
#pragma unroll
        for (int i = 0; i < DEF_Q; ++i) {
          if (pres[i]) {
            const u32 p = lane + 32u * i;
            const bool so_ = mul_gt(absdiff(sk[i], med_s), 1000u, mad_s, P.k_milli), shi = sk[i] > med_s;
            const bool dq = mul_gt(absdiff(du[i], med_d), 1000u, mad_d, P.k_milli), dhi = du[i] > med_d;
            fl[i] = (so_ ? CCLD_F_SKEW_OUT : 0) | (dq ? CCLD_F_DUR_OUT : 0) | (shi ? CCLD_F_SKEW_HI : 0) | (dhi ? CCLD_F_DUR_HI : 0);
            if (so_) { ++n_fs; atomicAdd(&R.votes[(u64)mem[p] * 4 + (shi ? 0 : 1)], 1u); }
            if (dq) { ++n_fd; atomicAdd(&R.votes[(u64)mem[p] * 4 + (dhi ? 2 : 3)], 1u); }
          }
        }
      }
    }
    n_fs = __reduce_add_sync(FULLM, n_fs); n_fd = __reduce_add_sync(FULLM, n_fd);
    // ---- outputs ----
    {
      u8* __restrict__ fp = D.flags + row.slot0 + (u64)so * n;
#pragma unroll
      for (int i = 0; i < DEF_Q; ++i) { const u32 p = lane + 32u * i; if (p < n) fp[p] = (u8)fl[i]; }
    }
    if (lane == 0) {
      const u64 G = D.n_groups;
      const i64 span = complete ? x_max - (i64)e_min : 0;
      if (hang) raise_alert(D, R.comm_id[c], row.seq_lo + so, age);
      D.gi64[(u64)GI_E_MIN * G + g] = complete ? (i64)e_min : 0; D.gi64[(u64)GI_ARRIVAL_SKEW * G + g] = complete ? (i64)(e_max - e_min) : 0;
      D.gi64[(u64)GI_T_MAX * G + g] = (i64)tmax; D.gi64[(u64)GI_T_MIN * G + g] = (i64)tmin; D.gi64[(u64)GI_SPAN * G + g] = span;
      D.gi64[(u64)GI_MED_SKEW * G + g] = (i64)med_s; D.gi64[(u64)GI_MAD_SKEW * G + g] = (i64)mad_s;
      D.gi64[(u64)GI_MED_DUR * G + g] = (i64)med_d; D.gi64[(u64)GI_MAD_DUR * G + g] = (i64)mad_d;
      D.gu32[(u64)GU_RANK_TMIN * G + g] = complete ? mem[pmin] : 0; D.gu32[(u64)GU_RANK_TMAX * G + g] = complete ? mem[pmax] : 0;
      D.gu32[(u64)GU_MAX_CHG * G + g] = complete ? (u32)(ck >> 32) : 0;
      D.gu32[(u64)GU_RANK_MAX_CHG * G + g] = complete ? mem[NONE - (u32)ck] : 0;
      D.gu32[(u64)GU_N_PRESENT * G + g] = npres; D.gu32[(u64)GU_GFLAGS * G + g] = gfl;
      D.gbw[g] = complete ? busbw_fast(bn, den, span) : 0.0;
      count_add(D.counters, complete ? C_COMPLETE : C_INCOMPLETE, 1u);
      if (barrier) count_add(D.counters, C_BARRIER, 1u);
      if (analysed) count_add(D.counters, C_ANALYSED, 1u);
      if (mismatch) count_add(D.counters, C_MISMATCH, 1u);
      count_add(D.counters, C_PRESENT, npres); count_add(D.counters, C_FLAG_SKEW, n_fs); count_add(D.counters, C_FLAG_DUR, n_fd);
    }
  }
}

}  // namespace ccld
