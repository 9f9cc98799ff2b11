// Per-op reductions, median / MAD, flags and votes for communicators of more than 1,024 ranks (sm_100a). Included by
// ccld_kernels.cuh.
//
// A group of thousands of members has its records spread over as many places of the upload, and its order statistics need
// every key several times. A cluster of eight CTAs takes a tile of LARGE_SEQS = 8 consecutive op counters of one communicator:
//
//   gather    CTA c takes an eighth of the members through all eight op counters. Lanes run along the op counter first: the
//             eight record indices of a member are one 32-byte sector of the member-major permutation, and in a rank-major
//             upload its eight records are neighbours too, so every gather of a warp fetches whole sectors. Times become 32-bit
//             keys against the group's first member (enter-time offset, duration), which go straight to the shared memory of CTA j, whose op
//             counter they belong to; extrema, op-set check and rate column are reduced on the way.
//   meet      One barrier of the cluster later CTA j has its op counter's keys, and everybody the eight CTAs' extrema. The bandwidths of
//             a CTA's members over the eight op counters are added up where they were gathered, so a member costs one atomic per tile.
//   select    medians of both metrics side by side: a histogram of 2,048 bins from the largest key's highest bit down names the
//             bin of the median, the few keys of that bin are put in a list, and a thread per listed key counts those before
//             it; then the same for the deviations. Five barriers per median of both metrics.
//
// Groups that are not complete and 32-bit clean go to k_reduce_large_deferred (one CTA per listed group, 64-bit, hang alerts).
//
// Two windows of one communicator of 4,096 ranks, 2 x 1,000 groups: 219 us. A CTA lives 35 us: 16 of them in the gather (four round
// trips to memory, two records per thread each; more do not fit the registers of three CTAs per SM), 10 in the two selections, the rest in
// barriers, merges and the row. With the keys staged where they were gathered and pulled over by their owners between two
// barriers, subtracted and stored once more, and lists ordered by two comparisons per pair, it took 229 (2,000 ranks 160 instead of 151, 3,000 199
// instead of 190); two kernels with the keys in memory between them 285.
#pragma once
#include <cooperative_groups.h>
#include "ccld_device.cuh"

namespace ccld {

constexpr int LQ_THREADS = 512, LQ_WARPS = LQ_THREADS / 32;
constexpr u32 LQ_BITS = 11, LQ_BINS = 1u << LQ_BITS;       // bins of a histogram level
constexpr u32 LQ_LIST = 256, LQ_PLACE_BITS = 8;            // keys a bin may hold to be settled by counting; bits of a place in their list
constexpr u32 LQ_LEVELS = (32 + LQ_BITS - 1) / LQ_BITS;    // after that many levels no bit is undecided
static_assert(LARGE_SEQS == 8 && LQ_WARPS == 16 && LQ_LIST == LQ_THREADS / 2, "a CTA of the cluster per op counter, eight warps per metric");
static_assert(LQ_LIST == 1u << LQ_PLACE_BITS && 32 - LQ_BITS + LQ_PLACE_BITS < 32, "what the first level leaves undecided and a place fit a word");
// A CTA gathers at most M = 64 Q members; the padding sets a row's lanes (op counter 0..7, member 0..3) on 32 different banks. Dynamic
// shared memory: the keys of my op counter (pairs), the durations of my members, and the histograms, which take the
// durations' place where that is large enough.
template <int Q> struct LargeTile {
  static constexpr bool STAGED = Q < 16;                   // 33 KB more per CTA would leave L1 28 KB: 289 us instead of 232 on 8,000 members
  static constexpr u32 M = 64 * Q, PITCH = M + 4, KEYS = LARGE_SEQS * M * 8, DURS = STAGED ? LARGE_SEQS * PITCH * 4 : 0, HIST = 2 * LQ_BINS * 4;
  static constexpr bool OVERLAY = DURS >= HIST;
  static constexpr u32 BYTES = KEYS + DURS + (OVERLAY ? 0 : HIST);
};

struct LargePick { u32 lo, sh, k, cnt; };                  // the k-th of cnt keys in [lo, lo + 2^sh)
struct LargeShared {
  uint4 list[2][LQ_LIST / 4];
  MidPart part[LQ_WARPS][LARGE_SEQS], mine[LARGE_SEQS], group;
  LargePick pick[LQ_LEVELS][2];                            // [level][metric]
  u32 wsum[LQ_WARPS], n_list[2], res[2], n_fs, n_fd, ranks[3];
  u64 gby[LARGE_SEQS]; i64 te0[LARGE_SEQS]; u32 gop[LARGE_SEQS];
  u32 state[LARGE_SEQS], rng[LARGE_SEQS];                  // per op counter: 1 clean, 2 a round; range of durations
  double bd[LARGE_SEQS];                                   // bytes * factor of an op counter that is a round, else 0
};

// The k-th smallest (0-based) of |a - ma| and of |d - md| over the n pairs in shared memory. ba, bd: the largest of them.
// All threads call it; the histograms ([2][LQ_BINS]) are zero on entry and on return.
template <int Q> __device__ __forceinline__ void large_pick(const uint2* __restrict__ keys, u32 n, u32 ma, u32 md, u32 k, u32 ba, u32 bd,
                                                            u32* hist, LargeShared& sh, u32* ra, u32* rd) {
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5, x = wid >> 3;             // eight warps scan a metric's bins
  u32 lo0 = 0, lo1 = 0, w0 = 32 - (u32)__clz(ba | 1u), w1 = 32 - (u32)__clz(bd | 1u);  // undecided bits
  u32 k0 = k, k1 = k, c0 = NONE, c1 = NONE;
  for (u32 level = 0; level < LQ_LEVELS; ++level) {
    const bool first = level == 0;
    const bool act0 = first || (w0 > 0 && c0 > LQ_LIST), act1 = first || (w1 > 0 && c1 > LQ_LIST);
    if (!act0 && !act1) break;                             // the same in every thread
    const u32 n0 = w0 > LQ_BITS ? w0 - LQ_BITS : 0u, n1 = w1 > LQ_BITS ? w1 - LQ_BITS : 0u;
    if (first) {                                           // every key counts, and none is larger than the bound
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const u32 i = threadIdx.x + (u32)q * LQ_THREADS;
        if (i >= n) break;
        const uint2 y = keys[i];
        atomicAdd(&hist[__usad(y.x, ma, 0u) >> n0], 1u);
        atomicAdd(&hist[LQ_BINS + (__usad(y.y, md, 0u) >> n1)], 1u);
      }
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const u32 i = threadIdx.x + (u32)q * LQ_THREADS;
        if (i >= n) break;
        const uint2 y = keys[i];
        const u32 a = __usad(y.x, ma, 0u) - lo0, d = __usad(y.y, md, 0u) - lo1;
        if (act0 && (a >> w0) == 0) atomicAdd(&hist[a >> n0], 1u);            // (w < 32 after the first level)
        if (act1 && (d >> w1) == 0) atomicAdd(&hist[LQ_BINS + (d >> n1)], 1u);
      }
    }
    __syncthreads();
    u32 loc[8], sum = 0;
    uint4* h = reinterpret_cast<uint4*>(&hist[x * LQ_BINS + (wid & 7) * 256 + lane * 8]);
    { const uint4 a = h[0], b = h[1]; loc[0] = a.x; loc[1] = a.y; loc[2] = a.z; loc[3] = a.w; loc[4] = b.x; loc[5] = b.y; loc[6] = b.z; loc[7] = b.w; }
    h[0] = make_uint4(0, 0, 0, 0); h[1] = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int q = 0; q < 8; ++q) sum += loc[q];
    u32 inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const u32 o = __shfl_up_sync(FULLM, inc, d); if (lane >= (u32)d) inc += o; }
    // what this level leaves undecided for a metric that takes no part, and a defined value for one that does
    if ((wid & 7) == 0 && lane == 0) sh.pick[level][x] = x ? LargePick{lo1, act1 ? 0u : w1, k1, c1} : LargePick{lo0, act0 ? 0u : w0, k0, c0};
    if (lane == 31) sh.wsum[wid] = inc;
    __syncthreads();
    const u32 off = __reduce_add_sync(FULLM, lane < (wid & 7) ? sh.wsum[(wid & 8) + lane] : 0u);
    const u32 kr = x ? k1 : k0, ex = off + inc - sum;
    if ((x ? act1 : act0) && kr >= ex && kr < ex + sum) {
      u32 cum = ex;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (kr >= cum && kr < cum + loc[q]) {
          const u32 bin = (wid & 7) * 256 + lane * 8 + q, ns = x ? n1 : n0;
          sh.pick[level][x] = LargePick{(x ? lo1 : lo0) + (bin << ns), ns, kr - cum, loc[q]};
        }
        cum += loc[q];
      }
    }
    __syncthreads();
    const LargePick p0 = sh.pick[level][0], p1 = sh.pick[level][1];
    lo0 = p0.lo; w0 = p0.sh; k0 = p0.k; c0 = p0.cnt; lo1 = p1.lo; w1 = p1.sh; k1 = p1.k; c1 = p1.cnt;
  }
  if (w0 | w1) {
    // the keys of the bins go into lists, each with its place below its undecided bits, so that no two are equal and one comparison
    // orders them; a list's places beyond its end hold the largest word
    u32* const l0 = reinterpret_cast<u32*>(sh.list[0]); u32* const l1 = reinterpret_cast<u32*>(sh.list[1]);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const u32 i = threadIdx.x + (u32)q * LQ_THREADS;
      if (i >= n) break;
      const uint2 y = keys[i];
      const u32 a = __usad(y.x, ma, 0u) - lo0, d = __usad(y.y, md, 0u) - lo1;
      if (w0 && (a >> w0) == 0) { const u32 at = atomicAdd(&sh.n_list[0], 1u); if (at < LQ_LIST) l0[at] = a << LQ_PLACE_BITS | at; }    // c0 <= LQ_LIST of them
      if (w1 && (d >> w1) == 0) { const u32 at = atomicAdd(&sh.n_list[1], 1u); if (at < LQ_LIST) l1[at] = d << LQ_PLACE_BITS | at; }
    }
    __syncthreads();
    {
      // a thread per listed key counts those before it; the key with k before it is the one
      const u32 c = x ? c1 : c0, w = x ? w1 : w0, kr = x ? k1 : k0, i = (wid & 7) * 32 + lane, c4 = min((c + 3) / 4, LQ_LIST / 4);
      if (w == 0) { if (i == 0) sh.res[x] = x ? lo1 : lo0; }
      else if ((wid & 7) * 32 < c) {
        const u32 v = (x ? l1 : l0)[i];
        u32 before = 0;
#pragma unroll 4
        for (u32 g = 0; g < c4; ++g) {
          const uint4 y = sh.list[x][g];
          before += y.x < v ? 1u : 0u; before += y.y < v ? 1u : 0u; before += y.z < v ? 1u : 0u; before += y.w < v ? 1u : 0u;
        }
        if (i < c && before == kr) sh.res[x] = (x ? lo1 : lo0) + (v >> LQ_PLACE_BITS);
      }
    }
    __syncthreads();
    lo0 = sh.res[0]; lo1 = sh.res[1];
    // the lists are empty again for the next call (whose lists are written several barriers on)
    { const u32 i = threadIdx.x & (LQ_LIST - 1); (x ? l1 : l0)[i] = NONE; if (threadIdx.x < 2) sh.n_list[threadIdx.x] = 0; }
  }
  *ra = lo0; *rd = lo1;
}

// The cluster's barrier in two halves; every thread of every CTA takes part in each.
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// A pair into the shared memory of CTA `cta` of the cluster, at the place that p is in mine.
__device__ __forceinline__ u32 cluster_address(const void* p, u32 cta) {
  u32 r; asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((u32)__cvta_generic_to_shared(p)), "r"(cta)); return r;
}
__device__ __forceinline__ void cluster_store(u32 address, u32 a, u32 b) { asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" :: "r"(address), "r"(a), "r"(b) : "memory"); }

// The duration of the pair that CTA `cta` keeps at the place of p.
__device__ __forceinline__ u32 cluster_duration(const uint2* p, u32 cta) {
  u32 d; asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(d) : "r"(cluster_address(p, cta) + 4) : "memory"); return d;
}

// CTAs per SM: three up to 4,096 members, although that leaves 40 registers and spills some 80 bytes (two instead, with two windows each:
// 261 and not 232 us for 2 x 2,000 groups of 1,100 members, for 2 x 1,000 of 2,000 155 and 147, of 2,049 173 and 161, of 3,000 199 and 190, of 4,096 224 and 222);
// above, two are what shared memory holds. Two records in flight per thread; four spill more, above 4,096 there is room for them.
template <int Q>
__global__ void __launch_bounds__(LQ_THREADS, Q == 16 ? 2 : 3) k_reduce_large(const WinDesc* wd, const Tile* tiles,
    TileSum* __restrict__ sums, Registry R, Params P, DeferList DL) {
  begin_after();
  extern __shared__ __align__(16) unsigned char large_raw[];
  __shared__ __align__(16) LargeShared sh;
  namespace cg = cooperative_groups;
  const Tile t = tiles[blockIdx.x / LARGE_SEQS];
  const u32 n = t.row.n;
  if (t.count == 0 || (n <= 2048 ? 4 : (n <= 4096 ? 8 : 16)) != Q) return;     // no work, or another instance's: the same in the whole cluster
  cluster_arrive();                                         // waited for before anything is stored elsewhere: the others have begun
  using L = LargeTile<Q>;
  constexpr u32 PITCH = L::PITCH;
  const u32 me = blockIdx.x % LARGE_SEQS;                   // my eighth of the members, and my op counter
  const WinDesc& D = wd[t.w];
  const RangeRow& row = t.row;
  const u32* __restrict__ mem = R.members + t.moff;
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const u32 M = (n + LARGE_SEQS - 1) / LARGE_SEQS, m0 = me * M, m_cnt = m0 >= n ? 0u : min(M, n - m0);
  uint2* const keys = reinterpret_cast<uint2*>(large_raw);                      // [member] enter time against base, duration: my op counter
  u32* const k_d = reinterpret_cast<u32*>(large_raw + L::KEYS);                 // [op counter][member of mine] durations
  u32* const hist = L::OVERLAY ? k_d : reinterpret_cast<u32*>(large_raw + L::KEYS + L::DURS);
  const auto clear_hist = [&] { for (u32 i = threadIdx.x; i < 2 * LQ_BINS / 4; i += LQ_THREADS) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0, 0, 0, 0); };
  if (!L::OVERLAY) clear_hist();
  if (threadIdx.x < 2 * LQ_LIST / 4) (&sh.list[0][0])[threadIdx.x] = make_uint4(NONE, NONE, NONE, NONE);
  if (threadIdx.x < 2) sh.n_list[threadIdx.x] = 0;
  if (threadIdx.x == 0) { sh.n_fs = 0; sh.n_fd = 0; }
  // ---- gather ----
  {
    const u32 j = lane & 7, pq = lane >> 3;                 // op counter of the tile, member of the quad
    const bool jv = j < t.count;
    const u32* perm = D.perm + row.slot0 + t.seq_off + (jv ? j : 0u);
    const i64* __restrict__ c_te = D.t_enter; const i64* __restrict__ c_tx = D.t_exit;
    const u64* __restrict__ c_by = D.bytes; const u8* __restrict__ c_op = D.op;
    const u32* __restrict__ c_sc = D.send_chg; const u32* __restrict__ c_rc = D.recv_chg;
    const u32 theirs = cluster_address(keys + m0, j);       // where CTA j keeps my members' keys
    MidTrack x;
    u32 idx[Q];
    const u32 i0 = jv ? *perm : NONE;
#pragma unroll
    for (int q = 0; q < Q; ++q) { const u32 m = (wid + LQ_WARPS * (u32)q) * 4 + pq; idx[q] = (jv && m < m_cnt) ? perm[(u64)(m0 + m) * row.n_seq] : NONE; }
    i64 te0 = 0; u64 by0 = 0; u32 op0 = 0;
    if (i0 != NONE) { te0 = __ldg(c_te + i0); by0 = __ldg(c_by + i0); op0 = __ldg(c_op + i0); } else x.bits = 1;
    const u64 base = (u64)te0 - 0x80000000ull;
    cluster_wait();
    constexpr int STEP = Q == 16 ? 4 : 2;                   // records in flight per thread
#pragma unroll
    for (int q0 = 0; q0 < Q; q0 += STEP) {
      i64 ta[STEP], tb[STEP]; u64 by[STEP]; u32 op[STEP], ch[STEP];
#pragma unroll
      for (int u = 0; u < STEP; ++u) {
        const u32 ix = idx[q0 + u] == NONE ? 0u : idx[q0 + u];
        ta[u] = __ldg(c_te + ix); tb[u] = __ldg(c_tx + ix); by[u] = __ldg(c_by + ix); op[u] = __ldg(c_op + ix); ch[u] = 0;
        if (c_sc != nullptr) { const u32 sc = __ldg(c_sc + ix), rc = __ldg(c_rc + ix); ch[u] = max(sc, rc); }
      }
#pragma unroll
      for (int u = 0; u < STEP; ++u) {
        const u32 m = (wid + LQ_WARPS * (u32)(q0 + u)) * 4 + pq, p = m0 + m;
        if (m >= m_cnt) continue;
        u32 a = 0, d = 0;
        if (idx[q0 + u] == NONE) { if (jv) x.bits |= 1; }
        else {
          const u64 ra = (u64)ta[u] - base, rb = (u64)tb[u] - base;
          a = (u32)ra; const u32 b = (u32)rb; d = b - a;
          if (((ra | rb) >> 32) != 0 || (ta[u] | tb[u]) < 0 || b < a) x.bits |= 1;       // beyond 32 bits, negative or in flight, exit before enter
          if (op[u] != op0 || by[u] != by0) x.bits |= 2;
          x.see(p, a, b, d, ch[u]);
          cluster_store(theirs + m * 8, a, d);
        }
        if (L::STAGED) k_d[j * PITCH + m] = d;
      }
    }
    MidPart mine = x.part();
    mid_merge(mine, mid_shfl_xor(mine, 8)); mid_merge(mine, mid_shfl_xor(mine, 16));
    if (lane < LARGE_SEQS) sh.part[wid][lane] = mine;
    if (wid == 0 && lane < LARGE_SEQS) { sh.te0[lane] = te0; sh.gby[lane] = by0; sh.gop[lane] = op0; }
  }
  __syncthreads();
  if (wid < LARGE_SEQS) {                                   // warp j: my part of op counter j
    MidPart x = sh.part[lane & (LQ_WARPS - 1)][wid];
#pragma unroll
    for (int h = 1; h < LQ_WARPS; h <<= 1) mid_merge(x, mid_shfl_xor(x, h));
    if (lane == 0) sh.mine[wid] = x;
  }
  cluster_arrive(); cluster_wait();                         // all keys and parts of the cluster are where they belong
  if (wid < LARGE_SEQS) {                                   // op counter j's extrema by warp j
    const u32 j = wid;
    MidPart x = *cg::this_cluster().map_shared_rank(&sh.mine[j], lane & 7);
#pragma unroll
    for (int h = 1; h < (int)LARGE_SEQS; h <<= 1) mid_merge(x, mid_shfl_xor(x, h));
    if (lane == 0) {
      const u32 gop = sh.gop[j]; const u64 gby = sh.gby[j];
      const bool clean = j < t.count && !(x.bits & 1), round = clean && !(gop == CCLD_OP_ALLREDUCE && gby < P.barrier_bytes);
      double num, den; bus_factor(gop, n, &num, &den);
      sh.state[j] = (clean ? 1u : 0u) | (round ? 2u : 0u); sh.rng[j] = (u32)(x.kmax >> 32) - (u32)(~x.n_kmin >> 32);
      sh.bd[j] = round ? (double)gby * num / den : 0.0;
      if (j == me) {
        sh.group = x;
        if (clean) { sh.ranks[0] = __ldg(mem + (u32)~x.n_kmin); sh.ranks[1] = __ldg(mem + (NONE - (u32)x.kmax)); sh.ranks[2] = __ldg(mem + (NONE - (u32)x.ck)); }
      }
    }
  }
  __syncthreads();
  if (L::STAGED) cluster_arrive();                          // I read nobody's shared memory any more; waited for at the end
  // ---- bandwidth of my members over the tile's op counters, where they were gathered ----
  u32 rounds = 0;
#pragma unroll
  for (u32 j = 0; j < LARGE_SEQS; ++j) rounds += sh.state[j] >> 1;
  if (rounds) {
    for (u32 m = threadIdx.x; m < m_cnt; m += LQ_THREADS) {
      double v = 0.0;
      u32 d[LARGE_SEQS];
#pragma unroll
      for (u32 j = 0; j < LARGE_SEQS; ++j) d[j] = L::STAGED ? k_d[j * PITCH + m] : cluster_duration(keys + m0 + m, j);
#pragma unroll
      for (u32 j = 0; j < LARGE_SEQS; ++j) if (d[j] != 0 && sh.bd[j] != 0.0) v += sh.bd[j] * rcp_u32(d[j]);
      const u32 rank = __ldg(mem + m0 + m);
      atomicAdd(&R.bw_sum[rank], v); atomicAdd(&R.bw_cnt[rank], rounds);
    }
  }
  if (!L::STAGED) cluster_arrive();
  // ---- my group ----
  const u32 emin = ~sh.group.n_emin, emax = sh.group.emax, tmx = (u32)(sh.group.kmax >> 32), tmn = (u32)(~sh.group.n_kmin >> 32);
  const u32 so = t.seq_off + me;
  const bool gvalid = me < t.count, gok = sh.state[me] & 1, barrier = gok && !(sh.state[me] & 2), analysed = gok && !barrier && n >= P.min_group;
  u32 ms = 0, ds = 0, md = 0, dm = 0;
  if (gok) {                                                // the same in the whole CTA
    u8* __restrict__ fp = D.flags + row.slot0 + (u64)so * n;
    if (analysed) {
      if (L::OVERLAY) { __syncthreads(); clear_hist(); __syncthreads(); }
      const u32 k = (n - 1) >> 1, ba = emax - emin, bd = tmx - tmn;
      large_pick<Q>(keys, n, emin, tmn, k, ba, bd, hist, sh, &ms, &md);
      large_pick<Q>(keys, n, emin + ms, tmn + md, k, max(ms, ba - ms), max(md, bd - md), hist, sh, &ds, &dm);
      // |x - med| * 1000 > k * MAD in whole numbers: |x - med| > floor(k * MAD / 1000); a quotient of 2^32 - 1 or more is never exceeded
      const u64 qs = (u64)ds * P.k_milli / 1000u, qd = (u64)dm * P.k_milli / 1000u;
      const u32 ts = qs > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qs, td = qd > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qd;
      const u32 ca = emin + ms, cd = tmn + md;
      u32 n_fs = 0, n_fd = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const u32 i = threadIdx.x + (u32)q * LQ_THREADS;
        if (i >= n) break;
        const uint2 y = keys[i];
        const bool os = __usad(y.x, ca, 0u) > ts, od = __usad(y.y, cd, 0u) > td, hs = y.x > ca, hd = y.y > cd;
        fp[i] = (u8)((os ? CCLD_F_SKEW_OUT : 0) | (od ? CCLD_F_DUR_OUT : 0) | (hs ? CCLD_F_SKEW_HI : 0) | (hd ? CCLD_F_DUR_HI : 0));
        if (os) { ++n_fs; atomicAdd(&R.votes[(u64)mem[i] * 4 + (hs ? 0 : 1)], 1u); }
        if (od) { ++n_fd; atomicAdd(&R.votes[(u64)mem[i] * 4 + (hd ? 2 : 3)], 1u); }
      }
      n_fs = __reduce_add_sync(FULLM, n_fs); n_fd = __reduce_add_sync(FULLM, n_fd);
      if (lane == 0) { if (n_fs) atomicAdd(&sh.n_fs, n_fs); if (n_fd) atomicAdd(&sh.n_fd, n_fd); }
      __syncthreads();
    } else {
      for (u32 i = threadIdx.x; i < n; i += LQ_THREADS) fp[i] = CCLD_F_NOT_ANALYSED;
    }
  }
  // ---- the row, the counters; the tile's summary by the first CTA ----
  if (threadIdx.x == 0) {
    if (gok) {
      const u64 G = D.n_groups, gr = row.group0 + so;
      i64* __restrict__ gi = D.gi64 + gr; u32* __restrict__ gu = D.gu32 + gr; double* __restrict__ gb = D.gbw + gr; u64* const counters = D.counters;
      const u32 span = sh.group.xmax - emin;
      const bool mismatch = (sh.group.bits & 2) != 0;
      double num, den; bus_factor(sh.gop[me], n, &num, &den);
      gi[(u64)GI_E_MIN * G] = (i64)((u64)sh.te0[me] - 0x80000000ull + emin); gi[(u64)GI_ARRIVAL_SKEW * G] = (i64)(u64)(emax - emin);
      gi[(u64)GI_T_MAX * G] = (i64)(u64)tmx; gi[(u64)GI_T_MIN * G] = (i64)(u64)tmn; gi[(u64)GI_SPAN * G] = (i64)(u64)span;
      gi[(u64)GI_MED_SKEW * G] = (i64)(u64)ms; gi[(u64)GI_MAD_SKEW * G] = (i64)(u64)ds;
      gi[(u64)GI_MED_DUR * G] = analysed ? (i64)((u64)tmn + md) : 0; gi[(u64)GI_MAD_DUR * G] = (i64)(u64)dm;
      gu[(u64)GU_RANK_TMIN * G] = sh.ranks[0]; gu[(u64)GU_RANK_TMAX * G] = sh.ranks[1];
      gu[(u64)GU_MAX_CHG * G] = (u32)(sh.group.ck >> 32); gu[(u64)GU_RANK_MAX_CHG * G] = sh.ranks[2];
      gu[(u64)GU_N_PRESENT * G] = n;
      gu[(u64)GU_GFLAGS * G] = CCLD_G_COMPLETE | (barrier ? CCLD_G_BARRIER : 0) | (mismatch ? CCLD_G_OPSET_MISMATCH : 0) | (analysed ? CCLD_G_ANALYSED : 0);
      *gb = span ? (double)sh.gby[me] * num * rcp_newton((double)span * den) : 0.0;
      count_add(counters, C_COMPLETE, 1); count_add(counters, C_PRESENT, n); count_add(counters, C_BARRIER, barrier); count_add(counters, C_ANALYSED, analysed);
      count_add(counters, C_MISMATCH, mismatch); count_add(counters, C_FLAG_SKEW, sh.n_fs); count_add(counters, C_FLAG_DUR, sh.n_fd);
    } else if (gvalid) {                                    // set aside for the 64-bit kernel
      const u32 e = atomicAdd(DL.count, 1u);
      DL.entries[e] = ((u64)t.w << 32) | (u64)(row.group0 + so);
    }
    if (me == 0) {
      TileSum ts = {0, NONE, rounds, n >= P.min_group ? rounds : 0u, 0};
      for (u32 j = 0; j < t.count; ++j) {
        if (sh.state[j] & 2) best_merge(ts.best_rng, ts.best_k, (u64)sh.rng[j], t.seq_off + j);
        if (!(sh.state[j] & 1)) ++ts.pad;
      }
      sums[blockIdx.x / LARGE_SEQS] = ts;
    }
  }
  cluster_wait();                                           // my shared memory stays until nobody reads it any more
}

// ------------------------------------------------------------------------------------------------
// the groups k_reduce_large set aside: one CTA per listed group; enter times and durations live in
// shared memory as 64-bit values, order statistics by most-significant-byte-first radix select
// ------------------------------------------------------------------------------------------------
constexpr int LARGE_DEF_THREADS = 1024;
constexpr int LARGE_DEF_GRID = 148;         // grid-stride over the list: one CTA per SM of a B200

// Reduction over the CTA (all threads call; blockDim.x a multiple of 32): warps reduce by shuffles, the first warp
// reduces the warps' partial results the same way, everyone reads the result from s_red[0].
template <class T, class Op>
__device__ T block_reduce(T v, Op op, T* s_red /*[32]*/) {
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) { T o = __shfl_xor_sync(0xFFFFFFFFu, v, d); v = op(v, o); }
  __syncthreads();
  if (lane == 0) s_red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    T x = lane < nw ? s_red[lane] : Op::identity();
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) { T o = __shfl_xor_sync(0xFFFFFFFFu, x, d); x = op(x, o); }
    if (lane == 0) s_red[0] = x;
  }
  __syncthreads();
  return s_red[0];
}
struct OpMaxU64 { __device__ u64 operator()(u64 a, u64 b) const { return a > b ? a : b; } static __device__ u64 identity() { return 0; } };
struct OpAddU32 { __device__ u32 operator()(u32 a, u32 b) const { return a + b; } static __device__ u32 identity() { return 0; } };
struct OpMinU32 { __device__ u32 operator()(u32 a, u32 b) const { return a < b ? a : b; } static __device__ u32 identity() { return NONE; } };

// k-th smallest (0-based) of key(i), i < n; max_key bounds the keys. All threads of the CTA call it.
template <class F>
__device__ u64 radix_select(F key, u32 n, u32 k, u64 max_key, u32* hist /*[256]*/, u32* s_pick /*[2]*/) {
  int top = max_key == 0 ? 0 : (63 - __clzll((long long)max_key)) >> 3;
  u64 prefix = 0, mask = 0; u32 krem = k;
  for (int b = top; b >= 0; --b) {
    for (u32 i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    for (u32 i = threadIdx.x; i < n; i += blockDim.x) {
      const u64 v = key(i);
      if ((v & mask) == prefix) {
        const u32 bin = (u32)(v >> (8 * b)) & 255u;
        const u32 m = __match_any_sync(__activemask(), bin);       // one atomic per distinct bin in the warp
        if ((threadIdx.x & 31) == (u32)(__ffs(m) - 1)) atomicAdd(&hist[bin], (u32)__popc(m));
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      u32 loc[8], sum = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) { loc[q] = hist[threadIdx.x * 8 + q]; sum += loc[q]; }
      u32 inc = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) { u32 o = __shfl_up_sync(0xFFFFFFFFu, inc, d); if ((threadIdx.x & 31) >= (u32)d) inc += o; }
      u32 ex = inc - sum;
      if (krem >= ex && krem < inc) {
        u32 cum = ex;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (krem >= cum && krem < cum + loc[q]) { s_pick[0] = threadIdx.x * 8 + q; s_pick[1] = krem - cum; }
          cum += loc[q];
        }
      }
    }
    __syncthreads();
    prefix |= (u64)s_pick[0] << (8 * b); mask |= 0xFFull << (8 * b); krem = s_pick[1];
    __syncthreads();
  }
  return prefix;
}

// What a pass over a group's records finds: members present, the first of them with its op and size (and the extremes of both over
// all), why the group may not be complete (2 in flight, 4 invalid times), the oldest op in flight, most changes, extremes of the times.
struct DefPart {
  u64 by = 0, by_lo = U64_MAX_, by_hi = 0, chk = 0, e_min = U64_MAX_, tmax = 0, tmin = U64_MAX_; i64 age = -1, x_max = INT64_MIN;
  u32 npres = 0, first = NONE, op = 0, op_lo = NONE, op_hi = 0, bits = 0;
};
// 64-bit extremes over the warp: the upper words decide, then the lower words of those that have the extreme upper word
__device__ __forceinline__ u64 redux_max(u64 v) {
  const u32 h = (u32)(v >> 32), top = __reduce_max_sync(FULLM, h), l = __reduce_max_sync(FULLM, h == top ? (u32)v : 0u);
  return (u64)top << 32 | l;
}
__device__ __forceinline__ u64 redux_min(u64 v) { return ~redux_max(~v); }
__device__ __forceinline__ i64 redux_max_signed(i64 v) { return (i64)(redux_max((u64)v ^ (1ull << 63)) ^ (1ull << 63)); }
__device__ __forceinline__ DefPart def_warp(const DefPart& a) {
  DefPart r;
  r.first = __reduce_min_sync(FULLM, a.first);
  const u32 src = (u32)__ffs(__ballot_sync(FULLM, a.first == r.first)) - 1u;              // (all lanes where no member is present)
  r.by = (u64)__shfl_sync(FULLM, (u32)a.by, src) | (u64)__shfl_sync(FULLM, (u32)(a.by >> 32), src) << 32; r.op = __shfl_sync(FULLM, a.op, src);
  r.npres = __reduce_add_sync(FULLM, a.npres); r.bits = __reduce_or_sync(FULLM, a.bits);
  r.by_lo = redux_min(a.by_lo); r.by_hi = redux_max(a.by_hi); r.op_lo = __reduce_min_sync(FULLM, a.op_lo); r.op_hi = __reduce_max_sync(FULLM, a.op_hi);
  r.chk = redux_max(a.chk); r.e_min = redux_min(a.e_min); r.tmax = redux_max(a.tmax); r.tmin = redux_min(a.tmin);
  r.age = redux_max_signed(a.age); r.x_max = redux_max_signed(a.x_max);
  return r;
}
// Over the CTA, which all threads call: the warps' parts meet in shared memory and every warp merges them for itself. Twelve
// reductions of a value each, with three barriers apiece, and two passes over the records took 10 instead of 7.1 us for one op in flight
// of a ring of 256.
__device__ __forceinline__ DefPart def_reduce(const DefPart& mine, DefPart* s_part /*[32]*/) {
  const DefPart w = def_warp(mine);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = w;
  __syncthreads();                                         // (the CTA's next group begins with a barrier)
  static_assert(LARGE_DEF_THREADS == 1024, "a warp's part per lane");
  return def_warp(s_part[threadIdx.x & 31]);
}

__global__ void __launch_bounds__(LARGE_DEF_THREADS) k_reduce_large_deferred(const WinDesc* wd, DeferList DL, Registry R, Params P, i64 now) {
  begin_after();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ u64 s_red64[32];
  __shared__ u32 s_red32[32];
  __shared__ u32 s_hist[256];
  __shared__ u32 s_pick[2];
  __shared__ DefPart s_part[32];
  const u32 total = *DL.count;
  for (u32 e = blockIdx.x; e < total; e += gridDim.x) {
    const u64 ent = DL.entries[e];
    const WinDesc& D = wd[(u32)(ent >> 32)];
    const u64 g = (u32)ent;
    const u32 c = owner_of(D.ranges, R.n_comms, g, threadIdx.x & 31);      // every warp for itself: no barrier
    const RangeRow row = D.ranges[c];
    const u32 n = row.n, so = (u32)(g - row.group0);
    const u32* mem = R.members + R.comm_moff[c];
    u64* s_te = (u64*)smem_raw;
    u64* s_du = s_te + n;
    const u64 G = D.n_groups;
    __syncthreads();
    const u64 slot = row.slot0 + (u64)so * n;                      // flags, group-major
    const u32 seq = row.seq_lo + so;
    const u32* pm = D.perm + perm_at(row, so, 0);     // member p at pm[p * n_seq]
    const u64 pst = row.n_seq;
    // one pass over the records, one reduction over everything it finds
    DefPart x;
    for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS) {
      const u32 idx = pm[p * pst];
      u64 te = 0, du = 0;
      if (idx != NONE) {
        const i64 ta = D.t_enter[idx], tb = D.t_exit[idx]; const u64 by = D.bytes[idx]; const u32 op = D.op[idx];
        u32 ch = 0;
        if (D.send_chg != nullptr) { const u32 sc = D.send_chg[idx], rc = D.recv_chg[idx]; ch = sc > rc ? sc : rc; }
        te = (u64)ta; du = (u64)(tb - ta);
        ++x.npres;
        if (p < x.first) { x.first = p; x.by = by; x.op = op; }
        x.by_lo = min(x.by_lo, by); x.by_hi = max(x.by_hi, by); x.op_lo = min(x.op_lo, op); x.op_hi = max(x.op_hi, op);
        if (tb == -1) { x.bits |= 2; x.age = max(x.age, now - ta); } else if (ta < 0 || tb < ta) x.bits |= 4;
        x.chk = max(x.chk, ((u64)ch << 32) | (u64)(NONE - p));
        x.e_min = min(x.e_min, te); x.tmax = max(x.tmax, du); x.tmin = min(x.tmin, du); x.x_max = max(x.x_max, tb);
      }
      s_te[p] = te; s_du[p] = du;
    }
    x = def_reduce(x, s_part);
    const u32 npres = x.npres, gop = x.op, mism = x.npres != 0 && (x.by_lo != x.by_hi || x.op_lo != x.op_hi);
    const u64 gbytes = x.by, chk = x.chk, e_min = x.e_min, tmax = x.tmax, tmin = x.tmin; const i64 age = x.age, x_max = x.x_max;
    const bool have_first = npres != 0, inflight = x.bits & 2, bad_time = x.bits & 4, complete = npres == n && !inflight && !bad_time;
    const bool barrier = have_first && gop == CCLD_OP_ALLREDUCE && gbytes < P.barrier_bytes;
    u32 gfl = (mism ? CCLD_G_OPSET_MISMATCH : 0) | (barrier ? CCLD_G_BARRIER : 0) | (inflight ? CCLD_G_INFLIGHT : 0) |
              (bad_time ? CCLD_G_BAD_TIME : 0) | (complete ? CCLD_G_COMPLETE : CCLD_G_INCOMPLETE);
    const bool analysed = complete && !barrier && n >= P.min_group;
    const bool hang = !complete && inflight && age > P.hang_ns && !barrier;
    if (analysed) gfl |= CCLD_G_ANALYSED;
    if (hang) gfl |= CCLD_G_HANG_ALERT;

    if (!complete) {
      for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS)
        D.flags[slot + p] = pm[p * pst] == NONE ? (CCLD_F_NOT_ANALYSED | CCLD_F_MISSING) : CCLD_F_NOT_ANALYSED;
      if (threadIdx.x == 0) {
        if (hang) raise_alert(D, R.comm_id[c], seq, age);
        for (int q = 0; q < GI_COUNT; ++q) D.gi64[(u64)q * G + g] = 0;
        for (int q = 0; q < GU_COUNT; ++q) D.gu32[(u64)q * G + g] = 0;
        D.gu32[(u64)GU_N_PRESENT * G + g] = npres; D.gu32[(u64)GU_GFLAGS * G + g] = gfl; D.gbw[g] = 0.0;
        count_add(D.counters, C_INCOMPLETE, 1); count_add(D.counters, C_BARRIER, barrier); count_add(D.counters, C_MISMATCH, mism);
        count_add(D.counters, C_PRESENT, npres);
      }
      continue;
    }
    // positions of the extrema: lowest ring position among equals
    u32 pmax = NONE, pmin = NONE; u64 askew = 0;
    for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS) {
      if (s_du[p] == tmax && p < pmax) pmax = p;
      if (s_du[p] == tmin && p < pmin) pmin = p;
      const u64 sk = s_te[p] - e_min; askew = sk > askew ? sk : askew;
    }
    pmax = block_reduce(pmax, OpMinU32(), s_red32);
    pmin = block_reduce(pmin, OpMinU32(), s_red32);
    askew = block_reduce(askew, OpMaxU64(), s_red64);
    const i64 span = x_max - (i64)e_min;
    double num, den; bus_factor(gop, n, &num, &den);
    const double bn = (double)gbytes * num;
    if (!barrier) {
      for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS) { atomicAdd(&R.bw_sum[mem[p]], busbw(bn, den, (i64)s_du[p])); atomicAdd(&R.bw_cnt[mem[p]], 1u); }
    }
    u64 med_s = 0, mad_s = 0, med_d = 0, mad_d = 0; u32 n_fs = 0, n_fd = 0;
    if (analysed) {
      const u32 k = (n - 1) >> 1;
      med_s = radix_select([&](u32 i) { return s_te[i] - e_min; }, n, k, askew, s_hist, s_pick);
      { const u64 m = med_s, dmax = m > askew - m ? m : askew - m;
        mad_s = radix_select([&](u32 i) { return absdiff(s_te[i] - e_min, m); }, n, k, dmax, s_hist, s_pick); }
      med_d = tmin + radix_select([&](u32 i) { return s_du[i] - tmin; }, n, k, tmax - tmin, s_hist, s_pick);
      { const u64 m = med_d, dmax = (m - tmin) > (tmax - m) ? (m - tmin) : (tmax - m);
        mad_d = radix_select([&](u32 i) { return absdiff(s_du[i], m); }, n, k, dmax, s_hist, s_pick); }
      for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS) {
        const u64 sk = s_te[p] - e_min, du = s_du[p];
        const bool so_ = mul_gt(absdiff(sk, med_s), 1000u, mad_s, P.k_milli), sh = sk > med_s;
        const bool dq = mul_gt(absdiff(du, med_d), 1000u, mad_d, P.k_milli), dh = du > med_d;
        D.flags[slot + p] = (so_ ? CCLD_F_SKEW_OUT : 0) | (dq ? CCLD_F_DUR_OUT : 0) | (sh ? CCLD_F_SKEW_HI : 0) | (dh ? CCLD_F_DUR_HI : 0);
        if (so_) { ++n_fs; atomicAdd(&R.votes[(u64)mem[p] * 4 + (sh ? 0 : 1)], 1u); }
        if (dq) { ++n_fd; atomicAdd(&R.votes[(u64)mem[p] * 4 + (dh ? 2 : 3)], 1u); }
      }
      n_fs = block_reduce(n_fs, OpAddU32(), s_red32);
      n_fd = block_reduce(n_fd, OpAddU32(), s_red32);
    } else {
      for (u32 p = threadIdx.x; p < n; p += LARGE_DEF_THREADS) D.flags[slot + p] = CCLD_F_NOT_ANALYSED;
    }
    if (threadIdx.x == 0) {
      D.gi64[(u64)GI_E_MIN * G + g] = (i64)e_min; D.gi64[(u64)GI_ARRIVAL_SKEW * G + g] = (i64)askew;
      D.gi64[(u64)GI_T_MAX * G + g] = (i64)tmax; D.gi64[(u64)GI_T_MIN * G + g] = (i64)tmin; D.gi64[(u64)GI_SPAN * G + g] = span;
      D.gi64[(u64)GI_MED_SKEW * G + g] = (i64)med_s; D.gi64[(u64)GI_MAD_SKEW * G + g] = (i64)mad_s;
      D.gi64[(u64)GI_MED_DUR * G + g] = (i64)med_d; D.gi64[(u64)GI_MAD_DUR * G + g] = (i64)mad_d;
      D.gu32[(u64)GU_RANK_TMIN * G + g] = mem[pmin]; D.gu32[(u64)GU_RANK_TMAX * G + g] = mem[pmax];
      D.gu32[(u64)GU_MAX_CHG * G + g] = (u32)(chk >> 32); D.gu32[(u64)GU_RANK_MAX_CHG * G + g] = mem[NONE - (u32)chk];
      D.gu32[(u64)GU_N_PRESENT * G + g] = npres; D.gu32[(u64)GU_GFLAGS * G + g] = gfl;
      D.gbw[g] = busbw(bn, den, span);
      count_add(D.counters, C_COMPLETE, 1); count_add(D.counters, C_BARRIER, barrier); count_add(D.counters, C_ANALYSED, analysed);
      count_add(D.counters, C_MISMATCH, mism); count_add(D.counters, C_PRESENT, npres);
      count_add(D.counters, C_FLAG_SKEW, n_fs); count_add(D.counters, C_FLAG_DUR, n_fd);
    }
  }
}

}  // namespace ccld
