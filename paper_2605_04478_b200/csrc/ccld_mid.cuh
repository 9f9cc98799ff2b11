// Per-op reductions, median / MAD, flags and votes for communicators of 129 to 1,024 ranks (sm_100a). Included by
// ccld_kernels.cuh.
//
// A CTA takes a tile of MID_SEQS consecutive op counters of one communicator. It first gathers the tile's records with lanes
// along the op counter, turning times into 32-bit keys against the group's first member, which wait in shared memory as
// [member][op counter] (pitch MID_SEQS + 1, so that both the gather's rows and a group's column are free of bank
// conflicts); extrema, op-set check and rate column are reduced on the way. Then a warp takes a group: 32 R keys in the
// registers of its lanes (R = 8, 16 or 32 per lane, one kernel each so that small communicators do not pay for the
// registers of large ones), sorted by a register / shuffle network without a barrier; the deviations of the sorted keys fall
// and rise, so a merge sorts them. Last, a thread per member adds up the tile's bandwidths.
// Groups that are not complete and 32-bit clean go to k_reduce_large_deferred.
//
// Bound by the latency of the gathers (record index, then values) and by issue: about 12 warp instructions per record, half
// of them the network. The kernel before it sorted 64-bit keys in shared memory, a barrier per step: 2 x 24 communicators
// of 172 ranks x 117 ops took 221 us (4.4 G records/s).
#pragma once

namespace ccld {

constexpr int MID_WARPS = MID_THREADS / 32;
constexpr u32 MID_PITCH = MID_SEQS + 1;
static_assert(MID_WARPS == MID_SEQS && MID_SEQS == 8, "a warp per group of a tile");
inline size_t mid_smem_bytes(u32 n) { return (size_t)n * MID_PITCH * 8; }

// merge of R keys that fall and then rise (bitonic), and the sorting network built on it
template <int R, class K> __device__ __forceinline__ void merge_r(K (&v)[R]) {
#pragma unroll
  for (int h = R / 2; h >= 1; h >>= 1) {
#pragma unroll
    for (int i = 0; i < R; ++i) if ((i & h) == 0) cswap(v[i], v[i | h]);
  }
}
template <int R, class K> __device__ __forceinline__ void sort_r(K (&v)[R]) {
#pragma unroll
  for (int b = 0; b < R; b += 8) {                                  // 19-exchange networks for the eights
    K t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = v[b + i];
    sort8(t);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[b + i] = t[i];
  }
#pragma unroll
  for (int w = 8; w < R; w <<= 1) {                                 // two runs of w: mirrored exchange, then half-cleaners in each
#pragma unroll
    for (int b = 0; b < R; b += 2 * w) {
#pragma unroll
      for (int i = 0; i < w; ++i) cswap(v[b + i], v[b + 2 * w - 1 - i]);
    }
#pragma unroll
    for (int h = w / 2; h >= 1; h >>= 1) {
#pragma unroll
      for (int i = 0; i < R; ++i) if ((i & h) == 0) cswap(v[i], v[i | h]);
    }
  }
}
// element r against element r of lane ^ mask, or against R - 1 - r of it
template <int R, class K> __device__ __forceinline__ void lane_exchange(K (&v)[R], int mask, bool keep_low) {
#pragma unroll
  for (int r = 0; r < R; ++r) { const K o = __shfl_xor_sync(FULLM, v[r], mask); v[r] = keep_low ? min(v[r], o) : max(v[r], o); }
}
template <int R, class K> __device__ __forceinline__ void lane_mirror(K (&v)[R], int mask, bool keep_low) {
#pragma unroll
  for (int r = 0; r < R / 2; ++r) {
    const K a = __shfl_xor_sync(FULLM, v[R - 1 - r], mask), b = __shfl_xor_sync(FULLM, v[r], mask);
    v[r] = keep_low ? min(v[r], a) : max(v[r], a);
    v[R - 1 - r] = keep_low ? min(v[R - 1 - r], b) : max(v[R - 1 - r], b);
  }
}
template <int R, class K> __device__ __forceinline__ K pick_r(const K (&v)[R], u32 k) {
  K x = v[0];
#pragma unroll
  for (int i = 1; i < R; ++i) x = k == (u32)i ? v[i] : x;
  return x;
}
// Lower median and lower-median absolute deviation of a warp's 32 R keys, n of them real and the rest the largest key. The
// keys may come in any order; sorted element i lives in lane i / R, register i % R.
template <int R> __device__ __forceinline__ void warp_median_mad(u32 (&v)[R], u32 n, u32 lane, u32* med, u32* mad) {
  sort_r<R>(v);
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    lane_mirror<R>(v, 2 * m - 1, (lane & m) == 0);
#pragma unroll
    for (int h = m >> 1; h >= 1; h >>= 1) lane_exchange<R>(v, h, (lane & h) == 0);
    merge_r<R>(v);
  }
  const u32 k = (n - 1) >> 1;
  const u32 m = __shfl_sync(FULLM, pick_r<R>(v, k % R), k / R);
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = lane * R + r < n ? __usad(v[r], m, 0u) : 0xFFFFFFFFu;        // falls to 0 at k, then rises
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) lane_exchange<R>(v, h, (lane & h) == 0);
  merge_r<R>(v);
  *med = m; *mad = __shfl_sync(FULLM, pick_r<R>(v, k % R), k / R);
}

// what a warp finds for its lanes' op counter while it gathers; every field merges by maximum or or
struct MidPart { u64 kmax, n_kmin, ck; u32 n_emin, emax, xmax, bits; };
__device__ __forceinline__ void mid_merge(MidPart& a, const MidPart& x) {
  a.kmax = x.kmax > a.kmax ? x.kmax : a.kmax; a.n_kmin = x.n_kmin > a.n_kmin ? x.n_kmin : a.n_kmin; a.ck = x.ck > a.ck ? x.ck : a.ck;
  a.n_emin = max(a.n_emin, x.n_emin); a.emax = max(a.emax, x.emax); a.xmax = max(a.xmax, x.xmax); a.bits |= x.bits;
}
__device__ __forceinline__ MidPart mid_shfl_xor(const MidPart& a, int h) {
  MidPart x;
  x.kmax = shfl_xor64(a.kmax, h); x.n_kmin = shfl_xor64(a.n_kmin, h); x.ck = shfl_xor64(a.ck, h);
  x.n_emin = __shfl_xor_sync(FULLM, a.n_emin, h); x.emax = __shfl_xor_sync(FULLM, a.emax, h); x.xmax = __shfl_xor_sync(FULLM, a.xmax, h);
  x.bits = __shfl_xor_sync(FULLM, a.bits, h);
  return x;
}

// The same while a thread goes along its members, in ascending order: values and positions in words of their own, so that a
// record costs a comparison and two selects per extreme. With 64-bit keys, twice that, k_reduce_mid took 71.3 us instead of 66.9 on
// two windows of groups of 172 and 33.6 instead of 31.3 on sixteen rings of 256.
struct MidTrack {
  u32 dmax = 0, pmax = NONE, dmin = NONE, pmin = NONE, cmax = 0, pc = NONE, first = NONE, n_emin = 0, emax = 0, xmax = 0, bits = 0;
  __device__ __forceinline__ void see(u32 p, u32 a, u32 b, u32 d, u32 ch) {
    first = min(first, p);
    if (d > dmax) { dmax = d; pmax = p; }
    if (d < dmin) { dmin = d; pmin = p; }
    if (ch > cmax) { cmax = ch; pc = p; }
    n_emin = max(n_emin, ~a); emax = max(emax, a); xmax = max(xmax, b);
  }
  __device__ __forceinline__ MidPart part() const {
    MidPart x; x.kmax = 0; x.n_kmin = 0; x.ck = 0; x.n_emin = n_emin; x.emax = emax; x.xmax = xmax; x.bits = bits;
    if (first != NONE) {                                      // no longer than the start value: the first member holds it
      x.kmax = ((u64)dmax << 32) | (u64)(NONE - (pmax == NONE ? first : pmax));          // longest, then the lowest position
      x.n_kmin = ~(((u64)dmin << 32) | (u64)(pmin == NONE ? first : pmin));              // shortest, then the lowest position
      x.ck = ((u64)cmax << 32) | (u64)(NONE - (pc == NONE ? first : pc));                // most changes, then the lowest position
    }
    return x;
  }
};

// CTAs per SM: up to 256 members three (four leave 64 registers and spill: 57.0 instead of 58.8 us on twenty rings of 172, but 20.9 instead of
// 18.9 on sixteen of 256 and 103 instead of 98 beside groups of 4 and 6), of 257 to 512 three (76.4 instead of 94.2 us with two on ten rings of 400,
// 82 instead of 100 on one of 500); with 32 keys per lane two are what the registers allow.
template <int R>
__global__ void __launch_bounds__(MID_THREADS, R == 32 ? 2 : 3) k_reduce_mid(const WinDesc* wd, const Tile* tiles,
    TileSum* __restrict__ sums, Registry R_, Params P, DeferList DL) {
  begin_after();
  extern __shared__ __align__(16) u32 mid_keys[];
  __shared__ MidPart s_part[MID_WARPS][MID_SEQS];
  __shared__ u64 s_base[MID_SEQS], s_gby[MID_SEQS];
  __shared__ u32 s_gop[MID_SEQS];
  __shared__ double s_bn[MID_SEQS], s_den[MID_SEQS];          // 0: the group adds no bandwidth
  __shared__ u32 s_rng[MID_SEQS], s_state[MID_SEQS];          // state: 1 round, 2 analysed, 4 set aside
  __shared__ u32 s_cnt[SC_COUNT];
  const Registry& Reg = R_;
  const Tile t = tiles[blockIdx.x];
  const u32 n = t.row.n;
  if (mid_npad(n) != 32u * R || t.count == 0) return;         // another instance's tile, or none (a window that gave up)
  const WinDesc& D = wd[t.w];
  const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const RangeRow& row = t.row;
  const u32* __restrict__ mem = Reg.members + t.moff;
  u32* __restrict__ k_a = mid_keys; u32* __restrict__ k_d = mid_keys + n * MID_PITCH;
  if (threadIdx.x < SC_COUNT) s_cnt[threadIdx.x] = 0;

  // ---- gather: op counter j of the tile in lanes j, j + 8, j + 16, j + 24, a member each; four members in flight ----
  {
    const u32 j = lane & 7, ml = lane >> 3;
    const bool jv = j < t.count;
    const u32* perm = D.perm + row.slot0 + t.seq_off + (jv ? j : 0u);
    const i64* __restrict__ c_te = D.t_enter; const i64* __restrict__ c_tx = D.t_exit;
    const u64* __restrict__ c_by = D.bytes; const u8* __restrict__ c_op = D.op;
    const u32* __restrict__ c_sc = D.send_chg; const u32* __restrict__ c_rc = D.recv_chg;
    MidTrack x;
    i64 te0 = 0; u64 by0 = 0; u32 op0 = 0;
    const u32 i0 = jv ? *perm : NONE;
    if (i0 != NONE) { te0 = c_te[i0]; by0 = c_by[i0]; op0 = c_op[i0]; } else x.bits = 1;
    const u64 base = (u64)te0 - 0x80000000ull;
    for (u32 p0 = wid * 4 + ml; p0 < n; p0 += 4 * 4 * MID_WARPS) {
      u32 idx[4]; i64 ta[4], tb[4]; u64 by[4]; u32 op[4], ch[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { const u32 p = p0 + q * 4 * MID_WARPS; idx[q] = (jv && p < n) ? perm[(u64)p * row.n_seq] : NONE; }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const u32 ix = idx[q] == NONE ? 0u : idx[q];
        ta[q] = c_te[ix]; tb[q] = c_tx[ix]; by[q] = c_by[ix]; op[q] = c_op[ix]; ch[q] = 0;
        if (c_sc != nullptr) { const u32 sc = c_sc[ix], rc = c_rc[ix]; ch[q] = max(sc, rc); }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const u32 p = p0 + q * 4 * MID_WARPS;
        if (p >= n) continue;
        u32 a = 0, d = 0;
        if (idx[q] == NONE) { if (jv) x.bits |= 1; }
        else {
          const u64 ra = (u64)ta[q] - base, rb = (u64)tb[q] - base;
          a = (u32)ra; const u32 b = (u32)rb; d = b - a;
          if (((ra | rb) >> 32) != 0 || (ta[q] | tb[q]) < 0 || b < a) x.bits |= 1;       // beyond 32 bits, negative or in flight, exit before enter
          if (op[q] != op0 || by[q] != by0) x.bits |= 2;
          x.see(p, a, b, d, ch[q]);
        }
        k_a[p * MID_PITCH + j] = a; k_d[p * MID_PITCH + j] = d;
      }
    }
    MidPart mine = x.part();
#pragma unroll
    for (int h = 8; h < 32; h <<= 1) mid_merge(mine, mid_shfl_xor(mine, h));
    if (lane < MID_SEQS) s_part[wid][lane] = mine;
    if (wid == 0 && lane < MID_SEQS) { s_base[lane] = base; s_gby[lane] = by0; s_gop[lane] = op0; }
  }
  __syncthreads();

  // ---- a warp per group: order statistics, flags, votes, the row ----
  {
    const u32 g = wid;
    double bn = 0.0, den = 1.0; u32 state = 0, rng = 0;
    if (g < t.count) {
      MidPart x = s_part[lane & 7][g];
#pragma unroll
      for (int h = 1; h < 8; h <<= 1) mid_merge(x, mid_shfl_xor(x, h));
      const u32 so = t.seq_off + g, emin = ~x.n_emin, tmx = (u32)(x.kmax >> 32), tmn = (u32)(~x.n_kmin >> 32);
      const u64 gby = s_gby[g]; const u32 gop = s_gop[g];
      if (x.bits & 1) {
        state = 4;
        if (lane == 0) { const u32 e = atomicAdd(DL.count, 1u); DL.entries[e] = ((u64)t.w << 32) | (u64)(row.group0 + so); }
      } else {
        const bool barrier = gop == CCLD_OP_ALLREDUCE && gby < P.barrier_bytes, mismatch = (x.bits & 2) != 0;
        const bool analysed = !barrier && n >= P.min_group;
        double num; bus_factor(gop, n, &num, &den);
        const double bnum = (double)gby * num;
        if (!barrier) { bn = bnum; rng = tmx - tmn; }
        state = (barrier ? 0u : 1u) | (analysed ? 2u : 0u);
        u32 ms = 0, ds = 0, md = 0, dm = 0, n_fs = 0, n_fd = 0;
        u8* __restrict__ fp = D.flags + row.slot0 + (u64)so * n;
        const u32* __restrict__ ca = k_a + g; const u32* __restrict__ cd = k_d + g;
        if (analysed) {
          u32 v[R];
#pragma unroll
          for (int q = 0; q < R; ++q) { const u32 p = (u32)q * 32 + lane; v[q] = p < n ? ca[p * MID_PITCH] - emin : 0xFFFFFFFFu; }
          warp_median_mad<R>(v, n, lane, &ms, &ds);
#pragma unroll
          for (int q = 0; q < R; ++q) { const u32 p = (u32)q * 32 + lane; v[q] = p < n ? cd[p * MID_PITCH] - tmn : 0xFFFFFFFFu; }
          warp_median_mad<R>(v, n, lane, &md, &dm);
          // |x - med| * 1000 > k * MAD in whole numbers: |x - med| > floor(k * MAD / 1000); a quotient of 2^32 - 1 or more is never exceeded
          const u64 qs = (u64)ds * P.k_milli / 1000u, qd = (u64)dm * P.k_milli / 1000u;
          const u32 ts = qs > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qs, td = qd > 0xFFFFFFFFull ? 0xFFFFFFFFu : (u32)qd;
#pragma unroll 4
          for (u32 p = lane; p < n; p += 32) {
            const u32 sk = ca[p * MID_PITCH] - emin, dd = cd[p * MID_PITCH] - tmn;
            const bool os = __usad(sk, ms, 0u) > ts, od = __usad(dd, md, 0u) > td, hs = sk > ms, hd = dd > md;
            fp[p] = (u8)((os ? CCLD_F_SKEW_OUT : 0) | (od ? CCLD_F_DUR_OUT : 0) | (hs ? CCLD_F_SKEW_HI : 0) | (hd ? CCLD_F_DUR_HI : 0));
            if (os) { ++n_fs; atomicAdd(&Reg.votes[(u64)mem[p] * 4 + (hs ? 0 : 1)], 1u); }
            if (od) { ++n_fd; atomicAdd(&Reg.votes[(u64)mem[p] * 4 + (hd ? 2 : 3)], 1u); }
          }
        } else {
          for (u32 p = lane; p < n; p += 32) fp[p] = CCLD_F_NOT_ANALYSED;
        }
        n_fs = __reduce_add_sync(FULLM, n_fs); n_fd = __reduce_add_sync(FULLM, n_fd);
        if (lane == 0) {
          const u64 G = D.n_groups, gr = row.group0 + so;
          i64* __restrict__ gi = D.gi64 + gr; u32* __restrict__ gu = D.gu32 + gr; double* __restrict__ gb = D.gbw + gr;
          const u32 span = x.xmax - emin;
          gi[(u64)GI_E_MIN * G] = (i64)(s_base[g] + emin); gi[(u64)GI_ARRIVAL_SKEW * G] = (i64)(u64)(x.emax - emin);
          gi[(u64)GI_T_MAX * G] = (i64)(u64)tmx; gi[(u64)GI_T_MIN * G] = (i64)(u64)tmn; gi[(u64)GI_SPAN * G] = (i64)(u64)span;
          gi[(u64)GI_MED_SKEW * G] = (i64)(u64)ms; gi[(u64)GI_MAD_SKEW * G] = (i64)(u64)ds;
          gi[(u64)GI_MED_DUR * G] = analysed ? (i64)((u64)tmn + md) : 0; gi[(u64)GI_MAD_DUR * G] = (i64)(u64)dm;
          gu[(u64)GU_RANK_TMIN * G] = mem[(u32)~x.n_kmin]; gu[(u64)GU_RANK_TMAX * G] = mem[NONE - (u32)x.kmax];
          gu[(u64)GU_MAX_CHG * G] = (u32)(x.ck >> 32); gu[(u64)GU_RANK_MAX_CHG * G] = mem[NONE - (u32)x.ck];
          gu[(u64)GU_N_PRESENT * G] = n;
          gu[(u64)GU_GFLAGS * G] = CCLD_G_COMPLETE | (barrier ? CCLD_G_BARRIER : 0) | (mismatch ? CCLD_G_OPSET_MISMATCH : 0) | (analysed ? CCLD_G_ANALYSED : 0);
          *gb = busbw(bnum, den, (i64)span);
          atomicAdd(&s_cnt[SC_COMP], 1u);
          if (barrier) atomicAdd(&s_cnt[SC_BAR], 1u);
          if (analysed) atomicAdd(&s_cnt[SC_AN], 1u);
          if (mismatch) atomicAdd(&s_cnt[SC_MIS], 1u);
          if (n_fs) atomicAdd(&s_cnt[SC_FS], n_fs);
          if (n_fd) atomicAdd(&s_cnt[SC_FD], n_fd);
        }
      }
    }
    if (lane == 0) { s_bn[g] = bn; s_den[g] = den; s_rng[g] = rng; s_state[g] = state; }
  }
  __syncthreads();

  // ---- per-member bandwidth over the tile's groups, and the tile's summary ----
  u32 rounds = 0;
#pragma unroll
  for (u32 g = 0; g < MID_SEQS; ++g) rounds += s_state[g] & 1;
  if (rounds) {
    for (u32 p = threadIdx.x; p < n; p += MID_THREADS) {
      double v = 0.0;
#pragma unroll
      for (u32 g = 0; g < MID_SEQS; ++g) {
        const u32 d = k_d[p * MID_PITCH + g];
        if ((s_state[g] & 1) && d != 0) v += s_bn[g] * rcp_newton((double)d * s_den[g]);
      }
      atomicAdd(&Reg.bw_sum[mem[p]], v); atomicAdd(&Reg.bw_cnt[mem[p]], rounds);
    }
  }
  if (threadIdx.x == 0) {
    TileSum ts = {0, NONE, rounds, 0, 0};
    for (u32 g = 0; g < t.count; ++g) {
      if (s_state[g] & 1) best_merge(ts.best_rng, ts.best_k, (u64)s_rng[g], t.seq_off + g);
      ts.n_an += (s_state[g] >> 1) & 1; ts.pad += s_state[g] >> 2;
    }
    sums[blockIdx.x] = ts;
    u64* const counters = D.counters;
    count_add(counters, C_COMPLETE, s_cnt[SC_COMP]); count_add(counters, C_BARRIER, s_cnt[SC_BAR]); count_add(counters, C_ANALYSED, s_cnt[SC_AN]);
    count_add(counters, C_MISMATCH, s_cnt[SC_MIS]); count_add(counters, C_PRESENT, s_cnt[SC_COMP] * n);
    count_add(counters, C_FLAG_SKEW, s_cnt[SC_FS]); count_add(counters, C_FLAG_DUR, s_cnt[SC_FD]);
  }
}

}  // namespace ccld
