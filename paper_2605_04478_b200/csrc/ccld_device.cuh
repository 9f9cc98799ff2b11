// Device-side data layout shared by the kernels and the host API of libccld (sm_100a).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/ccld.h"

namespace ccld {

typedef int64_t i64;
typedef uint64_t u64;
typedef uint32_t u32;
typedef uint8_t u8;
typedef unsigned long long ull;

constexpr u32 NONE = 0xFFFFFFFFu;
constexpr u64 U64_MAX_ = ~0ull;

// ---- launch geometry ----
constexpr int REC_THREADS = 128;       // record-streaming kernels: threads per CTA
constexpr int REC_PER_THREAD = 16;     //   each walks a run of consecutive records
constexpr int REC_PER_CTA = REC_THREADS * REC_PER_THREAD;
constexpr int SMALL_N = 8;             // communicators of up to 8 ranks: one thread per group
constexpr int SMALL_SEQS = 256;        //   threads per CTA: eight warps, each on a warp-tile of up to 32 op counters at a time
constexpr u32 FUSED_WT_PER_CTA = 16;   //   warp-tiles a CTA works through: two per warp, or one where that gives every tile of the batch a
                                       //   warp of its own at once
constexpr int WARP_N = 128;            // up to 128 ranks: a CTA per tile of op counters, n_pad / 8 lanes per group
constexpr int MID_ELEMS = 2048;        //   padded records per tile of a communicator of 9 to 128 ranks
constexpr int MID_N = 1024;            // up to 1024 ranks: a warp per group, keys in its registers (as far as 32 per lane go; ns per op
                                       //   counter against the cluster kernel's: 31 and 57 at 520 ranks, 40 and 62 at 768, 46 and 66 at 1,024)
constexpr int MID_THREADS = 256;
constexpr int MID_SEQS = 8;            //   op counters per tile
constexpr int LARGE_SEQS = 8;          // above: a cluster of eight CTAs per tile of 8 consecutive op counters

// First thing in every kernel: what the kernel before it in the stream wrote is visible from here on, and the next one may be
// brought to the SMs.
// A kernel therefore begins while the one before it still writes. What that one may have written - descriptors, ranges, work
// lists, slot tables, result rows, tick blocks; in the first kernel of a call also the caller's columns - is no read-only memory to
// it: such memory is read by ordinary loads through pointers that are not restrict, never by __ldg. (Two kernels back is far
// enough: that one had ended when the wait of the one before let the launch go.) __ldg and const restrict are for the
// registry's tables and, from the second kernel of a call on, for the caller's columns.
__device__ __forceinline__ void begin_after() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

struct Params {
  i64 tbase_init_ns, m_max_ns, hang_ns;
  u64 barrier_bytes;
  u32 theta_slow_milli, alpha_milli, beta_milli, m_max_rounds, slow_rep_threshold, k_milli, min_group, vote_rep_milli;
};

// Eq. 1 state of one communicator, carried from window to window.
struct CommState { u64 rounds; i64 t_first; i64 sum_m; u64 m; u64 slow_count; };

// Registered communicators (immutable after the first analysis) and cumulative per-rank statistics.
struct Registry {
  u32 n_comms, hash_mask, n_ranks, pad;
  const uint4* hash;        // open addressing: (communicator id, index, seq0, n), index NONE = empty
  const uint4* rank_tab;    // [n_ranks][2]: up to RANK_TAB_K inline (communicator id, index << 13 | position) pairs of a rank
  const u32* comm_id;       // [n_comms]
  const u32* comm_n;        // [n_comms] members
  const u32* comm_seq0;     // [n_comms]
  const u64* comm_moff;     // [n_comms] offset of the member list in `members`
  const u32* members;       // rank ids, ring order
  const u32* rank_ptr;      // [n_ranks+1] CSR over (communicator index, position) pairs of a rank
  const u32* ent_comm;
  const u32* ent_pos;
  const u32* const* comm_head;   // [n_comms] trees: [n] lowest position of each member's layer (REG_NO_LAYERS: not known); null for a ring
  CommState* state;         // [n_comms]
  u32* votes;               // [n_ranks][4] skew hi, skew lo, dur hi, dur lo
  u32* ops;                 // [n_ranks]
  u32* bw_cnt;              // [n_ranks]
  double* bw_sum;           // [n_ranks]
};

#define REG_NO_LAYERS reinterpret_cast<const u32*>(1)    // never dereferenced

// rank_tab: pairs beyond RANK_TAB_K do not fit inline; the last pair then holds (NONE, RANK_TAB_OVERFLOW) and the
// CSR lists are searched instead. Empty pairs are (NONE, NONE).
constexpr int RANK_TAB_K = 4;
constexpr u32 RANK_TAB_OVERFLOW = 0xFFFFFFFEu;
constexpr u32 RANK_TAB_POS_BITS = 13;  // positions < CCLD_MAX_COMM_SIZE = 8192

// Which op counters a communicator covers in a window and where its groups / slots start.
// tile0 / n_units: where the communicator's TileSum entries start (index into the window's part of its summary array) and how many it has.
struct RangeRow { u32 seq_lo, n_seq, row_idx, n; u64 group0, slot0; u32 tile0, n_units; };

enum { C_REJECTED = 0, C_COMPLETE, C_INCOMPLETE, C_BARRIER, C_ANALYSED, C_FLAG_SKEW, C_FLAG_DUR, C_MISMATCH,
       C_PRESENT, C_ALERTS, C_ERR, C_INTERNAL, C_MIXED, C_COUNT = 16 };
constexpr int N_CLASSES = 4;           // reduction code paths: n <= 8, <= 128, <= 1024, larger
// Classes 0 and 1 run in one fused kernel whose work list is ordered by (window, time chunk): a window's op
// counters are cut into T chunks per communicator, so that the tiles of one chunk - which gather from the same
// stretch of every rank's records - run together and share the fetched sectors in L2. A communicator's work units are spread evenly
// over the chunks (units_before), so that chunks are stretches of time for all communicators and yet every unit but a communicator's last one is full:
// chunks cut at op counters of their own left a warp-tile 22 or 29 of 32 op counters for 200, 600 and 1,000 per window.
// A chunk of the busiest communicator is one unit long: what the families share then stays in L2 however many ranks there are.
// k_reduce_fused with 96, 64, 32: twelve windows of 4,096 ranks 556, 549, 540 us; one of 16,384 ranks (the larger communicators beside it)
// 401, 382, 361; smaller jobs alike. With 16 the lists take 7 us longer to write and nothing is gained.
constexpr u32 CHUNK_REF = 32;          // op counters per chunk of the busiest communicator of a window
constexpr u32 CHUNK_MAX = 64;          // at most this many chunks per window (longer chunks beyond)
enum { T_GROUPS = 0, T_SLOTS, T_FCTA, T_FWT, T_FSUM, T_TILES2, T_TILES3, T_ROWS, T_FAILED, T_CHUNKS, T_WT_PER_CTA, T_MIXED,
       T_FUSED, T_COUNT = 13 };        // T_FUSED: slots of classes 0 and 1, in units of 32, each communicator's rounded up
// Whether most stretches (of 32 threads' records in the range pass) are among the `mixed` ones.
__host__ __device__ inline bool mostly_mixed(u64 mixed, u64 n_rec) { return mixed * 2 * 32 * REC_PER_THREAD > n_rec; }
constexpr u64 FAILED_CAPACITY = 1, FAILED_EXPECT = 2;      // T_FAILED: the window needs too many slots / its layout is not the expected one
enum { B_FCTA = 0, B_FWT, B_FSUM, B_T2, B_T3, B_COUNT };

// Work-list entries carry a copy of the communicator's range row and member-list offset, so that a
// tile needs no further lookups before its first gather.
struct alignas(16) Tile { u32 w, c, seq_off, count; RangeRow row; u64 moff, pad; };      // classes 2 and 3: one CTA (a cluster) each; summary index = tile index
struct alignas(16) WarpTile { u32 c, seq_off, count, sum_idx; RangeRow row; u64 moff; };      // class 0: up to 32 consecutive op counters of one communicator
struct alignas(16) FusedCta { u32 w, cls, c, seq_off, count, sum_idx, wt_first, wt_count; RangeRow row; u64 moff; };   // class 0: wt_*; class 1: c .. sum_idx, row, moff

// What a tile contributes to its communicator's window decision (Eq. 2 and the round counts).
struct TileSum { u64 best_rng; u32 best_k, n_rounds, n_an, pad; };   // best_k: op-counter offset in the range, NONE if no round

// What the fused kernel needs of a record, as one sector. Where the records of a rank are not neighbours in the upload, a gather of
// every column fetches a sector per value - 200 bytes per record -, so such windows are scattered record by record.
struct PackedRecord { u64 te, tx, by; u32 ch, op; };
static_assert(sizeof(PackedRecord) == 32, "one sector");
__device__ __forceinline__ void store_packed(uint4* at, const PackedRecord& r) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" :: "l"(at), "r"((u32)r.te), "r"((u32)(r.te >> 32)), "r"((u32)r.tx), "r"((u32)(r.tx >> 32)),
               "r"((u32)r.by), "r"((u32)(r.by >> 32)), "r"(r.ch), "r"(r.op) : "memory");
}
__device__ __forceinline__ PackedRecord load_packed(const uint4* at) {
  u32 a, b, c, d, e, f; PackedRecord r;
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d), "=r"(e), "=r"(f), "=r"(r.ch), "=r"(r.op) : "l"(at));
  r.te = (u64)a | (u64)b << 32; r.tx = (u64)c | (u64)d << 32; r.by = (u64)e | (u64)f << 32;
  return r;
}

// One window of a batch: input columns, scratch and result pointers (all device memory).
struct WinDesc {
  const u32 *rank, *comm, *seq;
  const u8* op;
  const u64* bytes;
  const i64 *t_enter, *t_exit;
  const u32 *send_chg, *recv_chg;   // may be null
  u64 n_rec;
  u64 slot_cap;                      // plan fails the window if it would need more slots
  u32 *rmin, *rmax;                  // [n_comms] op counter range seen
  RangeRow* ranges;                  // [n_comms]
  uint4* srow;                       // [n_comms] scatter rows: first slot low, high, op counters covered (0 = nothing to place), first op counter
  u64* totals;                       // [T_COUNT]
  uint2* chunks;                     // [CHUNK_MAX + 1] first CTA (x) and first warp-tile (y) of every chunk, relative to the window
  u64* totals_host;                  // [T_COUNT] the totals once more, in pinned host memory
  const u64* expect;                 // [T_COUNT] totals the host sized this window's results for without waiting (null: it waited)
  u32* poison;                       // set once a window's layout differs from what the host expected: every window planned later gives up too
  u64* counters;                     // [C_COUNT]
  // sized after the plan:
  u64 n_groups, n_slots;
  u32* perm;                         // [n_slots]
  uint4* packed;                     // [n_slots][2] the slots' records (PackedRecord); null: the fused kernel gathers through perm
  u8* flags;                         // [n_slots]
  i64* gi64;                         // [9][n_groups]
  u32* gu32;                         // [6][n_groups]
  double* gbw;                       // [n_groups]
  ccld_comm_verdict* comm_rows;      // [n_rows]
  ccld_hang_alert* alerts;           // [CCLD_MAX_ALERTS_PER_WINDOW]
  u32 base[B_COUNT];                 // this window's first entry in the batch-wide lists (B_*)
  u32 pad;
  TileSum* tsum[3];                  // this window's tile summaries: fused classes, class 2, class 3
};

enum { GI_E_MIN = 0, GI_ARRIVAL_SKEW, GI_T_MAX, GI_T_MIN, GI_SPAN, GI_MED_SKEW, GI_MAD_SKEW, GI_MED_DUR, GI_MAD_DUR, GI_COUNT };
enum { GU_RANK_TMIN = 0, GU_RANK_TMAX, GU_MAX_CHG, GU_RANK_MAX_CHG, GU_N_PRESENT, GU_GFLAGS, GU_COUNT };

__host__ __device__ inline u32 next_pow2(u32 n) { u32 p = 1; while (p < n) p <<= 1; return p; }
__host__ __device__ inline u32 comm_class(u32 n) { return n <= SMALL_N ? 0u : (n <= WARP_N ? 1u : (n <= MID_N ? 2u : 3u)); }
__host__ __device__ inline u32 mid_npad(u32 n) { u32 p = next_pow2(n); return p < 32 ? 32 : p; }
// op counters per work unit: a warp-tile (class 0) or a CTA tile (classes 1 to 3)
__host__ __device__ inline u32 tile_seqs(u32 n) {
  u32 c = comm_class(n);
  return c == 0 ? 32u : (c == 1 ? MID_ELEMS / mid_npad(n) : (c == 2 ? (u32)MID_SEQS : (u32)LARGE_SEQS));
}
__host__ __device__ inline u32 ceil_div(u32 a, u32 b) { return (a + b - 1) / b; }
// work units of a communicator's n_units that lie before chunk tau of T (tau <= T <= CHUNK_MAX): n_units * tau / T
__host__ __device__ inline u32 units_before(u32 n_units, u32 T, u32 tau) { return n_units / T * tau + n_units % T * tau / T; }

}  // namespace ccld
