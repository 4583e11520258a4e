// vocab_parallel.cu -- the scoring path for vocabulary-sharded logits and for
// given log-probs (sm_103a).
//
// When a teacher (or student) runs with tensor parallelism its logits are
// split by vocabulary columns across ranks.  Each rank reduces its shard of
// a row to a log-sum-exp pair (m, s) and, if the sampled token falls in its
// columns, the token's logit: 24 bytes per row for S and T together
// (partial_lse_kernel).  After the ranks exchange those, the pairs merge
// into the row's log-sum-exp (combine_kernel), which gives the same
// log-probs as the full row.  The rest of the path (turn statistics, stop
// rule, OPD loss, profile, carried state) then runs on the log-probs: in two
// passes over tiles of rows (scan_aggregate_kernel, scan_complete_kernel), or,
// for a small window after the small-window kernel, as one thread-block
// cluster whose tiles exchange their aggregates through distributed shared
// memory (scan_cluster_kernel).
#include <cooperative_groups.h>
#include <math.h>

#include <atomic>
#include <type_traits>

#include "row_scan.cuh"
#include "stride.h"
#include "stride_device.cuh"
#include "stride_internal.h"

namespace stride {

// Shard-pass launch shapes: CTAs of 128 threads with U 16-byte loads in flight
// per thread and tensor, U = 4 at 8 CTAs per SM or U = 5 at 7 (what the
// registers allow).  Five loads stream faster; eight CTAs hold more rows at
// once, which decides where it saves a wave.  GB300, us for passes, merge and
// scan, 4 at 8 / 5 at 7 (5 at 6 / 7 at 6): 6,000 rows in 4 shards of 37,984
// bf16 logits 520.6 / 520.2 (520.3 / 521.6), in 8 534.1 / 529.3 (529.5 /
// 527.3), in 4 of 8,000 138.7 / 132.5 (132.7 / 138.3); 800 rows 99.0 / 95.8,
// 1,500 168.3 / 159.7, 3,000 282.3 / 274.5; a wave more: 1,100 rows 117.8 /
// 135.8, 1,216 126.4 / 144.0, 2,400 225.0 / 237.5; 600 rows 84.2 / 87.6.  CTAs
// of 64 threads (4 at 16) 542, of 256 (4 at 4) 518 but 547 in 8 shards.
constexpr int kPartialThreads = 128;
constexpr int kPartialManyCtas = 8, kPartialManyLoads = 7;  // CTAs per SM with U = 4, with U = 5
constexpr int kPartialWarps = kPartialThreads / 32;

struct PartialParams {
  const void* S;
  const void* T;
  int64_t ld;
  int32_t V_shard;
  int64_t col0;
  const int32_t* tokens;
  int64_t rows;
  float* partials;  // [rows][6]
  int32_t* dev_status;
  int64_t first_wave;  // rows whose CTAs are resident from the start
};

// Bytes per tensor and first-wave CTA that the hints ahead of the wait ask
// for.  GB300, 6,000 rows in 4 shards of 37,984 bf16 logits, and in 8 of
// 18,992 (passes, merge and scan): plain launches 531 and 577 us; dependent
// ones with 0 / 4 / 8 / 16 / 32 KB 520 / 517 / 516 / 518 / 531 and 559 / 552 /
// 551 / 564 / 585: more than the wait lasts only evicts.
#ifndef STRIDE_PARTIAL_PREFETCH
#define STRIDE_PARTIAL_PREFETCH 8192
#endif
constexpr int64_t kPartialPrefetch = STRIDE_PARTIAL_PREFETCH;

// One CTA per row: (m, s) of S and T over this shard's columns, and the
// gathered logits when the token is one of them (NaN otherwise).
template <typename LT, bool VEC, int U>
__global__ void __launch_bounds__(kPartialThreads, U == 5 ? kPartialManyLoads : kPartialManyCtas)
    partial_lse_kernel(const PartialParams p) {
  __shared__ float s_red[4][kPartialWarps];
  const int64_t r = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const LT* srow = reinterpret_cast<const LT*>(p.S) + r * p.ld;
  const LT* trow = reinterpret_cast<const LT*>(p.T) + r * p.ld;
  // A programmatic dependent: the first wave's CTAs come in as the previous
  // kernel's leave, ask for the start of their rows in L2 (a hint, which
  // reads nothing) and wait for that kernel.
  if (r < p.first_wave && (tid == 0 || tid == 32))
    prefetch_l2(tid == 0 ? srow : trow, min((int64_t)p.V_shard * (int64_t)sizeof(LT), kPartialPrefetch));
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float mS = kMaxStart, sS = 0.f, mT = kMaxStart, sT = 0.f;
  stream_pair<LT, VEC, U>(srow, trow, 0, p.V_shard, tid, kPartialThreads, mS, sS, mT, sT);
  warp_merge2(mS, sS, mT, sT);
  if (lane == 0) {
    s_red[0][warp] = mS;
    s_red[1][warp] = sS;
    s_red[2][warp] = mT;
    s_red[3][warp] = sT;
  }
  __syncthreads();
  if (warp != 0) return;
  mS = lane < kPartialWarps ? s_red[0][lane] : kMaxStart;
  sS = lane < kPartialWarps ? s_red[1][lane] : 0.f;
  mT = lane < kPartialWarps ? s_red[2][lane] : kMaxStart;
  sT = lane < kPartialWarps ? s_red[3][lane] : 0.f;
  warp_merge2<kPartialWarps>(mS, sS, mT, sT);
  if (lane == 0) {
    const float nan = __int_as_float(0x7fc00000);
    const int32_t y = __ldg(p.tokens + r);
    const int64_t c = (int64_t)y - p.col0;
    float xs = nan, xt = nan;
    if (c >= 0 && c < p.V_shard) {
      xs = to_f32(srow[c]);
      xt = to_f32(trow[c]);
    }
    float* o = p.partials + r * 6;
    o[0] = mS;
    o[1] = sS;
    o[2] = mT;
    o[3] = sT;
    o[4] = xs;
    o[5] = xt;
  }
}

// One thread per row: merge the shards' pairs, take the logit from the shard
// that owns the token (exactly one must), form the log-probs.
__global__ void combine_kernel(const float* __restrict__ parts, int32_t n_shards, int64_t rows,
                               float* logp_s, float* logp_t, float* lse_s, float* lse_t,
                               int32_t* dev_status) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  float mS = kMaxStart, sS = 0.f, mT = kMaxStart, sT = 0.f;
  float xs = 0.f, xt = 0.f;
  int owners = 0;
  for (int k = 0; k < n_shards; ++k) {
    const float* q = parts + ((int64_t)k * rows + r) * 6;
    lse_merge(mS, sS, q[0], q[1]);
    lse_merge(mT, sT, q[2], q[3]);
    if (!isnan(q[4]) || !isnan(q[5])) {
      xs = q[4];
      xt = q[5];
      ++owners;
    }
  }
  const float ls = lse_finish(mS, sS), lt = lse_finish(mT, sT);
  const float nan = __int_as_float(0x7fc00000);
  if (owners != 1) {
    set_status(dev_status, STRIDE_DEV_TOKEN_RANGE);
    xs = nan;
    xt = nan;
  }
  if (logp_s) logp_s[r] = xs - ls;
  if (logp_t) logp_t[r] = xt - lt;
  if (lse_s) lse_s[r] = ls;
  if (lse_t) lse_t[r] = lt;
}

constexpr int kRestartTurn = 1;  // st, sd, sl restart at this row
constexpr int kRestartSum = 2;   // c restarts (a seeded row)

// A row's element inside a tile.  The running stop sum c is fp64 (the stop
// rule compares it with lambda); the open-turn sums of log pi_T, d and the
// loss term are fp32 inside the tile (summed in a tree: relative error a few
// 1e-7 of the summed magnitudes), in the cluster's fold of at most 16 tile
// aggregates, and where the tile's prefix meets a row; every stored sum is
// fp64, and so are all sums of a window that might leave fp32's range (`wide`).
// GB300 runs FP64 at 1/64 of the FP32 rate, and the tile scans' fp64 adds were
// what a small window's scan waited on (a 512-row window in one CTA: 6.6 us for
// the block scan).
template <typename F>
struct TileElem {
  double c;
  F st, sd, sl;
  int flags;
};

template <typename F>
__device__ __forceinline__ TileElem<F> tile_combine(const TileElem<F>& a, const TileElem<F>& b) {
  TileElem<F> r;
  r.c = (b.flags & kRestartSum) ? b.c : a.c + b.c;
  r.st = (b.flags & kRestartTurn) ? b.st : a.st + b.st;
  r.sd = (b.flags & kRestartTurn) ? b.sd : a.sd + b.sd;
  r.sl = (b.flags & kRestartTurn) ? b.sl : a.sl + b.sl;
  r.flags = a.flags | b.flags;
  return r;
}

// A tile's aggregate or prefix: with (for turn means) the sum c before the
// last turn mark, a turn's first row or a seeded one, counted from where c is.
template <typename F>
struct TileAgg {
  TileElem<F> e;
  double c0;
};

// c0 of a (earlier, whose c0 is a_c0) and b together.
template <typename F>
__device__ __forceinline__ double tile_c0(const TileElem<F>& a, double a_c0, const TileAgg<F>& b) {
  return !(b.e.flags & kRestartTurn) ? a_c0 : (b.e.flags & kRestartSum) ? b.c0 : a.c + b.c0;
}

template <typename F>
__device__ __forceinline__ TileElem<F> tile_shfl_up(const TileElem<F>& v, int d) {
  TileElem<F> o;
  o.c = __shfl_up_sync(0xffffffffu, v.c, d);
  o.st = __shfl_up_sync(0xffffffffu, v.st, d);
  o.sd = __shfl_up_sync(0xffffffffu, v.sd, d);
  o.sl = __shfl_up_sync(0xffffffffu, v.sl, d);
  o.flags = __shfl_up_sync(0xffffffffu, v.flags, d);
  return o;
}

template <typename F>
__device__ __forceinline__ TileElem<F> elem_combine(const TileElem<F>& a, const TileElem<F>& b) {
  return tile_combine(a, b);
}
template <typename F>
__device__ __forceinline__ TileElem<F> elem_shfl_up(const TileElem<F>& v, int d) {
  return tile_shfl_up(v, d);
}

// Inclusive and exclusive scan of one element per thread over the CTA's
// WARPS warps, in thread order: warp shuffles, then warp 0 scans the warps'
// totals once (each thread then combines with one prefix).  `id` is the
// identity; s_tot and s_pre hold WARPS elements.  With ANY the answer is
// whether any thread's `flag` is set (if so the scan is left there, in all).
template <int WARPS, bool ANY = false, typename E>
__device__ __forceinline__ bool block_scan(const E& v, const E& id, int lane, int warp, E* s_tot, E* s_pre,
                                           E& incl_out, E& excl_out, bool flag = false) {
  E incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const E o = elem_shfl_up(incl, d);
    if (lane >= d) incl = elem_combine(o, incl);
  }
  const E up1 = elem_shfl_up(incl, 1);
  if (lane == 31) s_tot[warp] = incl;
  if (!ANY)
    __syncthreads();
  else if (__syncthreads_or(flag))
    return true;
  if (warp == 0) {
    E t = lane < WARPS ? s_tot[lane] : id;
#pragma unroll
    for (int d = 1; d < WARPS; d <<= 1) {
      const E o = elem_shfl_up(t, d);
      if (lane >= d) t = elem_combine(o, t);
    }
    const E e = elem_shfl_up(t, 1);
    if (lane < WARPS) s_pre[lane] = (lane == 0) ? id : e;
  }
  __syncthreads();
  const E wpre = s_pre[warp];
  incl_out = elem_combine(wpre, incl);
  excl_out = (lane == 0) ? wpre : elem_combine(wpre, up1);
  return false;
}

// Largest j in [0, n) with a[j] <= r (a ascending, a[0] <= r).
__device__ __forceinline__ int smem_upper_le(const int64_t* a, int n, int64_t r) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a[mid] <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The scan on given log-probs, in two passes over tiles of R x kPassThreads
// consecutive rows, R rows per thread:
//   scan_aggregate_kernel  each tile's aggregate: the sums after its last
//                          seeded row and after its last turn start, and the
//                          carried state of every seeded row set aside
//                          (before anything writes the states);
//   scan_complete_kernel   the same rows again: prefixes inside the tile, the
//                          profile, and, once the first pass is complete, the
//                          predecessors' aggregates folded back to the
//                          nearest seeded tile and every row completed.
// The second pass is the first one's programmatic dependent, and what it does
// before its wait needs nothing of it, so the passes overlap: the time is one
// tile's lookups and scan, then one fold.  No flag, ticket or lookback:
// nothing waits on another CTA, nothing has to be cleared.
//
// What bounds it: latency, and FP64 issue (1/64 of the FP32 rate).  So a
// thread takes R rows one after the other (one fp64 add each), and only the
// threads' totals are scanned across the CTA; the open-turn sums are pairs
// of fp32 numbers inside a tile and meet the fp64 prefix where a turn ends.  The profile's
// sums are formed per thread and per run of equal deciles, in registers: a
// shared-memory fp64 atomicAdd per row is a compare-and-swap loop that a
// warp's rows, nearly all in one decile, went through in turn.
//
// GB300, 148,909 rows in 64 trajectories of 8 turns with the profile: a tile
// of 256 rows with a row per thread, shared-memory atomics per row and a
// lookback took 68.8 us (and its 19 MB clear 3.8 us); the passes take about
// 20.  The whole chain of a training step on given log-probs (state, profile
// cleared, scan, record, restart choice): 87.8 -> 27.5 us (with warp 0 alone
// finding a seeded tile near by, and the first pass at 48 registers, so that
// two CTAs of the second fit beside its two; 33.0 without both).
constexpr int kPassThreads = 256;
constexpr int kPassWarps = kPassThreads / 32;
// A tile folds its predecessors' aggregates itself (kPassThreads per round,
// back to the nearest seeded tile), or one CTA turns them into prefixes first,
// so that long trajectories' scans stay linear in their rows: above kDirectTiles
// tiles, whatever the trajectories, and above kDirectMean tiles per trajectory.
// GB300, state and scan in turn mode, us folded / prefixed: one trajectory of
// 262,144 rows 32.6 / 37.9, 524,288 (1,024 tiles) 56.2 / 56.8, 1,048,576 104.5 /
// 84.6, 2,097,152 (4,096 tiles) 213.9 / 144.5; in trajectories of 65,536 rows
// 43.1 / 55.1, 74.2 / 80.3 and 140.1 / 149.0 at the last three, of 2,326 rows
// 49.4 / 60.8, 79.0 / 94.7 and 148.2 / 172.1.
constexpr int64_t kDirectTiles = 4096, kDirectMean = 1024;
constexpr int kFromSeed = 8;  // the open turn's sums start at a seeded row

// A tile's aggregate, or, after scan_prefix_kernel, the prefix before it: a
// ScanSlot in agg[tile], and beside it, in the flags' place, the sum c before
// its last turn start (counted as c is: from the last seeded row, or the tile's
// first) and its kRestart marks.
struct alignas(16) TileMark {
  double c0;
  int marks;
};
struct TileSlot {
  ScanSlot sum;
  TileMark mark;
};

// Past this SM's L1.
__device__ __forceinline__ TileSlot load_tile(const BatchParams& p, int64_t tile) {
  const double2* s = reinterpret_cast<const double2*>(p.agg + tile);
  const double2 a = __ldcg(s), b = __ldcg(s + 1), m = __ldcg(reinterpret_cast<const double2*>(p.flags) + tile);
  return TileSlot{{a.x, a.y, b.x, b.y}, {m.x, (int)__double_as_longlong(m.y)}};
}

__device__ __forceinline__ void store_tile(const BatchParams& p, int64_t tile, const TileSlot& t) {
  p.agg[tile] = t.sum;
  reinterpret_cast<TileMark*>(p.flags)[tile] = t.mark;
}

// A tile's part of the layout: the offsets of its first turn and of the
// ROWS turns after it (every turn has a row at least), and of as many
// trajectories.
template <int ROWS>
struct TileLayout {
  int64_t turn_off[ROWS + 1];
  int64_t traj_row[ROWS + 1];
  int64_t traj_turn[ROWS + 1];
  int64_t first[2];  // first turn and first trajectory, -1 if the layout does not reach the tile's first row
  int begun[2];      // of the staged turns and trajectories, those that begin at or before the tile's last row
};

template <int ROWS>
__device__ __forceinline__ void stage_layout(const BatchParams& p, int64_t r0, int n_here, int tid,
                                             TileLayout<ROWS>& L) {
  const int lane = tid & 31, warp = tid >> 5;
  if (tid < 2) L.begun[tid] = 0;
  if (p.n_turns <= ROWS && p.n_traj <= ROWS) {  // all of it: no search
    if (tid == 0) {
      L.first[0] = p.n_turns > 0 ? 0 : -1;
      L.first[1] = 0;
    }
  } else if (warp == 0) {
    const bool ok = p.n_turns > 0 && __ldg(p.turn_row_off) <= r0;
    const int64_t k0 = ok ? warp_upper_le(p.turn_row_off, 0, p.n_turns - 1, r0, lane) : 0;
    if (lane == 0) L.first[0] = ok ? k0 : -1;
  } else if (warp == 1) {
    const bool ok = __ldg(p.traj_row_off) <= r0;
    const int64_t i0 = ok ? warp_upper_le(p.traj_row_off, 0, p.n_traj - 1, r0, lane) : 0;
    if (lane == 0) L.first[1] = ok ? i0 : -1;
  }
  __syncthreads();
  const int64_t k0 = L.first[0], i0 = L.first[1];
  if (k0 >= 0 && i0 >= 0) {
// (whole warps take part: ROWS is a multiple of the CTA's threads, the
    // offset after the last is one thread's)
#pragma unroll
    for (int i = 0; i <= ROWS; i += kPassThreads) {
      const int j = i + tid;
      if (i == ROWS && warp != 0) break;
      bool turn = false, traj = false;
      if (j <= ROWS) {
        if (k0 + j <= p.n_turns) {
          const int64_t o = __ldg(p.turn_row_off + k0 + j);
          L.turn_off[j] = o;
          turn = j < ROWS && k0 + j < p.n_turns && o < r0 + n_here;
        }
        if (i0 + j <= p.n_traj) {
          const int64_t o = __ldg(p.traj_row_off + i0 + j);
          L.traj_row[j] = o;
          L.traj_turn[j] = __ldg(p.traj_turn_off + i0 + j);
          traj = j < ROWS && i0 + j < p.n_traj && o < r0 + n_here;
        }
      }
      const int n_turn = __popc(__ballot_sync(0xffffffffu, turn)), n_traj = __popc(__ballot_sync(0xffffffffu, traj));
      if (lane == 0 && n_turn) atomicAdd(&L.begun[0], n_turn);
      if (lane == 0 && n_traj) atomicAdd(&L.begun[1], n_traj);
    }
  }
  __syncthreads();
}

// Row r's turn and trajectory.  `m` may hold an earlier row's: most rows
// share its.
template <int ROWS>
__device__ __forceinline__ void seek_row(const BatchParams& p, const TileLayout<ROWS>& L, int64_t r, RowMeta& m) {
  if (!m.bad && r < m.turn_end && r < m.traj_end) return;  // (rows are sought in ascending order)
  m.bad = true;
  m.traj = m.turn = m.local_turn = 0;
  m.traj_start = m.traj_end = m.turn_start = m.turn_end = 0;
  const int64_t k0 = L.first[0], i0 = L.first[1];
  if (k0 < 0 || i0 < 0) return;
  const int j = smem_upper_le(L.turn_off, max(L.begun[0], 1), r);
  const int ni = max(L.begun[1], 1);
  const int q = smem_upper_le(L.traj_row, ni, r);
  int64_t traj = i0 + q, tr_start = L.traj_row[q], tr_end = L.traj_row[q + 1];
  int64_t tu0 = L.traj_turn[q], tu1 = L.traj_turn[q + 1];
  if (r >= tr_end && q == ni - 1 && i0 + ni < p.n_traj) {
    // past the staged trajectories (more than ROWS empty ones in the tile's
    // rows): search the rest in global memory
    int64_t lo = i0 + ni, hi = p.n_traj - 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (__ldg(p.traj_row_off + mid) <= r) lo = mid; else hi = mid - 1;
    }
    traj = lo;
    tr_start = __ldg(p.traj_row_off + traj);
    tr_end = __ldg(p.traj_row_off + traj + 1);
    tu0 = __ldg(p.traj_turn_off + traj);
    tu1 = __ldg(p.traj_turn_off + traj + 1);
  }
  const int64_t turn = k0 + j;
  m.turn = (int32_t)turn;
  m.traj = (int32_t)traj;
  m.turn_start = L.turn_off[j];
  m.turn_end = L.turn_off[j + 1];
  m.local_turn = (int32_t)(turn - tu0);
  m.traj_start = tr_start;
  m.traj_end = tr_end;
  m.bad = !(m.turn_start <= r && r < m.turn_end) || !(tr_start <= r && r < tr_end) || !(tu0 <= turn && turn < tu1);
}

__device__ __forceinline__ RowMeta no_row() {
  RowMeta m;
  m.bad = true;
  m.traj = m.turn = m.local_turn = 0;
  m.traj_start = m.traj_end = m.turn_start = m.turn_end = 0;
  return m;
}

// A row's term of the running stop sum: its log pi_T, for turn means divided
// by the turn's length -- EXACT (after a scoring kernel, whose own scan is
// fp64) in fp64, else (log-probs as given) with one fp32 rounding, 6e-8 of the
// term.
template <bool EXACT>
struct StopTerm {
  using Length = double;
};
template <>
struct StopTerm<false> {
  using Length = float;
};

template <typename Length>
__device__ __forceinline__ double stop_term(const BatchParams& p, float lpt, Length n_k) {
  return p.mode == STRIDE_STOP_TURN_MEAN ? (double)((Length)lpt / n_k) : (double)lpt;
}

// A thread's R rows, what the layout alone says of them: rows tid * R + i of
// the tile.
constexpr int kRowLive = 1, kRowBad = 2, kRowSeeded = 4, kRowTurnStart = 8;

template <int R, bool EXACT>
struct Rows {
  RowMeta first;     // the first row's
  float lam;         // its trajectory's threshold
  int what[R];       // kRow bits
  typename StopTerm<EXACT>::Length length[R];  // of the row's turn
  int bin[R];        // the profile's decile
  float lps[R], lpt[R];
};

// Fills all but the log-probs; seed(j, z) is told the carried state of every
// seeded row j (zeros for a bad one).
template <int R, bool EXACT, int ROWS, typename Seed>
__device__ __forceinline__ void find_rows(const BatchParams& p, const TileLayout<ROWS>& L, int64_t t0, int n_here, int tid,
                                          Rows<R, EXACT>& x, Seed&& seed) {
  RowMeta m = no_row();
  x.first = m;
  x.lam = 0.f;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int j = tid * R + i;
    x.what[i] = 0;
    x.length[i] = 1;
    x.bin[i] = 0;
    if (j >= n_here) continue;
    const int64_t r = p.row_begin + t0 + j;
    seek_row(p, L, r, m);
    const bool seeded = t0 + j == 0 || r == m.traj_start || m.bad;
    const bool fturn = r == m.turn_start;
    x.what[i] = kRowLive | (m.bad ? kRowBad : 0) | (seeded ? kRowSeeded : 0) | (fturn ? kRowTurnStart : 0);
    x.length[i] = i == 0 || seeded || fturn ? max(m.turn_end - m.turn_start, (int64_t)1) : x.length[i > 0 ? i - 1 : 0];
    if (i == 0) {
      x.first = m;
      if (!m.bad) x.lam = p.lambda ? __ldg(p.lambda + m.traj) : p.lambda_all;
    }
    if (seeded) {
      ScanSlot z = {0.0, 0.0, 0.0, 0.0};
      if (!m.bad) {
        const stride_scan_state* sp = p.state + m.traj;
        z.c = __ldcg(&sp->cum);
        if (!fturn) {
          z.st = __ldcg(&sp->turn_sum_t);
          z.sd = __ldcg(&sp->turn_sum_d);
          z.sl = __ldcg(&sp->turn_sum_l);
        }
      }
      seed(j, z);
    }
    if (p.profile && !m.bad) {
      const int64_t pos = r - m.turn_start, n_k = m.turn_end - m.turn_start;  // Observation 1 decile
      x.bin[i] = n_k < (1 << 28) ? (int)(10u * (unsigned)pos / (unsigned)n_k) : (int)((10 * pos) / n_k);
    }
  }
}

template <int R, bool EXACT>
__device__ __forceinline__ void load_logps(const float* __restrict__ logp_s, const float* __restrict__ logp_t, int64_t t0,
                                           int tid, Rows<R, EXACT>& x) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int64_t w = t0 + tid * R + i;
    const bool live = (x.what[i] & kRowLive) != 0;
    x.lps[i] = live ? __ldcg(logp_s + w) : 0.f;
    x.lpt[i] = live ? __ldcg(logp_t + w) : 0.f;
  }
}

// A sum of fp32 terms as the fp32 sum and the sum of its rounding errors
// (Knuth's TwoSum): hi + lo is good to about 2^-45 of the summed magnitudes
// over a tile, at seven FP32 operations where an fp64 add costs as much as 64.
// Its range is fp32's.  So a tile (or, for the profile, a warp) that holds a
// log-prob of 2^50 or more, an infinity or a NaN (`wide`) takes fp64 sums
// instead: a sampled token masked with the lowest finite logit has log pi =
// -3.4e38, and two of them, or its product with another log-prob, are finite
// in fp64 alone.  Below 2^50 a difference is below 2^51, a product below
// 2^101 and the sum of a tile's 512 rows below 2^110.  GB300, 30,011 rows of
// 32,000 bf16 logits: pairs 519.3 us, fp64 in every tile 528.0.  Errors of the
// turns' sums there, in pairs / fp64, of the summed magnitudes: log pi_T and d
// none / none (48 bits hold them), logp_S * d 5e-16 / 3e-18.
struct Sum2 {
  float hi, lo;
};

__device__ __forceinline__ bool wide(float lps, float lpt) {
  constexpr float kMost = 1125899906842624.0f;  // 2^50
  return !(fabsf(lps) < kMost && fabsf(lpt) < kMost);
}

__device__ __forceinline__ void sum_add(double& a, double b) { a += b; }
__device__ __forceinline__ void sum_add(Sum2& a, const Sum2& b) {
  const float s = __fadd_rn(a.hi, b.hi), t = s - a.hi;
  const float e = (a.hi - (s - t)) + (b.hi - t);
  a.hi = s;
  a.lo += b.lo + e;
}

template <typename Sum>
__device__ __forceinline__ Sum sum_of(float x);
template <>
__device__ __forceinline__ double sum_of<double>(float x) { return (double)x; }
template <>
__device__ __forceinline__ Sum2 sum_of<Sum2>(float x) { return Sum2{x, 0.f}; }

// The product a b, exact; as a pair, of log-probs as given, rounded to fp32.
template <typename Sum, bool EXACT>
__device__ __forceinline__ Sum product(float a, float b) {
  if constexpr (std::is_same<Sum, double>::value) {
    return (double)a * (double)b;
  } else {
    const float hi = __fmul_rn(a, b);
    return Sum2{hi, EXACT ? fmaf(a, b, -hi) : 0.f};
  }
}

__device__ __forceinline__ double sum_value(double a) { return a; }
__device__ __forceinline__ double sum_value(const Sum2& a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ double sum_shfl_up(double a, int d) { return __shfl_up_sync(0xffffffffu, a, d); }
__device__ __forceinline__ Sum2 sum_shfl_up(const Sum2& a, int d) {
  return Sum2{__shfl_up_sync(0xffffffffu, a.hi, d), __shfl_up_sync(0xffffffffu, a.lo, d)};
}

__device__ __forceinline__ double sum_shfl_xor(double a, int d) { return __shfl_xor_sync(0xffffffffu, a, d); }
__device__ __forceinline__ Sum2 sum_shfl_xor(const Sum2& a, int d) {
  return Sum2{__shfl_xor_sync(0xffffffffu, a.hi, d), __shfl_xor_sync(0xffffffffu, a.lo, d)};
}

template <typename Sum>
__device__ __forceinline__ Sum warp_sum(Sum v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum_add(v, sum_shfl_xor(v, o));
  return v;
}

// Inclusive sum over the lanes from `head` (<= lane) to this one.
template <typename Sum>
__device__ __forceinline__ Sum seg_sum(Sum v, int head, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const Sum o = sum_shfl_up(v, d);
    if (lane - d >= head) sum_add(v, o);
  }
  return v;
}

// A thread's or tile's element without the carried state: sums since the last
// seeded row (c) and since the last turn start (st, sd, sl).
template <typename Sum>
struct PassElem {
  double c;
  Sum st, sd, sl;
  int flags;  // kRestart marks
  int seed;  // the last seeded row, from the tile's first; -1: none
};

template <typename Sum>
__device__ __forceinline__ void open_rows(Sum& v, const Sum& before, bool turn) {
  if (!turn) sum_add(v, before);
}

template <typename Sum>
__device__ __forceinline__ PassElem<Sum> elem_combine(const PassElem<Sum>& a, const PassElem<Sum>& b) {
  PassElem<Sum> r;
  r.c = (b.flags & kRestartSum) ? b.c : a.c + b.c;
  const bool turn = (b.flags & kRestartTurn) != 0;
  r.st = b.st;
  r.sd = b.sd;
  r.sl = b.sl;
  open_rows(r.st, a.st, turn);
  open_rows(r.sd, a.sd, turn);
  open_rows(r.sl, a.sl, turn);
  r.flags = ((a.flags | b.flags) & (kRestartSum | kRestartTurn)) | ((turn ? b.flags : a.flags) & kFromSeed);
  r.seed = max(a.seed, b.seed);
  return r;
}

template <typename Sum>
__device__ __forceinline__ PassElem<Sum> elem_shfl_up(const PassElem<Sum>& v, int d) {
  PassElem<Sum> o;
  o.c = __shfl_up_sync(0xffffffffu, v.c, d);
  o.st = sum_shfl_up(v.st, d);
  o.sd = sum_shfl_up(v.sd, d);
  o.sl = sum_shfl_up(v.sl, d);
  o.flags = __shfl_up_sync(0xffffffffu, v.flags, d);
  o.seed = __shfl_up_sync(0xffffffffu, v.seed, d);
  return o;
}

// Whether the thread's rows need fp64 sums (bad rows are NaN either way).
template <int R, bool EXACT>
__device__ __forceinline__ bool rows_wide(const Rows<R, EXACT>& x) {
  bool any = false;
#pragma unroll
  for (int i = 0; i < R; ++i) any |= (x.what[i] & (kRowLive | kRowBad)) == kRowLive && wide(x.lps[i], x.lpt[i]);
  return any;
}

// The thread's rows as one element.
// c0 and rest: the sum c before the last turn start of the thread's rows (0 if
// there is none, or a seeded row starts it), and from there on.
template <typename Sum, int R, bool EXACT>
__device__ __forceinline__ PassElem<Sum> rows_elem(const BatchParams& p, const Rows<R, EXACT>& x, int tid, double& c0,
                                                   double& rest) {
  const Sum zero = sum_of<Sum>(0.f);
  PassElem<Sum> e = {0.0, zero, zero, zero, 0, -1};
  c0 = rest = 0.0;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int what = x.what[i];
    if (!(what & kRowLive)) continue;
    const float nan = __int_as_float(0x7fc00000);
    const float lps = (what & kRowBad) ? nan : x.lps[i], lpt = (what & kRowBad) ? nan : x.lpt[i], dd = lps - lpt;
    const bool seeded = (what & kRowSeeded) != 0;
    if (seeded) {
      e.c = 0.0;
      e.seed = tid * R + i;
      e.flags |= kRestartSum;
    }
    if (what & (kRowSeeded | kRowTurnStart)) {
      c0 = e.c;
      rest = 0.0;
      e.st = e.sd = e.sl = zero;
      e.flags = (e.flags & kRestartSum) | kRestartTurn | (seeded ? kFromSeed : 0);
    }
    const double term = stop_term(p, lpt, x.length[i]);
    e.c += term;
    rest += term;
    sum_add(e.st, sum_of<Sum>(lpt));
    sum_add(e.sd, sum_of<Sum>(dd));
    sum_add(e.sl, product<Sum, EXACT>(lps, dd));
  }
  return e;
}

// The thread's rows into the CTA's profile: runs of equal deciles summed in
// registers, neighbouring threads' open runs of one decile together.
template <typename Sum, int R, bool EXACT>
__device__ __forceinline__ void rows_profile_in(const Rows<R, EXACT>& x, int lane, double* s_prof) {
  const Sum zero = sum_of<Sum>(0.f);
  int bin = -1, n = 0;
  Sum d = zero, t = zero;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    if ((x.what[i] & (kRowLive | kRowBad)) != kRowLive) continue;
    if (x.bin[i] != bin) {
      if (bin >= 0) {
        atomicAdd(s_prof + 3 * bin + 0, sum_value(d));
        atomicAdd(s_prof + 3 * bin + 1, sum_value(t));
        atomicAdd(s_prof + 3 * bin + 2, (double)n);
      }
      bin = x.bin[i];
      n = 0;
      d = t = zero;
    }
    sum_add(d, sum_of<Sum>(x.lps[i] - x.lpt[i]));
    sum_add(t, sum_of<Sum>(x.lpt[i]));
    ++n;
  }
  __syncwarp();
  const int prev = __shfl_up_sync(0xffffffffu, bin, 1);
  const unsigned m_run = __ballot_sync(0xffffffffu, lane == 0 || bin != prev);
  const int h = head_of(m_run, lane);
  d = seg_sum(d, h, lane);
  t = seg_sum(t, h, lane);
#pragma unroll
  for (int k = 1; k < 32; k <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, n, k);
    if (lane - k >= h) n += o;
  }
  if (bin >= 0 && (lane == 31 || ((m_run >> lane) & 2u))) {
    atomicAdd(s_prof + 3 * bin + 0, sum_value(d));
    atomicAdd(s_prof + 3 * bin + 1, sum_value(t));
    atomicAdd(s_prof + 3 * bin + 2, (double)n);
  }
}

template <int R, bool EXACT>
__device__ __forceinline__ void rows_profile(const Rows<R, EXACT>& x, int lane, double* s_prof) {
  if (__any_sync(0xffffffffu, rows_wide(x)))
    rows_profile_in<double>(x, lane, s_prof);
  else
    rows_profile_in<Sum2>(x, lane, s_prof);
}

// A slot that the first pass wrote, past this SM's L1.
__device__ __forceinline__ ScanSlot load_slot(const ScanSlot* s) {
  const double2 a = __ldcg(reinterpret_cast<const double2*>(s));
  const double2 b = __ldcg(reinterpret_cast<const double2*>(s) + 1);
  return ScanSlot{a.x, a.y, b.x, b.y};
}

// What the CTA's warps of the first pass exchange.  (A pair is as large as a
// double: the arrays serve either sum.)
struct AggregateShared {
  int last[2][kPassWarps];
  double c[2][kPassWarps];  // before the last turn start, and from there on
  double base[4];
  double open[3][kPassWarps];
};

// First pass: tile t's aggregate (TileSlot), and in incl[w] the carried state of
// every seeded row w.  z is the carried state of the thread's last seeded row.
// False, with nothing written, if the tile's sums need more than Sum.
template <typename Sum, int R, bool EXACT>
__device__ __forceinline__ bool aggregate_tile(const BatchParams& p, int64_t tile, int tid, const Rows<R, EXACT>& x,
                                               const ScanSlot& z, AggregateShared& sh) {
  auto& s_last = sh.last;
  auto& s_c = sh.c;
  auto& s_base = sh.base;
  auto& s_open = reinterpret_cast<Sum(&)[3][kPassWarps]>(sh.open);
  const int lane = tid & 31, warp = tid >> 5;
  if (tid < 4) s_base[tid] = 0.0;
  const Sum zero = sum_of<Sum>(0.f);
  double c0, c;
  const PassElem<Sum> e = rows_elem<Sum>(p, x, tid, c0, c);
  Sum st = e.st, sd = e.sd, sl = e.sl;
  // only what follows the last restart counts: from thread own_c on in the
  // running sum, from own_t on in the open turn's (-1: from the first)
  const unsigned b_sum = __ballot_sync(0xffffffffu, (e.flags & kRestartSum) != 0);
  const unsigned b_turn = __ballot_sync(0xffffffffu, (e.flags & kRestartTurn) != 0);
  if (lane == 0) {
    s_last[0][warp] = b_sum ? warp * 32 + 31 - __clz(b_sum) : -1;
    s_last[1][warp] = b_turn ? warp * 32 + 31 - __clz(b_turn) : -1;
  }
  if (std::is_same<Sum, double>::value)
    __syncthreads();
  else if (__syncthreads_or(rows_wide(x)))
    return false;
  int own_c = -1, own_t = -1;
#pragma unroll
  for (int w = 0; w < kPassWarps; ++w) {
    own_c = max(own_c, s_last[0][w]);
    own_t = max(own_t, s_last[1][w]);
  }
  if (tid == own_c) s_base[0] = z.c;
  if (tid == own_t && (e.flags & kFromSeed)) {
    s_base[1] = z.st;
    s_base[2] = z.sd;
    s_base[3] = z.sl;
  }
  c0 = warp * 32 + 31 < own_c || warp * 32 > own_t ? 0.0 : warp_sum(tid < own_c || tid > own_t ? 0.0 : tid < own_t ? e.c : c0);
  if (tid < own_t) {
    c = 0.0;
    st = sd = sl = zero;
  }
  if (warp * 32 + 31 >= own_t) {
    c = warp_sum(c);
    st = warp_sum(st);
    sd = warp_sum(sd);
    sl = warp_sum(sl);
  }
  if (lane == 0) {
    s_c[0][warp] = c0;
    s_c[1][warp] = c;
    s_open[0][warp] = st;
    s_open[1][warp] = sd;
    s_open[2][warp] = sl;
  }
  __syncthreads();
  if (warp == 0) {
    c0 = warp_sum(lane < kPassWarps ? s_c[0][lane] : 0.0);
    c = warp_sum(lane < kPassWarps ? s_c[1][lane] : 0.0);
    st = warp_sum(lane < kPassWarps ? s_open[0][lane] : zero);
    sd = warp_sum(lane < kPassWarps ? s_open[1][lane] : zero);
    sl = warp_sum(lane < kPassWarps ? s_open[2][lane] : zero);
    if (lane == 0) {
      c0 += s_base[0];
      store_tile(p, tile, TileSlot{{c0 + c, s_base[1] + sum_value(st), s_base[2] + sum_value(sd), s_base[3] + sum_value(sl)},
                                   {c0, (own_c >= 0 ? kRestartSum : 0) | (own_t >= 0 ? kRestartTurn : 0)}});
    }
  }
  return true;
}

template <int R, bool EXACT>
__global__ void __launch_bounds__(kPassThreads, EXACT && R > 1 ? 4 : 5) scan_aggregate_kernel(const BatchParams p,
                                                                     const float* __restrict__ logp_s,
                                                                     const float* __restrict__ logp_t, bool early) {
  constexpr int kRows = R * kPassThreads;
  __shared__ TileLayout<kRows> L;
  __shared__ AggregateShared sh;
  const int tid = threadIdx.x;
  const int64_t tile = blockIdx.x;
  const int64_t t0 = tile * kRows;
  const int n_here = (int)min((int64_t)kRows, p.n_rows - t0);
  Rows<R, EXACT> x;
  ScanSlot z = {0.0, 0.0, 0.0, 0.0};
  // Everything before this kernel is complete past the wait, and only then
  // may the second pass come in: what it reads before its own wait (the
  // layout, the log-probs, lambda) is complete too.  After a scoring kernel
  // (`early`), which lets this one in once its own predecessors are complete,
  // all but the log-probs is read while that kernel ends.
  if (!early) asm volatile("griddepcontrol.wait;" ::: "memory");
  stage_layout(p, p.row_begin + t0, n_here, tid, L);
  find_rows<R, EXACT>(p, L, t0, n_here, tid, x, [&](int j, const ScanSlot& s) {
    z = s;
    p.incl[t0 + j] = s;
  });
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  load_logps<R>(logp_s, logp_t, t0, tid, x);
  if (!aggregate_tile<Sum2>(p, tile, tid, x, z, sh)) aggregate_tile<double>(p, tile, tid, x, z, sh);
}

// Between the passes of a window of many tiles: the aggregates replaced by
// the prefixes before each tile.  One CTA, a run of tiles per thread.
constexpr int kPrefixThreads = 1024;

struct PrefixElem {
  double c, st, sd, sl, c0;
  int flags;
};

__device__ __forceinline__ PrefixElem prefix_elem(const TileSlot& t) {
  return PrefixElem{t.sum.c, t.sum.st, t.sum.sd, t.sum.sl, t.mark.c0, t.mark.marks};
}

__device__ __forceinline__ PrefixElem elem_combine(const PrefixElem& a, const PrefixElem& b) {
  PrefixElem r;
  const bool turn = (b.flags & kRestartTurn) != 0;
  r.c = (b.flags & kRestartSum) ? b.c : a.c + b.c;
  r.st = turn ? b.st : a.st + b.st;
  r.sd = turn ? b.sd : a.sd + b.sd;
  r.sl = turn ? b.sl : a.sl + b.sl;
  r.c0 = !turn ? a.c0 : (b.flags & kRestartSum) ? b.c0 : a.c + b.c0;
  r.flags = a.flags | b.flags;
  return r;
}

__device__ __forceinline__ PrefixElem elem_shfl_up(const PrefixElem& v, int d) {
  PrefixElem o;
  o.c = __shfl_up_sync(0xffffffffu, v.c, d);
  o.st = __shfl_up_sync(0xffffffffu, v.st, d);
  o.sd = __shfl_up_sync(0xffffffffu, v.sd, d);
  o.sl = __shfl_up_sync(0xffffffffu, v.sl, d);
  o.c0 = __shfl_up_sync(0xffffffffu, v.c0, d);
  o.flags = __shfl_up_sync(0xffffffffu, v.flags, d);
  return o;
}

__global__ void __launch_bounds__(kPrefixThreads) scan_prefix_kernel(const BatchParams p, int64_t n_tiles) {
  constexpr int kWarps = kPrefixThreads / 32;
  __shared__ PrefixElem s_tot[kWarps], s_pre[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const PrefixElem id = {0.0, 0.0, 0.0, 0.0, 0.0, 0};
  const int64_t per = (n_tiles + kPrefixThreads - 1) / kPrefixThreads;
  const int64_t j0 = min(tid * per, n_tiles), j1 = min(j0 + per, n_tiles);
  PrefixElem v = id, incl, before;
#pragma unroll 4
  for (int64_t j = j0; j < j1; ++j) v = elem_combine(v, prefix_elem(load_tile(p, j)));
  block_scan<kWarps>(v, id, lane, warp, s_tot, s_pre, incl, before);
#pragma unroll 4
  for (int64_t j = j0; j < j1; ++j) {
    const PrefixElem e = prefix_elem(load_tile(p, j));
    store_tile(p, j, TileSlot{{before.c, before.st, before.sd, before.sl}, {before.c0, before.flags}});
    before = elem_combine(before, e);
  }
}

// A trajectory's share of a thread's rows: the loss of its retained rows and
// its first crossing of lambda here.
template <typename Sum>
struct TrajPart {
  int32_t traj, count, cross_turn;  // traj -1: none
  Sum loss;
  int64_t cross_row;  // from the trajectory's first row; -1: none
};

template <typename Sum>
__device__ __forceinline__ void record_cross(stride_scan_state* sp, const TrajPart<Sum>& t) {
  atomicMin(reinterpret_cast<unsigned long long*>(&sp->stop_row), (unsigned long long)t.cross_row);
  atomicMin(reinterpret_cast<unsigned int*>(&sp->stop_turn), (unsigned int)t.cross_turn);
  sp->stopped = 1;
}

template <typename Sum>
__device__ __forceinline__ void record_loss(stride_scan_state* sp, const Sum& loss, int count) {
  atomicAdd(&sp->loss, sum_value(loss));
  atomicAdd(reinterpret_cast<unsigned long long*>(&sp->loss_tokens), (unsigned long long)count);
}

// The trajectories' records: neighbouring threads of one trajectory together
// (the lowest crossing, the sum of the losses).  Warp-wide.
template <typename Sum>
__device__ __forceinline__ void record_parts(const BatchParams& p, const TrajPart<Sum>& part, int lane) {
  __syncwarp();
  const int prev = __shfl_up_sync(0xffffffffu, part.traj, 1);
  const unsigned m_run = __ballot_sync(0xffffffffu, lane == 0 || part.traj != prev);
  const unsigned m_cross = __ballot_sync(0xffffffffu, part.cross_row >= 0);
  const int h = head_of(m_run, lane);
  const Sum loss = seg_sum(part.loss, h, lane);
  int count = part.count;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, count, d);
    if (lane - d >= h) count += n;
  }
  if (part.traj >= 0) {
    stride_scan_state* sp = p.state + part.traj;
    const unsigned mine = (0xffffffffu >> (31 - lane)) & (0xffffffffu << h);
    if (part.cross_row >= 0 && __ffs(m_cross & mine) - 1 == lane) record_cross(sp, part);
    if (count > 0 && (lane == 31 || ((m_run >> lane) & 2u))) record_loss(sp, loss, count);
  }
}

// Completes the thread's rows, given the exclusive prefix of its rows inside
// the tile, the tile's (pre), the carried state of the tile's seeded rows
// (seed(j), which covers excl.seed too), and by thread the sum c before the
// last turn start of its rows, counted as excl.c is (turn_c0).
template <typename Sum, int R, bool EXACT, int ROWS, typename Seed>
__device__ __forceinline__ void complete_rows(const BatchParams& p, const TileLayout<ROWS>& L, int64_t t0, int tid,
                                              const Rows<R, EXACT>& x, const PassElem<Sum>& excl, const double* pre,
                                              const double* turn_c0, Seed&& seed) {
  const int lane = tid & 31;
  const float nan = __int_as_float(0x7fc00000);
  const Sum zero = sum_of<Sum>(0.f);
  ScanSlot z = {0.0, 0.0, 0.0, 0.0};  // the last seeded row's before this thread
  if (excl.seed >= 0 && (x.what[0] & kRowLive)) z = seed(excl.seed);
  const double from = excl.seed >= 0 ? z.c : pre[0];
  double c = from + excl.c;
  double b_st = pre[1], b_sd = pre[2], b_sl = pre[3];  // what the open turn brought into the tile
  if (excl.flags & kRestartTurn) {
    const bool from = (excl.flags & kFromSeed) != 0;
    b_st = from ? z.st : 0.0;
    b_sd = from ? z.sd : 0.0;
    b_sl = from ? z.sl : 0.0;
  }
  Sum st = excl.st, sd = excl.sd, sl = excl.sl;
  TrajPart<Sum> part = {-1, 0, 0, zero, -1};
  bool kept = false;  // in turn mode the same for all of a turn's rows
  float lam = x.lam;
  RowMeta m = x.first;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int what = x.what[i];
    if (!(what & kRowLive)) break;
    const int j = tid * R + i;
    const int64_t w = t0 + j, r = p.row_begin + w;
    if (what & kRowBad) {
      set_status(p.dev_status, STRIDE_DEV_BAD_LAYOUT);
      if (p.out.logp_s) p.out.logp_s[w] = nan;  // a bad row's log-probs are NaN
      if (p.out.logp_t) p.out.logp_t[w] = nan;
      if (p.out.opd) p.out.opd[w] = nan;
      c = (double)nan;  // nothing after a bad row is meaningful
      continue;
    }
    if (i > 0) seek_row(p, L, r, m);
    const float lps = x.lps[i], lpt = x.lpt[i], dd = lps - lpt;
    const Sum l = product<Sum, EXACT>(lps, dd);
    const bool seeded = (what & kRowSeeded) != 0, fturn = (what & kRowTurnStart) != 0;
    stride_scan_state* sp = p.state + m.traj;
    if (seeded || fturn) {
      st = sd = sl = zero;
      b_st = b_sd = b_sl = 0.0;
    }
    if (seeded) {
      const ScanSlot own = seed(j);
      c = own.c;
      b_st = own.st;
      b_sd = own.sd;
      b_sl = own.sl;
    }
    if (part.traj != m.traj) {  // a new trajectory: the last one's share is complete
      if (part.traj >= 0) {
        if (part.cross_row >= 0) record_cross(p.state + part.traj, part);
        if (part.count > 0) record_loss(p.state + part.traj, part.loss, part.count);
      }
      if (i > 0) lam = p.lambda ? __ldg(p.lambda + m.traj) : p.lambda_all;
      part = TrajPart<Sum>{m.traj, 0, 0, zero, -1};
    }
    const bool turn_last = r == m.turn_end - 1;
    const bool token_sum = p.mode == STRIDE_STOP_TOKEN_SUM;
    const int64_t n_k = m.turn_end - m.turn_start;
    // retained unless the rule fired before the row (row_scan.cuh); a
    // trajectory's first token or turn always is
    if (token_sum) {
      kept = r == m.traj_start || !below(c, lam);
    } else if (i == 0 || seeded || fturn) {
      double c0 = c;  // the sum before the row's turn
      if (!fturn) {
        const int64_t at = m.turn_start - (p.row_begin + t0);  // its first row, from the tile's
        c0 = at < 0 ? pre[4] : from + turn_c0[at / R];
      }
      kept = m.local_turn == 0 || !fired_before_turn(p, m, c0, lam);
    }
    c += stop_term(p, lpt, x.length[i]);
    sum_add(st, sum_of<Sum>(lpt));
    sum_add(sd, sum_of<Sum>(dd));
    sum_add(sl, l);
    if (p.out.opd) p.out.opd[w] = dd;
    if (kept) {
      sum_add(part.loss, l);
      ++part.count;
    }
    if ((token_sum || turn_last) && part.cross_row < 0 && below(c, lam)) {
      part.cross_row = r - m.traj_start;
      part.cross_turn = m.local_turn;
    }
    const bool last = r == m.traj_end - 1 || r == p.row_end - 1;
    if (turn_last || last) {
      const double t_st = b_st + sum_value(st), t_sd = b_sd + sum_value(sd), t_sl = b_sl + sum_value(sl);
      if (turn_last && p.turn_stats) {
        stride_turn_stats ts;
        ts.sum_t = t_st;
        ts.sum_d = t_sd;
        ts.sum_l = t_sl;
        ts.cum = c;
        ts.mean_t = (float)(t_st / (double)n_k);
        ts.n = (int32_t)n_k;
        p.turn_stats[m.turn] = ts;
      }
      if (last) {
        sp->cum = c;
        sp->turn_sum_t = turn_last ? 0.0 : t_st;
        sp->turn_sum_d = turn_last ? 0.0 : t_sd;
        sp->turn_sum_l = turn_last ? 0.0 : t_sl;
        sp->rows_seen = r - m.traj_start + 1;
        sp->turn_idx = turn_last ? m.local_turn + 1 : m.local_turn;
        sp->turn_tokens = turn_last ? 0 : (int32_t)(r - m.turn_start + 1);
      }
    }
  }
  record_parts(p, part, lane);
}

// A small window's scan after the small-window kernel, one tile of TILE
// consecutive rows per CTA (one row per thread) and all tiles one
// thread-block cluster:
//   1. the CTA stages the offsets of the tile's turns and trajectories in
//      shared memory and every thread finds its row's there;
//   2. each row's element: the stop-sum term, log pi_T, d, logp_S * d, and
//      two restart marks -- the open-turn sums restart at a turn's first row,
//      the running sum at a seeded row (a trajectory's first row, or the
//      window's), whose element already holds the carried state;
//   3. a segmented inclusive scan of the tile's elements (warp shuffles, then
//      the warps' totals);
//   4. the tile's aggregate goes to the later tiles' shared memory, and after
//      one cluster barrier warp 0 folds its predecessors';
//   5. every row completes with its inclusive and exclusive prefixes: turn
//      statistics and carried state (row_tail);
//   6. each trajectory's retained loss and first crossing are gathered per
//      warp (record_parts), so its record takes one update per warp instead
//      of one per row (the rows of a token-sum segment below lambda all
//      contended for it).
// A tile that holds a log-prob beyond fp32 sums (`wide`) tells all the others
// with its aggregate, and the window's steps 2 to 6 are done again in fp64.
// The profile's runs of equal deciles are summed in registers while the
// aggregates are on their way.  GB300, against a second block scan for 6 and a
// shared-memory atomic per row for the profile: a 512-row window of 32,000
// fp32 logits 25.9 -> 25.7 us, with the profile 33.7 -> 30.7; 1,024 rows of
// 151,936 bf16 logits with the profile 107.4 -> 101.4.
// The tiles of a window of at most kClusterMaxTiles tiles run at once, as
// ONE thread-block cluster of one CTA per tile: each stores its aggregate
// into the shared memory of every later tile, and after one cluster barrier
// folds its predecessors' aggregates itself.  A second role of the barrier:
// the carried state is read before the dependency wait and written at a
// trajectory's last row, possibly by a later tile, so every CTA arrives once
// its reads are done and waits before any write.
constexpr int kClusterMaxTiles = 16;
// Rows per tile of the cluster scan (a build define, for sweeps).  A sweep of
// the lookback form that preceded it on GB300: the 512-row tiny step took 36.6
// / 36.7 / 37.4 / 39.0 us with tiles of 64 / 128 / 256 / 512 rows.
#ifndef STRIDE_CLUSTER_TILE_ROWS
#define STRIDE_CLUSTER_TILE_ROWS 128
#endif
constexpr int kClusterTileRows = STRIDE_CLUSTER_TILE_ROWS;
static_assert(kClusterTileRows % 32 == 0 && kClusterTileRows >= 64 && kClusterTileRows <= 1024,
              "whole warps, 2 to 32 of them");

// What a thread of the cluster scan knows of its row before the scan.
struct ClusterRow {
  RowMeta meta;
  int64_t r;
  float lps, lpt, lam;
  double cum0, st0, sd0, sl0;  // a seeded row's carried state
  bool live, seeded, fturn;
};

// Whether the window needs fp64 sums for this row: its 2,048 rows at most and
// a carried sum stay below 2^114 otherwise.
__device__ __forceinline__ bool row_wide(const ClusterRow& q) {
  if (!q.live || q.meta.bad) return false;
  constexpr double kMost = 1.3e33;  // (about 2^110)
  return wide(q.lps, q.lpt) || (q.seeded && !(fabs(q.st0) < kMost && fabs(q.sd0) < kMost && fabs(q.sl0) < kMost));
}

__device__ __forceinline__ Sum2 cluster_term(float x) { return Sum2{x, 0.f}; }
__device__ __forceinline__ double cluster_term(double x) { return x; }

// What the CTAs of the cluster scan exchange, and their warps.
template <typename F, int TILE>
struct ClusterShared {
  TileElem<F> wtot[TILE / 32], wpre[TILE / 32];
  TileAgg<F> caggs[kClusterMaxTiles];  // predecessors' aggregates
  TileAgg<F> agg, excl;                // the tile's aggregate and exclusive prefix (its flags unused)
  double c0[TILE];  // by row where a turn begins: the sum c before it (from the row where c restarts)
};

// Steps 2 to 6 with open-turn sums in F.  False, with nothing written, if any
// row of the window needs more than F.
namespace cg = cooperative_groups;
template <typename F, int TILE, typename Meanwhile>
__device__ __forceinline__ bool scan_cluster_rows(const BatchParams& p, const ClusterRow& q, int64_t tile, int64_t n_tiles,
                                                  int64_t r0, int n_here, ClusterShared<F, TILE>& sh, int* s_wide,
                                                  Meanwhile&& meanwhile) {
  constexpr int kWarps = TILE / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const RowMeta& meta = q.meta;
  const bool live = q.live, seeded = q.seeded, fturn = q.fturn, turn_mean = p.mode == STRIDE_STOP_TURN_MEAN;
  const int64_t r = q.r;

  // 2. the row's element: its terms in F (logp_S * d in fp32 rounded once); the
  //    stop-sum term in fp64, a turn mean's share lpt / n_k rounded once to
  //    fp32 first (GB300 issues an fp64 divide as a sequence of fp64
  //    operations at 1/64 of the fp32 rate; the rounding is 6e-8 of the term)
  TileElem<F> x = {0.0, 0, 0, 0, 0};
  double c_before = q.cum0, c0 = 0.0, ri_c = 0.0;
  F e_sl = 0;
  if (live) {
    const float lpt = q.lpt, dd = q.lps - lpt;
    const int64_t n_k = meta.turn_end - meta.turn_start;
    const double ec = turn_mean ? (double)(lpt / (float)(n_k > 0 ? n_k : 1)) : (double)lpt;
    e_sl = (F)q.lps * (F)dd;
    if (seeded && !meta.bad)
      x = TileElem<F>{q.cum0 + ec, (F)(q.st0 + (double)lpt), (F)(q.sd0 + (double)dd), (F)(q.sl0 + (double)e_sl),
                      kRestartSum | kRestartTurn};
    else  // (a bad row's are NaN: nothing after it is meaningful)
      x = TileElem<F>{ec, lpt, dd, e_sl, seeded ? kRestartSum | kRestartTurn : fturn ? kRestartTurn : 0};
  }

  // 3. segmented inclusive scan over the tile
  const TileElem<F> tile_id = {0.0, 0, 0, 0, 0};
  TileElem<F> tile_incl, tile_excl;
  block_scan<kWarps>(x, tile_id, lane, warp, sh.wtot, sh.wpre, tile_incl, tile_excl);

  // 4. the tile's exclusive prefix, from the cluster's other tiles
  if (turn_mean && (seeded || fturn)) {
    const double c0 = seeded ? q.cum0 : tile_excl.c;
    sh.c0[tid] = c0;
    if (meta.turn_end >= r0 + n_here) sh.agg.c0 = c0;  // the tile's last turn
  }
  if (tid == n_here - 1) sh.agg.e = tile_incl;
  __syncthreads();
  const cg::cluster_group cl = cg::this_cluster();
  constexpr bool kNarrow = std::is_same<F, float>::value;
  if (kNarrow) cluster_wait_acquire();  // every tile has started and read its carried state
  if (warp == 0) {
    const TileAgg<F> agg = sh.agg;
    for (int64_t j = tile + 1 + lane; j < n_tiles; j += 32) {
      TileAgg<F>* to = cl.map_shared_rank(sh.caggs, (unsigned)j) + tile;
      to->e = agg.e;
      if (turn_mean) to->c0 = agg.c0;
    }
  }
  if (kNarrow && __any_sync(0xffffffffu, row_wide(q)) && lane < n_tiles) *cl.map_shared_rank(s_wide, (unsigned)lane) = 1;
  __syncwarp();
  cluster_arrive_release();
  meanwhile();             // (while the aggregates are on their way)
  cluster_wait_acquire();  // every aggregate has arrived; nothing touches these arrays after
  if (kNarrow && *s_wide) return false;
  if (warp == 0) {
    // the predecessors' aggregates folded in tile order (a warp scan: the
    // stop sum fp64, the open-turn sums as inside a tile)
    const TileAgg<F> none = {{0.0, 0, 0, 0, 0}, 0.0};
    TileAgg<F> v = none;
    if (lane < tile) v = sh.caggs[lane];
#pragma unroll
    for (int d = 1; d < kClusterMaxTiles; d <<= 1) {
      const TileElem<F> o = tile_shfl_up(v.e, d);
      if (turn_mean) {
        const double c0 = __shfl_up_sync(0xffffffffu, v.c0, d);
        if (lane >= d) v.c0 = tile_c0(o, c0, v);
      }
      if (lane >= d) v.e = tile_combine(o, v.e);
    }
    if (lane == (tile > 0 ? (int)tile - 1 : 0)) sh.excl = tile > 0 ? v : none;
  }
  __syncthreads();

  // 5. complete every row
  if (live) {
    // the row's prefixes: the stop sum fp64, the open-turn sums in F
    const TileElem<F> pre = sh.excl.e;
    const TileElem<F> ri = tile_combine(pre, tile_incl);
    const double from = (tile_excl.flags & kRestartSum) ? 0.0 : pre.c;  // what c counts from, before this row
    if (!seeded) c_before = from + tile_excl.c;
    if (turn_mean && !meta.bad) {  // the sum before the row's turn
      const int64_t j = meta.turn_start - r0;
      c0 = j < 0 ? sh.excl.c0 : seeded ? q.cum0 : from + sh.c0[j];
    }
    RowCarry rc;
    rc.e = ScanElem{0.0, 0.0, 0.0, (double)e_sl, fturn};
    const ScanElem si{ri.c, (double)ri.st, (double)ri.sd, (double)ri.sl, 1};
    row_tail(p, r, meta, rc, si, c_before, c0, false, true);
    ri_c = ri.c;
  }

  // 6. the trajectories' stop records and losses, once per trajectory and warp
  using Sum = typename std::conditional<kNarrow, Sum2, double>::type;
  TrajPart<Sum> part = {-1, 0, 0, sum_of<Sum>(0.f), -1};
  if (live && !meta.bad) {
    const bool turn_last = (r == meta.turn_end - 1);
    const bool test = (p.mode == STRIDE_STOP_TOKEN_SUM) || turn_last;
    // retained unless the rule fired before the row (row_tail); a
    // trajectory's first token or turn always is
    const bool first = (p.mode == STRIDE_STOP_TOKEN_SUM) ? (r == meta.traj_start) : (meta.local_turn == 0);
    const bool kept = first || !(turn_mean ? fired_before_turn(p, meta, c0, q.lam) : below(c_before, q.lam));
    part.traj = meta.traj;
    part.count = kept ? 1 : 0;
    if (kept) part.loss = cluster_term(e_sl);
    if (test && below(ri_c, q.lam)) {
      part.cross_row = r - meta.traj_start;
      part.cross_turn = meta.local_turn;
    }
  }
  record_parts(p, part, lane);
  return true;
}

template <int TILE>
__global__ void __launch_bounds__(TILE) scan_cluster_kernel(const BatchParams p, const float* __restrict__ logp_s,
                                                            const float* __restrict__ logp_t, int64_t n_tiles) {
  __shared__ int64_t s_turn_off[TILE + 1];
  __shared__ int64_t s_traj_row[TILE + 1];   // traj_row_off
  __shared__ int64_t s_traj_turn[TILE + 1];  // traj_turn_off, widened
  __shared__ int64_t s_first[2];                      // first turn, first trajectory of the tile
  __shared__ ClusterShared<float, TILE> s_f32;
  __shared__ ClusterShared<double, TILE> s_f64;
  __shared__ int s_wide;  // set by any tile of the window
  __shared__ double s_prof[3 * STRIDE_PROFILE_BINS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Launched as a programmatic dependent of the kernel that wrote the
  // log-probs.  That kernel waited for its own predecessors before letting
  // this grid be scheduled, so the layout and the carried state may be read
  // before the wait; the log-probs only after it.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid < 3 * STRIDE_PROFILE_BINS) s_prof[tid] = 0.0;
  if (tid == 0) s_wide = 0;
  const int64_t tile = (int64_t)blockIdx.x;
  const int64_t t0 = tile * TILE;           // first window row of the tile
  const int64_t n_here = min((int64_t)TILE, p.n_rows - t0);
  const int64_t r0 = p.row_begin + t0;
  const int64_t w = t0 + tid;  // this thread's window row
  const int64_t r = p.row_begin + w;
  const bool live = tid < n_here;
  float lps = 0.f, lpt = 0.f;

  // 1. the tile's first turn (warp 0) and first trajectory (warp 1), then
  //    the offsets of the next TILE + 1 of each in shared memory (a layout
  //    of at most TILE turns and trajectories: all of them, no search --
  //    one dependent round trip less before the wait)
  if (p.n_turns <= TILE && p.n_traj <= TILE) {
    if (tid == 0) {
      s_first[0] = p.n_turns > 0 ? 0 : -1;
      s_first[1] = 0;
    }
  } else if (warp == 0) {
    const bool ok = p.n_turns > 0 && __ldg(p.turn_row_off) <= r0;
    const int64_t k0 = ok ? warp_upper_le(p.turn_row_off, 0, p.n_turns - 1, r0, lane) : 0;
    if (lane == 0) s_first[0] = ok ? k0 : -1;
  } else if (warp == 1) {
    const bool ok = __ldg(p.traj_row_off) <= r0;
    const int64_t i0 = ok ? warp_upper_le(p.traj_row_off, 0, p.n_traj - 1, r0, lane) : 0;
    if (lane == 0) s_first[1] = ok ? i0 : -1;
  }
  __syncthreads();
  const int64_t k0 = s_first[0], i0 = s_first[1];
  if (k0 >= 0 && i0 >= 0) {
    for (int j = tid; j <= TILE; j += TILE) {
      s_turn_off[j] = __ldg(p.turn_row_off + min(k0 + j, (int64_t)p.n_turns));
      s_traj_row[j] = __ldg(p.traj_row_off + min(i0 + j, (int64_t)p.n_traj));
      s_traj_turn[j] = __ldg(p.traj_turn_off + min(i0 + j, (int64_t)p.n_traj));
    }
  }
  __syncthreads();

  // 2. this thread's row: its turn and trajectory, and its element
  RowMeta meta;
  meta.bad = true;
  meta.traj = 0;
  meta.turn = 0;
  meta.local_turn = 0;
  meta.traj_start = meta.traj_end = meta.turn_start = meta.turn_end = 0;
  if (live && k0 >= 0 && i0 >= 0) {
    const int nk = (int)min((int64_t)TILE, (int64_t)p.n_turns - k0);
    const int j = smem_upper_le(s_turn_off, nk, r);
    const int ni = (int)min((int64_t)TILE, (int64_t)p.n_traj - i0);
    int q = smem_upper_le(s_traj_row, ni, r);
    int64_t traj = i0 + q, tr_start = s_traj_row[q], tr_end = s_traj_row[q + 1];
    int64_t tu0 = s_traj_turn[q], tu1 = s_traj_turn[q + 1];
    if (r >= tr_end && q == ni - 1 && i0 + ni < p.n_traj) {
      // past the staged trajectories (more than TILE empty ones
      // in the tile's rows): search the rest in global memory
      int64_t lo = i0 + ni, hi = p.n_traj - 1;
      while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (__ldg(p.traj_row_off + mid) <= r) lo = mid; else hi = mid - 1;
      }
      traj = lo;
      tr_start = __ldg(p.traj_row_off + traj);
      tr_end = __ldg(p.traj_row_off + traj + 1);
      tu0 = __ldg(p.traj_turn_off + traj);
      tu1 = __ldg(p.traj_turn_off + traj + 1);
    }
    const int64_t turn = k0 + j;
    meta.turn = (int32_t)turn;
    meta.traj = (int32_t)traj;
    meta.turn_start = s_turn_off[j];
    meta.turn_end = s_turn_off[j + 1];
    meta.local_turn = (int32_t)(turn - tu0);
    meta.traj_start = tr_start;
    meta.traj_end = tr_end;
    meta.bad = !(meta.turn_start <= r && r < meta.turn_end) || !(tr_start <= r && r < tr_end) ||
               !(tu0 <= turn && turn < tu1);
  }
  // a seeded row's carried state, and lambda, before the wait
  const bool seeded = live && ((w == 0) || (r == meta.traj_start) || meta.bad);
  const int fturn = (live && r == meta.turn_start) ? 1 : 0;
  double cum0 = 0.0, st0 = 0.0, sd0 = 0.0, sl0 = 0.0;
  if (seeded && !meta.bad) {
    const stride_scan_state* sp = p.state + meta.traj;
    cum0 = __ldcg(&sp->cum);
    st0 = fturn ? 0.0 : __ldcg(&sp->turn_sum_t);
    sd0 = fturn ? 0.0 : __ldcg(&sp->turn_sum_d);
    sl0 = fturn ? 0.0 : __ldcg(&sp->turn_sum_l);
  }
  int bin = 0;
  if (p.profile && live && !meta.bad) bin = (int)((10 * (r - meta.turn_start)) / (meta.turn_end - meta.turn_start));
  const float lam = (live && !meta.bad) ? (p.lambda ? __ldg(p.lambda + meta.traj) : p.lambda_all) : 0.f;
  cluster_arrive_release();  // this CTA's reads of the carried state are done
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (live) {
    lps = __ldcg(logp_s + w);
    lpt = __ldcg(logp_t + w);
  }
  if (live && meta.bad) {
    set_status(p.dev_status, STRIDE_DEV_BAD_LAYOUT);
    lps = lpt = __int_as_float(0x7fc00000);
    if (p.out.logp_s) p.out.logp_s[w] = lps;  // a bad row's log-probs are NaN
    if (p.out.logp_t) p.out.logp_t[w] = lps;
  }
  if (live && p.out.opd) p.out.opd[w] = lps - lpt;
  const ClusterRow x = {meta, r, lps, lpt, lam, cum0, st0, sd0, sl0, live, seeded, fturn != 0};
  Rows<1, false> row;  // for the profile
  row.what[0] = (live ? kRowLive : 0) | (meta.bad ? kRowBad : 0);
  row.bin[0] = bin;
  row.lps[0] = lps;
  row.lpt[0] = lpt;
  const bool done = scan_cluster_rows<float, TILE>(p, x, tile, n_tiles, r0, (int)n_here, s_f32, &s_wide, [&] {
    if (p.profile) rows_profile(row, lane, s_prof);
  });
  if (!done) scan_cluster_rows<double, TILE>(p, x, tile, n_tiles, r0, (int)n_here, s_f64, &s_wide, [] {});
  if (p.profile) {
    __syncthreads();
    if (tid < 3 * STRIDE_PROFILE_BINS && s_prof[tid] != 0.0) atomicAdd(p.profile + tid, s_prof[tid]);
  }
}

// What the CTA's warps of the second pass exchange.
struct CompleteShared {
  PassElem<double> tot[kPassWarps], wpre[kPassWarps];
  int near[2][kPassWarps], needs, folded;
  double fold[5][kPassWarps], pre[5], turn_c0[kPassThreads];
};
static_assert(sizeof(PassElem<Sum2>) == sizeof(PassElem<double>), "the arrays serve either sum");

// Second pass.  False, with nothing written, if the tile's sums need more
// than Sum.
template <typename Sum, int R, bool EXACT, int ROWS>
__device__ __forceinline__ bool complete_tile(const BatchParams& p, const TileLayout<ROWS>& L, int64_t tile, int tid,
                                              const Rows<R, EXACT>& x, bool prefixed, CompleteShared& sh) {
  auto* const s_tot = reinterpret_cast<PassElem<Sum>*>(sh.tot);
  auto* const s_wpre = reinterpret_cast<PassElem<Sum>*>(sh.wpre);
  auto& s_near = sh.near;
  auto& s_fold = sh.fold;
  auto& s_pre = sh.pre;
  auto& s_turn_c0 = sh.turn_c0;
  auto& s_needs = sh.needs;
  auto& s_folded = sh.folded;
  const int lane = tid & 31, warp = tid >> 5;
  const int64_t t0 = tile * ROWS;
  if (tid < 5) s_pre[tid] = 0.0;
  if (tid == 0) {
    s_needs = !(x.what[0] & kRowSeeded);
    s_folded = 0;
  }
  const Sum zero = sum_of<Sum>(0.f);
  const PassElem<Sum> id = {0.0, zero, zero, zero, 0, -1};
  PassElem<Sum> incl, excl;
  constexpr bool kNarrow = std::is_same<Sum, Sum2>::value;
  double c0, rest;
  const PassElem<Sum> own = rows_elem<Sum>(p, x, tid, c0, rest);
  if (block_scan<kPassWarps, kNarrow>(own, id, lane, warp, s_tot, s_wpre, incl, excl, kNarrow && rows_wide(x)))
    return false;
  if (own.flags & kRestartTurn) s_turn_c0[tid] = (own.flags & kRestartSum) ? c0 : excl.c + c0;

  // ---- the first pass's results
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Sums of the predecessors' aggregates back to the nearest one with a seeded
  // row (c), and to the nearest one with a turn start (the open turn's); c0 is
  // that one's, with the sums c before it back to the seeded row.  A seeded
  // tile among the 32 before this one is warp 0's alone to fold.
  const bool needs = s_needs;
  TileSlot a = {{0.0, 0.0, 0.0, 0.0}, {0.0, 0}};
  if (needs) {
    if (prefixed || tid < tile) a = load_tile(p, prefixed ? tile : tile - 1 - tid);
    const unsigned b_sum = __ballot_sync(0xffffffffu, (a.mark.marks & kRestartSum) != 0);
    const unsigned b_turn = __ballot_sync(0xffffffffu, (a.mark.marks & kRestartTurn) != 0);
    if (lane == 0) {
      s_near[0][warp] = b_sum ? warp * 32 + __ffs(b_sum) - 1 : kPassThreads;
      s_near[1][warp] = b_turn ? warp * 32 + __ffs(b_turn) - 1 : kPassThreads;
    }
    if (warp == 0 && (prefixed || b_sum)) {
      double f[5] = {a.sum.c, a.sum.st, a.sum.sd, a.sum.sl, a.mark.c0};
      if (!prefixed) {
        const int n_sum = __ffs(b_sum) - 1, n_turn = __ffs(b_turn) - 1;  // (a seeded row starts a turn: n_turn <= n_sum)
        if (p.mode == STRIDE_STOP_TURN_MEAN)
          f[4] = warp_sum(lane == n_turn ? f[4] : lane > n_turn && lane <= n_sum ? f[0] : 0.0);
        f[0] = warp_sum(lane <= n_sum ? f[0] : 0.0);
#pragma unroll
        for (int k = 1; k < 4; ++k) f[k] = warp_sum(lane <= n_turn ? f[k] : 0.0);
      }
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 5; ++k) s_pre[k] = f[k];
        s_folded = 1;
      }
    }
  }
  __syncthreads();
  if (needs && !s_folded) {
    double f[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    bool turn_open = true, any = false;
    for (int64_t hi = tile;;) {
      int n_sum = kPassThreads, n_turn = kPassThreads;
#pragma unroll
      for (int w = 0; w < kPassWarps; ++w) {
        n_sum = min(n_sum, s_near[0][w]);
        n_turn = min(n_turn, s_near[1][w]);
      }
      if (warp * 32 <= n_sum && hi > warp * 32) {
        any = true;
        if (tid <= n_sum) f[0] += a.sum.c;
        if (turn_open && tid <= n_turn) {
          f[1] += a.sum.st;
          f[2] += a.sum.sd;
          f[3] += a.sum.sl;
          if (tid == n_turn) f[4] = a.mark.c0;
        } else if (tid <= n_sum) {
          f[4] += a.sum.c;
        }
      }
      turn_open = turn_open && n_turn == kPassThreads;
      hi -= kPassThreads;
      if (n_sum < kPassThreads || hi <= 0) break;
      __syncthreads();  // (s_near has been read)
      a = TileSlot{{0.0, 0.0, 0.0, 0.0}, {0.0, 0}};
      if (tid < hi) a = load_tile(p, hi - 1 - tid);
      const unsigned b_sum = __ballot_sync(0xffffffffu, (a.mark.marks & kRestartSum) != 0);
      const unsigned b_turn = __ballot_sync(0xffffffffu, (a.mark.marks & kRestartTurn) != 0);
      if (lane == 0) {
        s_near[0][warp] = b_sum ? warp * 32 + __ffs(b_sum) - 1 : kPassThreads;
        s_near[1][warp] = b_turn ? warp * 32 + __ffs(b_turn) - 1 : kPassThreads;
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (k == 4 && p.mode != STRIDE_STOP_TURN_MEAN) break;
      const double v = any ? warp_sum(f[k]) : 0.0;
      if (lane == 0) s_fold[k][warp] = v;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        double v = lane < kPassWarps ? s_fold[k][lane] : 0.0;
#pragma unroll
        for (int o = kPassWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) s_pre[k] = v;
      }
    }
    __syncthreads();
  }
  complete_rows<Sum>(p, L, t0, tid, x, excl, s_pre, s_turn_c0, [&](int j) { return load_slot(p.incl + t0 + j); });
  return true;
}

template <int R, bool EXACT>
__global__ void __launch_bounds__(kPassThreads, 3) scan_complete_kernel(const BatchParams p,
                                                                       const float* __restrict__ logp_s,
                                                                       const float* __restrict__ logp_t, int64_t n_tiles,
                                                                       bool prefixed, bool validate) {
  constexpr int kRows = R * kPassThreads;
  __shared__ TileLayout<kRows> L;
  __shared__ CompleteShared sh;
  __shared__ double s_prof[3 * STRIDE_PROFILE_BINS];
  const int tid = threadIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t tile = blockIdx.x;
  const int64_t t0 = tile * kRows;
  const int n_here = (int)min((int64_t)kRows, p.n_rows - t0);
  if (tid < 3 * STRIDE_PROFILE_BINS) s_prof[tid] = 0.0;
  stage_layout(p, p.row_begin + t0, n_here, tid, L);
  Rows<R, EXACT> x;
  find_rows<R, EXACT>(p, L, t0, n_here, tid, x, [](int, const ScanSlot&) {});  // (the first pass set the states aside)
  load_logps<R>(logp_s, logp_t, t0, tid, x);
  if (p.profile) rows_profile(x, tid & 31, s_prof);
  if (!complete_tile<Sum2>(p, L, tile, tid, x, prefixed, sh)) complete_tile<double>(p, L, tile, tid, x, prefixed, sh);
  if (p.profile && tid < 3 * STRIDE_PROFILE_BINS && s_prof[tid] != 0.0) atomicAdd(p.profile + tid, s_prof[tid]);
  if (validate) validate_layout(p, tile * kPassThreads + tid, n_tiles * kPassThreads);
}

// Whether a shard pass takes the persistent kernel (score_batch_stream.cu)
// instead of one CTA per row: rows long enough that its ring pays (its rate is
// higher, a row's end costs it more), or so few that one CTA each leaves most
// of the device idle.  GB300, us for the passes, merge and scan, one CTA per
// row / persistent: shard rows of 152 KB (75,968 bf16) 400 rows 64 / 54, 3,000
// 286 / 271, 10,000 860 / 843; (37,984 fp32) 6,000 rows 1,046 / 1,012; of 76 KB
// 400 rows 73 / 63, 800 98 / 102, 6,000 522 / 532; of 38 KB 400 rows 85 / 78,
// 800 115 / 120; of 16 KB 64 rows 45 / 49, 6,000 275 / 337.
static bool shard_pass_persistent(int64_t rows, int dtype, int32_t V, int sms) {
  const int64_t bytes = (int64_t)V * (dtype == STRIDE_DTYPE_BF16 ? 2 : 4);
  return bytes <= ((int64_t)1 << 31) && (bytes >= (128 << 10) || (bytes >= (32 << 10) && rows <= 3 * (int64_t)sms));
}

cudaError_t launch_partial_lse(const void* S, const void* T, int dtype, bool vec, int64_t ld,
                               int32_t V_shard, int64_t col0, const int32_t* tokens, int64_t rows,
                               float* partials, int32_t* dev_status, cudaStream_t stream) {
  int dev = 0;
  cudaError_t qe = cudaSuccess;
  const int sms = current_device_sms(&dev, &qe);
  if (sms <= 0) return qe != cudaSuccess ? qe : cudaErrorInvalidDevice;
  if (shard_pass_persistent(rows, dtype, V_shard, sms) && (reinterpret_cast<uintptr_t>(partials) & 7u) == 0) {
    BatchParams q = {};
    q.S = S;
    q.T = T;
    q.ld = ld;
    q.V = V_shard;
    q.tokens = tokens;
    q.n_rows = rows;
    q.dev_status = dev_status;
    q.partials = partials;
    q.col0 = col0;
    q.timeout_ns = kWaitTimeoutNs;
    return launch_score_batch_stream(q, dtype, vec, stream);
  }
  // five loads, unless eight CTAs per SM save one of a few waves, or the rows
  // are too few to fill either
  const int64_t waves_many = (rows + kPartialManyCtas * sms - 1) / (kPartialManyCtas * sms);
  const int64_t waves_loads = (rows + kPartialManyLoads * sms - 1) / (kPartialManyLoads * sms);
  const bool loads = rows >= 5 * (int64_t)sms && (waves_loads == waves_many || waves_loads > 5);
  const PartialParams p{S, T, ld, V_shard, col0, tokens, rows, partials, dev_status,
                        (int64_t)(loads ? kPartialManyLoads : kPartialManyCtas) * sms};
  const bool bf16 = dtype == STRIDE_DTYPE_BF16;
  auto* kern = loads ? (bf16 ? (vec ? partial_lse_kernel<__nv_bfloat16, true, 5> : partial_lse_kernel<__nv_bfloat16, false, 5>)
                             : (vec ? partial_lse_kernel<float, true, 5> : partial_lse_kernel<float, false, 5>))
                     : (bf16 ? (vec ? partial_lse_kernel<__nv_bfloat16, true, 4> : partial_lse_kernel<__nv_bfloat16, false, 4>)
                             : (vec ? partial_lse_kernel<float, true, 4> : partial_lse_kernel<float, false, 4>));
  return launch_dependent(kern, (unsigned)rows, kPartialThreads, stream, p);
}

cudaError_t launch_combine_partials(const float* parts, int32_t n_shards, int64_t rows, float* logp_s,
                                    float* logp_t, float* lse_s, float* lse_t, int32_t* dev_status,
                                    cudaStream_t stream) {
  return launch_dependent(combine_kernel, (unsigned)((rows + 255) / 256), 256, stream, parts, n_shards, rows, logp_s, logp_t,
                          lse_s, lse_t, dev_status);
}

// Whether one cluster of n CTAs of the cluster scan can be placed on this
// device (looked up once per device and size; sizes above 8 need the
// non-portable cluster attribute, set here first).
bool scan_cluster_fits(int dev, int n, cudaStream_t stream) {
  constexpr int kMaxDev = 64;
  static std::atomic<int> fits[kMaxDev][kClusterMaxTiles + 1];  // 0 unknown, 1 yes, 2 no
  if (dev < 0 || dev >= kMaxDev || n < 1 || n > kClusterMaxTiles) return false;
  const int known = fits[dev][n].load(std::memory_order_acquire);
  if (known) return known == 1;
  auto kern = scan_cluster_kernel<kClusterTileRows>;
  bool ok = true;
  if (n > 8) ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  if (ok) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n);
    cfg.blockDim = dim3(kClusterTileRows);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)n;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    ok = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters >= 1;
  }
  if (!ok) (void)cudaGetLastError();  // a refused size is an answer, not an error to carry
  fits[dev][n].store(ok ? 1 : 2, std::memory_order_release);
  return ok;
}

namespace {

template <int R, bool EXACT>
cudaError_t launch_passes(const BatchParams& p, const float* logp_s, const float* logp_t, const ScanAfter& after,
                          cudaStream_t stream) {
  constexpr int kRows = R * kPassThreads;
  const int64_t n_tiles = (p.n_rows + kRows - 1) / kRows;
  const bool prefixed = n_tiles > kDirectTiles || n_tiles > kDirectMean * p.n_traj;
  cudaError_t e =
      launch_dependent(scan_aggregate_kernel<R, EXACT>, (unsigned)n_tiles, kPassThreads, stream, p, logp_s, logp_t, after.scoring);
  if (e == cudaSuccess && prefixed)
    e = launch_dependent(scan_prefix_kernel, 1, kPrefixThreads, stream, p, n_tiles);
  if (e == cudaSuccess)
    e = launch_dependent(scan_complete_kernel<R, EXACT>, (unsigned)n_tiles, kPassThreads, stream, p, logp_s, logp_t, n_tiles,
                         prefixed, !after.checked);
  return e;
}

}  // namespace

cudaError_t launch_scan_logprobs(const BatchParams& p, const float* logp_s, const float* logp_t,
                                 cudaStream_t stream, const ScanAfter& after) {
  int dev = 0;
  cudaError_t qe = cudaSuccess;
  const int sms = current_device_sms(&dev, &qe);
  if (sms <= 0) return qe != cudaSuccess ? qe : cudaErrorInvalidDevice;
  // a small window: one cluster
  const int64_t cluster_tiles = (p.n_rows + kClusterTileRows - 1) / kClusterTileRows;
  if (after.small && cluster_tiles <= kClusterMaxTiles && scan_cluster_fits(dev, (int)cluster_tiles, stream)) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cluster_tiles);
    cfg.blockDim = dim3(kClusterTileRows);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster_tiles;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, scan_cluster_kernel<kClusterTileRows>, p, logp_s, logp_t, cluster_tiles);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  // A row per thread while its tiles are one per SM, two from there on.
  // 148,909 rows as above (state to restart choice), 1 / 2 / 4 per thread:
  // 34.9 / 32.9 / 35.1 us (one token-sum trajectory: 40.3 / 32.4 / 30.4);
  // 38,000 rows: 24.7 each way.
  const bool one = p.n_rows <= (int64_t)sms * kPassThreads;
  if (after.scoring)
    return one ? launch_passes<1, true>(p, logp_s, logp_t, after, stream)
               : launch_passes<2, true>(p, logp_s, logp_t, after, stream);
  return one ? launch_passes<1, false>(p, logp_s, logp_t, after, stream)
             : launch_passes<2, false>(p, logp_s, logp_t, after, stream);
}

}  // namespace stride
