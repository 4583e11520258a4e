// warp_tile_scan.cuh -- the persistent kernel's scan: 32 consecutive window
// rows per warp.
//
// A row's log-probs go to the workspace as soon as the row is scored, and
// the row counts itself in at its tile's counter.  Whoever counts the
// tile's last row finds the rows' turns and trajectories, forms their scan
// elements, scans them with shuffles and publishes the tile's aggregate, and
// beside it the sum before its last turn start (publish_tile, which waits for
// nobody).  A scan warp then folds the earlier
// tiles' aggregates (row_scan.cuh lookback, over tiles) and completes the
// rows -- turn statistics, stop test, loss, profile, carried state
// (complete_tile).  All sums are fp64.
//
// Why tiles.  With one lookback per row the chain of inclusive prefixes ran
// 17 us behind the data, and every row paid the search of its turn and an
// fp64 divide on its own.  A tile shares both among 32 rows, its lookback
// spans 1,024 rows per pass, and the wait for the rows' elements is gone.
//
// Why two warps.  Publishing must not wait behind a lookback: a row warp
// that looked back itself held up its next rows, whose tiles' lookbacks then
// waited in turn (30,011 rows of 32,000 bf16 logits on GB300: 1,360 us so,
// 544 us with a scan warp; 919-924 us with one row warp and a scan per row).
//
// Progress.  Publishing waits for nobody; a tile that finds the scan warp's
// queue full is completed by the row warp itself.  Rows are started in ticket
// order and a row warp finishes its rows in that order, so a row warp that
// looks back from tile t has yet to finish only rows of tile t and later:
// the oldest unpublished tile always gets its rows.
#pragma once

#include "row_scan.cuh"

namespace stride {

constexpr int kTileRows = 32;      // window rows per tile (one warp)
constexpr int kCounterWord = 16;   // the tile's counter shares its flag's 128-byte line, in another sector

__device__ __forceinline__ uint32_t count_in(uint32_t* p) {
  uint32_t v;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Number of lanes j whose v is <= x, for v ascending over the lanes
// (0..32; a binary search by shuffles).
__device__ __forceinline__ int lanes_le(int v, int x) {
  int n = 0;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const int at = __shfl_sync(0xffffffffu, v, n + d - 1);
    if (at <= x) n += d;
  }
  const int last = __shfl_sync(0xffffffffu, v, 31);
  return n == 31 && last <= x ? 32 : n;
}

// Largest i in [0, n) with off[i] <= r, per lane, where off[base] <= r and
// `next` is the lanes' off[base + 1 + lane] - r0 (clamped).  Past the staged
// entries (many empty trajectories in a row, or a broken layout) each lane
// searches on.
__device__ __forceinline__ int64_t lane_upper_le(const int64_t* __restrict__ off, int64_t base, int64_t n, int64_t r0,
                                                 int lane) {
  const int64_t at = base + 1 + lane;
  int64_t d = (at < n ? __ldg(off + at) : INT64_MAX) - r0;
  if (at >= n) d = 1 << 20;
  const int rel = (int)(d < -1 ? -1 : (d > (1 << 20) ? (1 << 20) : d));
  const int c = lanes_le(rel, lane);
  int64_t lo = base + c;
  if (c == 32) {
    const int64_t r = r0 + lane;
    int64_t hi = n - 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (__ldg(off + mid) <= r) lo = mid; else hi = mid - 1;
    }
  }
  return lo;
}

// Inclusive sum over the lanes from `head` (<= lane) to this one.
__device__ __forceinline__ double seg_sum(double v, int head, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane - d >= head) v += o;
  }
  return v;
}

// A published tile on its way to the scan warp (shared memory, by lane).
struct TileCarry {
  double c[32], st[32], sd[32], sl[32];  // inclusive within the tile (seeded rows: from the carried state)
  double c_seed[32];                     // a seeded row's carried running sum
  float lps[32], lpt[32];
  int32_t turn[32], traj[32];
  uint32_t m_good, m_seed, m_turn;
  int64_t tile;
};

// Publishes tile t, whose rows' log-probs are all in the workspace, and
// leaves what complete_tile needs in tc.  Warp-wide; waits for nobody.
__device__ __forceinline__ void publish_tile(const BatchParams& p, int64_t t, int lane, TileCarry& tc) {
  const int64_t w = t * kTileRows + lane;   // window row
  const int64_t r0 = p.row_begin + t * kTileRows;
  const int64_t r = r0 + lane;
  const int n_here = (int)min((int64_t)kTileRows, p.n_rows - t * kTileRows);
  const bool live = lane < n_here;
  float lps = 0.f, lpt = 0.f;
  if (live) {
    lps = __ldcg(p.ws_logp_s + w);
    lpt = __ldcg(p.ws_logp_t + w);
  }

  // ---- the rows' turns and trajectories
  RowMeta meta;
  meta.bad = true;
  meta.traj = meta.turn = meta.local_turn = 0;
  meta.traj_start = meta.traj_end = meta.turn_start = meta.turn_end = 0;
  if (p.n_turns > 0 && __ldg(p.turn_row_off) <= r0 && __ldg(p.traj_row_off) <= r0) {
    const int64_t k0 = warp_upper_le(p.turn_row_off, 0, p.n_turns - 1, r0, lane);
    const int64_t i0 = warp_upper_le(p.traj_row_off, 0, p.n_traj - 1, r0, lane);
    const int64_t turn = lane_upper_le(p.turn_row_off, k0, p.n_turns, r0, lane);
    const int64_t traj = lane_upper_le(p.traj_row_off, i0, p.n_traj, r0, lane);
    const int32_t a = __ldg(p.traj_turn_off + traj), b = __ldg(p.traj_turn_off + traj + 1);
    meta.turn = (int32_t)turn;
    meta.traj = (int32_t)traj;
    meta.turn_start = __ldg(p.turn_row_off + turn);
    meta.turn_end = __ldg(p.turn_row_off + turn + 1);
    meta.traj_start = __ldg(p.traj_row_off + traj);
    meta.traj_end = __ldg(p.traj_row_off + traj + 1);
    meta.bad = !(meta.turn_start <= r && r < meta.turn_end) || !(meta.traj_start <= r && r < meta.traj_end) ||
               !(a <= turn && turn < b);
  }
  const bool good = live && !meta.bad;
  if (live && meta.bad) {
    set_status(p.dev_status, STRIDE_DEV_BAD_LAYOUT);
    lps = lpt = __int_as_float(0x7fc00000);
    if (p.out.logp_s) p.out.logp_s[w] = lps;
    if (p.out.logp_t) p.out.logp_t[w] = lps;
    if (p.out.opd) p.out.opd[w] = lps;
  }
  const float dd = lps - lpt;
  const int64_t n_k = good ? meta.turn_end - meta.turn_start : 1;
  const bool fturn = live && r == meta.turn_start;
  const bool seeded = live && (w == 0 || r == meta.traj_start || meta.bad);

  // ---- elements; a seeded row's holds the carried state
  double c = !live ? 0.0 : (p.mode == STRIDE_STOP_TURN_MEAN) ? (double)lpt / (double)n_k : (double)lpt;
  double st = (double)lpt, sd = (double)dd, sl = (double)lps * (double)dd;  // -log pi_S * r_t (Eq. 2)
  double c_seed = 0.0;
  if (seeded && good) {
    const stride_scan_state* sp = p.state + meta.traj;
    c_seed = __ldcg(&sp->cum);
    c += c_seed;
    if (!fturn) {
      st += __ldcg(&sp->turn_sum_t);
      sd += __ldcg(&sp->turn_sum_d);
      sl += __ldcg(&sp->turn_sum_l);
    }
  }
  const unsigned m_seed = __ballot_sync(0xffffffffu, seeded);
  const unsigned m_turn = __ballot_sync(0xffffffffu, fturn) | m_seed;
  const int h_seed = head_of(m_seed, lane), h_turn = head_of(m_turn, lane);
  c = seg_sum(c, max(h_seed, 0), lane);
  st = seg_sum(st, max(h_turn, 0), lane);
  sd = seg_sum(sd, max(h_turn, 0), lane);
  sl = seg_sum(sl, max(h_turn, 0), lane);

  // the sum before each row's turn, where that begins here
  const double c_prev = __shfl_up_sync(0xffffffffu, c, 1);
  const double c0 = __shfl_sync(0xffffffffu, seeded ? c_seed : lane > 0 ? c_prev : 0.0, max(h_turn, 0));

  // ---- the tile's aggregate out, the earlier tiles' prefix in
  uint32_t* flag = p.flags + t * kFlagStride;
  if (lane == n_here - 1) {
    const ScanElem agg{c, st, sd, sl, 0};
    if (m_seed)
      publish(p.incl + t, flag, agg, c0, kStIncl);
    else
      publish(p.agg + t, flag, agg, c0, kStAgg | (m_turn ? kFlagTurnStart : 0u));
  }
  tc.c[lane] = c;
  tc.st[lane] = st;
  tc.sd[lane] = sd;
  tc.sl[lane] = sl;
  tc.c_seed[lane] = c_seed;
  tc.lps[lane] = lps;
  tc.lpt[lane] = lpt;
  tc.turn[lane] = meta.turn;
  tc.traj[lane] = meta.traj;
  const unsigned m_good = __ballot_sync(0xffffffffu, good);
  if (lane == 0) {
    tc.m_good = m_good;
    tc.m_seed = m_seed;
    tc.m_turn = m_turn;
    tc.tile = t;
  }
  // this tile's share of the layout checks
  if (live) validate_layout(p, w, p.n_rows);
}

// Completes a published tile.  Warp-wide.
__device__ __forceinline__ void complete_tile(const BatchParams& p, const TileCarry& tc, int lane) {
  const int64_t t = tc.tile;
  const int64_t w = t * kTileRows + lane;
  const int64_t r = p.row_begin + w;
  const int n_here = (int)min((int64_t)kTileRows, p.n_rows - t * kTileRows);
  const unsigned m_seed = tc.m_seed, m_turn = tc.m_turn;
  const bool good = (tc.m_good >> lane) & 1u, seeded = (m_seed >> lane) & 1u;
  const int h_seed = head_of(m_seed, lane), h_turn = head_of(m_turn, lane);
  const float lps = tc.lps[lane], lpt = tc.lpt[lane], dd = lps - lpt;
  double c = tc.c[lane], st = tc.st[lane], sd = tc.sd[lane], sl = tc.sl[lane];
  RowMeta meta;
  meta.turn = tc.turn[lane];
  meta.traj = tc.traj[lane];
  meta.turn_start = meta.turn_end = meta.traj_start = meta.traj_end = 0;
  meta.local_turn = 0;
  float lam = 0.f;
  if (good) {
    meta.turn_start = __ldg(p.turn_row_off + meta.turn);
    meta.turn_end = __ldg(p.turn_row_off + meta.turn + 1);
    meta.traj_start = __ldg(p.traj_row_off + meta.traj);
    meta.traj_end = __ldg(p.traj_row_off + meta.traj + 1);
    meta.local_turn = meta.turn - __ldg(p.traj_turn_off + meta.traj);
    lam = p.lambda ? __ldg(p.lambda + meta.traj) : p.lambda_all;
  }
  const int64_t n_k = good ? meta.turn_end - meta.turn_start : 1;
  const bool fturn = good && r == meta.turn_start;

  ScanElem pre{0.0, 0.0, 0.0, 0.0, 0};
  double pre_c0 = 0.0;
  if (!(m_seed & 1u)) {
    bool timed_out = false;
    pre = lookback(p, t, lane, timed_out, pre_c0);
    if (timed_out && lane == 0) set_status(p.dev_status, STRIDE_DEV_TIMEOUT);
    if (h_seed < 0) c += pre.c;
    if (h_turn < 0) {
      st += pre.st;
      sd += pre.sd;
      sl += pre.sl;
    }
  }
  // the running sum before each row, and before its turn
  double c_before = __shfl_up_sync(0xffffffffu, c, 1);
  if (lane == 0) c_before = pre.c;
  if (seeded) c_before = tc.c_seed[lane];
  const double c0_here = __shfl_sync(0xffffffffu, c_before, max(h_turn, 0));
  const double c0 = h_turn < 0 ? pre_c0 : c0_here;
  if (!m_seed && lane == n_here - 1)
    publish(p.incl + t, p.flags + t * kFlagStride, ScanElem{c, st, sd, sl, 0}, c0, kStIncl);

  // ---- turn statistics, stop test, retention (row_scan.cuh states the rule)
  const bool turn_last = good && r == meta.turn_end - 1;
  const bool token_sum = p.mode == STRIDE_STOP_TOKEN_SUM;
  if (turn_last && p.turn_stats) {
    stride_turn_stats ts;
    ts.sum_t = st;
    ts.sum_d = sd;
    ts.sum_l = sl;
    ts.cum = c;
    ts.mean_t = (float)(st / (double)n_k);
    ts.n = (int32_t)n_k;
    p.turn_stats[meta.turn] = ts;
  }
  const bool cross = good && (token_sum || turn_last) && below(c, lam);
  const bool first = token_sum ? r == meta.traj_start : meta.local_turn == 0;
  const bool kept = good && (first || !(token_sum ? below(c_before, lam) : fired_before_turn(p, meta, c0, lam)));

  // ---- the trajectories' records, once per trajectory and tile
  const unsigned m_traj = __ballot_sync(0xffffffffu, !good || r == meta.traj_start);
  const unsigned m_cross = __ballot_sync(0xffffffffu, cross), m_kept = __ballot_sync(0xffffffffu, kept);
  const int h_traj = max(head_of(m_traj, lane), 0);
  const double loss = seg_sum(kept ? (double)lps * (double)dd : 0.0, h_traj, lane);
  const unsigned mine = (0xffffffffu >> (31 - lane)) & (0xffffffffu << h_traj);  // this row's trajectory up to it
  if (good) {
    stride_scan_state* sp = p.state + meta.traj;
    if (cross && __ffs(m_cross & mine) - 1 == lane) {
      atomicMin(reinterpret_cast<unsigned long long*>(&sp->stop_row), (unsigned long long)(r - meta.traj_start));
      atomicMin(reinterpret_cast<unsigned int*>(&sp->stop_turn), (unsigned int)meta.local_turn);
      sp->stopped = 1;
    }
    const int n_kept = __popc(m_kept & mine);
    if ((r == meta.traj_end - 1 || lane == n_here - 1) && n_kept > 0) {
      atomicAdd(&sp->loss, loss);
      atomicAdd(reinterpret_cast<unsigned long long*>(&sp->loss_tokens), (unsigned long long)n_kept);
    }
    if (r == meta.traj_end - 1 || r == p.row_end - 1) {
      sp->cum = c;
      sp->turn_sum_t = turn_last ? 0.0 : st;
      sp->turn_sum_d = turn_last ? 0.0 : sd;
      sp->turn_sum_l = turn_last ? 0.0 : sl;
      sp->rows_seen = r - meta.traj_start + 1;
      sp->turn_idx = turn_last ? meta.local_turn + 1 : meta.local_turn;
      sp->turn_tokens = turn_last ? 0 : (int32_t)(r - meta.turn_start + 1);
    }
  }
  if (p.profile) {
    // Observation 1 decile; runs of equal deciles (a turn's rows in order) are summed first
    const int bin = good ? (int)((10 * (r - meta.turn_start)) / n_k) : -1;
    const int prev = __shfl_up_sync(0xffffffffu, bin, 1);
    const unsigned m_run = __ballot_sync(0xffffffffu, lane == 0 || bin != prev);
    const int h_run = head_of(m_run, lane);
    const double bd = seg_sum((double)dd, h_run, lane), bt = seg_sum((double)lpt, h_run, lane);
    if (bin >= 0 && (lane == 31 || ((m_run >> lane) & 2u))) {
      atomicAdd(p.profile + 3 * bin + 0, bd);
      atomicAdd(p.profile + 3 * bin + 1, bt);
      atomicAdd(p.profile + 3 * bin + 2, (double)(lane - h_run + 1));
    }
  }
}

}  // namespace stride
