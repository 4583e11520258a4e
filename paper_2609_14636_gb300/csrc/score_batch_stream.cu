// score_batch_stream.cu -- persistent, warp-specialised batch scoring kernel
// (sm_103a).
//
// One CTA per SM runs until the window's rows are exhausted.  Its warps have
// fixed roles:
//
//   warp 0, producer   takes row tickets (atomicAdd, so rows are processed in
//                      ticket order) and streams each row's student and
//                      teacher logits, chunk by chunk, into a ring of
//                      kStages shared-memory stages with 1-D bulk async copies
//                      (cp.async.bulk ... mbarrier::complete_tx).  The ring
//                      keeps kStages x 2 x kChunk bytes in flight per SM
//                      without spending registers on them.
//   warps 6..21,       read each stage from shared memory into single-pass
//   consumers          online log-sum-exp pairs (stride_device.cuh), release
//                      the stage, and at a row's last chunk post their pairs
//                      for the row's row warp.
//   warps 1..4, row    rows taken round-robin (row n by row warp n mod 4).
//   warps              While the row streams: token, gathered logits, the
//                      row's ragged ends (the logits before its first
//                      16-byte boundary and after its last whole vector).  Once the consumers'
//                      pairs land: their merge, log-probs and outputs, then
//                      the row is counted in at its 32-row tile; the warp
//                      that counts a tile's last row publishes the tile
//                      (warp_tile_scan.cuh) and queues it for the scan warp.
//   warp 5, scan warp  completes the queued tiles: lookback, turn
//                      statistics, stop test, carried state.
//
// With short rows the row warps only leave the log-probs, and the scan follows
// as two passes over them (vocab_parallel.cu): scan_inside below.
//
// Rows of any length should be bound by HBM.  With one row warp, which also
// searched the row's turn and formed its scan element, a row cost about 4.7
// us of dependent latency, more than its bytes take below about 100,000 bf16
// logits.  GB300, before -> four row warps and a scan warp -> now: 30,011 rows
// of 32,000 bf16 logits 919 -> 544 -> 522 us (7,360 GB/s), 3,000 rows 107 ->
// 85.7 -> 70.0; 3,001 rows of 151,936 267.5 -> 263.5 -> 262.0 us; 20,000 rows
// of 151,936 in two windows 1,654 -> 1,645 -> 1,636 us (7,430 GB/s): with long
// rows what was left is the shorter tail of a window's scan.  (Carrying the sum
// before the open turn through the lookback costs a window
// 0.4 us at its end: 20,000 rows in windows of 1,500 1,852 -> 1,858 us.)
//
// Hand-offs inside the CTA use mbarriers only (no named barriers): full/empty
// per stage, and per row slot (kSlots rows in flight) start / red_done /
// slot_free.  Every wait is bounded by a
// %globaltimer budget; on expiry the CTA sets STRIDE_DEV_TIMEOUT, stops
// issuing, waits (bounded) for the copies it has in flight, and returns.
#include <math.h>

#include <atomic>

#include "mbarrier.cuh"
#include "row_scan.cuh"
#include "stride.h"
#include "stride_device.cuh"
#include "stride_internal.h"
#include "warp_tile_scan.cuh"

// Ring shape: 3 stages of 32 KB per tensor (192 KB in flight per SM).  A
// sweep on GB300 over stages x chunk bytes at up to 218 KB of ring (the
// batch-scoring workload, two boxes, alternating runs) put 3 x 32 KB 0.4-
// 0.5 % ahead of 6 x 16 KB and 3 x 36 KB level with it; 2 x 48 KB, 4 x 27 KB,
// 5 x 20 KB and 8 x 12 KB were slower, 12 x 8 KB 14 % slower.
#ifndef STRIDE_BULK_STAGES
#define STRIDE_BULK_STAGES 3
#endif
#ifndef STRIDE_BULK_CHUNK
#define STRIDE_BULK_CHUNK 32768
#endif
#ifndef STRIDE_BULK_EVICT_FIRST
#define STRIDE_BULK_EVICT_FIRST 1
#endif

namespace stride {

constexpr int kStages = STRIDE_BULK_STAGES;   // ring depth
constexpr int kChunk = STRIDE_BULK_CHUNK;     // bytes per tensor per stage
constexpr int kSlots = 8;                     // rows in flight per CTA
constexpr int kConsumerWarps = 16;
constexpr int kConsumers = kConsumerWarps * 32;
constexpr int kRowWarps = 4;
constexpr int kScanWarp = 1 + kRowWarps;
constexpr int kFirstConsumerWarp = 2 + kRowWarps;
constexpr int kStreamThreads = 32 * kFirstConsumerWarp + kConsumers;
constexpr int kInfoEnd = -1;
constexpr int kInfoLast = 1 << 16;
// Bytes per tensor and CTA that the hints ahead of the wait ask for.  GB300,
// 3,001 rows of 151,936 bf16 logits, and 20,000 in windows of 4,096: none
// 262.3 and 1,689 us, 64 KB 261.5 and 1,686, 128 KB 262.6 and 1,684, 256 KB
// 264.3 and 1,683 (267.0 and 1,713 us before the 32-row tiles and before the
// state's initialisation was in the programmatic chain).
constexpr int64_t kStreamPrefetch = 64 << 10;
static_assert(kChunk % 16 == 0, "bulk copies move multiples of 16 bytes");
constexpr int kQueue = 8;  // published tiles waiting for the scan warp
static_assert(kSlots % kRowWarps == 0, "a row warp keeps its own slots");

struct alignas(128) StreamShared {
  uint64_t full[kStages];
  uint64_t empty[kStages];
  uint64_t start[kSlots];
  uint64_t red_done[kSlots];
  uint64_t slot_free[kSlots];
  int32_t stage_info[kStages];
  uint2 stage_vecs[kStages];  // 16-byte vectors of S and of T
  int64_t slot_tile[kSlots];  // window row, -1 past the last
  float4 red[kSlots][kConsumerWarps];  // the consumer warps' (mS, sS, mT, sT)
  uint64_t queue_full[kQueue];
  uint32_t queue_head;          // entries claimed by the row warps
  uint32_t queue_tail;          // entries completed by the scan warp
  uint32_t rows_done[kRowWarps];
  int32_t abort;
  TileCarry queue[kQueue];      // tile -1: a row warp has finished
  TileCarry own[kRowWarps];     // a row warp's tile that found the queue full
};

constexpr size_t kStreamHeader = (sizeof(StreamShared) + 127) & ~size_t(127);
constexpr size_t kStreamSmem = kStreamHeader + 2 * (size_t)kStages * kChunk;
static_assert(kStreamSmem <= 227 * 1024, "ring and header exceed the shared memory of one CTA");

__device__ __forceinline__ void raise_abort(StreamShared& sh, const BatchParams& p) {
  *reinterpret_cast<volatile int32_t*>(&sh.abort) = 1;
  set_status(p.dev_status, STRIDE_DEV_TIMEOUT);
}

// Claims the next entry of the queue to the scan warp, -1 if it is full.
__device__ __forceinline__ int queue_claim(StreamShared& sh) {
  uint32_t n = *reinterpret_cast<volatile uint32_t*>(&sh.queue_head);
  while (true) {
    if (n - *reinterpret_cast<volatile uint32_t*>(&sh.queue_tail) >= (uint32_t)kQueue) return -1;
    const uint32_t was = atomicCAS(&sh.queue_head, n, n + 1);
    if (was == n) break;
    n = was;
  }
  __threadfence_block();  // the entry's last reader has left it (it moved queue_tail after its last read)
  return (int)(n % kQueue);
}

// The logits of a row that bulk copies move: whole 16-byte vectors from the
// row's first 16-byte boundary on.  The up to P - 1 logits before (`head`)
// and after them are the row warp's.  EDGE = false: every row starts on a
// boundary.
template <typename LT, bool EDGE>
struct RowBody {
  int head;       // logits before the first vector
  uint32_t vecs;  // 16-byte vectors
  __device__ __forceinline__ RowBody(const LT* row, int V) : head(0) {
    constexpr int P = LogitTraits<LT>::kPerVec;
    if (EDGE) head = min((int)(((16u - (unsigned)(reinterpret_cast<uintptr_t>(row) & 15u)) & 15u) / sizeof(LT)), V);
    vecs = (uint32_t)((V - head) / P);
  }
  // Vectors of chunk c (every chunk but the last has `chunk` of them).
  __device__ __forceinline__ uint32_t chunk_vecs(uint32_t c, uint32_t chunk) const {
    const uint32_t off = c * chunk;
    return off < vecs ? min(chunk, vecs - off) : 0u;
  }
  // The row's logits outside its body, one per lane; false past the last.
  __device__ __forceinline__ bool edge(const LT* row, int V, int lane, float& x) const {
    constexpr int P = LogitTraits<LT>::kPerVec;
    const int j = (lane < head ? 0 : (int)vecs * P) + lane;
    const bool in = j < V;
    x = in ? to_f32(row[j]) : 0.f;
    return in;
  }
};

template <typename LT, bool EDGE>
__global__ void __launch_bounds__(kStreamThreads, 1) score_batch_stream_kernel(const BatchParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamShared& sh = *reinterpret_cast<StreamShared*>(smem_raw);
  unsigned char* bufS = smem_raw + kStreamHeader;
  unsigned char* bufT = bufS + (size_t)kStages * kChunk;
  volatile int32_t* abort = &sh.abort;

  constexpr int P = LogitTraits<LT>::kPerVec;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  // A row's chunks: as few as fit the stages, of equal size, so that its last
  // stage is as full as the others.  (V / P vectors is the most a row's body
  // can have; a row of less than a vector still passes one empty stage.)
  const uint32_t max_vecs = (uint32_t)(p.V / P);
  const uint32_t n_chunks = max((max_vecs * 16u + kChunk - 1) / kChunk, 1u);
  const uint32_t chunk = (max_vecs + n_chunks - 1) / n_chunks;  // vectors
  const uint64_t tmo = p.timeout_ns;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], kConsumerWarps);
    }
    for (int q = 0; q < kSlots; ++q) {
      mbar_init(&sh.start[q], 1);
      mbar_init(&sh.red_done[q], kConsumerWarps);
      mbar_init(&sh.slot_free[q], 1);
    }
    for (int i = 0; i < kQueue; ++i) mbar_init(&sh.queue_full[i], 1);
    for (int i = 0; i < kRowWarps; ++i) sh.rows_done[i] = 0;
    sh.queue_head = sh.queue_tail = 0;
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // Launched as a programmatic dependent of the workspace clear: the set-up
  // above, and the start of one of the first rows on its way to L2 (not the
  // teacher's from the multi-teacher row table, which is not there yet), may
  // overlap the previous kernels' end; nothing global is read or written
  // before the clear (and everything before it) has completed.  Dependents
  // may be scheduled at once: they wait for this grid in turn.
  if (tid == 32 || (tid == 64 && !p.T_rows)) {
    const LT* row = reinterpret_cast<const LT*>(tid == 32 ? p.S : p.T) + (int64_t)blockIdx.x * p.ld;
    prefetch_l2(row, min((int64_t)p.V * (int64_t)sizeof(LT), kStreamPrefetch));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint64_t policy;
#if STRIDE_BULK_EVICT_FIRST
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
#else
      asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
#endif
      uint32_t it = 0;  // stages issued
      int64_t seq = 0;  // rows started by this CTA
      bool ok = true;
      // (a shard pass has no workspace, hence no ticket: rows in turn)
      uint32_t t = p.partials ? blockIdx.x : atomicAdd(p.ticket, 1u);
      while ((int64_t)t < p.n_rows) {
        const int q = (int)(seq % kSlots);
        const uint32_t use = (uint32_t)(seq / kSlots);
        if (use > 0 && !mbar_wait(&sh.slot_free[q], (use - 1) & 1u, tmo, abort)) {
          ok = false;
          break;
        }
        sh.slot_tile[q] = (int64_t)t;
        mbar_arrive(&sh.start[q]);
        const LT* srow = reinterpret_cast<const LT*>(p.S) + (int64_t)t * p.ld;
        const LT* trow = teacher_row<LT>(p, (int64_t)t);
        const RowBody<LT, EDGE> body_s(srow, p.V), body_t(trow, p.V);
        const unsigned char* src_s = reinterpret_cast<const unsigned char*>(srow + body_s.head);
        const unsigned char* src_t = reinterpret_cast<const unsigned char*>(trow + body_t.head);
        for (uint32_t c = 0; c < n_chunks; ++c) {
          // the next row's ticket arrives while the last chunk waits for its stage
          if (c == n_chunks - 1) t = p.partials ? t + gridDim.x : atomicAdd(p.ticket, 1u);
          const int s = (int)(it % kStages);
          const uint32_t k = it / kStages;
          if (k > 0 && !mbar_wait(&sh.empty[s], (k - 1) & 1u, tmo, abort)) {
            ok = false;
            break;
          }
          const uint32_t n_s = body_s.chunk_vecs(c, chunk), n_t = body_t.chunk_vecs(c, chunk);
          const size_t off = (size_t)c * chunk * 16;
          sh.stage_info[s] = q | (c == n_chunks - 1 ? kInfoLast : 0);
          sh.stage_vecs[s] = make_uint2(n_s, n_t);
          mbar_arrive_expect_tx(&sh.full[s], (n_s + n_t) * 16u);
          if (n_s) bulk_g2s(bufS + (size_t)s * kChunk, src_s + off, n_s * 16u, &sh.full[s], policy);
          if (n_t) bulk_g2s(bufT + (size_t)s * kChunk, src_t + off, n_t * 16u, &sh.full[s], policy);
          ++it;
        }
        if (!ok) break;
        ++seq;
      }
      if (ok) {
        // end markers: for the consumers in the next stage, for the row
        // warps in their next slots
        const int s = (int)(it % kStages);
        const uint32_t k = it / kStages;
        if (k == 0 || mbar_wait(&sh.empty[s], (k - 1) & 1u, tmo, abort)) {
          sh.stage_info[s] = kInfoEnd;
          mbar_arrive(&sh.full[s]);
        } else {
          ok = false;
        }
        for (int i = 0; ok && i < kRowWarps; ++i, ++seq) {
          const int q = (int)(seq % kSlots);
          const uint32_t use = (uint32_t)(seq / kSlots);
          if (use > 0 && !mbar_wait(&sh.slot_free[q], (use - 1) & 1u, tmo, abort)) {
            ok = false;
            break;
          }
          sh.slot_tile[q] = -1;
          mbar_arrive(&sh.start[q]);
        }
      }
      if (!ok) {
        raise_abort(sh, p);
        // wait (bounded) for the last copies issued into each stage
        for (int s = 0; s < kStages; ++s) {
          const uint32_t uses = it / kStages + ((uint32_t)s < it % kStages ? 1u : 0u);
          if (uses > 0) {
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait(&sh.full[s], (uses - 1) & 1u) && globaltimer_ns() - t0 < tmo) {
            }
          }
        }
      }
    }
    return;
  }

  if (warp >= kFirstConsumerWarp) {
    // ----------------------------------------------------------- consumers
    const int cw = warp - kFirstConsumerWarp;
    const int ct = tid - 32 * kFirstConsumerWarp;
    uint32_t it = 0;
    float mS = kMaxStart, sS = 0.f, mT = kMaxStart, sT = 0.f;
    while (true) {
      const int s = (int)(it % kStages);
      const uint32_t k = it / kStages;
      if (!mbar_wait_warp(&sh.full[s], k & 1u, tmo, abort)) {
        raise_abort(sh, p);
        break;
      }
      const int info = sh.stage_info[s];
      if (info == kInfoEnd) break;
      const uint2 nv = sh.stage_vecs[s];
      const int n_s = (int)nv.x, n_t = EDGE ? (int)nv.y : n_s;  // (they differ by one vector at most, in the last chunk)
      const uint4* vs = reinterpret_cast<const uint4*>(bufS + (size_t)s * kChunk);
      const uint4* vt = reinterpret_cast<const uint4*>(bufT + (size_t)s * kChunk);
      int v = ct;
      for (; v + kConsumers < (EDGE ? min(n_s, n_t) : n_s); v += 2 * kConsumers) {
        const uint4 a[2] = {vs[v], vs[v + kConsumers]};
        const uint4 b[2] = {vt[v], vt[v + kConsumers]};
        LogitTraits<LT>::template chunk<2>(a, mS, sS);
        LogitTraits<LT>::template chunk<2>(b, mT, sT);
      }
      for (; v < (EDGE ? max(n_s, n_t) : n_s); v += kConsumers) {
        if (!EDGE || v < n_s) {
          const uint4 a[1] = {vs[v]};
          LogitTraits<LT>::template chunk<1>(a, mS, sS);
        }
        if (!EDGE || v < n_t) {
          const uint4 b[1] = {vt[v]};
          LogitTraits<LT>::template chunk<1>(b, mT, sT);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.empty[s]);
      ++it;
      if (info & kInfoLast) {
        // Row end: each warp posts its pair under the row's slot; the row
        // warp merges them once all 16 have arrived.  red[q] is reused only
        // after that warp has read it (slot_free).
        const int q = info & 0xffff;
        warp_merge2(mS, sS, mT, sT);
        if (lane == 0) {
          sh.red[q][cw] = make_float4(mS, sS, mT, sT);
          mbar_arrive(&sh.red_done[q]);
        }
        mS = kMaxStart;
        sS = 0.f;
        mT = kMaxStart;
        sT = 0.f;
      }
    }
    return;
  }

  if (warp == kScanWarp) {
    // ----------------------------------------------------------- scan warp
    if (!p.scan_inside) return;
    int running = kRowWarps;
    uint32_t seen = 0;
    for (uint32_t n = 0; running > 0;) {
      const int i = (int)(n % kQueue);
      if (!mbar_wait_warp(&sh.queue_full[i], (n / kQueue) & 1u, tmo, abort)) {
        // a long wait is an error only if no row was finished meanwhile
        uint32_t done = 0;
        for (int k = 0; k < kRowWarps; ++k) done += *reinterpret_cast<volatile uint32_t*>(&sh.rows_done[k]);
        done = __shfl_sync(0xffffffffu, done, 0);
        if (done != seen && !__any_sync(0xffffffffu, *abort)) {
          seen = done;
          continue;
        }
        if (lane == 0) raise_abort(sh, p);
        break;
      }
      if (sh.queue[i].tile < 0)
        --running;
      else
        complete_tile(p, sh.queue[i], lane);
      ++n;
      __syncwarp();
      __threadfence_block();
      if (lane == 0) *reinterpret_cast<volatile uint32_t*>(&sh.queue_tail) = n;
    }
    return;
  }

  // ---------------------------------------------------------------- row warps
  const float nan = __int_as_float(0x7fc00000);
  for (int64_t seq = warp - 1;; seq += kRowWarps) {
    const int q = (int)(seq % kSlots);
    const uint32_t use = (uint32_t)(seq / kSlots);
    if (!mbar_wait_warp(&sh.start[q], use & 1u, tmo, abort)) {
      if (lane == 0) raise_abort(sh, p);
      break;
    }
    const int64_t w = sh.slot_tile[q];  // window row
    if (w < 0) break;
    const LT* srow = reinterpret_cast<const LT*>(p.S) + w * p.ld;
    const LT* trow = teacher_row<LT>(p, w);
    const int64_t y = (int64_t)__ldg(p.tokens + w) - p.col0;
    const bool y_ok = y >= 0 && y < p.V;
    float xs = nan, xt = nan;
    if (y_ok) {
      xs = to_f32(srow[y]);
      xt = to_f32(trow[y]);
    }
    // the row's ragged ends: the logits before and after its whole vectors
    float es, et;
    const bool in_s = RowBody<LT, EDGE>(srow, p.V).edge(srow, p.V, lane, es);
    const bool in_t = RowBody<LT, EDGE>(trow, p.V).edge(trow, p.V, lane, et);
    if (!mbar_wait_warp(&sh.red_done[q], use & 1u, tmo, abort)) {
      if (lane == 0) raise_abort(sh, p);
      break;
    }
    float mS = kMaxStart, sS = 0.f, mT = kMaxStart, sT = 0.f;
    if (lane < kConsumerWarps) {
      const float4 v = sh.red[q][lane];
      mS = v.x;
      sS = v.y;
      mT = v.z;
      sT = v.w;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.slot_free[q]);  // the slot has been read
    if (in_s) lse_one(es, mS, sS);
    if (in_t) lse_one(et, mT, sT);
    warp_merge2(mS, sS, mT, sT);
    if (p.partials) {
      if (lane == 0) {
        float2* o = reinterpret_cast<float2*>(p.partials + w * 6);
        o[0] = make_float2(mS, sS);
        o[1] = make_float2(mT, sT);
        o[2] = make_float2(xs, xt);
      }
      continue;
    }
    uint32_t counted = 0;
    const int64_t t = w / kTileRows;
    if (lane == 0) {
      const float lse_s = lse_finish(mS, sS), lse_t = lse_finish(mT, sT);
      const float lps = xs - lse_s, lpt = xt - lse_t;
      if (!y_ok) set_status(p.dev_status, STRIDE_DEV_TOKEN_RANGE);
      const stride_row_outputs& o = p.out;
      if (o.logp_s) o.logp_s[w] = lps;
      if (o.logp_t) o.logp_t[w] = lpt;
      if (o.opd && p.scan_inside) o.opd[w] = lps - lpt;  // (the scan on log-probs writes it otherwise)
      if (o.lse_s) o.lse_s[w] = lse_s;
      if (o.lse_t) o.lse_t[w] = lse_t;
      if (o.x_s) o.x_s[w] = xs;
      if (o.x_t) o.x_t[w] = xt;
      p.ws_logp_s[w] = lps;
      p.ws_logp_t[w] = lpt;
      if (p.scan_inside) counted = count_in(p.flags + t * kFlagStride + kCounterWord) + 1;
    }
    if (!p.scan_inside) continue;
    counted = __shfl_sync(0xffffffffu, counted, 0);
    if ((int64_t)counted == min((int64_t)kTileRows, p.n_rows - t * kTileRows)) {
      int i = lane == 0 ? queue_claim(sh) : 0;
      i = __shfl_sync(0xffffffffu, i, 0);
      // lane 0 has acquired the tile's other rows (count_in) and the queue's
      // entry (queue_claim); a shuffle orders no memory, so this passes both on
      __syncwarp();
      TileCarry& tc = i < 0 ? sh.own[warp - 1] : sh.queue[i];
      publish_tile(p, t, lane, tc);
      __syncwarp();
      if (i < 0)
        complete_tile(p, tc, lane);
      else if (lane == 0)
        mbar_arrive(&sh.queue_full[i]);
      __syncwarp();
    }
    if (lane == 0) *reinterpret_cast<volatile uint32_t*>(&sh.rows_done[warp - 1]) = (uint32_t)(seq / kRowWarps) + 1;
  }
  // nothing more from this row warp (its rows are done: it may wait here)
  if (lane == 0 && p.scan_inside) {
    int i;
    const uint64_t t0 = globaltimer_ns();
    while ((i = queue_claim(sh)) < 0 && !*abort) {
      __nanosleep(200);
      if (globaltimer_ns() - t0 > tmo) raise_abort(sh, p);
    }
    if (i >= 0) {
      sh.queue[i].tile = -1;
      mbar_arrive(&sh.queue_full[i]);
    }
  }
}

// Whether the window's scan runs inside the kernel, behind the data, with a
// tail of its last tiles' lookups and lookback; or after it, 3 us later at the
// window's end but without the row warps' counting and publishing, which short
// rows wait for.  GB300, us inside / after: 3,000 rows of 32,000 bf16 logits
// 85.7 / 70.0, of 48,000 101.8 / 95.2, of 64,000 118.3 / 120.9, of 151,936
// 257.8 / 261.2; of 32,000 fp32 127.3 / 119.2, of 48,000 168.8 / 169.4; 30,011
// rows of 32,000 bf16 546 / 522.
constexpr int kScanInsideLogits = 56 << 10;

bool stream_scan_inside(int V) { return V >= kScanInsideLogits; }

size_t stream_clear_bytes(int64_t n_rows, int V) {
  if (!stream_scan_inside(V)) return 256;
  return 256 + (size_t)((n_rows + kTileRows - 1) / kTileRows) * kFlagStride * sizeof(uint32_t);
}

cudaError_t launch_score_batch_stream(const BatchParams& p, int dtype, bool aligned, cudaStream_t stream) {
  // The dynamic shared-memory limit is a per-device function attribute: set
  // once per device and kernel (setting it again is harmless, so two threads
  // racing here both succeed).
  static std::atomic<bool> attr_done[64][4];
  int dev = 0;
  cudaError_t e = cudaSuccess;
  const int sms = current_device_sms(&dev, &e);
  if (sms <= 0) return e != cudaSuccess ? e : cudaErrorInvalidDevice;
  const bool bf16 = dtype == STRIDE_DTYPE_BF16;
  auto kern = bf16 ? (aligned ? score_batch_stream_kernel<__nv_bfloat16, false> : score_batch_stream_kernel<__nv_bfloat16, true>)
                   : (aligned ? score_batch_stream_kernel<float, false> : score_batch_stream_kernel<float, true>);
  std::atomic<bool>& done = attr_done[dev][(bf16 ? 0 : 2) + (aligned ? 0 : 1)];
  if (!done.load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmem);
    if (e != cudaSuccess) return e;
    done.store(true, std::memory_order_release);
  }
  const int64_t grid = p.n_rows < sms ? p.n_rows : sms;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kStreamThreads);
  cfg.dynamicSmemBytes = kStreamSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace stride
