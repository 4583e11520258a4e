// score_step.cu -- one decode step over the live rollouts of a batch (sm_103a).
//
// Algorithm 1's inner loop scores one generated token per rollout per step.
// A step holds only a few hundred rows, too few for one CTA per row to fill
// 152 SMs, so each row is split over the C CTAs of one thread-block cluster:
// every CTA streams a slice of the vocabulary of both the student and the
// teacher row into online log-sum-exp pairs, the pairs meet in rank 0 through
// distributed shared memory, and rank 0 forms the token's log-probs and
// advances the rollout's carried state (open-turn sums, turn close with
// Eq. 4, stop test of Eq. 5 or Sec. 5.5).  No workspace, no atomics, no
// spin-waits: the cluster barrier is hardware.
//
// Two row layouts share the kernel:
//  * masked (stride_score_step): row b is rollout b of the batch; a rollout
//    whose state says stopped exits before reading a byte;
//  * compacted (stride_score_step_compact): the caller packs the live
//    rollouts' rows, row b is rollout rollout_idx[b], whose state and lambda
//    are read through that index.  As rollouts stop the step shrinks, and the
//    cluster size grows with it, so a small step still fills the GPU.
//
// Launch shape.  CTAs of 128 threads (8 per SM) or 512 threads (2 per SM),
// both at most 64 registers per thread; the cluster size C and the CTA size
// come from the step's row count (choose_shape below): as many CTAs per row
// as still run at once.
//
// Steps are launched with programmatic dependent launch.  A CTA lets the next
// kernel be scheduled once its own stream is done, so the next step's CTAs
// come in as this step's leave; each asks for the start of its slice in L2
// (a hint, which reads nothing) and then waits (griddepcontrol.wait) for this
// kernel's completion before its first global read, so the caller's inputs
// and the carried state are always complete when read.  The loads' ramp thus
// overlaps the previous step's merges and state updates.  GB300, steps of a
// 32-step graph (151,936 bf16 logits), one box, before the overlap -> now, with
// the launch shapes of choose_shape, the loop's last batch in one and the
// merges of stride_device.cuh: 1 row 3.66 -> 3.14 us, 8 rows 5.52 -> 4.48, 24
// rows 7.36 -> 6.4, 61 rows 10.8 -> 8.9, 128 rows 16.2 -> 13.7, 256 rows 27.1 ->
// 24.9; of 32,000 logits 2.95 -> 2.57, 3.72 -> 3.64, 4.55 -> 4.3, 5.98 -> 4.74,
// 8.2 -> 5.65, 10.6 -> 8.1.  The overlap alone took 61 rows from 11.0 to 9.8 and
// 256 from 27.0 to 25.8 on another box; letting the next step in at the start instead makes its hints
// compete with this step's loads (61 rows 9.8 -> 10.4), and in mid-stream costs
// a split of the loop (11.9).
#include <cooperative_groups.h>
#include <math.h>

#include <atomic>

#include "stride.h"
#include "stride_device.cuh"
#include "stride_internal.h"

namespace cg = cooperative_groups;

namespace stride {

#ifndef STRIDE_STEP_UNROLL
#define STRIDE_STEP_UNROLL 4
#endif

constexpr int kStepUnroll = STRIDE_STEP_UNROLL;
constexpr int kStepMaxCluster = 16;
constexpr int kStepSmallCluster = 14;  // of 128-thread CTAs: clusters of 16 were slower at every row count
// Bytes of a step that the hints ahead of the wait ask for, over all its
// CTAs.  12 / 20 / 28 / 40 MB, us per step: 61 rows 9.4 / 9.3 / 9.2 / 9.4, 76
// rows 11.2 / 10.6 / 10.3 / 10.4, 128 rows 14.2 / 14.0 / 13.9 / 14.4, 256 rows
// 25.0 / 24.9 / 24.9 / 25.0: more than the wait lasts only evicts.
constexpr int64_t kStepPrefetch = 28 << 20;
// Two CTA shapes, both at most 64 registers per thread: 128 threads, 8 CTAs
// per SM (the shape of steps with many rows), and 512 threads, 2 per SM (more
// threads per row when a step has too few rows to fill the GPU with
// 128-thread CTAs even in the largest clusters).
constexpr int kStepThreadsSmall = 128;
constexpr int kStepThreadsLarge = 512;
template <int THREADS>
struct StepShape {
  static constexpr int kWarps = THREADS / 32;
  static constexpr int kMinBlocks = 1024 / THREADS;  // 64 registers per thread
};

namespace {

__device__ __forceinline__ void write_row_nan(const StepParams& p, int b) {
  const float nan = __int_as_float(0x7fc00000);
  const stride_row_outputs& o = p.out;
  if (o.logp_s) o.logp_s[b] = nan;
  if (o.logp_t) o.logp_t[b] = nan;
  if (o.opd) o.opd[b] = nan;
  if (o.lse_s) o.lse_s[b] = nan;
  if (o.lse_t) o.lse_t[b] = nan;
  if (o.x_s) o.x_s[b] = nan;
  if (o.x_t) o.x_t[b] = nan;
  if (p.stopped_now) p.stopped_now[b] = 0;
  if (p.turn_out) p.turn_out[b] = stride_turn_stats{0.0, 0.0, 0.0, 0.0, 0.f, 0};
}

}  // namespace

// The 80-byte state as ten 8-byte L2 loads (no L1: the previous step's
// cluster wrote it on another SM), issued together.
__device__ __forceinline__ stride_scan_state load_state(const stride_scan_state* sp) {
  static_assert(sizeof(stride_scan_state) == 80, "state layout");
  union {
    stride_scan_state s;
    unsigned long long w[10];
  } u;
  const unsigned long long* src = reinterpret_cast<const unsigned long long*>(sp);
#pragma unroll
  for (int i = 0; i < 10; ++i) u.w[i] = __ldcg(src + i);
  return u.s;
}

template <typename LT, bool VEC, bool COMPACT, int THREADS>
__global__ void __launch_bounds__(THREADS, StepShape<THREADS>::kMinBlocks) score_step_kernel(const StepParams p) {
  constexpr int kStepWarps = StepShape<THREADS>::kWarps;
  __shared__ float s_red[4][kStepWarps];
  __shared__ float4 s_part[kStepMaxCluster];  // rank 0: every rank's (mS, sS, mT, sT), written by the ranks
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int b = (int)(blockIdx.x / (unsigned)C);  // row of this step
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  // first barrier phase: arriving here and waiting before the first remote
  // store guarantees every CTA of the cluster has started (its shared memory
  // exists); the wait comes after the stream, so it costs nothing
  cluster_arrive_relaxed();

  const LT* srow = reinterpret_cast<const LT*>(p.S) + (int64_t)b * p.ld;
  const LT* trow = reinterpret_cast<const LT*>(p.T) + (int64_t)b * p.ld;

  // vocabulary slice of this rank (whole 16-byte vectors on the vector path;
  // the last rank also takes the ragged tail)
  int c0, c1;
  if (VEC) {
    constexpr int P = LogitTraits<LT>::kPerVec;
    const int nv = p.V / P;
    const int per = (nv + C - 1) / C;
    c0 = min(nv, rank * per) * P;
    c1 = (rank == C - 1) ? p.V : min(nv, (rank + 1) * per) * P;
  } else {
    const int per = (p.V + C - 1) / C;
    c0 = min(p.V, rank * per);
    c1 = min(p.V, (rank + 1) * per);
  }

  // The start of the slice on its way to L2 while the previous kernel ends
  // (the stopped flag may be about to change: it only saves a useless hint).
  if (tid == 0 || tid == 32) {
    const bool skip = !COMPACT && *reinterpret_cast<const volatile int32_t*>(&p.state[b].stopped) != 0;
    const int64_t most = kStepPrefetch / (2 * (int64_t)gridDim.x);
    if (!skip) prefetch_l2((tid == 0 ? srow : trow) + c0, min((int64_t)(c1 - c0) * (int64_t)sizeof(LT), most));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (!COMPACT) {
    // A stopped rollout's whole cluster leaves before reading a logit (every
    // CTA reads the flag, which only this step's rank 0 writes, after the
    // cluster's last remote store).
    if (__ldcg(&p.state[b].stopped)) {
      if (rank == 0 && tid == 0) write_row_nan(p, b);
      return;
    }
  }

  // The token id (and, compacted, the rollout id) is loaded now, the token's
  // logits and the rollout's state after the stream, so rank 0 streams as
  // early as the other ranks (a gather before the stream held rank 0 back by
  // about 0.7 us on average, GB300 timeline) and the state's latency hides
  // behind the merge and the cluster barrier.  A compacted row streams
  // without first reading its rollout's state: the caller passes live
  // rollouts, and a row whose state turns out stopped is discarded.
  int32_t y = 0, r = b;
  if (rank == 0 && tid == 0) {
    y = __ldg(p.tokens + b);
    if (COMPACT) r = __ldg(p.rollout_idx + b);
  }

  float mS = kMaxStart, sS = 0.f, mT = kMaxStart, sT = 0.f;
  stream_pair<LT, VEC, kStepUnroll>(srow, trow, c0, c1, tid, THREADS, mS, sS, mT, sT);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  float xs = __int_as_float(0x7fc00000), xt = xs, lam = 0.f;
  bool valid = false, closes = false;
  stride_scan_state st;
  if (rank == 0 && tid == 0) {
    if (y >= 0 && y < p.V) {
      xs = to_f32(srow[y]);
      xt = to_f32(trow[y]);
    }
    valid = !COMPACT || (r >= 0 && r < p.n_state);
    if (valid) {
      st = load_state(p.state + r);
      lam = p.lambda ? __ldg(p.lambda + r) : p.lambda_all;
      closes = __ldg(p.turn_end + b) != 0;
    }
  }
  warp_merge2(mS, sS, mT, sT);
  if (lane == 0) {
    s_red[0][warp] = mS;
    s_red[1][warp] = sS;
    s_red[2][warp] = mT;
    s_red[3][warp] = sT;
  }
  __syncthreads();
  cluster_wait_acquire();  // (first phase) every CTA of the cluster has started
  if (warp == 0) {
    mS = lane < kStepWarps ? s_red[0][lane] : kMaxStart;
    sS = lane < kStepWarps ? s_red[1][lane] : 0.f;
    mT = lane < kStepWarps ? s_red[2][lane] : kMaxStart;
    sT = lane < kStepWarps ? s_red[3][lane] : 0.f;
    warp_merge2<kStepWarps>(mS, sS, mT, sT);
    if (lane == 0) {
      float4* dst = cluster.map_shared_rank(s_part, 0);
      dst[rank] = make_float4(mS, sS, mT, sT);
    }
  }
  // second phase: the ranks' stores are released to rank 0, the other
  // ranks leave (nobody reads their shared memory)
  cluster_arrive_release();
  if (rank != 0) return;
  cluster_wait_acquire();

  if (warp == 0) {
    mS = kMaxStart;
    sS = 0.f;
    mT = kMaxStart;
    sT = 0.f;
    if (lane < C) {
      const float4 q = s_part[lane];
      mS = q.x;
      sS = q.y;
      mT = q.z;
      sT = q.w;
    }
    warp_merge2<kStepMaxCluster>(mS, sS, mT, sT);
    if (lane == 0) {
      if (!valid) {
        set_status(p.dev_status, STRIDE_DEV_BAD_LAYOUT);
        write_row_nan(p, b);
      } else if (COMPACT && st.stopped) {
        write_row_nan(p, b);
      } else {
        const float lse_s = lse_finish(mS, sS);
        const float lse_t = lse_finish(mT, sT);
        const float lps = xs - lse_s;
        const float lpt = xt - lse_t;
        const float dd = lps - lpt;
        if (!(y >= 0 && y < p.V)) set_status(p.dev_status, STRIDE_DEV_TOKEN_RANGE);
        const stride_row_outputs& o = p.out;
        if (o.logp_s) o.logp_s[b] = lps;
        if (o.logp_t) o.logp_t[b] = lpt;
        if (o.opd) o.opd[b] = dd;
        if (o.lse_s) o.lse_s[b] = lse_s;
        if (o.lse_t) o.lse_t[b] = lse_t;
        if (o.x_s) o.x_s[b] = xs;
        if (o.x_t) o.x_t[b] = xt;

        // carried state (Algorithm 1 inner loop)
        const double term = (double)lps * (double)dd;  // -log pi_S * r_t (Eq. 2); every scored token is retained
        st.turn_sum_t += (double)lpt;
        st.turn_sum_d += (double)dd;
        st.turn_sum_l += term;
        st.loss += term;
        st.loss_tokens += 1;
        st.turn_tokens += 1;
        const int64_t pos = st.rows_seen;
        st.rows_seen += 1;
        uint8_t fired = 0;
        if (p.mode == STRIDE_STOP_TOKEN_SUM) {
          st.cum += (double)lpt;
          if (st.cum < (double)lam) fired = 1;
        }
        stride_turn_stats ts{0.0, 0.0, 0.0, 0.0, 0.f, 0};
        if (closes) {
          const double mean = st.turn_sum_t / (double)st.turn_tokens;  // Eq. 4
          if (p.mode == STRIDE_STOP_TURN_MEAN) {
            st.cum += mean;  // Eq. 5
            if (st.cum < (double)lam) fired = 1;
          }
          ts.sum_t = st.turn_sum_t;
          ts.sum_d = st.turn_sum_d;
          ts.sum_l = st.turn_sum_l;
          ts.cum = st.cum;
          ts.mean_t = (float)mean;
          ts.n = st.turn_tokens;
          st.turn_idx += 1;
          st.turn_tokens = 0;
          st.turn_sum_t = 0.0;
          st.turn_sum_d = 0.0;
          st.turn_sum_l = 0.0;
        }
        if (fired) {
          st.stopped = 1;
          st.stop_row = pos;
          // the turn the firing token belongs to (closed or still open)
          st.stop_turn = closes ? st.turn_idx - 1 : st.turn_idx;
        }
        p.state[r] = st;
        if (p.stopped_now) p.stopped_now[b] = fired;
        if (p.turn_out) p.turn_out[b] = ts;
      }
    }
  }
}

namespace {

// Forced launch shape (0 = automatic), set by stride_force_step_shape.
std::atomic<int> g_force_threads{0};
std::atomic<int> g_force_cluster{0};

constexpr int kMaxDev = 64;

// Cluster sizes above 8 need the non-portable attribute, set once per device
// for each kernel (one set of statics per template instance).
template <typename LT, bool VEC, bool COMPACT, int THREADS>
cudaError_t allow_large_clusters(int dev) {
  static std::atomic<int> done[kMaxDev];
  if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(score_step_kernel<LT, VEC, COMPACT, THREADS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) done[dev].store(1, std::memory_order_release);
  return e;
}

// How many clusters of C CTAs of THREADS threads the device holds at once
// (GB300's GPCs hold whole clusters: 14 of 16 CTAs of 512 threads, 72 of 4),
// looked up once per device and size.
template <int THREADS>
int resident_clusters(int dev, int C) {
  static std::atomic<int> known[kMaxDev][kStepMaxCluster + 1];  // count + 1, 0 = not looked up yet
  int n = known[dev][C].load(std::memory_order_relaxed);
  if (n > 0) return n - 1;
  auto kern = score_step_kernel<__nv_bfloat16, true, true, THREADS>;  // (the others have the same bounds)
  int clusters = 0;
  if (C <= 8 || allow_large_clusters<__nv_bfloat16, true, true, THREADS>(dev) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(THREADS);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();  // a refused size is an answer, not an error to carry
      clusters = 0;
    }
  }
  known[dev][C].store(clusters + 1, std::memory_order_relaxed);
  return clusters;
}

// The most CTAs of THREADS threads per row that still run at once, with the
// share of the device's CTAs (percent) that clusters of their size can use
// before some row waits for another's to end: what the sweeps below found.
template <int THREADS>
int one_wave_cluster(int dev, int sms, int64_t rows) {
  const bool large = THREADS == kStepThreadsLarge;
  const int64_t slots = (int64_t)StepShape<THREADS>::kMinBlocks * sms;
  for (int C = large ? kStepMaxCluster : kStepSmallCluster; C > 1; --C) {
    const int share = large ? (C >= 7 ? 82 : C >= 5 ? 87 : C == 4 ? 95 : C == 3 ? 83 : 100) : (C > 10 ? 83 : 90);
    if (rows * C * 100 <= share * slots && rows <= resident_clusters<THREADS>(dev, C)) return C;
  }
  return 1;
}

// Launch shape of a step with `rows` rows: as many CTAs per row as still run
// at once, of 512 threads or of 128.  One cluster too many makes the step
// wait for a second wave: 24 rows in clusters of 9 / 10 / 11 CTAs of 512
// threads 6.3 / 6.8 / 8.1 us, 108 rows in 10 / 11 of 128 threads 12.4 / 15.7.
// GB300, us per step of graphs over 151,936 bf16 logits, each size in its
// best cluster:
//   rows         8   16   22   28   36   44   52   56   60   68   76   92  108  124  144  152  168
//   512 threads 4.7  5.4  5.8  6.4  7.0  7.7  8.2  9.4  9.4  9.4 10.9 12.9 13.8 14.1 15.1 15.5 23.3
//   128 threads 5.4  6.0  6.4  6.7  7.2  8.2  8.8  9.1  9.3  9.6 10.5 11.6 12.4 14.0 16.2 16.6 18.0
// so 512 threads from 5 CTAs a row on, and below that where 4 or 2 CTAs a row
// all but fill the device -- not in the masked form, whose stopped rows leave
// their CTAs idle (62 rows 9.4 / 8.7, 136 rows 13.6 / 13.0).
//
// The shares and fills are those rows' own.  Other rows follow them, against the
// best of 23 fixed shapes (12 row counts from 1 to 256; percent slower, 32,000
// bf16 / 32,000 fp32 / 151,936 fp32): 24 rows 7 / 13 / 12, 61 rows 5 / 9 / 1, 76
// rows 16 / 18 / 5, 108 rows 30 / 21 / 10, 256 rows 5 / 2 / 7, the others within
// 3 (1 row of 32,000 bf16: 5); faster everywhere than the fixed shapes before.
struct Shape {
  int threads, cluster;
};

Shape choose_shape(int64_t rows, bool compact, int dev, int sms) {
  const int ft = g_force_threads.load(std::memory_order_relaxed);
  const int fc = g_force_cluster.load(std::memory_order_relaxed);
  if (ft > 0 || fc > 0) return Shape{ft > 0 ? ft : kStepThreadsSmall, fc > 0 ? fc : 1};
  const int large = one_wave_cluster<kStepThreadsLarge>(dev, sms, rows);
  const int64_t fill = rows * large * 100 / (StepShape<kStepThreadsLarge>::kMinBlocks * (int64_t)sms);
  if (large > 4 || (compact && ((large == 4 && fill >= 83) || (large == 2 && fill >= 90))))
    return Shape{kStepThreadsLarge, large};
  return Shape{kStepThreadsSmall, one_wave_cluster<kStepThreadsSmall>(dev, sms, rows)};
}

template <typename LT, bool VEC, bool COMPACT, int THREADS>
cudaError_t launch_step_pdl(const StepParams& p, int C, int dev, cudaStream_t stream) {
  if (C > 8) {
    const cudaError_t e = allow_large_clusters<LT, VEC, COMPACT, THREADS>(dev);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.B * (unsigned)C);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, score_step_kernel<LT, VEC, COMPACT, THREADS>, p);
}

template <bool COMPACT, int THREADS>
cudaError_t launch_step_form(const StepParams& p, int dtype, bool vec, int C, int dev, cudaStream_t stream) {
  if (dtype == STRIDE_DTYPE_BF16)
    return vec ? launch_step_pdl<__nv_bfloat16, true, COMPACT, THREADS>(p, C, dev, stream)
               : launch_step_pdl<__nv_bfloat16, false, COMPACT, THREADS>(p, C, dev, stream);
  return vec ? launch_step_pdl<float, true, COMPACT, THREADS>(p, C, dev, stream)
             : launch_step_pdl<float, false, COMPACT, THREADS>(p, C, dev, stream);
}

}  // namespace

int set_step_shape_override(int threads, int C) {
  if (C < 0 || C > kStepMaxCluster) return -1;
  if (threads != 0 && threads != kStepThreadsSmall && threads != kStepThreadsLarge) return -1;
  g_force_threads.store(threads, std::memory_order_relaxed);
  g_force_cluster.store(C, std::memory_order_relaxed);
  return 0;
}

cudaError_t launch_score_step(const StepParams& p, int dtype, bool vec, cudaStream_t stream) {
  int dev = 0;
  cudaError_t e = cudaSuccess;
  const int sms = current_device_sms(&dev, &e);
  if (sms <= 0) return e != cudaSuccess ? e : cudaErrorInvalidDevice;
  Shape sh = choose_shape(p.B, p.rollout_idx != nullptr, dev, sms);
  // a few whole vectors per thread of a rank at least
  while (sh.cluster > 1 && (int64_t)p.V < (int64_t)sh.threads * sh.cluster) sh.cluster >>= 1;
  if (sh.threads == kStepThreadsLarge && (int64_t)p.V < (int64_t)kStepThreadsLarge * 2) sh.threads = kStepThreadsSmall;
  const bool compact = p.rollout_idx != nullptr;
  if (sh.threads == kStepThreadsLarge)
    e = compact ? launch_step_form<true, kStepThreadsLarge>(p, dtype, vec, sh.cluster, dev, stream)
                : launch_step_form<false, kStepThreadsLarge>(p, dtype, vec, sh.cluster, dev, stream);
  else
    e = compact ? launch_step_form<true, kStepThreadsSmall>(p, dtype, vec, sh.cluster, dev, stream)
                : launch_step_form<false, kStepThreadsSmall>(p, dtype, vec, sh.cluster, dev, stream);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace stride
