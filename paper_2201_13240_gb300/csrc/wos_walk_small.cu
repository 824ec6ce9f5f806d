// wos_walk_small.cu -- the sums of small FP32 solves, whose walk kernels run one walk per lane.
#include "wos_walk_impl.cuh"

namespace wos {

struct SumRun {
  uint32_t p, n;        // point, walks
  float sh, d1, d2;     // the first walk's value, and the sums of differences from it and of their squares
};

// Per-point sums of a small solve from its walks' totals (item_acc, in item order).
//
// What bounds it: nothing much (12 bytes per walk, ~25 rounds of a warp per 128 walks); it exists
// so that the walks of a small solve can run one per lane on the whole chip.  The persistent
// kernel gives a warp 128 walks, four per lane one after another, so a 2^18-walk solve used
// 2048 warps of the ~3000 that fit and lasted four walks and the longest one's tail.  Measured:
// 3,000 points x 64 walks on a mesh 476 -> 266 ms, 32^2 x 256 of the 2D square 494 -> 461 us.
//
// The sums are FP32 partial sums per lane, shifted by the lane's first walk of the point, over the walks
// that lane would have run had one warp taken 128 consecutive walks, each lane that is free claiming
// the next one (lanes free at the same iteration in lane order, GATHERED: once four lanes are free).
// So they do not depend on which warp ran which walk, and they are the sums that small solves had
// when the walk kernels formed them.  Larger solves add in other orders, and kernels compiled for 2D or
// B-spline problems, and batches of such, in FP64 (sums_in_fp64): on the two sides of kSpreadItems walks
// those problems' sums differ by the rounding of FP32 partial sums.
template <bool GATHERED>
__global__ void __launch_bounds__(128) walk_sum_kernel(const float* __restrict__ acc, const uint32_t* __restrict__ iters,
                                                       const uint32_t* __restrict__ point,
                                                       const float* __restrict__ scale, uint64_t all,
                                                       const int64_t* walk_end, int64_t npts, double* sum,
                                                       double* sumsq, unsigned long long* count) {
  if (walk_end != nullptr) all = (uint64_t)__ldg(&walk_end[npts - 1]);  // per-point walk counts
  if (all > kSpreadItems) return;  // the walk kernel, or the other of two launches, added these up itself
  const uint32_t total = (uint32_t)all;
  const uint32_t lane = threadIdx.x & 31, base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kChunkMin;
  if (base >= total) return;
  const uint32_t n = min((uint32_t)kChunkMin, total - base);
  // The warp's walks, staged: a claim takes consecutive ones, so its loads have no bank conflicts (from
  // registers by eight shuffles and selects, with the point a global load in every round, 2^20 walks took
  // 28 us, so 22).
  __shared__ float walk_acc[4][kChunkMin];
  __shared__ uint32_t walk_iters[4][kChunkMin], walk_point[4][kChunkMin];
  const uint32_t warp = threadIdx.x >> 5;
  for (uint32_t i = lane; i < n; i += 32) {
    walk_acc[warp][i] = acc[base + i];
    walk_iters[warp][i] = iters[base + i];
    walk_point[warp][i] = point[base + i];
  }
  __syncwarp();
  // A lane's sums over consecutive walks of one point are a run; runs wait in shared memory until the
  // walks are through, so that their FP64 arithmetic is done by all lanes at once, and runs of one
  // point meet in one atomic (flushed as they end, by a lane or two: 2.6e5 points x 4 walks of the 3D
  // cube 808 us, so 680; 30 points x 8192 walks 386 us, so 299).
  __shared__ SumRun runs[4][kChunkMin];
  SumRun* run = runs[warp];
  uint32_t n_runs = 0;  // of the warp
  SumRun r = {0xffffffffu, 0u, 0.0f, 0.0f, 0.0f};
  auto add = [&](bool on, uint32_t i) {
    const uint32_t q = on ? walk_point[warp][i] : r.p;
    const bool ends = on && r.n != 0u && q != r.p;
    const unsigned done = __ballot_sync(kFull, ends);
    if (ends) run[n_runs + __popc(done & ((1u << lane) - 1u))] = r;
    n_runs += __popc(done);
    if (!on) return;
    const float v = walk_acc[warp][i];
    if (q != r.p) r = SumRun{q, 0u, v, 0.0f, 0.0f};
    const float dv = v - r.sh;
    r.d1 += dv;
    r.d2 += dv * dv;
    ++r.n;
  };
  add(lane < n, lane);
  uint32_t free_at = (lane < n) ? walk_iters[warp][lane] : 0u;  // iteration at which the lane has no walk
  for (uint32_t next = 32; next < n;) {
    // the iteration of the next claim
    uint32_t t = __reduce_min_sync(kFull, free_at);
    if (GATHERED) {
      uint32_t rest = free_at;
      for (int got = __popc(__ballot_sync(kFull, rest == t)); got < 4;) {
        if (rest == t) rest = 0xffffffffu;
        t = __reduce_min_sync(kFull, rest);
        got += __popc(__ballot_sync(kFull, rest == t));
      }
    }
    const unsigned claim = __ballot_sync(kFull, free_at <= t);
    const uint32_t j = next + __popc(claim & ((1u << lane) - 1u));
    const bool takes = (claim >> lane & 1u) && j < n;
    add(takes, j);
    if (takes) free_at = t + walk_iters[warp][j];
    next += __popc(claim);
  }
  const unsigned last = __ballot_sync(kFull, r.n != 0u);
  if (r.n != 0u) run[n_runs + __popc(last & ((1u << lane) - 1u))] = r;
  n_runs += __popc(last);
  __syncwarp();
  for (uint32_t at = 0; at < n_runs; at += 32) {
    const bool on = at + lane < n_runs;
    double s1 = 0.0, s2 = 0.0;
    uint32_t m = 0, p = run[at].p;
    if (on) {
      const SumRun q = run[at + lane];
      const double e0 = (double)scale[q.p], c = (double)q.sh, w = (double)q.n;
      s1 = w * c + (double)q.d1;
      s2 = w * c * c + 2.0 * c * (double)q.d1 + (double)q.d2;
      s1 = s1 * e0;
      s2 = s2 * e0 * e0;
      m = q.n;
      p = q.p;
    }
    // many walks per point: the warp's runs are of one point as a rule, and meet in one atomic each
    const bool one = __all_sync(kFull, p == __shfl_sync(kFull, p, 0));
    if (one) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        s1 += __shfl_down_sync(kFull, s1, off);
        s2 += __shfl_down_sync(kFull, s2, off);
        m += __shfl_down_sync(kFull, m, off);
      }
    }
    if (one ? lane == 0 : on) {
      atomicAdd(&sum[p], s1);
      atomicAdd(&sumsq[p], s2);
      atomicAdd(&count[p], (unsigned long long)m);
    }
  }
}

cudaError_t launch_walk_sums(const WalkLaunch& L, bool gathered, cudaStream_t stream) {
  const uint64_t most = (L.total_items < kSpreadItems) ? L.total_items : kSpreadItems;
  const uint64_t blocks = (most + 4 * kChunkMin - 1) / (4 * kChunkMin);
  auto* kernel = gathered ? walk_sum_kernel<true> : walk_sum_kernel<false>;
  kernel<<<(unsigned)blocks, 128, 0, stream>>>(L.item_acc, L.item_iters, L.item_point, L.point_scale, L.total_items,
                                               L.walk_end, L.npts, L.sum, L.sumsq, L.count);
  return cudaGetLastError();
}

}  // namespace wos
