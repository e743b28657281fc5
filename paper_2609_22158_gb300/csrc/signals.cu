// Step signals from evidence cues (Sec. 4.1 "New-step Scoring" and "Previous-step Updating"): each step's
// Thought, Action and Observation fields are represented by up to 64 evidence cues (sorted, distinct
// 32-bit ids), and sim(a, b) is the overlap similarity of two cue sets, |A n B| / |A u B| (0 when both
// are empty).  For every target step k in [k0, n_steps):
//   gain_k = 1 - max_{u<k} sim(Th_k || Obs_k, Th_u || Obs_u)   (gain = 1 for the first step)
//   red_k  = max_{u<k} sim(Act_k, Act_u)                        (red = 0 for the first step)
// where a concatenation of fields is the union of their cues; and for the newest step t = n_steps - 1
//   obs_sim[k] = sim(Obs_t, Obs_k), k < t                      (Eq. 3's input; obs_sim[t] = 0).
//
// The work is O(t x 128) set-membership tests per target step, a few microseconds of one SM late in an episode.  A
// CTA takes a target step (one more takes obs_sim) with a warp per earlier step, up to 32; a call with few
// targets and many earlier steps spreads each over a cluster of 8 CTAs.  The target's lists sit in shared memory, padded
// to a power of two and Thought and Observation merged into one; a warp holds its earlier step's lists in registers
// (two cues of each field per lane, the next step's already on their way), so a test is seven shared-memory probes of
// three instructions and all of a lane's are in flight together.  Maxima do not depend on the order (deterministic).
// 120 steps, the newest as target: 7.5 us (eight warps of one CTA searching in global memory: 77.4; one CTA and
// unpadded, unmerged lists: 20.6); 400 steps, all of them targets: 348 -> 76 us.  A count outside
// [0, 64] or a cue list that is not strictly increasing sets STEPKV_EDATA and the values that depend on it are not
// written.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace stepkv {

constexpr int kSigCluster = 8;
constexpr int kSigMaxWarps = 32;

struct SignalArgs {
  const uint32_t* cues;  // [n_steps][3][STEPKV_MAX_CUES]
  const int32_t* n_cues; // [n_steps][3]
  int n_steps;
  int k0;
  float* gain;           // [n_steps] (entries k >= k0 written) or NULL
  float* red;
  float* obs_sim;        // [n_steps] or NULL
  int32_t* status;
};

// One step's cue lists over a warp: lane i holds cues 2 i and 2 i + 1 of each field (any value past the count).
struct StepCues {
  uint2 x[3];
  int n[3];
};
__device__ __forceinline__ void load_step(const SignalArgs& a, int k, int lane, StepCues& s) {
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    // 4-byte loads: the caller's lists are only word-aligned
    const uint32_t* p = a.cues + ((size_t)k * 3 + f) * STEPKV_MAX_CUES + 2 * lane;
    s.x[f] = make_uint2(__ldg(p), __ldg(p + 1));
    s.n[f] = __ldg(&a.n_cues[k * 3 + f]);
  }
}
// Every count in [0, 64] and every list strictly increasing (sorted, distinct); counts clamped.
__device__ __forceinline__ bool check_step(StepCues& s, int lane) {
  bool ok = true;
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    ok &= s.n[f] >= 0 && s.n[f] <= STEPKV_MAX_CUES;
    s.n[f] = min(max(s.n[f], 0), STEPKV_MAX_CUES);
    const uint32_t before = __shfl_up_sync(0xffffffffu, s.x[f].y, 1);
    if (lane > 0 && 2 * lane < s.n[f]) ok &= before < s.x[f].x;
    if (2 * lane + 1 < s.n[f]) ok &= s.x[f].x < s.x[f].y;
  }
  return __all_sync(0xffffffffu, ok);
}

// Entries below x (with_equal: or equal to it) among the n of the sorted list p, which is padded with 0xFFFFFFFF to N
// (a power of two) entries.
template <int N>
__device__ __forceinline__ int count_below(const uint32_t* p, int n, uint32_t x, bool with_equal = false) {
  int pos = 0;
#pragma unroll
  for (int step = N / 2; step > 0; step >>= 1)
    if (p[pos + step - 1] < x || (with_equal && p[pos + step - 1] == x)) pos += step;
  if (p[pos] < x || (with_equal && p[pos] == x)) ++pos;  // pos can reach N
  return min(pos, n);
}
// This lane's two membership tests of a field's nx cues against a padded list of n, as a mask (bit i: cue 2 lane + i is
// there).
template <int N>
__device__ __forceinline__ int hits(const uint32_t* p, int n, const uint2& x, int nx, int lane) {
  const int i0 = count_below<N>(p, n, x.x), i1 = count_below<N>(p, n, x.y);
  const bool h0 = i0 < n && p[i0] == x.x, h1 = i1 < n && p[i1] == x.y;
  return (h0 && 2 * lane < nx ? 1 : 0) | (h1 && 2 * lane + 1 < nx ? 2 : 0);
}
// A field's list into shared memory, padded.
__device__ __forceinline__ void put_list(uint32_t* p, const uint2& x, int n, int lane) {
  p[2 * lane] = 2 * lane < n ? x.x : 0xFFFFFFFFu;
  p[2 * lane + 1] = 2 * lane + 1 < n ? x.y : 0xFFFFFFFFu;
}

__device__ __forceinline__ float jaccard(int inter, int na, int nb) {
  const int uni = na + nb - inter;
  return uni > 0 ? (float)inter / (float)uni : 0.f;
}

__global__ void __launch_bounds__(kSigMaxWarps * 32) step_signals_kernel(const __grid_constant__ SignalArgs a) {
  constexpr int C = STEPKV_MAX_CUES;
  __shared__ float s_g[kSigMaxWarps], s_r[kSigMaxWarps];
  __shared__ uint32_t s_list[3][C];               // the target's lists
  __shared__ uint32_t s_both[2 * C];              // its Thought and Observation merged (a cue of both twice)
  __shared__ uint32_t s_obs[kSigMaxWarps][C];     // each warp's earlier step: its Observation's list
  __shared__ int s_bad;
  __shared__ float s_best[2];                     // the CTA's maxima and error flag, read by its cluster
  pdl_wait();
  pdl_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int NC = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int target = (int)blockIdx.x / NC;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  const int u0 = rank * n_warps + warp, u_step = NC * n_warps;
  const bool is_sim = target >= a.n_steps - a.k0;  // the obs_sim block: the newest step against all before
  const int k = is_sim ? a.n_steps - 1 : a.k0 + target;
  // every warp reads the target's lists (the first keeps them for all), and its first earlier step's
  StepCues tgt, next;
  load_step(a, k, lane, tgt);
  if (u0 < k) load_step(a, u0, lane, next);
  const bool tgt_ok = check_step(tgt, lane);
  if (!tgt_ok) {  // the same in every warp and CTA: nothing of this target can be written
    if (threadIdx.x == 0 && rank == 0) {
      record_status(a.status, STEPKV_EDATA);
      if (is_sim) a.obs_sim[k] = 0.f;
    }
    return;
  }
  if (threadIdx.x == 0) s_bad = 0;
  if (warp == 0) {
#pragma unroll
    for (int f = 0; f < 3; ++f) put_list(s_list[f], tgt.x[f], tgt.n[f], lane);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) s_both[4 * lane + i] = 0xFFFFFFFFu;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t t = i ? tgt.x[0].y : tgt.x[0].x, o = i ? tgt.x[2].y : tgt.x[2].x;
      const int j = 2 * lane + i;
      if (j < tgt.n[0]) s_both[j + count_below<C>(s_list[2], tgt.n[2], t)] = t;
      if (j < tgt.n[2]) s_both[j + count_below<C>(s_list[0], tgt.n[0], o, true)] = o;
    }
  }
  __syncthreads();
  // |X| of the target's X = Thought u Observation
  const int n_both = tgt.n[0] + tgt.n[2];
  int size_x = 0;
  if (!is_sim)
    size_x = n_both - __reduce_add_sync(0xffffffffu, __popc(hits<C>(s_list[2], tgt.n[2], tgt.x[0], tgt.n[0], lane)));
  float best_g = 0.f, best_r = 0.f;
  for (int u = u0; u < k; u += u_step) {
    StepCues s = next;
    if (u + u_step < k) load_step(a, u + u_step, lane, next);
    if (!check_step(s, lane)) {
      if (lane == 0) s_bad = 1;
      continue;
    }
    if (is_sim) {
      const int inter = __reduce_add_sync(0xffffffffu, __popc(hits<C>(s_list[2], tgt.n[2], s.x[2], s.n[2], lane)));
      if (lane == 0) a.obs_sim[u] = jaccard(inter, tgt.n[2], s.n[2]);
      continue;
    }
    // Y = Thought_u u Observation_u: a cue of both fields counts once
    uint32_t* obs = s_obs[warp];
    __syncwarp();
    put_list(obs, s.x[2], s.n[2], lane);
    __syncwarp();
    const int th_both = hits<C>(obs, s.n[2], s.x[0], s.n[0], lane);
    const int th_in = hits<2 * C>(s_both, n_both, s.x[0], s.n[0], lane);
    const int ob_in = hits<2 * C>(s_both, n_both, s.x[2], s.n[2], lane);
    const int ac_in = hits<C>(s_list[1], tgt.n[1], s.x[1], s.n[1], lane);
    // three sums of at most 128 in one reduction
    const int sums = __reduce_add_sync(0xffffffffu, (__popc(th_in & ~th_both) + __popc(ob_in)) | (__popc(th_both) << 10) |
                                                        (__popc(ac_in) << 20));
    const int size_y = s.n[0] + s.n[2] - ((sums >> 10) & 1023);
    best_g = fmaxf(best_g, jaccard(sums & 1023, size_x, size_y));
    best_r = fmaxf(best_r, jaccard(sums >> 20, tgt.n[1], s.n[1]));
  }
  if (lane == 0) {
    s_g[warp] = best_g;
    s_r[warp] = best_r;
  }
  __syncthreads();
  if (warp == 0) {
    float g = lane < n_warps ? s_g[lane] : 0.f, r = lane < n_warps ? s_r[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, o));
      r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    }
    if (lane == 0) {
      s_best[0] = s_bad ? INFINITY : g;
      s_best[1] = r;
    }
  }
  if (NC > 1) cluster.sync();
  if (threadIdx.x == 0 && rank == 0) {
    float g = 0.f, r = 0.f;
    for (int c = 0; c < NC; ++c) {
      const float* best = cluster.map_shared_rank(s_best, c);
      g = fmaxf(g, best[0]);
      r = fmaxf(r, best[1]);
    }
    const bool bad = g == INFINITY;  // some earlier step's lists
    if (bad) record_status(a.status, STEPKV_EDATA);
    if (is_sim) {
      a.obs_sim[k] = 0.f;
    } else if (!bad) {
      if (a.gain) a.gain[k] = 1.f - g;
      if (a.red) a.red[k] = r;
    }
  }
  if (NC > 1) cluster.sync();  // no CTA exits while the first may still read its maxima
}

stepkv_status_t signals_run(const uint32_t* cues, const int32_t* n_cues, int n_steps, int k0, float* gain, float* red,
                            float* obs_sim, int32_t* status, cudaStream_t stream) {
  SignalArgs a;
  memset(&a, 0, sizeof(a));
  a.cues = cues;
  a.n_cues = n_cues;
  a.n_steps = n_steps;
  a.k0 = k0;
  a.gain = gain;
  a.red = red;
  a.obs_sim = obs_sim;
  a.status = status;
  const int blocks = (n_steps - k0) + (obs_sim != nullptr ? 1 : 0);
  if (blocks == 0) return STEPKV_OK;
  int n_sm = 0;
  cudaError_t e = device_sm_count(&n_sm);
  if (e == cudaSuccess) {
    const int earlier = n_steps - 1;  // of the newest target
    const int nc = earlier > kSigMaxWarps && blocks * kSigCluster <= n_sm ? kSigCluster : 1;
    const int warps = std::max(1, std::min(kSigMaxWarps, (earlier + nc - 1) / nc));
    e = launch_cluster(step_signals_kernel, dim3(blocks * nc), dim3(warps * 32), nc, 0, stream, a);
  }
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return STEPKV_ECUDA;
  }
  return STEPKV_OK;
}

}  // namespace stepkv
