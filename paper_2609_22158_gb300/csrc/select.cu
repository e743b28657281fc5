// Stages 2-4 -- step reduction, score fusion and global top-B selection.
//   T_i   = mean of the saliency rows (layers x KV heads), normalised by its maximum over prunable
//           tokens (appendix "Combination with token-level importance": H_i in [0, H_max]);
//   r_k   = valid_k + gain_k - lambda red_k                                  (Eq. 2)
//   c_k  <- c_k + min(1, eta sim(Obs_t, Obs_k)) for k < t, c_t = 0            (Eq. 3, Alg. 1 Phases 1-2)
//   S_k   = clip(w_r clip(r_k, r_min, r_max) + w_c log(1 + c_k), 0, S_max)    (Eq. 4)
//   P_i   = alpha T_i + beta S_{s(i)}                                        (Eq. 5)
//   K     = top B_t prunable tokens by (P desc, index asc), B_t from Eq. 1   (Alg. 1 Phase 3)
//
// GB300 design: the tokens live in shared memory (saliency, then the order-preserving 32-bit key of P,
// and a 16-bit step id) -- in one 1024-thread CTA up to 2048 tokens, else in a cluster of 8 CTAs.
// The exact B-th largest key is found by a linear bin of P and then digits of the key within that bin, over
// shared-memory histograms whose sums meet through distributed shared memory; retained
// slots are written in ascending order by warp ballot + prefix counts.  Per-step statistics use
// integer atomics only (fixed-point sums), so every output is bit-reproducible run to run.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace stepkv {

// Two shapes of the same algorithm: one 1024-thread CTA for short trajectories (no cluster barriers),
// else a cluster of 8 such CTAs whose histograms and counts meet through distributed shared memory.  One CTA up to 2048
// tokens: at 4096 it is 2.9 us behind the cluster, at 8192 10 us.  1024 threads a CTA: a fused pass over T = 32768 takes
// 257.7 us, 260.8 with 512 (the token loops are chains of short latencies, which more warps overlap and unrolling does
// not: 258.1-258.6 us, the code is fetched cold).
constexpr int kSelSingleMaxT = 2048;
constexpr int kSelClusterCtas = 8;
constexpr int kSelThreads = 1024;
constexpr uint32_t kNanKey = 0x007FFFFEu;  // just below the key of -inf

struct SelectArgs {
  const float* T_in;                  // token saliency as floats, or
  const unsigned long long* t_acc;    // as fixed-point sums: T_i = t_acc[i] * acc_to_T
  float acc_to_T;
  int T;
  int chunk;                          // tokens per CTA
  int s_in_smem;                      // S_k kept in shared memory (all CTAs compute all steps)
  const int32_t* step_id;
  const uint8_t* prot;
  stepkv_steps_t steps;
  stepkv_params_t prm;
  stepkv_budget_t budget;
  stepkv_select_out_t out;
  float* S;                           // [n_steps] step utilities (workspace)
  int32_t* acc_cnt;                   // [n_steps] workspace accumulators (zeroed here)
  unsigned long long* acc_sum;
  uint32_t* acc_max;
  int32_t* acc_kept;
  int32_t* status;
  // In-place compaction by hole filling (NULL plan: none).  The write pass also lays out the plan the move
  // kernel follows: plan[0] = number of holes H (slots below n_kept that are not retained), plan[1 + j] =
  // the j-th hole in slot order; the j-th mover is kept_idx[n_kept - H + j].  All rows below n_kept get their own
  // step id / position here; the move kernel overwrites those of the filled holes.
  int32_t* plan;
  const int32_t* pos_in;
  int32_t* step_id_out;
  int32_t* pos_out;
};

// One CTA's summary, pushed into every CTA of the cluster.
struct SelSummary {
  float max_T, min_T;  // over prunable tokens (min_T: NaN where one is)
  int n;               // prunable tokens
  int err;
};

// Several independent trajectories in one launch: cluster (or CTA) c selects for trajectory c, so the
// latency-bound passes of different trajectories run side by side on different SMs.
constexpr int kMaxSelBatch = 16;
struct SelectBatch {
  SelectArgs t[kMaxSelBatch];
};
static_assert(sizeof(SelectBatch) <= 32000, "kernel parameter space");

// Inclusive suffix sum over the warp: lane l gets v[l] + v[l + 1] + ... + v[31].
__device__ __forceinline__ int warp_suffix_sum(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_down_sync(0xffffffffu, v, o);
    if (lane + o < 32) v += y;
  }
  return v;
}

// Warp-wide flush of per-lane step statistics (lane: `act`, its step `sid`, count, fixed-point sum,
// max bits): one set of atomics per warp when every active lane holds the same step, else one per
// lane.  Integer atomics only, so the totals do not depend on the order of arrival.
__device__ __forceinline__ void step_stat_flush(bool act, int sid, int cnt_v, unsigned long long sum_v,
                                                uint32_t max_v, int32_t* cnt, unsigned long long* sum,
                                                uint32_t* mx) {
  const unsigned am = __ballot_sync(0xffffffffu, act);
  if (!am) return;
  const int lane = threadIdx.x & 31;
  const int sid0 = __shfl_sync(0xffffffffu, sid, __ffs(am) - 1);
  if (__all_sync(0xffffffffu, !act || sid == sid0)) {
    const int c = __reduce_add_sync(0xffffffffu, act ? cnt_v : 0);
    unsigned long long v = act ? sum_v : 0ull;
    const uint32_t m = mx ? __reduce_max_sync(0xffffffffu, act ? max_v : 0u) : 0u;
    if (sum) {
#pragma unroll 1
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    if (lane == 0) {
      atomicAdd(&cnt[sid0], c);
      if (sum) atomicAdd(&sum[sid0], v);
      if (mx) atomicMax(&mx[sid0], m);
    }
  } else if (act) {
    atomicAdd(&cnt[sid], cnt_v);
    if (sum) atomicAdd(&sum[sid], sum_v);
    if (mx) atomicMax(&mx[sid], max_v);
  }
}

__device__ __forceinline__ float step_reuse(const SelectArgs& a, int k, int t_last) {
  float c = 0.f;                                                                     // Alg. 1: c_t = 0
  if (k != t_last) {
    c = a.steps.reuse_in[k];
    if (a.steps.obs_sim) c += fminf(1.f, a.prm.eta * a.steps.obs_sim[k]);          // Eq. 3
  }
  return c;
}
__device__ __forceinline__ float step_utility(const SelectArgs& a, int k, int t_last) {
  const stepkv_params_t& p = a.prm;
  const float r = a.steps.valid[k] + a.steps.gain[k] - p.lambda * a.steps.red[k];  // Eq. 2
  const float rc = fminf(fmaxf(r, p.r_min), p.r_max);
  return fminf(fmaxf(p.w_r * rc + p.w_c * log1pf(step_reuse(a, k, t_last)), 0.f), p.s_max);  // Eq. 4
}

template <int NC>
struct ClusterOps {
  cg::cluster_group cluster;
  __device__ ClusterOps() : cluster(cg::this_cluster()) {}
  __device__ int rank() const { return (int)cluster.block_rank(); }
  __device__ void sync() { cluster.sync(); }
  // Every thread of the kernel: started() once at its beginning, then all_started() before the first access to another
  // CTA's shared memory, which exists only once that CTA runs.
  __device__ void started() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
  __device__ void all_started() { asm volatile("barrier.cluster.wait;" ::: "memory"); }
  template <typename P>
  __device__ P* peer(P* p, int r) { return cluster.map_shared_rank(p, r); }
};
template <>
struct ClusterOps<1> {
  __device__ int rank() const { return 0; }
  __device__ void sync() { __syncthreads(); }
  __device__ void started() {}
  __device__ void all_started() {}
  template <typename P>
  __device__ P* peer(P* p, int) { return p; }
};

// What bounds a selection is latency: barriers, distributed-shared-memory round trips, and code that runs once per
// launch and is fetched cold (so loops stay rolled).  There are as few of each as
// the result allows:
//  - the first digit is a linear bin of the priority between its bounds (the corners of alpha T^ + beta S over the
//    extreme T^ and S), so the bins spread over the values the trajectory has; the keys of the threshold's bin span about
//    BITS bits, and one more pass over the key's offset within the bin ranks them exactly (further passes where the bin
//    reaches down to where floats are dense).  Fixed digits of the key took three passes, the first of which only told
//    a few exponents apart.  Where the step utilities spread the priority by less than a 16th of what the saliency does, the
//    passes begin with the leading digit of the key's offset from the lowest: the saliency is heavy-tailed, and with linear
//    bins a selection by it alone (log-normal, all outputs) took up to five passes, T = 2049 / 9000 / 32768: 17.1 / 20.9 /
//    25.0 us; with key digits 11.6 / 15.2 / 17.8 (fixed digits 14.0 / 19.1 / 24.1).  Linear bins are the better ones from
//    there on (alpha = 0.8, beta = 0.2, saliencies over 30 decades, T = 32768: 23.4 us; key digits 26.8);
//  - the passes end where all keys left in the threshold's bin are kept, mostly one key: two or three digits of a priority
//    say no more than which tokens stay.  Ranking a few keys directly in one exchange instead of a last digit was up to
//    0.8 us ahead where the code was warm, but its code costs a fused pass 2-4 us (T = 32768: 256.7 -> 260.7 us, 258.4
//    where it is not even run);
//  - every exchange is a push into the other CTAs' shared memory before a cluster barrier, so only the 32 fine counts
//    of each digit are fetched after one;
//  - a CTA's output offset comes out of the same counts (those of the CTAs before it above each digit), so no
//    barrier is spent on it; the barrier that lets CTAs exit is split around the writes.
// Against three fixed digits with a gather after every barrier: a fused pass over T = 32768 263.5 -> 256.0 us, over
// T = 65536 864.6 -> 856, T = 2048 35.6 -> 31.9, an in-place boundary 102.1 -> 96.9, a selection alone with all outputs
// 26.6 -> 22.6.
// BITS: 13, or 11 where the tokens leave no room for 2 x 8192 bins.
template <int NC, int NT, int BITS>
__global__ void __launch_bounds__(NT, 1) select_kernel(const __grid_constant__ SelectBatch batch) {
  const SelectArgs& a = batch.t[blockIdx.x / NC];
  constexpr int NW = NT / 32;
  constexpr int U = 4;  // tokens of a thread in flight
  constexpr int kBins = 1 << BITS, kCoarse = kBins / 32;
  ClusterOps<NC> cl;
  const int rank = cl.rank();
  extern __shared__ __align__(16) uint8_t smem_raw[];
  // layout: [2][kBins] int histograms | [2][NC][kCoarse] every CTA's coarse counts | [chunk] T, then the ordered key of
  // P | [chunk] u16 step id (0xFFFF = protected) | S_k (when s_in_smem).  A token's entries are touched by one thread only.
  int* hist = reinterpret_cast<int*>(smem_raw);
  int* coarse = hist + 2 * kBins;
  uint32_t* sKey = reinterpret_cast<uint32_t*>(coarse + 2 * NC * kCoarse);
  float* sT = reinterpret_cast<float*>(sKey);
  uint16_t* sSid = reinterpret_cast<uint16_t*>(sKey + a.chunk);
  float* sS = reinterpret_cast<float*>(sSid + a.chunk);
  __shared__ SelSummary all[NC];
  __shared__ float w_max[NW], w_min[NW], s_lo[NW], s_hi[NW];
  __shared__ int w_n[NW], w_err[NW], w_strict[NW], w_eq[NW], bcast[5];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = a.T, n_steps = a.steps.n_steps, t_last = n_steps - 1;
  const int base = rank * a.chunk;
  const int len = max(0, min(a.chunk, T - base));
  const bool want_stats = a.out.step_count || a.out.step_sal_sum || a.out.step_sal_max;
  const bool want_kept = a.out.step_kept != nullptr;
  const bool s_in_smem = a.s_in_smem != 0;
  // warp w owns the consecutive slots [s0, s1) of this CTA, lanes take consecutive slots
  const int seg = ((len + NW - 1) / NW + 31) & ~31;
  const int s0 = min(len, warp * seg), s1 = min(len, s0 + seg);
  const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;

  // Launched with programmatic dependent launch: everything up to pdl_wait() reads only the call's inputs and writes
  // only this kernel's workspace and outputs, so it may overlap the tail of the kernel that produces the saliency.
  pdl_launch_dependents();
  cl.started();
  int lN = 0, lerr = 0;
#pragma unroll 1
  for (int i0 = s0 + lane; i0 < s1; i0 += 32 * U) {
    uint8_t pv[U];
    int sv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u;
      if (i < s1) {
        pv[u] = __ldg(&a.prot[base + i]);
        sv[u] = __ldg(&a.step_id[base + i]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u;
      if (i < s1) {
        const bool bad = !pv[u] && (sv[u] < 0 || sv[u] >= n_steps);
        lN += !pv[u];
        lerr |= bad;
        sSid[i] = pv[u] ? (uint16_t)0xFFFFu : (uint16_t)(bad ? 0 : sv[u]);
      }
    }
  }
#pragma unroll 1
  for (int i = tid; i < 2 * kBins / 4; i += NT) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
  // Phases 1 and 2 of Algorithm 1 (Eqs. 2-4).  Every CTA computes all S_k, for their bounds and, where they fit, into
  // shared memory; CTA 0 publishes them.
  float b_lo = INFINITY, b_hi = -INFINITY;  // bounds of beta S_k
#pragma unroll 1
  for (int k = tid; k < n_steps; k += NT) {
    const float sk = step_utility(a, k, t_last);
    if (s_in_smem) sS[k] = sk;
    b_lo = fminf(b_lo, a.prm.beta * sk);
    b_hi = fmaxf(b_hi, a.prm.beta * sk);
    if (rank == 0) {
      a.S[k] = sk;
      if (a.out.step_util) a.out.step_util[k] = sk;  // reuse_out may alias reuse_in: written after the barrier
    }
    if (k % NC == rank) {
      a.acc_cnt[k] = 0;
      a.acc_sum[k] = 0ull;
      a.acc_max[k] = 0u;
      a.acc_kept[k] = 0;
    }
  }
  if (a.plan && rank == 0 && tid == 0) a.plan[0] = 0;  // hole count
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    b_lo = fminf(b_lo, __shfl_xor_sync(full, b_lo, o));
    b_hi = fmaxf(b_hi, __shfl_xor_sync(full, b_hi, o));
  }
  lN = __reduce_add_sync(full, lN);
  lerr = __any_sync(full, lerr);
  if (lane == 0) {
    s_lo[warp] = b_lo;
    s_hi[warp] = b_hi;
    w_n[warp] = lN;
    w_err[warp] = lerr;
  }
  pdl_wait();  // t_acc / T_in come from the preceding kernel
  float lmax = -INFINITY, lmin = INFINITY;
#pragma unroll 1
  for (int i0 = s0 + lane; i0 < s1; i0 += 32 * U) {
    float tv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u;
      if (i < s1) tv[u] = a.t_acc ? __ull2float_rn(__ldcg(&a.t_acc[base + i])) * a.acc_to_T : __ldcg(&a.T_in[base + i]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u;
      if (i < s1) {
        sT[i] = tv[u];
        if (sSid[i] != 0xFFFFu) {
          lmax = fmaxf(lmax, tv[u]);
          lmin = min_nan(lmin, tv[u]);
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lmax = fmaxf(lmax, __shfl_xor_sync(full, lmax, o));
    lmin = min_nan(lmin, __shfl_xor_sync(full, lmin, o));
  }
  if (lane == 0) {
    w_max[warp] = lmax;
    w_min[warp] = lmin;
  }
  cl.all_started();  // the pushes below reach into every CTA (long since true: the tokens have been read meanwhile)
  __syncthreads();
  if (warp == 0) {
    float m = lane < NW ? w_max[lane] : -INFINITY, mi = lane < NW ? w_min[lane] : INFINITY;
    b_lo = lane < NW ? s_lo[lane] : INFINITY;
    b_hi = lane < NW ? s_hi[lane] : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m = fmaxf(m, __shfl_xor_sync(full, m, o));
      mi = min_nan(mi, __shfl_xor_sync(full, mi, o));
      b_lo = fminf(b_lo, __shfl_xor_sync(full, b_lo, o));
      b_hi = fmaxf(b_hi, __shfl_xor_sync(full, b_hi, o));
    }
    const int n = __reduce_add_sync(full, lane < NW ? w_n[lane] : 0);
    const int err = __reduce_or_sync(full, lane < NW ? w_err[lane] : 0);
    if (lane < NC) {
      SelSummary* dst = cl.peer(&all[rank], lane);
      dst->max_T = m;
      dst->min_T = mi;
      dst->n = n;
      dst->err = err;
    }
    if (lane == 0) {
      s_lo[0] = b_lo;
      s_hi[0] = b_hi;
    }
  }
  cl.sync();  // every CTA's summary is here; S_k, histograms and zeroed accumulators are ready
  if (rank == 0 && a.steps.reuse_out) {
#pragma unroll 1
    for (int k = tid; k < n_steps; k += NT) a.steps.reuse_out[k] = step_reuse(a, k, t_last);
  }
  float gmax = -INFINITY, gmin = INFINITY;
  int N = 0, err = 0, n_pre = 0;  // n_pre: prunable tokens of the CTAs before this one
#pragma unroll
  for (int r = 0; r < NC; ++r) {
    gmax = fmaxf(gmax, all[r].max_T);
    gmin = min_nan(gmin, all[r].min_T);
    if (r < rank) n_pre += all[r].n;
    N += all[r].n;
    err |= all[r].err;
  }
  if (err) {
    if (rank == 0 && tid == 0) {
      record_status(a.status, STEPKV_EDATA);
      *a.out.n_kept = 0;
      if (a.out.n_budget) { a.out.n_budget[0] = N; a.out.n_budget[1] = 0; }
    }
    if (NC > 1) cl.sync();
    return;
  }
  // ---- budget (Eq. 1): B = max(1, floor(num N / den)) or a count, then |K| = min(B, N)
  int B = 0;
  if (N > 0) {
    if (a.budget.mode == STEPKV_BUDGET_RATIO)
      B = (int)max(1ll, ((long long)a.budget.ratio_num * N) / a.budget.ratio_den);
    else
      B = a.budget.count;
    B = min(B, N);
  }
  const int total_kept = T - N + B;
  const bool overflow = total_kept > a.out.kept_cap;
  // In place: the step ids and positions of the rows below total_kept, holes included (the move kernel overwrites
  // those), copied by warps w0 .. of every CTA, a CTA's own slots.
  auto copy_metadata = [&](int w0) {
    if (!a.plan || overflow) return;
    for (int i = (warp - w0) * 32 + lane; i < len && base + i < total_kept; i += (NW - w0) * 32) {
      const int gi = base + i;
      const int sid = a.step_id_out ? __ldg(&a.step_id[gi]) : 0, pos = a.pos_in ? __ldg(&a.pos_in[gi]) : gi;
      if (a.step_id_out) a.step_id_out[gi] = sid;
      if (a.pos_out) a.pos_out[gi] = pos;
    }
  };
  const bool norm = a.prm.sal_norm == STEPKV_NORM_MAX && gmax > 0.f && N > 0;
  const float inv_max = norm ? 1.0f / gmax : 1.0f;
  // fixed-point scale for per-step sums of normalised saliency: values <= vmax, at most N terms
  const float vmax = norm ? 1.0f : fmaxf(gmax, 1e-30f);
  const int e_max = (int)(__float_as_uint(vmax) >> 23) - 126;  // vmax < 2^e_max (vmax is normal and positive)
  const int log2N = 32 - __clz(max(N, 1));            // N < 2^log2N
  const int fx_shift = min(62 - log2N - e_max, 126);  // every partial sum < 2^62

  // ---- priorities (Eq. 5) and their bounds; bins of the first digit
  const float t_lo = gmin * inv_max, t_hi = gmax * inv_max;
  float P_lo = fminf(fmaf(a.prm.alpha, t_lo, s_lo[0]), fmaf(a.prm.alpha, t_hi, s_lo[0]));
  float P_hi = fmaxf(fmaf(a.prm.alpha, t_lo, s_hi[0]), fmaf(a.prm.alpha, t_hi, s_hi[0]));
  // Where a priority can lie outside them (a saliency that is not finite, an overflow) the bounds become the infinities:
  // all keys share the first bin and their whole 32 bits follow.  A priority that is not a number ranks below -inf.
  if (!(fabsf(gmin) < INFINITY && fabsf(gmax) < INFINITY && fabsf(P_lo) < INFINITY && fabsf(P_hi) < INFINITY)) {
    P_lo = -INFINITY;
    P_hi = INFINITY;
  }
  // The first digit: linear in the priority where the step utilities spread it, else (scale 0: one bin) digits of the key
  // from the start, which are logarithmic: the saliency alone is heavy-tailed, and most of it would share the first bins.
  float scale = 0.999999f * (float)kBins / (P_hi - P_lo);
  if (!(scale < INFINITY && 16.f * (s_hi[0] - s_lo[0]) >= fabsf(a.prm.alpha) * (t_hi - t_lo))) scale = 0.f;
  auto first_bin = [&](uint32_t key) {  // monotone in the priority
    return min(max((int)((ordered_to_float(key) - P_lo) * scale), 0), kBins - 1);
  };
  const float* Sk = s_in_smem ? sS : a.S;
  {
    // A lane accumulates its tokens' statistics while their step does not change (slots of a step are mostly
    // contiguous) and flushes with integer atomics.
    int run_sid = -1, run_c = 0;
    unsigned long long run_s = 0ull;
    uint32_t run_m = 0u;
#pragma unroll 1
    for (int i = s0 + lane; i < s1; i += 32) {
      const int gi = base + i;
      const float x = sT[i] * inv_max;
      const int sid = sSid[i];
      uint32_t key = 0u;
      float P = -INFINITY;
      if (sid != 0xFFFF) {
        P = fmaf(a.prm.alpha, x, a.prm.beta * Sk[sid]);
        key = P == P ? float_to_ordered(P) : kNanKey;
        if (want_stats) {
          const float xc = fmaxf(x, 0.f);
          if (sid != run_sid) {
            if (run_c) {
              atomicAdd(&a.acc_cnt[run_sid], run_c);
              atomicAdd(&a.acc_sum[run_sid], run_s);
              atomicMax(&a.acc_max[run_sid], run_m);
            }
            run_sid = sid;
            run_c = 0;
            run_s = 0ull;
            run_m = 0u;
          }
          ++run_c;
          run_s += to_fixed(xc, fx_shift);
          run_m = max(run_m, __float_as_uint(xc));
        }
      }
      if (a.out.priority) a.out.priority[gi] = P;
      if (a.out.token_sal) a.out.token_sal[gi] = x;
      sKey[i] = key;
    }
    if (want_stats) step_stat_flush(run_c > 0, run_sid, run_c, run_s, run_m, a.acc_cnt, a.acc_sum, a.acc_max);
  }

  // ---- exact B-th largest key among the prunable tokens
  uint32_t kth = 0u;  // B == N: every prunable token's key is above 0
  int need_eq = 0;
  int strict_pre = n_pre, eq_pre = 0;  // tokens above / at the threshold in the CTAs before this one
  if (B == 0) {
    kth = 0xFFFFFFFFu;
    strict_pre = 0;
  } else if (B < N) {
    strict_pre = 0;
    int remaining = B, star = 0;  // star: the threshold's linear bin
    // keys as offsets from k_lo (one below the lowest: kNanKey below -inf), `left` bits of the threshold's undecided
    uint32_t k_lo = float_to_ordered(P_lo) - 1u, k_hi = float_to_ordered(P_hi) + 1u, prefix = 0u;
    int left = 32 - __clz((int)(k_hi - k_lo));
    const int first_pass = scale > 0.f ? 0 : 1;
#pragma unroll 1
    for (int pass = first_pass;; ++pass) {
      int* h = hist + (pass & 1) * kBins;
      int* ac = coarse + (pass & 1) * NC * kCoarse;
      const int bits = pass == 0 ? BITS : min(BITS, left), sh = left - bits;  // sh: of the key offset (later passes)
      const int n_coarse = pass == 0 ? kCoarse : max(1, (1 << bits) >> 5);
      if (pass >= 2) {  // the buffers were zeroed for two passes
#pragma unroll 1
        for (int i = tid; i < kBins / 4; i += NT) reinterpret_cast<int4*>(h)[i] = make_int4(0, 0, 0, 0);
        __syncthreads();
      }
#pragma unroll 1
      for (int i0 = s0; i0 < s1; i0 += 32) {
        const int i = i0 + lane;
        bool hit = i < s1 && sSid[i] != 0xFFFF;
        int bin = 0;
        if (hit) {
          const uint32_t key = sKey[i];
          bin = first_bin(key);
          if (pass > 0) {
            const uint32_t off = key - k_lo;
            hit = bin == star && (left >= 32 || (off >> left) == prefix);
            bin = (int)((off >> sh) & ((1u << bits) - 1u));
          }
        }
        const unsigned hm = __ballot_sync(full, hit);
        if (hm == 0u) continue;
        // tokens of one warp mostly fall into bins of their own; equal priorities share one addition
        const int b0 = __shfl_sync(full, bin, __ffs(hm) - 1);
        if (__all_sync(full, !hit || bin == b0)) {
          if (lane == 0) atomicAdd(&h[b0], __popc(hm));
        } else if (hit) {
          atomicAdd(&h[bin], 1);
        }
      }
      __syncthreads();
      // sums of 32 consecutive bins, NW warps over the coarse bins, pushed into every CTA (lane i holds sum i)
      constexpr int kPerWarp = kCoarse / NW;
      if (warp * kPerWarp < n_coarse) {
        int mine = 0;
#pragma unroll 4
        for (int i = 0; i < kPerWarp; ++i) {
          const int v = __reduce_add_sync(full, h[(warp * kPerWarp + i) * 32 + lane]);
          if (lane == i) mine = v;
        }
        if (lane < kPerWarp) {
#pragma unroll
          for (int r = 0; r < NC; ++r) cl.peer(ac, r)[rank * kCoarse + warp * kPerWarp + lane] = mine;
        }
      }
      cl.sync();  // every CTA's histogram and coarse counts of this pass are complete
      if (warp == 0) {
        // The digit in two steps (keys in descending order): the coarse bin that holds the remaining-th largest key
        // (lane l: coarse bins PL l .. PL l + PL - 1), then the bin within it (lane l: fine bin l).
        constexpr int PL = kCoarse / 32;  // 8, or 2 with 11 bits
        static_assert(kCoarse % 64 == 0, "a lane's coarse counts are read in pairs");
        int cnt[PL];
#pragma unroll
        for (int i = 0; i < PL; ++i) cnt[i] = 0;
        if (lane * PL < n_coarse) {
#pragma unroll
          for (int r = 0; r < NC; ++r) {
#pragma unroll
            for (int i = 0; i < PL; i += 2) {
              const int2 v = *reinterpret_cast<const int2*>(&ac[r * kCoarse + lane * PL + i]);
              cnt[i] += lane * PL + i < n_coarse ? v.x : 0;
              cnt[i + 1] += lane * PL + i + 1 < n_coarse ? v.y : 0;
            }
          }
        }
        int mine = 0;
#pragma unroll
        for (int i = 0; i < PL; ++i) mine += cnt[i];
        int above = warp_suffix_sum(mine, lane) - mine;  // keys in the coarse bins of the lanes after this one
        int cs = -1, above_c = 0;
#pragma unroll
        for (int i = PL - 1; i >= 0; --i) {
          if (cs < 0 && above < remaining && remaining <= above + cnt[i]) {
            cs = lane * PL + i;
            above_c = above;
          }
          above += cnt[i];
        }
        const unsigned mc = __ballot_sync(full, cs >= 0);
        const int src = mc ? __ffs(mc) - 1 : 0;
        const int cstar = max(0, __shfl_sync(full, cs, src));
        above_c = __shfl_sync(full, above_c, src);
        int f = 0, f_p = 0;
#pragma unroll
        for (int r = 0; r < NC; ++r) {
          const int v = cl.peer(h, r)[cstar * 32 + lane];
          f += v;
          if (r < rank) f_p += v;
        }
        int pre = 0;  // in the coarse bins above c*, of the CTAs before this one
#pragma unroll 1
        for (int i = cstar + 1 + lane; i < n_coarse; i += 32)
#pragma unroll
          for (int r = 0; r < NC; ++r)
            if (r < rank) pre += ac[r * kCoarse + i];
        const int sf = warp_suffix_sum(f, lane);
        const unsigned mf = __ballot_sync(full, above_c + sf - f < remaining && remaining <= above_c + sf);
        const int lf = mf ? __ffs(mf) - 1 : 0;
        const int above_f = __shfl_sync(full, above_c + sf - f, lf);
        pre = __reduce_add_sync(full, pre + (lane > lf ? f_p : 0));
        if (lane == lf) {
          // the counts always hold the remaining-th key; the guard only keeps every index in range
          const bool found = mc != 0 && mf != 0;
          if (!found) record_status(a.status, STEPKV_EDATA);
          bcast[0] = found ? cstar * 32 + lf : 0;
          bcast[1] = found ? above_f : 0;
          bcast[2] = pre;
          bcast[3] = f_p;
          bcast[4] = found ? f : 0;
        }
      } else if (pass == first_pass) {
        copy_metadata(1);  // while the first warp searches
      }
      __syncthreads();
      const int digit = bcast[0];
      remaining -= bcast[1];
      strict_pre += bcast[2];
      eq_pre = bcast[3];
      const int in_bin = bcast[4];
      if (pass == 0) {
        // the keys of the bin lie within its bounds, widened by its rounding and two keys
        star = digit;
        const float w = 1.0f / scale;
        const uint32_t lo = float_to_ordered(P_lo + ((float)star - 0.02f) * w) - 2u;
        const uint32_t hi = float_to_ordered(P_lo + ((float)star + 1.02f) * w) + 2u;
        if (star > 0) k_lo = max(k_lo, lo);
        if (star < kBins - 1) k_hi = min(k_hi, hi);
        left = 32 - __clz((int)(k_hi - k_lo));
      } else {
        prefix = (prefix << bits) | (uint32_t)digit;
        left = sh;
      }
      if (left == 0) {
        kth = k_lo + prefix;
        need_eq = remaining;
        break;
      }
      // All keys of the bin are kept (mostly it is one key): they lie above its lower bound less one, which the undecided
      // bits do not change, if no key outside the linear bin does.
      if (in_bin == remaining && pass > 0 && first_bin(k_lo + (prefix << left)) == star) {
        kth = k_lo + (prefix << left) - 1u;
        strict_pre += eq_pre;
        eq_pre = 0;
        break;
      }
    }
  }
  if (B == 0 || B == N) copy_metadata(0);
  if (NC > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");  // no more reads of other CTAs' memory

  // ---- counts per warp: kept for sure (protected or strictly above the threshold) and ties
  int strict_w = 0, eq_w = 0;
#pragma unroll 1
  for (int i = s0 + lane; i < s1; i += 32) {
    const bool pr = sSid[i] == 0xFFFF;
    strict_w += pr || sKey[i] > kth;
    eq_w += !pr && sKey[i] == kth;
  }
  strict_w = __reduce_add_sync(full, strict_w);
  eq_w = __reduce_add_sync(full, eq_w);
  if (lane == 0) {
    w_strict[warp] = strict_w;
    w_eq[warp] = eq_w;
  }
  __syncthreads();
  const int seg_s = lane < NW ? w_strict[lane] : 0, seg_e = lane < NW ? w_eq[lane] : 0;
  const int strict_before = __reduce_add_sync(full, lane < warp ? seg_s : 0);
  const int eq_before = __reduce_add_sync(full, lane < warp ? seg_e : 0);
  const int eq_cta = __reduce_add_sync(full, seg_e);
  // a CTA keeps its protected and strictly greater tokens and the ties that fall within the first need_eq in slot order
  const int prot_pre = min(base, T) - n_pre;
  const int out_off = prot_pre + strict_pre + min(need_eq, eq_pre);
  const int granted_cta = max(0, min(need_eq - eq_pre, eq_cta));
  if (rank == 0 && tid == 0) {
    *a.out.n_kept = total_kept;
    if (a.out.n_budget) { a.out.n_budget[0] = N; a.out.n_budget[1] = B; }
    if (overflow) record_status(a.status, STEPKV_ENOSPACE);
  }

  // ---- ordered write of the retained slots
  if (!overflow) {
    int tie_rank = eq_pre + eq_before;                                    // cluster-wide tie rank
    int out_pos = out_off + strict_before + min(granted_cta, eq_before);  // next output slot
    int holes = 0;  // in-place plan: holes among this lane's slots
    int run_sid = -1, run_c = 0;
#pragma unroll 1
    for (int i0 = s0; i0 < s1; i0 += 32) {
      const int i = i0 + lane, gi = base + i;
      const bool in = i < s1;
      const int sid = in ? sSid[i] : 0xFFFF;
      const uint32_t key = in ? sKey[i] : 0u;
      const bool pr = in && sid == 0xFFFF, is_eq = in && !pr && key == kth;
      const unsigned em = __ballot_sync(full, is_eq);
      const bool keep = pr || (in && (key > kth || (is_eq && tie_rank + __popc(em & lt) < need_eq)));
      const unsigned km = __ballot_sync(full, keep);
      const int kept_before = out_pos + __popc(km & lt);  // retained slots below this one, cluster-wide
      if (keep) a.out.kept_idx[kept_before] = gi;
      if (a.plan && in && !keep && gi < total_kept) {  // hole number gi - kept_before, filled by the mover of that number
        a.plan[1 + gi - kept_before] = gi;
        ++holes;
      }
      out_pos += __popc(km);
      tie_rank += __popc(em);
      if (want_kept && keep && !pr) {
        if (sid != run_sid) {
          if (run_c) atomicAdd(&a.acc_kept[run_sid], run_c);
          run_sid = sid;
          run_c = 0;
        }
        ++run_c;
      }
    }
    if (want_kept) step_stat_flush(run_c > 0, run_sid, run_c, 0ull, 0u, a.acc_kept, nullptr, nullptr);
    if (a.plan) {
      holes = __reduce_add_sync(full, holes);
      if (lane == 0 && holes) atomicAdd(&a.plan[0], holes);
    }
  }
  if (NC > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  if (want_stats || want_kept) {
    cl.sync();  // all step accumulators final
    const float fx_unit = __int_as_float((127 - fx_shift) << 23);  // 2^-fx_shift, -85 < fx_shift <= 126
#pragma unroll 1
    for (int k = rank * NT + tid; k < n_steps; k += NC * NT) {
      if (a.out.step_count) a.out.step_count[k] = __ldcg(&a.acc_cnt[k]);
      if (a.out.step_sal_sum) a.out.step_sal_sum[k] = __ull2float_rn(__ldcg(&a.acc_sum[k])) * fx_unit;
      if (a.out.step_sal_max) a.out.step_sal_max[k] = __uint_as_float(__ldcg(&a.acc_max[k]));
      if (a.out.step_kept) a.out.step_kept[k] = __ldcg(&a.acc_kept[k]);
    }
  }
}

// -------------------------------------------------------------------------------------------------
// T_out[j] = inv_div * sum over rows (fixed order): the token-saliency input of stepkv_select when the
// caller supplies per-(layer, head) saliency rows.  Four rows in flight per thread.
__global__ void mean_rows_kernel(const float* __restrict__ rows, int n_rows, int64_t row_stride, float inv_div, int T,
                                 float* __restrict__ T_out) {
  pdl_wait();
  pdl_launch_dependents();
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < T; j += gridDim.x * blockDim.x) {
    float s = 0.f;
    int r = 0;
    for (; r + 4 <= n_rows; r += 4) {
      const float a0 = __ldg(&rows[(int64_t)r * row_stride + j]);
      const float a1 = __ldg(&rows[(int64_t)(r + 1) * row_stride + j]);
      const float a2 = __ldg(&rows[(int64_t)(r + 2) * row_stride + j]);
      const float a3 = __ldg(&rows[(int64_t)(r + 3) * row_stride + j]);
      s = (((s + a0) + a1) + a2) + a3;
    }
    for (; r < n_rows; ++r) s += __ldg(&rows[(int64_t)r * row_stride + j]);
    T_out[j] = s * inv_div;
  }
}

// SnapKV-style estimator (Sec. 4.2: T_i from an existing token-level estimator): each row pooled along the
// token axis over the window [j - h, j + h] clipped to [0, T) -- its maximum, or the mean of its in-range
// values -- then T_out[j] = inv_div * the sum over rows in row order.  A CTA takes 256 tokens and stages
// eight rows' 256 + 2h values (the tile and its halo) in shared memory at a time, the next eight already on their way
// in registers: 24 rows x 32768 tokens, width 7: 27.6 -> 5.1 us against one row per pair of barriers (width 31: 31.5 ->
// 7.0 us).
constexpr int kPoolTile = 256;
constexpr int kRowsInFlight = 8;

template <bool IS_MAX>
__global__ void __launch_bounds__(kPoolTile) pool_mean_rows_kernel(const float* __restrict__ rows, int n_rows,
                                                                   int64_t row_stride, float inv_div, int T, int h,
                                                                   float* __restrict__ T_out) {
  extern __shared__ float tile[];  // [kRowsInFlight][kPoolTile + 2h]
  pdl_wait();
  pdl_launch_dependents();
  const int j0 = blockIdx.x * kPoolTile, j = j0 + (int)threadIdx.x;
  const int span = kPoolTile + 2 * h;
  // this token's window as tile indices (tile index x holds token j0 - h + x)
  const int lo = max(0, j - h) - (j0 - h), hi = min(T - 1, j + h) - (j0 - h);
  // a thread stages tile index threadIdx.x and, for the halo, kPoolTile + threadIdx.x (2h < kPoolTile)
  const int src0 = j0 - h + (int)threadIdx.x, src1 = src0 + kPoolTile;
  const bool ok0 = src0 >= 0 && src0 < T, has1 = (int)threadIdx.x < 2 * h, ok1 = has1 && src1 < T;
  float x0[kRowsInFlight], x1[kRowsInFlight];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int i = 0; i < kRowsInFlight; ++i) {
      const float* row = rows + (int64_t)(r0 + i) * row_stride;
      x0[i] = r0 + i < n_rows && ok0 ? __ldg(row + src0) : 0.f;
      x1[i] = r0 + i < n_rows && ok1 ? __ldg(row + src1) : 0.f;
    }
  };
  fetch(0);
  float acc = 0.f;
  for (int r0 = 0; r0 < n_rows; r0 += kRowsInFlight) {
    __syncthreads();  // the previous rows' tiles have been read
#pragma unroll
    for (int i = 0; i < kRowsInFlight; ++i) {
      tile[i * span + threadIdx.x] = x0[i];
      if (has1) tile[i * span + kPoolTile + threadIdx.x] = x1[i];
    }
    __syncthreads();
    if (r0 + kRowsInFlight < n_rows) fetch(r0 + kRowsInFlight);
    if (j < T) {
      const int nr = min(kRowsInFlight, n_rows - r0);
      float v[kRowsInFlight];
#pragma unroll
      for (int i = 0; i < kRowsInFlight; ++i) v[i] = tile[i * span + lo];
      for (int x = lo + 1; x <= hi; ++x) {
#pragma unroll
        for (int i = 0; i < kRowsInFlight; ++i) v[i] = IS_MAX ? fmaxf(v[i], tile[i * span + x]) : v[i] + tile[i * span + x];
      }
#pragma unroll
      for (int i = 0; i < kRowsInFlight; ++i)
        if (i < nr) acc += IS_MAX ? v[i] : v[i] / (float)(hi - lo + 1);
    }
  }
  if (j < T) T_out[j] = acc * inv_div;
}

stepkv_status_t pool_mean_rows_run(const float* rows, int n_rows, int64_t row_stride, float inv_div, int T, int h,
                                   bool is_max, float* T_out, cudaStream_t stream) {
  const int blocks = (T + kPoolTile - 1) / kPoolTile;
  const size_t smem = (size_t)kRowsInFlight * (kPoolTile + 2 * h) * sizeof(float);
  const cudaError_t e =
      is_max ? launch_kernel(pool_mean_rows_kernel<true>, dim3(blocks), dim3(kPoolTile), smem, stream, rows, n_rows,
                             row_stride, inv_div, T, h, T_out)
             : launch_kernel(pool_mean_rows_kernel<false>, dim3(blocks), dim3(kPoolTile), smem, stream, rows, n_rows,
                             row_stride, inv_div, T, h, T_out);
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return STEPKV_ECUDA;
  }
  return STEPKV_OK;
}

stepkv_status_t mean_rows_run(const float* rows, int n_rows, int64_t row_stride, float inv_div, int T, float* T_out,
                              cudaStream_t stream) {
  const int blocks = std::max(1, std::min((T + 255) / 256, 4096));
  cudaError_t e = launch_kernel(mean_rows_kernel, dim3(blocks), dim3(256), 0, stream, rows, n_rows, row_stride, inv_div,
                             T, T_out);
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return STEPKV_ECUDA;
  }
  return STEPKV_OK;
}

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

size_t select_ws_bytes(int T, int n_steps) {
  (void)T;
  const size_t n = (size_t)std::max(n_steps, 1);
  return align256(n * 4) + align256(n * 4) + align256(n * 8) + align256(n * 4) + align256(n * 4);
}

static SelectArgs make_select_args(const SelectSpec& sp) {
  SelectArgs a;
  memset(&a, 0, sizeof(a));
  a.T_in = sp.T_in;
  a.t_acc = sp.t_acc;
  a.acc_to_T = (float)sp.acc_to_T;
  a.T = sp.T;
  a.step_id = sp.step_id;
  a.prot = sp.prot;
  a.steps = sp.steps;
  a.prm = sp.params;
  a.budget = sp.budget;
  a.out = sp.out;
  const size_t n = (size_t)std::max(sp.steps.n_steps, 1);
  uint8_t* w = static_cast<uint8_t*>(sp.ws);
  a.S = reinterpret_cast<float*>(w);
  w += align256(n * 4);
  a.acc_cnt = reinterpret_cast<int32_t*>(w);
  w += align256(n * 4);
  a.acc_sum = reinterpret_cast<unsigned long long*>(w);
  w += align256(n * 8);
  a.acc_max = reinterpret_cast<uint32_t*>(w);
  w += align256(n * 4);
  a.acc_kept = reinterpret_cast<int32_t*>(w);
  a.status = sp.status;
  a.plan = sp.plan;
  a.pos_in = sp.pos_in;
  a.step_id_out = sp.step_id_out;
  a.pos_out = sp.pos_out;
  return a;
}

// Shared memory of one trajectory's CTA: histograms, coarse counts, keys + step ids of its chunk, and S_k when it fits.
constexpr size_t kSelSmemMax = 232448 - 2048;
static size_t select_smem(int chunk, int nc, int bits, int n_steps, int* s_in_smem) {
  const size_t bins = (size_t)1 << bits;
  const size_t fixed = (2 * bins + 2 * nc * (bins / 32)) * 4 + (size_t)chunk * 6;
  *s_in_smem = fixed + (size_t)n_steps * 4 <= kSelSmemMax ? 1 : 0;
  return fixed + (*s_in_smem ? (size_t)n_steps * 4 : 0);
}

stepkv_status_t select_run_batch(const SelectSpec* specs, int n, cudaStream_t stream) {
  for (int b0 = 0; b0 < n; b0 += kMaxSelBatch) {
    const int nb = std::min(kMaxSelBatch, n - b0);
    int T_max = 0;
    for (int i = 0; i < nb; ++i) T_max = std::max(T_max, specs[b0 + i].T);
    const int nc = T_max <= kSelSingleMaxT ? 1 : kSelClusterCtas;
    int unused;
    const int bits = select_smem(((T_max + nc - 1) / nc + 15) & ~15, nc, 13, 0, &unused) <= kSelSmemMax ? 13 : 11;
    SelectBatch batch;
    memset(&batch, 0, sizeof(batch));
    size_t smem = 0;
    for (int i = 0; i < nb; ++i) {
      SelectArgs a = make_select_args(specs[b0 + i]);
      a.chunk = ((a.T + nc - 1) / nc + 15) & ~15;
      smem = std::max(smem, select_smem(a.chunk, nc, bits, a.steps.n_steps, &a.s_in_smem));
      batch.t[i] = a;
    }
    void (*kern)(SelectBatch) = nc == 1      ? select_kernel<1, 1024, 13>
                                : bits == 13 ? select_kernel<kSelClusterCtas, kSelThreads, 13>
                                             : select_kernel<kSelClusterCtas, kSelThreads, 11>;
    cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kern), (int)smem);
    if (e == cudaSuccess)
      e = nc == 1 ? launch_kernel(kern, dim3(nb), dim3(1024), smem, stream, batch, true)
                  : launch_cluster(kern, dim3(nc * nb), dim3(kSelThreads), nc, smem, stream, batch, true);
    if (e != cudaSuccess) {
      set_last_cuda_error(e);
      return STEPKV_ECUDA;
    }
  }
  return STEPKV_OK;
}

stepkv_status_t select_run(const float* T_in, const unsigned long long* t_acc, double acc_to_T, int T,
                           const int32_t* step_id, const uint8_t* prot, const stepkv_steps_t& steps,
                           const stepkv_params_t& params, const stepkv_budget_t& budget,
                           const stepkv_select_out_t& out, void* ws, int32_t* status, cudaStream_t stream) {
  const SelectSpec sp{T_in, t_acc, acc_to_T, T, step_id, prot, steps, params, budget, out, ws, status};
  return select_run_batch(&sp, 1, stream);
}

}  // namespace stepkv
