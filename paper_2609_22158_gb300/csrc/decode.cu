// Decode attention over the compacted cache: after a compression boundary the agent keeps decoding,
// and every new token attends to the retained rows C_hat = C_prot || C_traj[K] (Eq. 1).  For each
// layer and query head g (KV head g / G):
//   out[g][:] = sum_{j < n} softmax_j( q[g] . K[g/G][j] / sqrt(d) ) V[g/G][j][:]
//
// GB300 design: HBM-bound (the K and V rows are read once per token, 1.08 GB for 32 layers x 8 heads x
// 8272 rows), so the work per row must stay far below what a scheduler issues while the row streams in.
// Both contractions run on the tensor cores, straight from the rows as they lie in memory (tcgen05 would need its
// 128-row operand tiles for the G <= 8 query heads of a pair, and V transposed; mma.sync takes 16 rows, its tensor
// pipe is 20% busy here):
//   S = Q K^T: the heads are the rows of A, 8 keys the columns of B.  A lane's 16-byte vector of a key
//     row is the B fragment of two k-steps; which of the d elements a k-step covers is free as long as
//     Q is loaded the same way.
//   O = P V: the probabilities of 16 keys are A (the accumulator layout of S is already A's layout), a
//     V row vector gives the B fragments of 8 column tiles after one byte permute per two elements.
// The probabilities stay exact to 24 bits: p = hi + mid + lo, three bf16 terms in groups of A's rows (G <= 4: one MMA
// holds all three; G <= 8: two MMAs).  Every MMA starts from a zero accumulator and is added to the running sums with
// fp32 adds, because the tensor core's own accumulation truncates: the output's error against 64-bit values is 3.8e-7
// at 8272 rows (5.2e-7 with fp32 FMAs and a logit rounded before its exponent).
// Each warp copies whole rows (16 keys and values a step) into a ring of its own with cp.async and needs no other
// warp: 13 instructions per key row instead of 79, so the reads bound it.  32 layers x 8 heads x 8272 rows, G = 4:
// 208 -> 164 us (6.6 TB/s, the rate of a large copy); 8 query heads per KV head 449 -> 172 us.  Reading the fragments straight from global
// memory, 64 bytes of each of 8 rows per load, ran at 215 us: full 128-byte lines matter.
//
// Two splits, chosen by the number of (layer, KV head) pairs and keys (decode_plan): each warp streams an equal range
// of the list of all pairs' 16-key blocks, or (few pairs or keys) each pair is split over CTAs whose warps
// interleave its blocks.  A second kernel merges the partial states of a pair in key order (deterministic); where one CTA
// takes a whole pair there is none.
// The number of keys may be read on the device (n_kept of a compaction), so no host sync is needed.
//
// Accumulated attention (the H2O-style token saliency, Sec. 4.2: T_i may come from an existing
// token-level importance estimator): with mass rows given, the first kernel also stores every key's logits, and
// the second (or the pair's one CTA) adds (1/G) sum_g softmax_j(q_g . k_j / sqrt(d)) to mass[j] for each key from the heads' log-sum-exp:
// one writer per element and call, a fixed order over g, so the result is deterministic.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace stepkv {

constexpr int kDecWarps = 8;
constexpr int kDecThreads = kDecWarps * 32;
constexpr int kDecBlock = 16;           // keys per warp step
// Per warp: two stages of 16 key and 16 value rows at d = 128, four at d = 64.  32 layers x 8 heads x 8272 rows, G = 4:
// 168.4 us; 24 KB 171.8; 12 warps of 16 KB 168.0 (and every G > 4 shape 5-7% slower: spills); 6 warps of 32 KB 175.1.
constexpr int kDecRingBytes = 16 << 10;
constexpr int kDecSplitKeys = 512;      // workspace sizing: one partial per 512 keys of a pair

struct DecodeArgs {
  const uint16_t* q[kMaxDecodeLayers];
  const uint16_t* K[kMaxDecodeLayers];
  const uint16_t* V[kMaxDecodeLayers];
  float* out[kMaxDecodeLayers];
  int64_t head_stride;  // elements
  int Hkv;
  int G;
  int pairs;
  int n_groups;         // CTAs per pair (split form)
  int n_warps;          // warps of the launch (stream form), 0: split form
  int chunks;           // accumulated attention: blocks of the merge kernel per pair
  int prefetch;         // split form: decode_prefetch before the wait
  const int32_t* n_dev;
  int n_host;
  int n_cap;
  float c;              // log2(e) / sqrt(d)
  float* part;          // partial states [slot][G][d + 4]: m c, l, -, -, acc[d]
  float* logits;        // [pairs][n_cap][G] (accumulated-attention mode, else NULL): q . k of every key
  float* mass[kMaxDecodeLayers];  // per layer [Hkv][mass_stride]: accumulated attention (+=), or NULL
  int64_t mass_stride;
  int32_t* status;
};

static_assert(sizeof(DecodeArgs) <= 32000, "kernel parameter space");

// early: before the wait (the count may still change, so it must not stay in L1).
__device__ __forceinline__ int decode_n(const DecodeArgs& a, bool early = false) {
  if (!a.n_dev) return a.n_host;
  return early ? __ldcg(a.n_dev) : *a.n_dev;
}

// Keys per CTA of the split form.
__device__ __forceinline__ int decode_share(int n, int groups) {
  return ((n + groups - 1) / groups + kDecBlock - 1) & ~(kDecBlock - 1);
}

// D = A B for one m16n8k16 tile of bf16 operands, from a zero accumulator.
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Two fp32 values as a bf16 pair (lo = x, hi = y), rounded to nearest even.
__device__ __forceinline__ uint32_t bf16x2_rn(float x, float y) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
  return r;
}
// p = hi + mid + lo exactly (24 bits): each term the rounding of what the terms before leave.
__device__ __forceinline__ void split3(float x, float y, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = bf16x2_rn(x, y);
  x -= __uint_as_float(hi << 16);
  y -= __uint_as_float(hi & 0xFFFF0000u);
  mid = bf16x2_rn(x, y);
  x -= __uint_as_float(mid << 16);
  y -= __uint_as_float(mid & 0xFFFF0000u);
  lo = bf16x2_rn(x, y);
}

// Merge the state (m2, l2, acc2) into (m, l, acc), m in log2 units; -inf marks an empty state.
template <int E>
__device__ __forceinline__ void merge_state(float& m, float& l, float (&acc)[E], float m2, float l2,
                                            const float (&acc2)[E]) {
  const float mn = fmaxf(m, m2);
  if (mn == -INFINITY) return;
  const float a = ex2_approx(m - mn), b = ex2_approx(m2 - mn);
  l = l * a + l2 * b;
#pragma unroll
  for (int e = 0; e < E; ++e) acc[e] = acc[e] * a + acc2[e] * b;
  m = mn;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint4 ld_shared16(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}

// A ring stage holds 16 key rows, then 16 value rows, as they lie in memory, with the 16-byte vectors of a row permuted
// (vector ^ mask of the row) so that the fragment reads do not conflict: eight lanes of a key read take four vectors of
// rows r and r + 1, eight lanes of a value read take two vectors of rows r, r + 2, r + 4 and r + 6.
__device__ __forceinline__ int decode_k_swizzle(int row) { return (row & 1) << 2; }
__device__ __forceinline__ int decode_v_swizzle(int row) { return row & 6; }

// One warp's state over the keys of a pair: running maximum of q . k (row `head`), this lane's part of the
// sum, and the weighted values.  acc[s][t] holds elements 64 s + 16 c4 + t and + 8 of row r8 (GP = 4: the hi + lo terms
// in rows 0-3, the mid terms in rows 4-7).
template <int D, int GP>
struct DecodeState {
  static constexpr int NCH = D / 32;    // 16-byte vectors of a key row per lane
  static constexpr int NSET = D / 64;   // 16-byte vectors of a value row per lane
  float m, l;
  uint64_t acc[NSET][8];

  __device__ __forceinline__ void clear() {
    m = -INFINITY;
    l = 0.f;
#pragma unroll
    for (int s = 0; s < NSET; ++s)
#pragma unroll
      for (int t = 0; t < 8; ++t) acc[s][t] = 0ull;
  }

  // Keys kb .. kb + 15 (those at or past k_end masked), their rows in the ring stage `ring` (decode_k_swizzle,
  // decode_v_swizzle).  Returns the logits q . k of keys kb + 8t + 2 c4 + x in s.
  __device__ __forceinline__ void block(uint32_t ring, const uint32_t (&qa)[2 * NCH][2], int kb, int k_end, float c,
                                        int lane, float (&s)[2][2]) {
    const int r8 = lane >> 2, c4 = lane & 3;
    const uint32_t kbase = ring + r8 * (2 * D), kx = decode_k_swizzle(r8);
    const uint32_t vbase = ring + 16 * 2 * D + 2 * c4 * (2 * D);
    // each k-step's product from zero, then fp32 adds as a tree
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      uint64_t x[2 * NCH];
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        const uint4 k = ld_shared16(kbase + t * 16 * D + (((c4 + 4 * i) ^ kx) << 4));
        float d[4];
        mma_16816(d, qa[2 * i][0], qa[2 * i][0], qa[2 * i][1], qa[2 * i][1], k.x, k.y);
        x[2 * i] = f2_pack(d[0], d[1]);
        mma_16816(d, qa[2 * i + 1][0], qa[2 * i + 1][0], qa[2 * i + 1][1], qa[2 * i + 1][1], k.z, k.w);
        x[2 * i + 1] = f2_pack(d[0], d[1]);
      }
#pragma unroll
      for (int w = NCH; w > 0; w >>= 1)
#pragma unroll
        for (int i = 0; i < w; ++i) x[i] = f2_add(x[i], x[i + w]);
      f2_unpack(x[0], s[t][0], s[t][1]);
    }
    if (kb + kDecBlock > k_end) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (kb + 8 * t + 2 * c4 + x >= k_end) s[t][x] = -INFINITY;
    }
    float mb = fmax3(fmaxf(s[0][0], s[0][1]), s[1][0], s[1][1]);
    mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
    mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, 2));
    if (__any_sync(0xffffffffu, mb > m)) {
      const float mn = fmaxf(m, mb);
      const float sc = m == mn ? 1.f : ex2_approx((m - mn) * c);  // (both -inf: no key of this head yet)
      const uint64_t sc2 = f2_pack(sc, sc);
      l *= sc;
#pragma unroll
      for (int s2 = 0; s2 < NSET; ++s2)
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[s2][t] = f2_mul(acc[s2][t], sc2);
      m = mn;
    }
    const float mc = m == -INFINITY ? 0.f : m * c;
    float p[2][2];
    uint32_t ph[2], pm[2], pl[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      p[t][0] = ex2_approx(fmaf(s[t][0], c, -mc));
      p[t][1] = ex2_approx(fmaf(s[t][1], c, -mc));
      split3(p[t][0], p[t][1], ph[t], pm[t], pl[t]);
    }
    l += (p[0][0] + p[0][1]) + (p[1][0] + p[1][1]);
    uint32_t a0 = ph[0], a1 = pm[0], a2 = ph[1], a3 = pm[1];
    if (GP == 4) {
      const bool top = lane < 16;
      a0 = top ? ph[0] : pm[0];
      a1 = top ? pl[0] : 0u;
      a2 = top ? ph[1] : pm[1];
      a3 = top ? pl[1] : 0u;
    }
#pragma unroll
    for (int s2 = 0; s2 < NSET; ++s2) {
      uint32_t v[4][4];  // [key 2 c4, 2 c4 + 1, 2 c4 + 8, 2 c4 + 9][pair of elements]
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int row = (x & 1) + 8 * (x >> 1);  // beyond 2 c4
        const uint4 r = ld_shared16(vbase + row * (2 * D) + (((r8 + 8 * s2) ^ decode_v_swizzle(2 * c4 + row)) << 4));
        v[x][0] = r.x;
        v[x][1] = r.y;
        v[x][2] = r.z;
        v[x][3] = r.w;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const uint32_t sel = (t & 1) ? 0x7632u : 0x5410u;
        const uint32_t b0 = __byte_perm(v[0][t >> 1], v[1][t >> 1], sel), b1 = __byte_perm(v[2][t >> 1], v[3][t >> 1], sel);
        float d[4];
        mma_16816(d, a0, a1, a2, a3, b0, b1);
        uint64_t o = f2_add(f2_pack(d[0], d[1]), f2_pack(d[2], d[3]));
        if (GP == 8) {
          mma_16816(d, pl[0], 0u, pl[1], 0u, b0, b1);
          o = f2_add(o, f2_pack(d[0], d[1]));
        }
        acc[s2][t] = f2_add(acc[s2][t], o);
      }
    }
  }

  // The warp's state written out: m c and l of head g at ml[g * ml_stride + {0, 1}], the values at vals + g * v_stride.
  __device__ __forceinline__ void store(float* ml, int ml_stride, float* vals, int v_stride, float c, int G, int lane) {
    const int r8 = lane >> 2, c4 = lane & 3, head = GP == 4 ? (r8 & 3) : r8;
    float ls = l;
    ls += __shfl_xor_sync(0xffffffffu, ls, 1);
    ls += __shfl_xor_sync(0xffffffffu, ls, 2);
    const bool writes = head < G && (GP == 8 || lane < 16);
#pragma unroll
    for (int s2 = 0; s2 < NSET; ++s2) {
      float x[8], y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        f2_unpack(acc[s2][t], x[t], y[t]);
        if (GP == 4) {
          x[t] += __shfl_xor_sync(0xffffffffu, x[t], 16);
          y[t] += __shfl_xor_sync(0xffffffffu, y[t], 16);
        }
      }
      if (writes) {
        float4* dst = reinterpret_cast<float4*>(vals + head * v_stride + 64 * s2 + 16 * c4);
        dst[0] = make_float4(x[0], x[1], x[2], x[3]);
        dst[1] = make_float4(x[4], x[5], x[6], x[7]);
        dst[2] = make_float4(y[0], y[1], y[2], y[3]);
        dst[3] = make_float4(y[4], y[5], y[6], y[7]);
      }
    }
    if (writes && c4 == 0) {
      ml[head * ml_stride] = ls == ls ? m * c : INFINITY;  // a NaN sum is not to be merged as an empty state (all logits NaN)
      ml[head * ml_stride + 1] = ls;
    }
  }
};

// A head's weighted value over its sum l: 0 without keys (l = 0), NaN where a logit is one or +inf (l is NaN).  The one
// expression of every form: the output is the same bit for bit with and without accumulated attention.
__device__ __forceinline__ float decode_quotient(float v, float l) { return l > 0.f ? v / l : v * l; }

// Element e of a head's output.  The three terms of a probability do not add up to an infinity when they multiply an
// infinite value (a term may be zero or negative): a NaN whose weights are numbers is replaced by what the infinities
// among the values say, and stays one where they are of both signs or a value is itself a NaN.
template <int D>
__device__ __forceinline__ float decode_output(float o, float l, const uint16_t* Vh, int n, int e) {
  if (o == o || !(l < INFINITY)) return o;
  bool pos = false, neg = false;
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const uint32_t w = Vh[(size_t)j * D + e];
    if ((w & 0x7F80u) != 0x7F80u) continue;
    if (w & 0x7Fu) return o;
    (w >> 15 ? neg : pos) = true;
  }
  return pos == neg ? o : pos ? INFINITY : -INFINITY;
}

// The last warp of a split-form CTA sends for the first 32 KB of the CTA's keys and of its values into L2 while the kernel
// before it finishes: with a call per layer that is the merge of the layer before, which leaves DRAM idle for ~3 us.  L2
// holds what memory holds, so rows still being written are read right after the wait; the number of keys may still
// change, so here it only tells where the share probably lies.  8 heads x 8272 rows, calls in a row: 13.7 -> 13.0 us (64
// KB or the whole share: no better), with another kernel between them 14.9 -> 15.0; 32 layers in a captured step 393 ->
// 368 us (307 with the merge's dry run).
// Only where the CTAs fill half the machine and have more rows than their rings (else the reads are short, and the warp
// that prefetches starts late: 1500 rows, 32 CTAs, another kernel between the calls 8.9 -> 9.3 us; 548 rows 5.9 -> 6.9),
// and not with accumulated attention, whose mass blocks read in that gap (one layer 22.9 -> 24.4 us).
constexpr int kDecPrefetchBytes = 32 << 10;
template <int D>
__device__ __forceinline__ void decode_prefetch(const DecodeArgs& a) {
  constexpr int kPieces = 16;  // per tensor
  const int t = (int)threadIdx.x - (kDecThreads - 2 * kPieces);
  if (t < 0) return;
  const int n = max(0, min(decode_n(a, true), a.n_cap));
  const int pair = blockIdx.x / a.n_groups, grp = blockIdx.x - pair * a.n_groups;
  const int layer = pair / a.Hkv, h = pair - layer * a.Hkv;
  const int share = decode_share(n, a.n_groups);
  const int k_begin = min(n, grp * share);
  const int rows = min(min(n - k_begin, share), kDecPrefetchBytes / (2 * D));
  const int per = (rows + kPieces - 1) / kPieces, r0 = min(rows, (t >> 1) * per), r1 = min(rows, r0 + per);
  const uint16_t* base = ((t & 1) ? a.V[layer] : a.K[layer]) + (size_t)h * a.head_stride;
  if (r1 > r0) bulk_prefetch_l2(base + (size_t)(k_begin + r0) * D, (uint32_t)(r1 - r0) * 2 * D);
}

// Adds the group-mean softmax weight of keys [j0, j1) of a pair to its masses, from the stored logits and the heads'
// log-sum-exp (one writer per key).  A chain of L2 loads, so four keys of a thread go at a time (25 layers x 32 heads x 1500
// rows, G = 1: 115.8 -> 106.7 us).
__device__ __forceinline__ void decode_add_mass(const DecodeArgs& a, int pair, const float* s_lse, int j0, int j1) {
  const int layer = pair / a.Hkv, h = pair - layer * a.Hkv, G = a.G;
  const float inv_G = 1.f / (float)G;
  float* mrow = a.mass[layer] + (size_t)h * a.mass_stride;
  const float* lg = a.logits + (size_t)pair * a.n_cap * G;
  constexpr int U = 4;  // keys of a thread in flight
#pragma unroll 1
  for (int j = j0 + (int)threadIdx.x; j < j1; j += U * (int)blockDim.x) {
    float sum[U], was[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      sum[u] = 0.f;
      was[u] = j + u * (int)blockDim.x < j1 ? mrow[j + u * (int)blockDim.x] : 0.f;
    }
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = j + u * (int)blockDim.x < j1 ? __ldcg(lg + (size_t)(j + u * (int)blockDim.x) * G + g) : 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u) sum[u] += ex2_approx(fmaf(x[u], a.c, -s_lse[g]));
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j + u * (int)blockDim.x < j1) mrow[j + u * (int)blockDim.x] = was[u] + sum[u] * inv_G;
  }
}
__device__ __forceinline__ float decode_lse(float m, float l) { return l > 0.f ? m + __log2f(l) : INFINITY; }

// GP: head rows per group of A's rows, 4 (G <= 4: three split terms in one MMA) or 8 (two MMAs).
// MASS: the accumulated-attention variant (a separate instantiation, so the plain decode keeps its registers).
// FORM kStream: each warp streams an equal contiguous range of the list of all pairs' 16-key blocks and leaves a partial state
// per pair it touches (slot warp + pair).  kSplit: n_groups CTAs of their own work on each pair and leave a partial state
// each.  kSplitSmall: one CTA per pair with 4, 2 or 1 warps, several on an SM, where there are more pairs than SMs.  A merge
// kernel joins the states and adds to the masses; one CTA per pair does both itself (64 layers x 8 heads x 64 rows with
// masses, G = 4: 17.0 -> 14.1 us, 300 rows 30.9 -> 28.4).
enum DecodeForm { kStream, kSplit, kSplitSmall };
constexpr int kDecSmallWarps = 4;  // of a kSplitSmall CTA at most
// Warps an SM holds of kSplitSmall: 12 rings of 16 KB and 168 registers, 8 with the registers of 8 query heads at d = 128.
constexpr int decode_small_warps_per_sm(int D, int GP) { return D == 128 && GP == 8 ? 8 : 12; }
template <int D, int GP, bool MASS, DecodeForm FORM>
__global__ void __launch_bounds__(FORM == kSplitSmall ? kDecSmallWarps * 32 : kDecThreads,
                                  FORM == kSplitSmall ? decode_small_warps_per_sm(D, GP) / kDecSmallWarps : 1)
decode_kernel(const __grid_constant__ DecodeArgs a) {
  using State = DecodeState<D, GP>;
  const int NW = FORM == kSplitSmall ? (int)(blockDim.x >> 5) : kDecWarps, NT = NW * 32;
  constexpr int NCH = State::NCH;
  constexpr int kStageBytes = 2 * kDecBlock * D * 2;
  constexpr int kStages = kDecRingBytes / kStageBytes;
  extern __shared__ __align__(16) uint8_t dec_smem[];     // per-warp rings

  if constexpr (FORM == kSplit && !MASS)
    if (a.prefetch) decode_prefetch<D>(a);
  pdl_wait();
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r8 = lane >> 2, c4 = lane & 3;                // fragment row (or column) and position in it
  const int head = GP == 4 ? (r8 & 3) : r8;               // the head of this lane's rows r8 and r8 + 8
  const int G = a.G;
  const float c = a.c;
  int n = decode_n(a);
  if (n > a.n_cap) {
    if (threadIdx.x == 0 && blockIdx.x == 0) record_status(a.status, STEPKV_ENOSPACE);
    n = a.n_cap;
  }
  if (n < 1) {
    if (threadIdx.x == 0 && blockIdx.x == 0) record_status(a.status, STEPKV_EDATA);
    n = 0;
  }
  uint8_t* my_ring = dec_smem + warp * kDecRingBytes;
  const uint32_t ring0 = smem_u32(my_ring);
  // A warp copies whole rows (256 or 128 consecutive bytes each); rows past `last` are read as row `last` (in range,
  // finite) and their probabilities set to zero.
  constexpr int VPR = D / 8, RPI = 32 / VPR;              // vectors per row, rows per copy instruction
  const int cp_row = lane / VPR, cp_vec = lane & (VPR - 1);
  auto issue = [&](uint32_t dst, const uint16_t* Kh, const uint16_t* Vh, int kb, int last) {
#pragma unroll
    for (int i = 0; i < kDecBlock / RPI; ++i) {
      const int row = i * RPI + cp_row;
      const size_t src = (size_t)min(kb + row, last) * D + cp_vec * 8;
      cp_async16(dst + row * (2 * D) + ((cp_vec ^ decode_k_swizzle(row)) << 4), Kh + src);
      cp_async16(dst + (16 + row) * (2 * D) + ((cp_vec ^ decode_v_swizzle(row)) << 4), Vh + src);
    }
  };
  // A fragments of Q: k-step 2i + x covers elements 4x .. 4x + 3 of every lane's vector c4 + 4i (rows r8 and r8 + 8
  // hold the same head, so a1 = a0 and a3 = a2)
  uint32_t qa[2 * NCH][2];
  auto load_q = [&](int layer, int h) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (head < G) v = __ldg(reinterpret_cast<const uint4*>(a.q[layer] + (size_t)(h * G + head) * D) + c4 + 4 * i);
      qa[2 * i][0] = v.x;
      qa[2 * i][1] = v.y;
      qa[2 * i + 1][0] = v.z;
      qa[2 * i + 1][1] = v.w;
    }
  };
  auto store_logits = [&](int pair, int kb, int k_end, const float (&s)[2][2]) {
    if (head >= G || (GP == 4 && lane >= 16)) return;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int j = kb + 8 * t + 2 * c4 + x;
        if (j < k_end) a.logits[((size_t)pair * a.n_cap + j) * G + head] = s[t][x];
      }
  };
  State st;
  st.clear();

  if constexpr (FORM == kStream) {
    const int nb = (n + kDecBlock - 1) / kDecBlock;       // blocks per pair
    const int total = a.pairs * nb;
    const int per = (total + a.n_warps - 1) / a.n_warps;
    const int w = blockIdx.x * NW + warp;
    const int lo = min(total, w * per), hi = min(total, lo + per);
    if (lo >= hi) return;
    // the copies run kStages blocks ahead of the arithmetic, across pair boundaries
    int i_pair = lo / nb, i_kb = (lo - i_pair * nb) * kDecBlock, i_left = hi - lo;
    const uint16_t *Kh, *Vh;
    auto bases = [&](int pair) {
      const int layer = pair / a.Hkv, h = pair - layer * a.Hkv;
      Kh = a.K[layer] + (size_t)h * a.head_stride;
      Vh = a.V[layer] + (size_t)h * a.head_stride;
    };
    bases(i_pair);
    auto issue_next = [&](uint32_t dst) {
      if (i_left > 0) {
        issue(dst, Kh, Vh, i_kb, n - 1);
        --i_left;
        i_kb += kDecBlock;
        if (i_kb >= n && i_left > 0) {
          i_kb = 0;
          bases(++i_pair);
        }
      }
      cp_async_commit();
    };
    int pair = i_pair, kb = i_kb, stage = 0;
#pragma unroll
    for (int s = 0; s < kStages; ++s) issue_next(ring0 + s * kStageBytes);
    load_q(pair / a.Hkv, pair - pair / a.Hkv * a.Hkv);
    for (int left = hi - lo;;) {
      cp_async_wait<kStages - 1>();
      __syncwarp();
      float s[2][2];
      const uint32_t ring = ring0 + stage * kStageBytes;
      st.block(ring, qa, kb, n, c, lane, s);
      __syncwarp();
      issue_next(ring);
      if (MASS) store_logits(pair, kb, n, s);
      stage = stage + 1 == kStages ? 0 : stage + 1;
      kb += kDecBlock;
      --left;
      if (kb >= n || left == 0) {
        float* dst = a.part + (size_t)(w + pair) * G * (D + 4);
        st.store(dst, D + 4, dst + 4, D + 4, c, G, lane);
        if (left == 0) break;
        st.clear();
        ++pair;
        kb = 0;
        load_q(pair / a.Hkv, pair - pair / a.Hkv * a.Hkv);
      }
    }
  } else {
    __shared__ float s_ml[FORM == kSplitSmall ? kDecSmallWarps : kDecWarps][GP][2], s_lse[GP];
    const int pair = blockIdx.x / a.n_groups, grp = blockIdx.x - pair * a.n_groups;
    const int layer = pair / a.Hkv, h = pair - layer * a.Hkv;
    const int share = decode_share(n, a.n_groups);
    const int k_begin = min(n, grp * share), k_end = min(n, k_begin + share);
    const uint16_t* Kh = a.K[layer] + (size_t)h * a.head_stride;
    const uint16_t* Vh = a.V[layer] + (size_t)h * a.head_stride;
    int kb = k_begin + warp * kDecBlock, i_kb = kb, stage = 0;
    auto issue_next = [&](uint32_t dst) {
      if (i_kb < k_end) issue(dst, Kh, Vh, i_kb, k_end - 1);
      i_kb += NW * kDecBlock;
      cp_async_commit();
    };
#pragma unroll
    for (int s = 0; s < kStages; ++s) issue_next(ring0 + s * kStageBytes);
    load_q(layer, h);
    for (; kb < k_end; kb += NW * kDecBlock) {
      cp_async_wait<kStages - 1>();
      __syncwarp();
      float s[2][2];
      const uint32_t ring = ring0 + stage * kStageBytes;
      st.block(ring, qa, kb, k_end, c, lane, s);
      __syncwarp();
      issue_next(ring);
      if (MASS) store_logits(pair, kb, k_end, s);
      stage = stage + 1 == kStages ? 0 : stage + 1;
    }
    cp_async_wait<0>();
    __syncwarp();
    st.store(&s_ml[warp][0][0], 2, reinterpret_cast<float*>(my_ring), D, c, G, lane);  // the ring is empty now
    __syncthreads();
    // the warps merged in order, four elements of one head per thread
    constexpr int V4 = D / 4;
    for (int t = threadIdx.x; t < G * V4; t += NT) {
      const int g = t / V4, e0 = (t - g * V4) * 4;
      float mm = -INFINITY, ll = 0.f, aa[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll (FORM == kSplitSmall ? 1 : kDecWarps)
      for (int w = 0; w < NW; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(dec_smem + w * kDecRingBytes) + g * D + e0);
        const float a2[4] = {v.x, v.y, v.z, v.w};
        merge_state<4>(mm, ll, aa, s_ml[w][g][0], s_ml[w][g][1], a2);
      }
      if (a.n_groups == 1) {
        float o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = decode_output<D>(decode_quotient(aa[e], ll), ll, Vh, n, e0 + e);
        *reinterpret_cast<float4*>(a.out[layer] + (size_t)(h * G + g) * D + e0) = make_float4(o[0], o[1], o[2], o[3]);
      } else {
        float* dst = a.part + ((size_t)blockIdx.x * G + g) * (D + 4);
        if (e0 == 0) {
          dst[0] = mm;
          dst[1] = ll;
        }
        *reinterpret_cast<float4*>(dst + 4 + e0) = make_float4(aa[0], aa[1], aa[2], aa[3]);
      }
      if (MASS && e0 == 0) s_lse[g] = decode_lse(mm, ll);
    }
    if constexpr (MASS) {
      if (a.n_groups == 1) {
        __syncthreads();  // also: this CTA's logits are written
        decode_add_mass(a, pair, s_lse, 0, n);
      }
    }
  }
}

// The partial slots of a pair, in key order: of the stream form those of the warps whose ranges reach into the pair,
// else its CTAs' (all of them, empty shares included, so that the number of keys need not be read first).
__device__ __forceinline__ void decode_slots(const DecodeArgs& a, int pair, int& first, int& count, bool early = false) {
  if (a.n_warps == 0) {
    first = pair * a.n_groups;
    count = a.n_groups;
    return;
  }
  const int n = max(0, min(decode_n(a, early), a.n_cap));
  const int nb = (n + kDecBlock - 1) / kDecBlock;
  const int per = (a.pairs * nb + a.n_warps - 1) / a.n_warps;
  first = count = 0;
  if (nb == 0) return;
  const int w0 = pair * nb / per, w1 = ((pair + 1) * nb - 1) / per;
  first = w0 + pair;
  count = w1 - w0 + 1;
}

// Merge of the partial states.  Blocks [0, pairs * G) take one (pair, head) each: warp w merges slots w, w + 4, ... in
// order, then the warps meet in order, and out = acc / l.  With accumulated attention,
// `chunks` more blocks per pair each take a contiguous share of the keys: the heads' log-sum-exp from all slots, then
// the group-mean softmax mass of every key of the share is added (one writer per key).
// A merge is a chain of latencies of code that runs once, and its blocks lie idle while the decode kernel works: so a
// block first goes through it without its loads and its store (but for one load, for the address translation), which
// brings in the code and the parameters, and only then waits.  And the loads of a warp's next four slots are in flight
// before the first is merged.  One layer of 8 heads x 8272 rows, calls in a row: 13.0 -> 10.1 us, with another kernel
// between them 15.0 -> 12.6; 4240 rows 10.3 -> 8.2; 2 heads x 16000 rows 9.2 -> 8.2; 8 layers 50.9 -> 48.5; 32 layers 168.8
// -> 168.2.  (Eight slots: 9.7, but 8 query heads or fewer rows slower, 32 layers 170.5.  An unrolled loop left to the
// compiler: 10.8-11.5, 2 heads up to 10.9.)  With accumulated attention the blocks are too many to lie idle (one layer
// 22.6 -> 24.1 us with the dry run), so those wait at once.
constexpr int kDecMergeThreads = 128;

template <int D, bool MASS>
__global__ void __launch_bounds__(kDecMergeThreads) decode_merge_kernel(const __grid_constant__ DecodeArgs a) {
  constexpr int PER = D / 32, NW = kDecMergeThreads / 32, kSlotsInFlight = 4;
  __shared__ float s_ml[NW][2];
  __shared__ float s_v[NW][D];
  __shared__ float s_lse[8];
  const int G = a.G, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = (int)blockIdx.x;
  int first, count;
  if (!MASS || item < a.pairs * G) {
    const int pair = item / G, g = item - pair * G;
    const int layer = pair / a.Hkv, h = pair - layer * a.Hkv;
#pragma unroll 1
    for (int rep = MASS ? 1 : 0; rep < 2; ++rep) {
      const bool live = MASS || rep == 1;
      if (live) {
        pdl_wait();
        pdl_launch_dependents();
      }
      decode_slots(a, pair, first, count, !live);
      float mm = -INFINITY, ll = 0.f, aa[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) aa[e] = 0.f;
      if (!live && lane == 0) s_ml[warp][0] = __ldcg(a.part);
#pragma unroll 1
      for (int i0 = warp; i0 < count; i0 += kSlotsInFlight * NW) {
        float2 ml[kSlotsInFlight];
        float a2[kSlotsInFlight][PER];
#pragma unroll
        for (int u = 0; u < kSlotsInFlight; ++u) {
          const float* src = a.part + ((size_t)(first + i0 + u * NW) * G + g) * (D + 4);
          const bool ok = live && i0 + u * NW < count;
          ml[u] = ok ? __ldcg(reinterpret_cast<const float2*>(src)) : make_float2(-INFINITY, 0.f);
#pragma unroll
          for (int e = 0; e < PER; ++e) a2[u][e] = ok ? __ldcg(src + 4 + e * 32 + lane) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kSlotsInFlight; ++u) merge_state<PER>(mm, ll, aa, ml[u].x, ml[u].y, a2[u]);
      }
      if (lane == 0) {
        s_ml[warp][0] = mm;
        s_ml[warp][1] = ll;
      }
#pragma unroll
      for (int e = 0; e < PER; ++e) s_v[warp][e * 32 + lane] = aa[e];
      __syncthreads();
      if ((int)threadIdx.x < D) {
        float m1 = -INFINITY, l1 = 0.f, v1[1] = {0.f};
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float v2[1] = {s_v[w][threadIdx.x]};
          merge_state<1>(m1, l1, v1, s_ml[w][0], s_ml[w][1], v2);
        }
        float* out = a.out[layer] + (size_t)(h * G + g) * D + threadIdx.x;
        const float o = decode_quotient(v1[0], l1);
        if (live) {
          const uint16_t* Vh = a.V[layer] + (size_t)h * a.head_stride;
          *out = decode_output<D>(o, l1, Vh, max(0, min(decode_n(a), a.n_cap)), (int)threadIdx.x);
        }
      }
      __syncthreads();
    }
    return;
  }
  pdl_wait();
  pdl_launch_dependents();
  const int rest = item - a.pairs * G, pair = rest / a.chunks, chunk = rest - pair * a.chunks;
  decode_slots(a, pair, first, count);
  for (int g = warp; g < G; g += NW) {
    float mm = -INFINITY, ll = 0.f, none[1] = {0.f};
    for (int i = lane; i < count; i += 32) {
      const float2 ml = __ldcg(reinterpret_cast<const float2*>(a.part + ((size_t)(first + i) * G + g) * (D + 4)));
      merge_state<1>(mm, ll, none, ml.x, ml.y, none);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, mm, o), l2 = __shfl_xor_sync(0xffffffffu, ll, o);
      merge_state<1>(mm, ll, none, m2, l2, none);
    }
    if (lane == 0) s_lse[g] = decode_lse(mm, ll);
  }
  __syncthreads();
  const int n = max(0, min(decode_n(a), a.n_cap));
  const int per = (n + a.chunks - 1) / a.chunks;
  const int j0 = chunk * per;
  decode_add_mass(a, pair, s_lse, j0, min(n, j0 + per));
}

size_t decode_ws_bytes(int n_layers, int Hkv, int Hq, int d, int n_cap) {
  const int n_splits = std::max(1, (n_cap + kDecSplitKeys - 1) / kDecSplitKeys);
  return (size_t)n_layers * Hq * n_splits * (d + 4) * sizeof(float);
}

size_t decode_mass_ws_bytes(int n_layers, int Hkv, int Hq, int d, int n_cap) {
  // partials (256-byte aligned), then the key logits of every head
  const size_t part = (decode_ws_bytes(n_layers, Hkv, Hq, d, n_cap) + 255) & ~(size_t)255;
  return part + (size_t)n_layers * Hq * std::max(1, n_cap) * sizeof(float);
}

// How a launch splits `pairs` (layer, KV head) pairs of up to n_cap keys.  The stream form balances every SM and fills
// its ring once, but a warp must have blocks enough to be worth a partial state, and the workspace holds
// pairs x ceil(n_cap / 512) of them: it is taken where that allows three quarters of the machine's warps.  Else each pair
// is split over as many CTAs as one wave and the workspace hold: one layer of 8 heads x 8272 rows takes 9.6 us per call
// in a captured step (27.3 us with 512-key splits and 16-byte loads into registers; a cluster of 16 CTAs per pair with
// the merge through distributed shared memory 24 us, since only 7 such clusters fit at a time; the last CTA of a pair
// merging, found by an atomic count, 18.5 us).
// More pairs than SMs, and too few keys to stream: CTAs of four, two or one warps, the most with which all of them run at
// once.  Eight warps a CTA hold an SM to themselves: 64 layers x 32 heads x 64 rows, G = 1: 45.0 -> 21.1 us; 40 layers x 32
// heads x 300 rows 51.3 -> 37.8; 40 layers x 8 heads x 300 rows, G = 4: 19.9 -> 15.6; 20 layers x 8 heads x 2500 rows 47.6
// -> 42.8 (the CUDA-core kernel with 512-key splits: 21.6, 42.8, 23.7, 57.2).  Where not even one-warp CTAs run at once, four
// warps are the best for longer pairs (2048 pairs x 512 rows: 86 us, two warps 90, one 103) and two for shorter (x 150:
// 37.5, 35.2, 37.2).
struct DecodePlan {
  int n_warps;       // > 0: stream form with that many warps
  int groups;        // else CTAs per pair
  int small;         // > 0: one CTA per pair, of that many warps (kSplitSmall)
};
static DecodePlan decode_plan(int pairs, int n_cap, int n_sm, int small_warps_per_sm) {
  DecodePlan p{0, 1, 0};
  const int splits = std::max(1, (n_cap + kDecSplitKeys - 1) / kDecSplitKeys);  // partial slots per pair
  // stream form: warps + pairs slots
  const int warps = std::min(n_sm * kDecWarps, pairs * (splits - 1) / kDecWarps * kDecWarps);
  if (warps >= n_sm * kDecWarps * 3 / 4) p.n_warps = warps;
  else if (pairs <= n_sm) p.groups = std::min(splits, n_sm / pairs);
  else if (pairs > n_sm * small_warps_per_sm) p.small = n_cap > 256 ? 4 : 2;
  else
    for (p.small = kDecSmallWarps; n_sm * (small_warps_per_sm / p.small) < pairs;) p.small /= 2;
  return p;
}

template <int D, int GP, bool MASS, DecodeForm FORM>
static cudaError_t decode_launch(const DecodeArgs& a, int warps, cudaStream_t stream) {
  void (*kern)(DecodeArgs) = decode_kernel<D, GP, MASS, FORM>;
  const int smem = warps * kDecRingBytes;
  const int grid = FORM == kStream ? a.n_warps / kDecWarps : a.pairs * a.n_groups;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kern), smem);
  // Both kernels launch dependently (each waits for the one before it before it uses anything that may still be
  // written): a captured decode step of 32 one-layer calls took 390 us when neither did anything before its wait, 406
  // with the first launched plainly, 541 with both; with the prefetch and the merge's dry run it takes 307.
  if (e == cudaSuccess) e = launch_kernel(kern, dim3(grid), dim3(warps * 32), smem, stream, a, true);
  if (e != cudaSuccess || (FORM != kStream && a.n_groups == 1)) return e;
  const int blocks = a.pairs * (a.G + (MASS ? a.chunks : 0));
  return launch_kernel(decode_merge_kernel<D, MASS>, dim3(blocks), dim3(kDecMergeThreads), 0, stream, a, true);
}

template <int D, int GP, bool MASS>
static cudaError_t decode_dispatch_form(const DecodeArgs& a, int small, cudaStream_t stream) {
  if (a.n_warps > 0) return decode_launch<D, GP, MASS, kStream>(a, kDecWarps, stream);
  return small > 0 ? decode_launch<D, GP, MASS, kSplitSmall>(a, small, stream)
                   : decode_launch<D, GP, MASS, kSplit>(a, kDecWarps, stream);
}
template <int D, int GP>
static cudaError_t decode_dispatch(const DecodeArgs& a, int small, cudaStream_t stream) {
  return a.logits ? decode_dispatch_form<D, GP, true>(a, small, stream) : decode_dispatch_form<D, GP, false>(a, small, stream);
}

stepkv_status_t decode_run(int n_layers, const void* const* q, const void* const* K, const void* const* V,
                           int64_t head_stride, int Hkv, int Hq, int d, const int32_t* n_dev, int n_host, int n_cap,
                           float* const* out, void* ws, int32_t* status, cudaStream_t stream, float* const* mass,
                           int64_t mass_stride) {
  const int G = Hq / Hkv;
  int n_sm = 0;
  cudaError_t e = device_sm_count(&n_sm);
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return STEPKV_ECUDA;
  }
  float* part = static_cast<float*>(ws);
  float* logits = nullptr;
  if (mass != nullptr)  // after one launch's partial states, as decode_mass_ws_bytes has it
    logits = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) +
                                      ((decode_ws_bytes(std::min(n_layers, kMaxDecodeLayers), Hkv, Hq, d, n_cap) + 255) &
                                       ~(size_t)255));
  for (int l0 = 0; l0 < n_layers; l0 += kMaxDecodeLayers) {
    const int nl = std::min(kMaxDecodeLayers, n_layers - l0);
    DecodeArgs a;
    memset(&a, 0, sizeof(a));
    for (int l = 0; l < nl; ++l) {
      a.q[l] = static_cast<const uint16_t*>(q[l0 + l]);
      a.K[l] = static_cast<const uint16_t*>(K[l0 + l]);
      a.V[l] = static_cast<const uint16_t*>(V[l0 + l]);
      a.out[l] = out[l0 + l];
      a.mass[l] = mass != nullptr ? mass[l0 + l] : nullptr;
    }
    a.logits = logits;  // the chunk's pairs index their own slice of the logit scratch from 0
    a.mass_stride = mass_stride;
    a.head_stride = head_stride;
    a.Hkv = Hkv;
    a.G = G;
    const DecodePlan p = decode_plan(nl * Hkv, n_cap, n_sm, decode_small_warps_per_sm(d, G <= 4 ? 4 : 8));
    a.pairs = nl * Hkv;
    a.n_groups = p.groups;
    a.n_warps = p.n_warps;
    a.prefetch = p.small == 0 && 2 * a.pairs * p.groups >= n_sm && (int64_t)(n_cap / p.groups) * (4 * d) > kDecWarps * kDecRingBytes;
    a.chunks = std::max(1, std::min(8, (n_cap + 1023) / 1024));
    a.n_dev = n_dev;
    a.n_host = n_host;
    a.n_cap = n_cap;
    a.c = (float)(1.4426950408889634 / sqrt((double)d));
    a.part = part;
    a.status = status;
    if (d == 128)
      e = G <= 4 ? decode_dispatch<128, 4>(a, p.small, stream) : decode_dispatch<128, 8>(a, p.small, stream);
    else
      e = G <= 4 ? decode_dispatch<64, 4>(a, p.small, stream) : decode_dispatch<64, 8>(a, p.small, stream);
    if (e != cudaSuccess) {
      set_last_cuda_error(e);
      return STEPKV_ECUDA;
    }
  }
  return STEPKV_OK;
}

}  // namespace stepkv
