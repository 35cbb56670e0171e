// Drafting and pruning (Sec. 4.4.2 "Drafting Source", Sec. 4.4.4 "Draft Graph
// Pruning"): from the target distribution of the current block build the draft
// blocks that the next verification step will score.
//
//   draft_topk_kernel   per (row, vocabulary slice) of a still-masked position:
//                       the K largest logits with their token ids (value desc,
//                       id asc), the slice maximum and sum of exponentials.  A
//                       slice is held in registers, like in the decision step.
//   draft_build_kernel  one CTA per sequence: merges the slices into the K
//                       candidates c_ij and probabilities of every position,
//                       ranks the positions (Eq. token-position-sort), builds
//                       every draft formula, scores it by geometric means,
//                       keeps the D* best and writes their blocks and parent
//                       lists.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace spiffy {
namespace {

constexpr int kThreads = 128;  // top-k kernel
constexpr int kVecs = 8;       // 128-bit vectors per thread
constexpr int kMaxK = 4;       // vocabulary ranks
constexpr int kBuildThreads = 1024;  // a warp per block position
constexpr int kRelated = 64;         // formulas whose subset relation fits its table
constexpr int kAtHand = 4;
constexpr int kFormulaBytes = 4096;  // shared memory for what is known about so many
constexpr int kGraphInts = 6144;     // shared-memory copy of the draft graph (24 KB)

struct __align__(16) TopPartial {
  float m, s;          // slice maximum, sum of exp(x - m)
  float val[kMaxK];    // the K largest values, -inf when the slice has fewer
  int idx[kMaxK];      // their token ids
  int pad[2];
};

// The maximum over the warp's lanes, on every lane (NaN loses).
__device__ __forceinline__ float warp_max(float x) {
  float m;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}

// (value desc, id asc): is (v2, i2) ahead of (v1, i1)?
__device__ __forceinline__ bool ahead(float v2, int i2, float v1, int i1) {
  return v2 > v1 || (v2 == v1 && i2 < i1);
}

template <typename T>
struct Unpack;
template <>
struct Unpack<__nv_bfloat16> {
  static constexpr int kPerVec = 8;
  static __device__ __forceinline__ void get(uint4 v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  static __device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
};
template <>
struct Unpack<float> {
  static constexpr int kPerVec = 4;
  static __device__ __forceinline__ void get(uint4 v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  static __device__ __forceinline__ float load1(const float* p) { return *p; }
};

// grid = (slices, B*L rows), 128 threads.
template <typename T>
__global__ void __launch_bounds__(kThreads)
draft_topk_kernel(const T* __restrict__ logits, int64_t row_stride, int V, int64_t chunk,
                  int splits, int K, const int32_t* __restrict__ state, int mask_id,
                  TopPartial* __restrict__ partials, int32_t* __restrict__ clear_status, int L) {
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();
  pdl_launch_dependents();  // the build kernel (one CTA per sequence) may take its SM and stage the graph
#endif
  const int row = blockIdx.y;
  if (clear_status && blockIdx.x == 0 && threadIdx.x == 0 && row % L == 0) clear_status[row / L] = 0;
  if (state[row] != mask_id) return;
  const int split = blockIdx.x;
  const int64_t begin = (int64_t)split * chunk;
  const int64_t end = min((int64_t)V, begin + chunk);
  constexpr int EPV = Unpack<T>::kPerVec;
  const T* base = logits + (int64_t)row * row_stride;
  const int nvec = begin < end ? (int)((end - begin) / EPV) : 0;
  const int ntail = begin < end ? (int)(end - begin) - nvec * EPV : 0;
  const uint4* p = reinterpret_cast<const uint4*>(base + begin);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // the thread's elements: vectors t, t + 128, ..., then (thread 0) the ragged tail
  constexpr int NE = kVecs * EPV + EPV;
  float x[NE];
#pragma unroll
  for (int u = 0; u < kVecs; ++u) {
    float f[EPV];
    if (tid + u * kThreads < nvec) {
      Unpack<T>::get(ld_stream(p + tid + u * kThreads), f);
    } else {
#pragma unroll
      for (int e = 0; e < EPV; ++e) f[e] = -INFINITY;
    }
#pragma unroll
    for (int e = 0; e < EPV; ++e) x[u * EPV + e] = f[e];
  }
#pragma unroll
  for (int e = 0; e < EPV; ++e)
    x[kVecs * EPV + e] =
        (tid == 0 && e < ntail) ? Unpack<T>::load1(base + begin + (int64_t)nvec * EPV + e) : -INFINITY;
  // The largest element of every vector: a round then looks at these, and only the thread that
  // holds the winner looks into the vector it lies in.
  constexpr int kGroups = kVecs + 1;
  float top[kGroups];
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    top[u] = x[u * EPV];
#pragma unroll
    for (int e = 1; e < EPV; ++e) top[u] = fmaxf(top[u], x[u * EPV + e]);
  }
  auto largest = [&]() {  // NaN loses
    float t = -INFINITY;
#pragma unroll
    for (int u = 0; u < kGroups; ++u) t = fmaxf(t, top[u]);
    return t;
  };
  __shared__ float w_max[kThreads / 32], w_sum[kThreads / 32];
  __shared__ float w_val[kThreads / 32][kMaxK];
  __shared__ int w_idx[kThreads / 32][kMaxK];
  float tv = largest();
  float wm = warp_max(tv);
  if (lane == 0) w_max[warp] = wm;
  __syncthreads();
  float m = w_max[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) m = fmaxf(m, w_max[w]);
  {  // sum of exp(x - m), before anything is knocked out
    const float ml = (m == -INFINITY) ? 0.f : m * kLog2e;
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < NE; ++k) s += ex2(fmaf(x[k], kLog2e, -ml));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) w_sum[warp] = s;
  }
  // the warp's K best, by itself
  for (int r = 0; r < K; ++r) {
    int mine = 0x7fffffff, at_u = -1, at_e = 0;
    if (tv == wm && wm != -INFINITY) {
#pragma unroll
      for (int u = kGroups - 1; u >= 0; --u)  // descending: ties end on the lowest token
        if (top[u] == wm) at_u = u;
#pragma unroll
      for (int u = 0; u < kGroups; ++u)
        if (u == at_u) {
#pragma unroll
          for (int e = EPV - 1; e >= 0; --e)
            if (x[u * EPV + e] == wm) at_e = e;
        }
      mine = at_u < kVecs ? (int)begin + (tid + at_u * kThreads) * EPV + at_e : (int)begin + nvec * EPV + at_e;
    }
    const int best = (int)__reduce_min_sync(0xffffffffu, (unsigned)mine);
    if (lane == 0) { w_val[warp][r] = wm; w_idx[warp][r] = best; }
    if (r + 1 < K) {
      if (mine == best && at_u >= 0) {  // taken: knock it out
#pragma unroll
        for (int u = 0; u < kGroups; ++u)
          if (u == at_u) {
            float t = -INFINITY;
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
              if (e == at_e) x[u * EPV + e] = -INFINITY;
              t = fmaxf(t, x[u * EPV + e]);
            }
            top[u] = t;
          }
        tv = largest();
      }
      wm = warp_max(tv);
    }
  }
  __syncthreads();
  if (warp != 0) return;
  // the K best of the four warps' lists: lane 4 w + t holds entry t of warp w
  float v = -INFINITY;
  int i = 0x7fffffff;
  if (lane < kThreads / 32 * kMaxK && lane % kMaxK < K) {
    v = w_val[lane / kMaxK][lane % kMaxK];
    i = w_idx[lane / kMaxK][lane % kMaxK];
  }
  TopPartial out;
  out.m = m;
  out.s = w_sum[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) out.s += w_sum[w];
#pragma unroll
  for (int r = 0; r < kMaxK; ++r) {
    const float bv = warp_max(v);
    const int bi = bv == -INFINITY ? 0x7fffffff
                                   : (int)__reduce_min_sync(0xffffffffu, v == bv ? (unsigned)i : 0x7fffffffu);
    out.val[r] = r < K ? bv : -INFINITY;
    out.idx[r] = r < K ? bi : 0x7fffffff;
    if (i == bi) v = -INFINITY;
  }
  out.pad[0] = out.pad[1] = 0;
  if (tid == 0) partials[(int64_t)row * splits + split] = out;
}

struct BuildArgs {
  const TopPartial* partials;
  int splits, L, K, D, budget, parent_cap, mask_id;
  const int32_t* state;        // [B][L]
  const int32_t* formula_off;  // [D+1]
  const int32_t* formula_i;
  const int32_t* formula_j;
  const int32_t* child_off;    // [D+1]
  const int32_t* child_idx;
  int32_t* tokens;      // [B][budget+1][L]
  int32_t* kept;        // [B][budget]
  float* score;         // [B][D]
  int32_t* parent_off;  // [B][budget+2]
  int32_t* parent_idx;  // [B][parent_cap]
  int32_t* dev_status;  // [B]
  int fill_parents;     // entries of parent_idx past the lists are written as 0
};

// Is the candidate set of formula a a strict subset of formula c's?  a < 0 is
// the current block (the empty set).
__device__ bool strict_subset(const BuildArgs& g, int a, int c) {
  const int c0 = g.formula_off[c], c1 = g.formula_off[c + 1];
  if (a < 0) return c1 > c0;
  const int a0 = g.formula_off[a], a1 = g.formula_off[a + 1];
  if (a1 - a0 >= c1 - c0) return false;
  for (int e = a0; e < a1; ++e) {
    bool found = false;
    for (int f = c0; f < c1; ++f)
      found |= g.formula_i[e] == g.formula_i[f] && g.formula_j[e] == g.formula_j[f];
    if (!found) return false;
  }
  return true;
}

// grid = B sequences, build_threads() threads: a warp per block position, two positions a warp beyond 32;
// dynamic shared memory, see build_smem_bytes.
//
// A chain of small steps in one CTA: what bounds it is how many dependent accesses it is long and how many
// instructions it meets for the first time (some five cycles each), not how much it does.  All that does not
// depend on the logits is worked out ahead of the wait: the graph copied to shared memory, each formula as a
// set of bits, which formulas contain which, the block's masked positions.  Behind the wait a warp merges each
// position's slices and takes its logarithms, a second step sorts the positions, and one warp, a formula a
// lane, does the rest without another barrier, in loops that are not unrolled.  32 positions x 16 slices, ten
// formulas: 4600 cycles to the wait and 14200 behind it with 1024 threads at eight barriers, formulas looked up
// through generic pointers pair by pair, logarithms inside the chains and merges by shuffles; 4500 and 7000
// now (the call 13.0 -> 9.4 us).  The whole chain gone through once beforehand, to have its instructions at
// hand, takes longer than the top-k kernel leaves time for (22 us).
__global__ void __launch_bounds__(kBuildThreads)
draft_build_kernel(BuildArgs g) {
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int threads = blockDim.x, warps = threads >> 5;
  const int L = g.L, K = g.K, D = g.D;
  extern __shared__ __align__(16) unsigned char draft_smem[];
  // of graphs of up to kRelated formulas
  struct Formulas {
    uint64_t sets[kRelated][kMaxK];           // bit i of word j: a formula has candidate (i, j)
    unsigned subsets[kRelated][kRelated / 32];  // bit a of row c: formula a < c is a strict subset of c
    int ranks_needed[kRelated];               // position ranks a formula asks for; INT_MAX: never built
    float log[kRelated + 1];                  // ln of a local score
    float local[kRelated + 1];                // the last one stands for children that do not exist: never built
    alignas(16) float total[kRelated];
  };
  static_assert(sizeof(Formulas) <= kFormulaBytes, "dynamic shared memory");
  Formulas& fs = *reinterpret_cast<Formulas*>(draft_smem);
  // of larger ones
  float* local = reinterpret_cast<float*>(draft_smem);  // [D]
  float* total = local + D;                             // [D]
  int* keep = reinterpret_cast<int*>(total + D);        // [D] whether a formula is kept
  int* node_formula = keep + D;                         // [budget + 1] formula of each node, -1 for node 0 / padding
  int* n_parents = node_formula + g.budget + 1;         // [budget + 1]
  __shared__ int now[64];                          // the current block
  __shared__ float top_p[64];                      // largest probability of a position, -1 of an unmasked one
  __shared__ float by_rank_log[64 * kMaxK];        // by position rank and vocabulary rank: ln of a candidate's
  __shared__ int by_rank_tok[64 * kMaxK];          // probability (-inf: none), its token
  __shared__ int pos_of_rank[64];
  __shared__ int32_t graph_smem[kGraphInts];
  const int32_t* state = g.state + (int64_t)b * L;
  // The draft graph is a constant of the model (calibrated offline), not the product of earlier work on the
  // stream; and the top-k kernel waited before it let this one start, so that the state is complete.
  // All loads that depend on nothing go out first.
  const int npairs = g.formula_off[D], nkids = g.child_off[D];
  const int f_mine = tid <= D ? g.formula_off[tid] : 0, c_mine = tid <= D ? g.child_off[tid] : 0;
  const int32_t t0 = lane < L ? state[lane] : ~g.mask_id, t1 = lane + 32 < L ? state[lane + 32] : ~g.mask_id;
  for (int i = tid; i < 64 * kMaxK; i += threads) {
    by_rank_log[i] = -INFINITY;
    by_rank_tok[i] = 0;
  }
  const bool staged = 2 * (D + 1) + 2 * npairs + nkids <= kGraphInts, one_warp = staged && D <= kRelated;
  int32_t* const f_off = graph_smem;
  int32_t* const c_off = f_off + D + 1;
  int32_t* const f_i = c_off + D + 1;
  int32_t* const f_j = f_i + npairs;
  int32_t* const c_idx = f_j + npairs;
  if (staged) {
    if (tid <= D) { f_off[tid] = f_mine; c_off[tid] = c_mine; }
    for (int i = tid + threads; i <= D; i += threads) { f_off[i] = g.formula_off[i]; c_off[i] = g.child_off[i]; }
    for (int i = tid; i < npairs; i += threads) { f_i[i] = g.formula_i[i]; f_j[i] = g.formula_j[i]; }
    for (int i = tid; i < nkids; i += threads) {
      const int x = g.child_idx[i];
      c_idx[i] = one_warp && (x < 0 || x >= D) ? kRelated : x;
    }
    g.formula_off = f_off; g.child_off = c_off; g.formula_i = f_i; g.formula_j = f_j; g.child_idx = c_idx;
  }
  const uint64_t masked_bits = (uint64_t)__ballot_sync(0xffffffffu, t0 == g.mask_id) |
                               (uint64_t)__ballot_sync(0xffffffffu, t1 == g.mask_id) << 32;
  const int masked = __popcll(masked_bits);
  if (warp == 0) {
    now[lane] = t0;
    now[lane + 32] = t1;
  }
  __syncthreads();
  if (one_warp) {
    if (tid == 0) fs.local[kRelated] = -INFINITY;
    for (int i = tid; i < kRelated; i += threads) fs.total[i] = -INFINITY;
    for (int q = tid; q < D; q += threads) {
      uint64_t set[kMaxK] = {};
      const int e0 = f_off[q], e1 = f_off[q + 1];
      int need = e1 > e0 ? 0 : 0x7fffffff;
#pragma unroll 1
      for (int e = e0; e < e1; ++e) {
        const int i = f_i[e], j = f_j[e];
        const bool exists = i >= 0 && i < 64 && j >= 0 && j < K;
        need = exists ? max(need, i + 1) : 0x7fffffff;
#pragma unroll
        for (int t = 0; t < kMaxK; ++t)
          if (exists && t == j) set[t] |= 1ull << i;
      }
#pragma unroll
      for (int t = 0; t < kMaxK; ++t) fs.sets[q][t] = set[t];
      fs.ranks_needed[q] = need;
    }
    __syncthreads();
    for (int w = warp; w < D * (kRelated / 32); w += warps) {  // a warp per word, its lanes over the smaller formulas
      const int c = w / (kRelated / 32), a = w % (kRelated / 32) * 32 + lane;
      bool sub = a < c && f_off[a + 1] - f_off[a] < f_off[c + 1] - f_off[c];
      if (sub) {
#pragma unroll
        for (int t = 0; t < kMaxK; ++t) sub &= (fs.sets[a][t] & ~fs.sets[c][t]) == 0ull;
      }
      const unsigned word = __ballot_sync(0xffffffffu, sub);
      if (lane == 0) fs.subsets[c][w % (kRelated / 32)] = word;
    }
    __syncthreads();
  }
  // Of up to 32 formulas of up to four candidates and children each, lane q of the first two warps has those of
  // formula q at hand: places in by_rank_log (-1: no more), indices in fs.local.
  bool at_hand = false;
  int place[kAtHand], kid[kAtHand], n_places = 0, needed = 0x7fffffff;
  if (one_warp && D <= 32 && warp <= 1) {
    const int q = min(lane, D - 1), e0 = f_off[q], k0 = c_off[q], n_kids = c_off[q + 1] - k0;
    n_places = f_off[q + 1] - e0;
    needed = fs.ranks_needed[q];
    at_hand = __all_sync(0xffffffffu, n_places <= kAtHand && n_kids <= kAtHand);
#pragma unroll
    for (int u = 0; u < kAtHand; ++u) {
      place[u] = u < n_places && needed <= 64 ? f_i[e0 + u] * kMaxK + f_j[e0 + u] : -1;
      kid[u] = u < n_kids ? c_idx[k0 + u] : kRelated;
    }
  }
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();  // the top-k kernel's partial results are visible, the outputs free
#endif
  int32_t* tokens = g.tokens + (int64_t)b * (g.budget + 1) * L;

  // 1. candidates c_ij and their probabilities: one warp per position
  float cand_log[2] = {};  // lane r: that of vocabulary rank r, of the warp's first and second position
  int cand_tok[2] = {};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int l = warp + h * warps;  // two rounds are enough for 64 positions, as there are min(L, 32) warps at least
    if (l >= L) break;
    const TopPartial* p = g.partials + ((int64_t)b * L + l) * g.splits;
    const bool is_masked = (masked_bits >> l & 1ull) != 0ull;
    float m = -INFINITY, s = 0.f;
    float hv[kMaxK];
    int hi[kMaxK];
#pragma unroll
    for (int t = 0; t < kMaxK; ++t) { hv[t] = -INFINITY; hi[t] = 0x7fffffff; }
    if (g.splits <= 32) {
      // one slice per lane, fetched whole in one trip: its maximum and sum, and its K
      // candidates, which the top-k kernel left sorted
      if (is_masked && lane < g.splits) {
        const uint4* q = reinterpret_cast<const uint4*>(p + lane);
        const uint4 q0 = __ldcg(q), q1 = __ldcg(q + 1), q2 = __ldcg(q + 2);
        m = __uint_as_float(q0.x);
        s = __uint_as_float(q0.y);
        hv[0] = __uint_as_float(q0.z); hv[1] = __uint_as_float(q0.w);
        hv[2] = __uint_as_float(q1.x); hv[3] = __uint_as_float(q1.y);
        hi[0] = (int)q1.z; hi[1] = (int)q1.w; hi[2] = (int)q2.x; hi[3] = (int)q2.y;
      }
    } else if (is_masked) {
      // maximum and sum over the slices, fixed order
      for (int k = lane; k < g.splits; k += 32) {
        const float m2 = __ldcg(&p[k].m), s2 = __ldcg(&p[k].s), M = fmaxf(m, m2);
        s = s * ((m == M) ? 1.f : ex2((m - M) * kLog2e)) + s2 * ((m2 == M) ? 1.f : ex2((m2 - M) * kLog2e));
        m = M;
      }
      // every lane sorts the candidates it reads (each is read once)
      for (int c = lane; c < g.splits * K; c += 32) {
        float v = __ldcg(&p[c / K].val[c % K]);
        int i = __ldcg(&p[c / K].idx[c % K]);
        if (v == -INFINITY) continue;
#pragma unroll
        for (int t = 0; t < kMaxK; ++t)  // insertion into the sorted list
          if (ahead(v, i, hv[t], hi[t])) {
            const float tv = hv[t]; const int ti = hi[t];
            hv[t] = v; hi[t] = i; v = tv; i = ti;
          }
      }
    }
    // every draft starts as the current block
    for (int n = lane; n <= g.budget; n += 32) tokens[n * L + l] = now[l];
    float p_top = -1.f;
    if (is_masked) {
      const float M = warp_max(m);
      s *= m == M ? 1.f : ex2((m - M) * kLog2e);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      // the K best of the slices' candidates (value desc, id asc): K rounds pick the best
      // head over the lanes and pop it; lane r keeps the best of round r
      float mine = -INFINITY;
      int mine_tok = 0x7fffffff;
#pragma unroll 1
      for (int r = 0; r < K; ++r) {
        const float bv = warp_max(hv[0]);
        const int bi = (int)__reduce_min_sync(0xffffffffu, hv[0] == bv ? (unsigned)hi[0] : 0x7fffffffu);
        if (hi[0] == bi) {  // this lane's head won, if there is any: pop it
#pragma unroll
          for (int t = 0; t + 1 < kMaxK; ++t) { hv[t] = hv[t + 1]; hi[t] = hi[t + 1]; }
          hv[kMaxK - 1] = -INFINITY;
          hi[kMaxK - 1] = 0x7fffffff;
        }
        if (lane == r) {
          mine = bv;
          mine_tok = bi;
        }
      }
      p_top = mine == -INFINITY ? 0.f : ex2((mine - M) * kLog2e) / s;
      if (!(p_top >= 0.f)) p_top = 0.f;  // a row without a distribution: behind the others, a rank of its own
      cand_tok[h] = mine_tok;
      cand_log[h] = p_top > 0.f ? logf(fmaxf(p_top, 1e-45f)) : -INFINITY;
      if (lane == 0 && (!(fabsf(M) < INFINITY) || !(s > 0.f) || !(s < INFINITY)) && g.dev_status)
        atomicOr(g.dev_status + b, SPIFFY_DEV_NONFINITE);
    }
    if (lane == 0) top_p[l] = p_top;
  }
  __syncthreads();
  // 2. token position ranks (Eq. token-position-sort): by maximum probability, ties to the lower position
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int l = warp + h * warps;
    if (l >= L) break;
    const float pl = top_p[l];
    if (pl < 0.f) continue;  // unmasked
    int rank = 0;
#pragma unroll
    for (int j0 = 0; j0 < 64; j0 += 32) {
      if (j0 >= L) break;
      const int j = j0 + lane;
      const float pj = j < L ? top_p[j] : -1.f;
      rank += __popc(__ballot_sync(0xffffffffu, pj >= 0.f && (pj > pl || (pj == pl && j < l))));
    }
    if (lane == 0) pos_of_rank[rank] = l;
    if (lane < K) {
      by_rank_log[rank * kMaxK + lane] = cand_log[h];
      by_rank_tok[rank * kMaxK + lane] = cand_tok[h];
    }
  }
  __syncthreads();
  int32_t* out_off = g.parent_off + (int64_t)b * (g.budget + 2);
  int32_t* out_idx = g.parent_idx + (int64_t)b * g.parent_cap;
  int32_t* out_kept = g.kept + (int64_t)b * g.budget;

  if (one_warp) {
    // Two warps with the same numbers: what follows from them is written by one or the other.
    if (warp > 1) return;
    const bool lists = warp == 0, drafts = warp == 1;
    if (at_hand) {  // 3. and 4. as below, the look-ups all at once
      float x = -INFINITY, lg = -INFINITY;
      if (needed <= masked) {
        float v[kAtHand];
#pragma unroll
        for (int u = 0; u < kAtHand; ++u) v[u] = place[u] >= 0 ? by_rank_log[max(place[u], 0)] : 0.f;
        x = expf((((v[0] + v[1]) + v[2]) + v[3]) / (float)n_places);
        lg = x > 0.f ? logf(fmaxf(x, 1e-45f)) : -INFINITY;
      }
      if (lane < D) {
        fs.local[lane] = x;
        fs.log[lane] = lg;
      }
      __syncwarp();
      int n = 0;
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < kAtHand; ++u) {
        const bool counts = fs.local[kid[u]] != -INFINITY;
        sum += counts ? fs.log[kid[u]] : 0.f;
        n += counts;
      }
      if (x != -INFINITY && n > 0) x = sqrtf(x * expf(sum / (float)n));
      if (lane < D) {
        fs.total[lane] = x;
        if (lists) g.score[(int64_t)b * D + lane] = x;
      }
    } else {
#pragma unroll 1
      for (int q = lane; q < D; q += 32) {  // 3. local scores: geometric means of the candidates' probabilities
        const int e0 = f_off[q], e1 = f_off[q + 1];
        float x = -INFINITY, lg = -INFINITY;
        if (fs.ranks_needed[q] <= masked) {
          float logsum = 0.f;
#pragma unroll 2
          for (int e = e0; e < e1; ++e) logsum += by_rank_log[f_i[e] * kMaxK + f_j[e]];
          x = expf(logsum / (float)(e1 - e0));  // 0 where a candidate has no probability
          lg = x > 0.f ? logf(fmaxf(x, 1e-45f)) : -INFINITY;
        }
        fs.local[q] = x;
        fs.log[q] = lg;
      }
      __syncwarp();
#pragma unroll 1
      for (int q = lane; q < D; q += 32) {  // 4. score = GM(local, GM(children's)); without buildable children local
        float x = fs.local[q];
        if (x != -INFINITY) {
          float logsum = 0.f;
          int n = 0;
          const int e1 = c_off[q + 1];
#pragma unroll 2
          for (int e = c_off[q]; e < e1; ++e) {
            const int y = c_idx[e];
            if (fs.local[y] == -INFINITY) continue;
            logsum += fs.log[y];
            ++n;
          }
          if (n > 0) x = sqrtf(x * expf(logsum / (float)n));
        }
        fs.total[q] = x;
        if (lists) g.score[(int64_t)b * D + q] = x;
      }
    }
    __syncwarp();
    uint64_t keep_bits = 0;  // 5. the D* best (score desc, formula index asc) keep their formula order
#pragma unroll 1
    for (int q = lane; q < D + lane; q += 32) {  // all lanes
      const float mine = q < D ? fs.total[q] : -INFINITY;
      int rank = 0;
#pragma unroll 1
      for (int x = 0; x < D; x += 4) {  // behind the last one -inf
        const float4 t = *reinterpret_cast<const float4*>(fs.total + x);
        rank += ((t.x > mine) | ((t.x == mine) & (x < q))) + ((t.y > mine) | ((t.y == mine) & (x + 1 < q))) +
                ((t.z > mine) | ((t.z == mine) & (x + 2 < q))) + ((t.w > mine) | ((t.w == mine) & (x + 3 < q)));
      }
      keep_bits |= (uint64_t)__ballot_sync(0xffffffffu, mine != -INFINITY && rank < g.budget) << (q - lane);
    }
    // 6., 7. kept drafts' tokens, and parent lists: every earlier kept node whose candidate set is a
    // strict subset, the current block (node 0, the empty set) among them
    int base = 0;
#pragma unroll 1
    for (int q = lane; q < D + lane; q += 32) {
      const uint64_t before = keep_bits & ((1ull << q) - 1ull);
      const int node = 1 + __popcll(before);
      // (scores that are no numbers have no order, and more of them than the budget may have been kept)
      const bool kept = (keep_bits >> q & 1ull) != 0ull && node <= g.budget;
      if (kept && drafts) {
        out_kept[node - 1] = q;
        const int e1 = f_off[q + 1];
#pragma unroll 1
        for (int e = f_off[q]; e < e1; ++e) tokens[node * L + pos_of_rank[f_i[e]]] = by_rank_tok[f_i[e] * kMaxK + f_j[e]];
      }
      if (!lists) continue;
      uint64_t parents = kept ? ((uint64_t)fs.subsets[q][0] | (uint64_t)fs.subsets[q][1] << 32) & before : 0ull;
      const int count = kept ? 1 + __popcll(parents) : 0;
      int upto = count;
#pragma unroll 1
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, upto, off);
        if (lane >= off) upto += y;
      }
      int at = base + upto - count;
      base += __shfl_sync(0xffffffffu, upto, 31);
      if (kept) {
        out_off[node] = min(at, g.parent_cap);
        if (at < g.parent_cap) out_idx[at] = 0;
#pragma unroll 1
        for (; parents; parents &= parents - 1) {
          ++at;
          if (at < g.parent_cap) out_idx[at] = 1 + __popcll(keep_bits & ((parents & (0ull - parents)) - 1ull));
        }
      }
    }
    const int nodes = min(__popcll(keep_bits), g.budget);
    if (drafts)
      for (int n = nodes + lane; n < g.budget; n += 32) out_kept[n] = -1;
    if (lists) {
      if (lane == 0) {
        out_off[0] = 0;
        if (base > g.parent_cap && g.dev_status) atomicOr(g.dev_status + b, SPIFFY_DEV_BADGRAPH);
      }
      for (int n = nodes + lane; n <= g.budget; n += 32) out_off[n + 1] = min(base, g.parent_cap);
      if (g.fill_parents)
        for (int i = base + lane; i < g.parent_cap; i += 32) out_idx[i] = 0;
    }
    return;
  }

  // Larger graphs: the same steps, by all threads.
  for (int q = tid; q < D; q += threads) {
    const int e0 = g.formula_off[q], e1 = g.formula_off[q + 1];
    bool ok = e1 > e0;
    float logsum = 0.f;
    for (int e = e0; e < e1 && ok; ++e) {
      const int i = g.formula_i[e], j = g.formula_j[e];
      if (i < 0 || i >= masked || j < 0 || j >= K) { ok = false; break; }
      logsum += by_rank_log[i * kMaxK + j];
    }
    local[q] = !ok ? -INFINITY : expf(logsum / (float)(e1 - e0));
  }
  __syncthreads();
  for (int q = tid; q < D; q += threads) {
    float sc = local[q];
    if (sc != -INFINITY) {
      float logsum = 0.f;
      int n = 0;
      for (int e = g.child_off[q]; e < g.child_off[q + 1]; ++e) {
        const int x = g.child_idx[e];
        if (x < 0 || x >= D || local[x] == -INFINITY) continue;
        logsum += local[x] > 0.f ? logf(fmaxf(local[x], 1e-45f)) : -INFINITY;
        ++n;
      }
      if (n > 0) sc = sqrtf(sc * expf(logsum / (float)n));
    }
    total[q] = sc;
    g.score[(int64_t)b * D + q] = sc;
  }
  __syncthreads();
  for (int q = tid; q < D; q += threads) {
    int rank = 0;
    const float sq = total[q];
    for (int x = 0; x < D; ++x) rank += (total[x] > sq || (total[x] == sq && x < q)) ? 1 : 0;
    keep[q] = (sq != -INFINITY && rank < g.budget) ? 1 : 0;
  }
  for (int n = tid; n <= g.budget; n += threads) node_formula[n] = -1;
  __syncthreads();
  for (int q = tid; q < D; q += threads) {
    if (!keep[q]) continue;
    int slot = 0;
    for (int x = 0; x < q; ++x) slot += keep[x];
    if (slot < g.budget) node_formula[slot + 1] = q;
  }
  __syncthreads();
  for (int n = tid; n < g.budget; n += threads) out_kept[n] = node_formula[n + 1];
  for (int n = 1 + tid; n <= g.budget; n += threads) {
    const int q = node_formula[n];
    if (q < 0) continue;
    for (int e = g.formula_off[q]; e < g.formula_off[q + 1]; ++e) {
      const int i = g.formula_i[e];
      tokens[n * L + pos_of_rank[i]] = by_rank_tok[i * kMaxK + g.formula_j[e]];
    }
  }
  // parent lists: one warp per child, its lanes over the candidate parents
  auto is_parent = [&](int a, int c) {
    if (a >= c || (a > 0 && node_formula[a] < 0)) return false;
    return strict_subset(g, a == 0 ? -1 : node_formula[a], node_formula[c]);
  };
  for (int c = warp; c <= g.budget; c += warps) {
    int n = 0;
    if (c > 0 && node_formula[c] >= 0)
      for (int a0 = 0; a0 < c; a0 += 32) n += __popc(__ballot_sync(0xffffffffu, is_parent(a0 + lane, c)));
    if (lane == 0) n_parents[c] = n;
  }
  __syncthreads();
  for (int c = warp; c <= g.budget; c += warps) {
    int start = 0;
    for (int x = lane; x < c; x += 32) start += n_parents[x];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) start += __shfl_xor_sync(0xffffffffu, start, off);
    if (lane == 0) {
      out_off[c] = min(start, g.parent_cap);
      if (c == g.budget) out_off[c + 1] = min(start + n_parents[c], g.parent_cap);
      if (start + n_parents[c] > g.parent_cap && g.dev_status) atomicOr(g.dev_status + b, SPIFFY_DEV_BADGRAPH);
    }
    if (g.fill_parents && c == g.budget)
      for (int i = start + n_parents[c] + lane; i < g.parent_cap; i += 32) out_idx[i] = 0;
    if (c > 0 && node_formula[c] >= 0) {
      int w = start;
      for (int a0 = 0; a0 < c; a0 += 32) {
        const bool par = is_parent(a0 + lane, c);
        const unsigned mask = __ballot_sync(0xffffffffu, par);
        const int at = w + __popc(mask & ((1u << lane) - 1u));
        if (par && at < g.parent_cap) out_idx[at] = a0 + lane;
        w += __popc(mask);
      }
    }
  }
}

int64_t draft_chunk(const spiffy_draft_desc& d, int* splits) {
  const int64_t epv = d.logits_dtype == SPIFFY_BF16 ? 8 : 4;
  const int64_t most = (int64_t)kThreads * kVecs * epv;
  const int64_t n = (d.vocab + most - 1) / most;
  int64_t chunk = (d.vocab + n - 1) / n;
  chunk = (chunk + epv - 1) / epv * epv;
  *splits = (int)n;
  return chunk;
}

// A warp per block position, and 16 at least, for the formulas: 64 of them and one position take 8.6 us with 512 threads, 11.0
// with 1024 before the kernel's chain was shortened and 20.0 with a warp for the one position (ten formulas 5.9, 8.9, 6.6).
// All threads work on graphs of more formulas than one warp takes, and their pairs of kept drafts: 1024, us with 512
// and 1024: 65 formulas, one position 10.0 9.3; 200, eight 24.1 20.7; 1000, all kept, eight 1537 1085.  Not where two
// blocks of 512 an SM have sequences to work on (100 formulas, 300 sequences 40.5 and 47.1).
int build_threads(const spiffy_draft_desc& d) {
  if (d.n_formulas > kRelated && d.batch <= sm_count()) return kBuildThreads;
  return std::min(kBuildThreads, std::max(kBuildThreads / 2, 32 * d.block_len));
}

size_t build_smem_bytes(const spiffy_draft_desc& d) {
  return std::max(d.n_formulas <= kRelated ? (size_t)kFormulaBytes : (size_t)0,
                  (size_t)d.n_formulas * 12 + (size_t)(d.budget + 1) * 8);  // a graph of few formulas may be too long to stage
}

}  // namespace

size_t draft_workspace_bytes(const spiffy_draft_desc& d) {
  int splits = 1;
  draft_chunk(d, &splits);
  return (size_t)d.batch * d.block_len * splits * sizeof(TopPartial);
}

spiffy_status launch_draft(const spiffy_draft_desc& d, const void* logits, const int32_t* state,
                           const int32_t* formula_off, const int32_t* formula_i,
                           const int32_t* formula_j, const int32_t* child_off,
                           const int32_t* child_idx, int32_t* tokens, int32_t* kept, float* score,
                           int32_t* parent_off, int32_t* parent_idx, int32_t* dev_status, void* ws,
                           bool fresh, cudaStream_t stream) {
  int splits = 1;
  const int64_t chunk = draft_chunk(d, &splits);
  TopPartial* partials = static_cast<TopPartial*>(ws);
  int32_t* clear = fresh ? dev_status : nullptr;
  const dim3 grid(splits, d.batch * d.block_len);
  cudaError_t e;
  if (d.logits_dtype == SPIFFY_BF16)
    e = launch_pdl(draft_topk_kernel<__nv_bfloat16>, grid, dim3(kThreads), (size_t)0, stream,
                   static_cast<const __nv_bfloat16*>(logits), (int64_t)d.row_stride, (int)d.vocab, chunk,
                   splits, (int)d.top_k, state, (int)d.mask_token_id, partials, clear, (int)d.block_len);
  else
    e = launch_pdl(draft_topk_kernel<float>, grid, dim3(kThreads), (size_t)0, stream,
                   static_cast<const float*>(logits), (int64_t)d.row_stride, (int)d.vocab, chunk, splits,
                   (int)d.top_k, state, (int)d.mask_token_id, partials, clear, (int)d.block_len);
  count_launch();
  if (e != cudaSuccess) return SPIFFY_ECUDA;
  BuildArgs g;
  g.partials = partials; g.splits = splits; g.L = d.block_len; g.K = d.top_k; g.D = d.n_formulas;
  g.budget = d.budget; g.parent_cap = d.parent_cap; g.mask_id = d.mask_token_id;
  g.state = state; g.formula_off = formula_off; g.formula_i = formula_i; g.formula_j = formula_j;
  g.child_off = child_off; g.child_idx = child_idx; g.tokens = tokens; g.kept = kept; g.score = score;
  g.parent_off = parent_off; g.parent_idx = parent_idx; g.dev_status = dev_status; g.fill_parents = fresh ? 1 : 0;
  e = launch_pdl(draft_build_kernel, dim3(d.batch), dim3(build_threads(d)), build_smem_bytes(d), stream, g);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

}  // namespace spiffy
