// Device code of the decision step shared by its kernels: the vocabulary-slice
// reduce (Algorithm 1, steps 1-2: per position the top token and its softmax
// probability), the fixed-order merge of slices, and the unmasking rule of
// Sec. 3.1 (step 3).
//
// The argmax compares logit values exactly ((value desc, index asc) order);
// probabilities only enter the confidence.  All merges run in a fixed order, so
// repeated calls -- and the different kernels that use this code -- give
// identical bits.
#pragma once
#include <math.h>

#include <type_traits>

#include "common.cuh"

namespace spiffy {
namespace {


// 128 threads holding 8 vectors each measured best among 64..512 threads and
// 2..16 vectors (smaller slices pay more per CTA, larger ones leave too few
// CTAs in flight per SM).
constexpr int kReduceThreads = 128;
constexpr int kUnroll = 8;  // 128-bit vectors per thread, all loaded at once

struct __align__(16) Partial {
  float m;    // slice maximum (-inf for an empty slice)
  float s;    // sum over the slice of exp(x - m)
  int idx;    // lowest index attaining m
  int pad;
};

// Clears the status words of a call whose caller left them arbitrary
// (SPIFFY_FRESH_STATUS); part of the call's first kernel, which sets no bit itself: the CTA
// of row i, of which there are more than sequences, clears word i.
struct StatusClear {
  int32_t* a;  // [B], null when there is nothing to clear
  int32_t* b;
  int batch;   // 0: nothing to clear
  // one thread per row below `batch` calls it, and not the one whose chain the CTA waits for
  __device__ __forceinline__ void run(int row) const {
    if (a) a[row] = 0;
    if (b) b[row] = 0;
  }
};
inline StatusClear status_clear(const spiffy_decide_desc& d, bool fresh, int32_t* a, int32_t* b) {
  return fresh ? StatusClear{a, b, d.batch} : StatusClear{nullptr, nullptr, 0};
}

// acc += {2^(x0 * log2e - ml), 2^(x1 * log2e - ml)}; k2 = {log2e, log2e}, nml2 = {-ml, -ml}
__device__ __forceinline__ uint64_t add_exp2(uint64_t acc, float x0, float x1, uint64_t k2,
                                             uint64_t nml2) {
  float a0, a1;
  unpack2(fma2(pack2(x0, x1), k2, nml2), a0, a1);
  return add2(acc, pack2(ex2(a0), ex2(a1)));
}

// (value desc, index asc) merge of two partial results.
__device__ __forceinline__ void merge(float& m, float& s, int& idx, float m2,
                                      float s2, int idx2) {
  if (m2 > m || (m2 == m && idx2 < idx)) idx = idx2;
  // the sum that belongs to the larger maximum stays as it is
  const float f = m == m2 ? 1.f : ex2(-fabsf(m - m2) * kLog2e);
  s = m2 > m ? __fmaf_rn(s, f, s2) : __fmaf_rn(s2, f, s);  // spelled out: every instance rounds the same way
  m = fmaxf(m, m2);
}

template <typename T>
struct Elem;

template <>
struct Elem<__nv_bfloat16> {
  static constexpr int kPerVec = 8;
  static constexpr uint32_t kNegInf = 0xff80ff80u;  // two bf16 -inf
  static __device__ __forceinline__ float lo(uint32_t w) { return __uint_as_float(w << 16); }
  static __device__ __forceinline__ float hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
  static __device__ __forceinline__ __nv_bfloat162 pk(uint32_t w) {
    return *reinterpret_cast<const __nv_bfloat162*>(&w);
  }
  // exact maximum of one vector / of a group of vectors, on the packed bf16 pipe
  static __device__ __forceinline__ float vmax(uint4 v) {
    const __nv_bfloat162 p = __hmax2(__hmax2(pk(v.x), pk(v.y)), __hmax2(pk(v.z), pk(v.w)));
    return fmaxf(__low2float(p), __high2float(p));
  }
  // true when some element of the vector equals x (x is one of the inputs, hence a bf16 value)
  static __device__ __forceinline__ bool holds(uint4 v, float x) {
    const __nv_bfloat162 xx = __float2bfloat162_rn(x);
    return (__heq2_mask(pk(v.x), xx) | __heq2_mask(pk(v.y), xx) | __heq2_mask(pk(v.z), xx) |
            __heq2_mask(pk(v.w), xx)) != 0u;
  }
  static __device__ __forceinline__ float gmax(const uint4 (&v)[kUnroll]) {
    __nv_bfloat162 p = __hmax2(__hmax2(pk(v[0].x), pk(v[0].y)), __hmax2(pk(v[0].z), pk(v[0].w)));
#pragma unroll
    for (int k = 1; k < kUnroll; ++k)
      p = __hmax2(p, __hmax2(__hmax2(pk(v[k].x), pk(v[k].y)), __hmax2(pk(v[k].z), pk(v[k].w))));
    return fmaxf(__low2float(p), __high2float(p));
  }
  // acc (two running sums) += 2^(x * log2e - ml) over the vector, even elements into the
  // low lane, odd ones into the high lane
  static __device__ __forceinline__ uint64_t sum_terms(uint4 v, uint64_t k2, uint64_t nml2,
                                                       uint64_t acc) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) acc = add_exp2(acc, lo(w[i]), hi(w[i]), k2, nml2);
    return acc;
  }
  // position of the first element equal to x, kPerVec if there is none
  static __device__ __forceinline__ int first_equal(uint4 v, float x) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    int j = kPerVec;
#pragma unroll
    for (int i = 3; i >= 0; --i) {
      j = (hi(w[i]) == x) ? 2 * i + 1 : j;
      j = (lo(w[i]) == x) ? 2 * i : j;
    }
    return j;
  }
  static __device__ __forceinline__ float load1(const __nv_bfloat16* p) {
    return __bfloat162float(*p);
  }
};

template <>
struct Elem<float> {
  static constexpr int kPerVec = 4;
  static constexpr uint32_t kNegInf = 0xff800000u;
  static __device__ __forceinline__ float vmax(uint4 v) {
    return fmaxf(fmaxf(__uint_as_float(v.x), __uint_as_float(v.y)),
                 fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
  }
  static __device__ __forceinline__ bool holds(uint4 v, float x) { return vmax(v) == x; }
  static __device__ __forceinline__ float gmax(const uint4 (&v)[kUnroll]) {
    float g = -INFINITY;
#pragma unroll
    for (int k = 0; k < kUnroll; ++k)
      g = fmaxf(g, fmaxf(fmaxf(__uint_as_float(v[k].x), __uint_as_float(v[k].y)),
                         fmaxf(__uint_as_float(v[k].z), __uint_as_float(v[k].w))));
    return g;
  }
  static __device__ __forceinline__ uint64_t sum_terms(uint4 v, uint64_t k2, uint64_t nml2,
                                                       uint64_t acc) {
    acc = add_exp2(acc, __uint_as_float(v.x), __uint_as_float(v.y), k2, nml2);
    return add_exp2(acc, __uint_as_float(v.z), __uint_as_float(v.w), k2, nml2);
  }
  static __device__ __forceinline__ int first_equal(uint4 v, float x) {
    int j = kPerVec;
    j = (__uint_as_float(v.w) == x) ? 3 : j;
    j = (__uint_as_float(v.z) == x) ? 2 : j;
    j = (__uint_as_float(v.y) == x) ? 1 : j;
    j = (__uint_as_float(v.x) == x) ? 0 : j;
    return j;
  }
  static __device__ __forceinline__ float load1(const float* p) { return *p; }
};

// 16 aligned bytes in one access, as another CTA may be polling for them.
__device__ __forceinline__ void store16(void* p, uint64_t lo, uint64_t hi) {
  asm volatile("{\n.reg .b128 t;\nmov.b128 t, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p), "l"(lo),
               "l"(hi)
               : "memory");
}

// The maximum over the warp's lanes; NaNs lose, as in fmaxf.
__device__ __forceinline__ float warp_max(float x) {
  float m;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}

// One CTA of kReduceThreads threads reduces one vocabulary slice
// [split * chunk, min(V, (split + 1) * chunk)) of the logits row at `base` to
// (maximum, sum of exp(x - maximum), lowest index attaining the maximum).  A
// slice is at most kReduceThreads * kUnroll vectors, so that every thread holds
// its whole share in registers: all loads go out at once, the slice maximum is
// found first and the exponentials are then taken against it directly.  All
// threads of the CTA call it together; thread 0 stores the result.  `k` is
// log2(e) for the plain softmax; the sampled decision passes log2(e) / T and
// gets the sum of exp((x - maximum) / T).  `tag`, if not 0, goes into the result's spare word
// in the one 16-byte access that writes it: a reader that polls for the tag has the rest with it.
// `out` may be null: thread 0 has the result anyway.  `keep`, in shared memory, gets the slice's
// vectors, number i at kept_at(i).  kGroups: the CTA is that many groups of kReduceThreads threads, each
// with a slice of its own (named barriers 1 ...); "thread 0" is then the group's first.
__device__ __forceinline__ int kept_at(int i) { return i ^ ((i >> 3) & 7); }  // no bank conflicts at stride 8 either
template <typename T, int kGroups = 1>
__device__ __forceinline__ Partial reduce_slice(const T* __restrict__ base, int V, int64_t chunk,
                                             int split, Partial* __restrict__ out,
                                             const float k = kLog2e, const int tag = 0, uint4* keep = nullptr) {
  const int64_t begin = (int64_t)split * chunk;
  const int64_t end = min((int64_t)V, begin + chunk);
  constexpr int EPV = Elem<T>::kPerVec;
  constexpr uint32_t NI = Elem<T>::kNegInf;
  const int nvec = begin < end ? (int)((end - begin) / EPV) : 0;  // <= kReduceThreads * kUnroll
  const int ntail = begin < end ? (int)(end - begin) - nvec * EPV : 0;  // < EPV, last slice only
  const uint4* p = reinterpret_cast<const uint4*>(base + begin);
  const int group = kGroups == 1 ? 0 : (int)threadIdx.x / kReduceThreads;
  const int tid = (int)threadIdx.x - group * kReduceThreads, warp = tid >> 5, lane = tid & 31;
  auto sync = [&]() {
    if constexpr (kGroups == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kReduceThreads) : "memory");
  };

  // 1. the thread's vectors t, t + kReduceThreads, ...; thread 0 also takes the ragged tail
  uint4 v[kUnroll];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u)
    v[u] = (tid + u * kReduceThreads < nvec) ? ld_stream(p + tid + u * kReduceThreads)
                                             : make_uint4(NI, NI, NI, NI);
  float tail[EPV];
#pragma unroll
  for (int e = 0; e < EPV; ++e)
    tail[e] = (tid == 0 && e < ntail) ? Elem<T>::load1(base + begin + (int64_t)nvec * EPV + e) : -INFINITY;
  if (keep) {
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) keep[kept_at(tid + u * kReduceThreads)] = v[u];
  }
  // 2. slice maximum: lanes, warps
  float m = Elem<T>::gmax(v);
#pragma unroll
  for (int e = 0; e < EPV; ++e) m = fmaxf(m, tail[e]);
  const float mine = m;
  m = warp_max(m);
  __shared__ float warp_ms[kGroups][kReduceThreads / 32], warp_ss[kGroups][kReduceThreads / 32];
  __shared__ int slice_idxs[kGroups];
  float *const warp_m = warp_ms[group], *const warp_s = warp_ss[group];
  int& slice_idx = slice_idxs[group];
  if (lane == 0) warp_m[warp] = m;
  if (tid == 0) slice_idx = 0x7fffffff;
  sync();
  m = warp_m[0];
#pragma unroll
  for (int w = 1; w < kReduceThreads / 32; ++w) m = fmaxf(m, warp_m[w]);
  // 3. the lowest index that attains m: only the threads whose own maximum it is search for it
  if (mine == m && m != -INFINITY) {
    int idx = 0x7fffffff;
#pragma unroll
    for (int e = EPV - 1; e >= 0; --e)
      if (e < ntail && tail[e] == m) idx = (int)begin + nvec * EPV + e;  // thread 0 alone has a tail
#pragma unroll
    for (int u = kUnroll - 1; u >= 0; --u)
      if (Elem<T>::holds(v[u], m)) idx = (int)begin + (tid + u * kReduceThreads) * EPV + Elem<T>::first_equal(v[u], m);
    atomicMin(&slice_idx, idx);
  }
  // 4. sum of exp(x - m)
  const float ml = (m == -INFINITY) ? 0.f : m * k;  // an all -inf slice sums to 0
  const uint64_t k2 = pack2(k, k), nml2 = pack2(-ml, -ml);
  uint64_t acc = pack2(0.f, 0.f);
#pragma unroll
  for (int u = kUnroll - 1; u >= 0; --u) acc = Elem<T>::sum_terms(v[u], k2, nml2, acc);
  float s;
  {
    float s0, s1;
    unpack2(acc, s0, s1);
    s = s0 + s1;
  }
  if (ntail > 0 && tid == 0) {
#pragma unroll
    for (int e = EPV - 1; e >= 0; --e) s += ex2(fmaf(tail[e], k, -ml));  // -inf beyond the tail: adds 0
  }
  // fixed order: lanes (butterfly), then warps
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) warp_s[warp] = s;
  sync();
  Partial r = {m, s, 0, tag};
  if (tid == 0) {
    s = warp_s[0];
    for (int w = 1; w < kReduceThreads / 32; ++w) s += warp_s[w];
    r = Partial{m, s, slice_idx, tag};
    if (out && tag == 0) *out = r;
    if (out && tag != 0)
      store16(out, (uint64_t)__float_as_uint(m) | (uint64_t)__float_as_uint(s) << 32,
              (uint64_t)(uint32_t)slice_idx | (uint64_t)(uint32_t)tag << 32);
  }
  return r;
}

// Sixteen bytes that another CTA may be writing, in one access.
__device__ __forceinline__ int4 load16(const void* p) {
  uint64_t a, b;
  asm volatile("{\n.reg .b128 t;\nld.relaxed.gpu.global.b128 t, [%2];\nmov.b128 {%0, %1}, t;\n}"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
  return make_int4((int)(uint32_t)a, (int)(uint32_t)(a >> 32), (int)(uint32_t)b, (int)(uint32_t)(b >> 32));
}

// How finalize_row comes by a row's slices.  Complete: they are all there, written by an earlier kernel.
// They are read at L2, as this CTA may have been resident while that kernel wrote them.
struct CompleteSlices {
  static constexpr bool kWaits = false, kShared = false;
};
struct SharedSlices {  // ... in this CTA's shared memory
  static constexpr bool kWaits = false, kShared = true;
};
// They are being written: a slice is there when its spare word is `tag`.  At most `polls` looks at a batch
// of slices; `missing` when they ran out, and the row's results mean nothing.
struct TaggedSlices {
  static constexpr bool kWaits = true, kShared = false;
  int tag;
  unsigned polls;
  bool missing = false;
};

// kLanes (8, 4, 2 or 1) neighbouring lanes merge the slices of one row and lane
// 0 of the group gets the row's confidence and top token (Algorithm 1, steps
// 1-2).  The order is fixed and the same for every kLanes: eight accumulators
// (accumulator j takes slices j, j + 8, ...) are combined by the butterfly
// 4, 2, 1 with the lower index first; a lane holds the accumulators j = sub,
// sub + kLanes, ... and does the butterfly steps that stay inside it locally.
// Returns false on lane 0 when the row is masked and not usable.  kAtOnce: slices of a lane on their way at
// a time, at least (the order of the merge does not depend on it).
template <int kLanes, class Source = CompleteSlices, int kAtOnce = 4>
__device__ __forceinline__ bool finalize_row(const Partial* __restrict__ p, int splits, int sub,
                                             int32_t state, int mask_id, float& conf, int32_t& tok,
                                             Source&& from = Source{}) {
  constexpr bool kWaits = std::remove_reference_t<Source>::kWaits, kShared = std::remove_reference_t<Source>::kShared;
  constexpr int kAcc = 8 / kLanes;
  float m[kAcc], s[kAcc];
  int idx[kAcc];
#pragma unroll
  for (int a = 0; a < kAcc; ++a) {
    m[a] = -INFINITY;
    s[a] = 0.f;
    idx[a] = 0x7fffffff;
  }
  // this lane's slices are sub, sub + kLanes, sub + 2 kLanes, ...; slice number t
  // goes to accumulator t mod kAcc.  They are fetched kBatch at a time, all
  // loads of a batch in flight together; a missing slice merges as the identity.
  constexpr int kBatch = kAcc > kAtOnce ? kAcc : kAtOnce;
  static_assert(kBatch % kAcc == 0, "slice number t of a lane goes to accumulator t mod kAcc");
  for (int t0 = 0; sub + kLanes * t0 < splits; t0 += kBatch) {
    Partial q[kBatch];
    auto fetch = [&]() {
      bool all = true;
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int k = sub + kLanes * (t0 + u);
        q[u] = Partial{-INFINITY, 0.f, 0x7fffffff, 0};
        if (k < splits && state == mask_id) {  // the slices of an unmasked row were never written
          const int4* at = reinterpret_cast<const int4*>(p + k);
          const int4 w = kShared ? *at : kWaits ? load16(at) : __ldcg(at);
          q[u] = Partial{__int_as_float(w.x), __int_as_float(w.y), w.z, w.w};
        }
      }
      if constexpr (kWaits) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
          if (sub + kLanes * (t0 + u) < splits && state == mask_id) all &= q[u].pad == from.tag;
      }
      return all;
    };
    if constexpr (kWaits) {
      unsigned polls = from.polls;
      while (!from.missing && !fetch())
        if (polls-- == 0) from.missing = true;
    } else {
      fetch();
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      merge(m[u % kAcc], s[u % kAcc], idx[u % kAcc], q[u].m, q[u].s, q[u].idx);
  }
#pragma unroll
  for (int oa = kAcc / 2; oa > 0; oa >>= 1) {  // butterfly steps 4.. down to kLanes
#pragma unroll
    for (int a = 0; a < kAcc; ++a)
      if (a < oa) merge(m[a], s[a], idx[a], m[a + oa], s[a + oa], idx[a + oa]);
  }
#pragma unroll
  for (int off = kLanes / 2; off > 0; off >>= 1) {  // the remaining steps cross lanes
    const float m2 = __shfl_xor_sync(0xffffffffu, m[0], off);
    const float s2 = __shfl_xor_sync(0xffffffffu, s[0], off);
    const int i2 = __shfl_xor_sync(0xffffffffu, idx[0], off);
    merge(m[0], s[0], idx[0], m2, s2, i2);
  }
  const bool masked = state == mask_id;
  conf = masked ? fminf(1.0f, 1.0f / s[0]) : -INFINITY;  // the sum can round just below one
  tok = masked ? idx[0] : state;
  // a usable row has a finite maximum and a finite, positive sum (the sum is one or more up to rounding)
  return !(masked && (!(fabsf(m[0]) < INFINITY) || !(s[0] > 0.f) || !(s[0] < INFINITY)));
}

// One warp applies the unmasking rule of Sec. 3.1 (Algorithm 1, step 3) to one
// node; lane k owns positions k and k + 32.  conf: the node's L confidences,
// -inf at unmasked positions.  Returns the bit mask of positions to unmask.
// kMarks: a NaN marks a masked row without a usable distribution (the sampled decision's; the greedy
// one's confidences are numbers).  It is passed over, and where a node has no other masked row the first
// masked position is taken, so that decoding always advances.
// Few positions are taken one after the other, each the most confident of those left, the first of
// several (a maximum and two votes, whatever L); more than kRounds, or a quarter of the block, by their ranks
// (a look at every position, whatever S).  Rounds and ranks, decision and walk, us: 2 x 33 nodes x 12 positions, six
// of them taken 8.95 8.35, eight 9.44 8.40; 4 x 64 x 8, two 10.3 10.5, four 11.0 10.5, eight 11.4 10.5; 16 x 32, eight
// 7.4 7.2; 8 x 64, eight 7.2 8.4.
template <bool kMarks = false>
__device__ __forceinline__ uint64_t unmask_rule(const float* conf, const int32_t* state, int L,
                                                int mask_id, int rule, int top_s, float tau,
                                                int lane) {
  constexpr int kRounds = 8;
  const unsigned full = 0xffffffffu;
  auto masked = [&](int l) { return l < L && state[min(l, L - 1)] == mask_id; };
  float c[2];  // -inf: not to be taken
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int l = lane + 32 * h;
    c[h] = masked(l) ? conf[l] : -INFINITY;
    if (kMarks && c[h] != c[h]) c[h] = -INFINITY;
  }
  const bool tops = rule == SPIFFY_RULE_TOPS;
  uint64_t bits = 0;
  if (!tops)  // strict, Sec. 3.1
    bits = (uint64_t)__ballot_sync(full, c[0] > tau) | (uint64_t)__ballot_sync(full, c[1] > tau) << 32;
  if (tops && (top_s > kRounds || L <= 4 * top_s)) {
    // rank among the usable positions by (confidence desc, position asc)
    bool take[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int l = lane + 32 * h;
      int rank = 0;
      if (c[h] != -INFINITY) {
        for (int j = 0; j < L; ++j) {
          const float cj = conf[j];  // a NaN is ahead of nothing
          rank += (cj > c[h] || (cj == c[h] && j < l)) ? 1 : 0;
        }
      }
      take[h] = c[h] != -INFINITY && rank < top_s;
    }
    bits = (uint64_t)__ballot_sync(full, take[0]) | (uint64_t)__ballot_sync(full, take[1]) << 32;
  } else if (!bits) {  // the threshold rule: the single most confident position, where none passes
#pragma unroll 1
    for (int left = tops ? top_s : 1; left > 0; --left) {
      const float best = warp_max(fmaxf(c[0], c[1]));
      if (best == -INFINITY) break;  // all taken
      const unsigned lo = __ballot_sync(full, c[0] == best), hi = __ballot_sync(full, c[1] == best);
      const int at = lo ? __ffs(lo) - 1 : __ffs(hi) + 31;
      bits |= 1ull << at;
      if (lane == at) c[0] = -INFINITY;
      if (lane + 32 == at) c[1] = -INFINITY;
    }
  }
  if (kMarks && !bits) {  // no usable row
    const uint64_t any = (uint64_t)__ballot_sync(full, masked(lane)) | (uint64_t)__ballot_sync(full, masked(lane + 32)) << 32;
    bits = any & (0ull - any);
  }
  return bits;
}

}  // namespace
}  // namespace spiffy
