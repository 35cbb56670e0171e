// What the two tensor-core attention kernels share: the description of a problem as
// the kernels get it, the mask of a key tile, and small device helpers.
#pragma once
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tma_map.cuh"

namespace spiffy {

using namespace sm100;

constexpr int BM = 128;  // rows of an M-tile (a pair of CTAs: 64 each)
constexpr int BN = 128;  // keys per key tile
// An accumulator is rescaled only when its row's maximum grew by more than 2^8 (exact: accumulator
// and sum always share one reference maximum).
constexpr float kRescaleLog2 = 8.0f;

struct Params {
  int B, N, L, Hq, Hkv, group;
  int P, P2;    // context keys: first and second segment
  int TNL;      // (node, position) pairs per M-tile
  int NL;       // N * L
  int TP1, TP;  // context key tiles: of the first segment, of both
  int log_cs;   // CTAs of a cluster that share an M-tile's key tiles: 1, 2, 4 or 8
  // A launch that takes a part of the call only, in one row of CTAs: its first M-tile, counted over all
  // (sequence, key/value head) pairs at `slots` each (the M-tiles of one, rounded up to even); 0: the
  // grid's y and z are key/value head and sequence.
  int first, slots;
  float scale_log2;
  __nv_bfloat16* out;
  int32_t* status;
  uint32_t spin_limit;  // polls of one mbarrier wait
  int early_trigger;    // let the next kernel of the stream begin its set-up while this one runs
  int independent;      // the kernel before this one writes none of its inputs: waited for at the end
};

// The operands of one attention problem: Q, two context segments, block keys.
struct Maps {
  CUtensorMap q, kp, vp, kp2, vp2, kb, vb;
};
// One launch runs one problem, or two side by side (the nodes and the trailing rows of a
// full-sequence model): the CTAs from x_split on along grid.x work on the second.
template <int NP>
struct Problems {
  Maps maps[NP];
  Params p[NP];
  int x_split;
};

// Which M-tile, head and sequence: `unit` is the M-tile among those of the CTA's row of the grid.
struct Place {
  int mt, g, b;
};
// (Two problems are one launch always: spared the look, 2 % of a short call.)
template <int NP>
__device__ __forceinline__ Place place_of(const Params& p, int unit) {
  if (NP == 2 || p.slots == 0) return {unit, (int)blockIdx.y, (int)blockIdx.z};
  const int at = p.first + unit, bg = at / p.slots;
  return {at - bg * p.slots, bg % p.Hkv, bg / p.Hkv};
}
template <int NP>
__device__ __forceinline__ bool no_such_tile(const Params& p, int unit) {
  return NP == 1 && p.slots != 0 && (p.first + unit) % p.slots * p.TNL >= p.NL;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Bounded wait that ignores the abort flag: for what must not be in flight when the block ends.
__device__ __forceinline__ void mbar_wait_quiet(uint64_t* bar, uint32_t parity) {
#pragma unroll 1
  for (uint32_t i = 0; i < kSpinLimit; ++i)
    if (mbar_try_wait(bar, parity)) return;
}

// Row r of an M-tile sees the columns [lo, hi) of key tile t (tile-relative).
struct Window {
  int lo, hi;
};
__device__ __forceinline__ Window visible_window(const Params& p, int t, int kb_start, int node) {
  Window w;
  if (t < p.TP) {  // context: every row sees every key that exists
    w.lo = 0;
    w.hi = t < p.TP1 ? min(BN, p.P - t * BN) : min(BN, p.P2 - (t - p.TP1) * BN);
  } else {  // block keys: the row's own node only
    w.lo = node * p.L - (kb_start + (t - p.TP) * BN);
    w.hi = w.lo + p.L;
  }
  return w;
}

// attention_pair.cu: `grid` CTAs, two neighbouring ones to an M-tile.
template <int NP>
spiffy_status launch_attention_pair(const Problems<NP>& pr, int head_dim, dim3 grid, cudaStream_t stream);

}  // namespace spiffy
