// Packed draft-graph attention (Sec. 4.3; mask of Fig. 3) on the sm_100a tensor
// cores: bf16 operands, head dimension 128 or 64.
//
// Work decomposition.  For one sequence b and one key/value head g, the query
// rows are all (node n, position l, query head of the group) triples; they all
// read the same P context keys, and a row of node n additionally reads the L
// keys of node n's own block.  An M-tile is TNL consecutive (n, l) positions
// times the `group` query heads of g (TNL = 128 / group, so at most 128 rows);
// a CTA owns one M-tile, or two neighbouring ones (see the kernel), and walks
// over key tiles of 128 keys: first the context tiles,
// then the tiles covering the block keys of the nodes its rows belong to.  The
// mask is never materialised: a context tile is visible to every row, and in a
// block-key tile row r sees exactly the columns of its own node, a contiguous
// column range computed from indices.
//
// Pipeline inside a CTA (384 threads):
//   warps 0, 3  TMA producers: Q once and the K tiles, and the V tiles, into two rings
//               (seven 32 KB tiles of shared memory in all, or fourteen of 16 KB at
//               head dimension 64).  Q and the first K tile are asked for before
//               the rest of the CTA has finished setting up.
//   warp 1      allocates tensor memory and issues the score products
//               S = Q K^T (tcgen05.mma, fp32 in TMEM)
//   warp 2      issues O += P V.  A warp each, because an issuing warp
//               is held for as long as its products run: with one for both, every
//               wait for one kind of operand kept the tensor pipe from the other.
//               All of them run converged and leave the instruction itself to an
//               elected lane, and what is counted is counted along: one lane, whose
//               operands go through uniform registers one by one, and a producer that
//               divided by its ring's length took 5 to 15 % longer (28 heads on 4, 512
//               positions over 1024 keys 14.5 -> 13.6 us; 2 x 32 x 32 positions x 32 heads
//               over 4096 keys 135 -> 127; 4096 keys, 8 heads of 4, 256 positions 24.5 -> 20.7).
//   warps 4-11  two softmax warpgroups, one thread per row each.  A unit of work is
//               one (M-tile, key tile) pair; units alternate between the
//               warpgroups, each of which keeps its own running (maximum, sum) and
//               accumulator O: with two M-tiles one M-tile's, with one M-tile
//               those of every other key tile, merged once at the end.  A thread
//               reads its scores from TMEM, writes P (bf16) to TMEM as the A
//               operand of the second product, and rescales its O only when the
//               maximum grew by more than 2^8 (exact: O and the sum always share
//               one reference maximum).  32-column chunks of a block-key tile that
//               no row of a warp may see are skipped.
// S and P have TMEM columns of their own, and there is one S: it is free again as
// soon as a warpgroup holds it in registers, so the scores of the next unit are
// formed while the exponentials of this one are taken, P V of this one runs under
// the exponentials of the next, and the hand-over keeps the two warpgroups half a
// unit apart.  Measured, 2 x 32 x 32 positions x 32 heads over 4096 keys: 127 us; of
// the 132 it once was, 109 were left when all arithmetic of the softmax was taken out: what bounds a
// long run is the round trip of the one S buffer (products 512 cycles, wake-up of
// the warpgroup, read, wake-up of the issuing thread: about 1500 per unit against
// 1024 of products).  P written over its S instead, with two of each, an issuing
// thread per stream and P V started on the first half of P: 192 us, the streams
// fall into step.  Two S buffers, P and two O do not fit tensor memory.
// Most CTAs run few units, and much of their time is instructions executed once:
// loops that are not the inner ones stay rolled (a kernel of 87 KB instead of 60
// cost 2 us of 19 at 9 units).
// With few CTAs the key tiles of an M-tile are split over the 2, 4 or 8 CTAs of a
// cluster.  Each finishes its share of the rows: it sends its partial of
// the others' rows into their shared memory, one bulk copy each, and merges what it
// gets.
//
// Head dimension 64 halves every tile (one 64-column half instead of two) and the
// products, not the exponentials.  The CUDA-core kernel, which this one stands in for
// there, keeps P in fp32: here P enters the second product as two bf16 terms, its
// upper half and what that leaves (to 2^-16 of a value, in the tensor memory that the
// narrower O leaves), so that the result's error against float64 is the CUDA cores'
// (0.166 % in the 2-norm, the rounding of the output, over 50 to 4096 keys; with one
// term 0.18 to 0.23 %).  The second term costs 5 to 20 % (4 x 32 x 32 positions x 32
// heads over 4096 keys: 232 -> 262 us when it came; CUDA cores 4596).
//
// Every wait is bounded; a wait that gives up raises SPIFFY_DEV_TIMEOUT in the
// caller's status word and the CTA winds down without touching its output.
#include "attention_tc.cuh"

namespace spiffy {
namespace {

constexpr int kThreads = 384;  // a warpgroup with the producer and the MMA warp, two softmax warpgroups
// Registers per thread: 168 at launch (65536 / 384 in steps of 8); the softmax warps, which hold
// 128 scores each with two M-tiles, take over what the first warpgroup does not need.
constexpr int kRegsIssue = 40, kRegsSoftmax = 232;
static_assert(kRegsIssue + 2 * kRegsSoftmax <= 3 * 168, "within what the block was launched with");
constexpr int kHalfBytes = BN * 128;           // one 64-column half of a tile: 128 rows x 128 B
constexpr uint32_t kTmemCols = 512;
// S: 128 columns; warpgroup w: P (bf16 pairs) at 128 + 64 w, O at 256 + w * head dim, and at head
// dimension 64, P's second term at 384 + 64 w
constexpr uint32_t kColS = 0, kColP = 128, kColO = 256, kColRest = 384;
static_assert(kColRest + 2 * 64 <= kTmemCols && kColO + 2 * 64 <= kColRest, "tensor memory at head dimension 64");
// Shared memory: NQ Q tiles, a K ring of 3 stages and a V ring of 4 - NQ, seven tiles of
// 32 KB in all; at head dimension 64 fourteen of 16 KB.  (The same amount for all: two
// CTAs must not share an SM, each holds all of its tensor memory until it exits.)
template <int NQ, int HD>
struct Smem {
  static constexpr int tile = BN * HD * 2;  // bytes
  static constexpr int ks = HD == 128 ? 3 : 6, vs = 14 * 64 / HD - NQ - ks;
  static constexpr int q = 0;
  static constexpr int k = q + NQ * tile;
  static constexpr int v = k + ks * tile;
  static constexpr int bars = v + vs * tile;
  static constexpr int n_bars = 1 + 2 * ks + 2 * vs + 4 + 2 + 2 + 2;
  static constexpr int tmem = bars + 8 * n_bars;
  static constexpr int abort_flag = tmem + 8;
  static constexpr int rows = abort_flag + 8;  // int [NQ][128]: where a row of an M-tile is stored
  static constexpr int total = rows + NQ * BM * 4;
};
constexpr int most(int a, int b) { return a > b ? a : b; }
constexpr int kSmemBytes = most(most(Smem<1, 64>::total, Smem<2, 64>::total), most(Smem<1, 128>::total, Smem<2, 128>::total)) +
                           1024;  // slack for 1024-byte alignment
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");

// The maximum of one thread's scores of a row (raw bits, -inf where masked).
__device__ __forceinline__ float row_max(const uint32_t (&s)[BN]) {
  float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
  for (int c = 0; c < BN; c += 8) {
    mx0 = max3(mx0, __uint_as_float(s[c]), __uint_as_float(s[c + 1]));
    mx1 = max3(mx1, __uint_as_float(s[c + 2]), __uint_as_float(s[c + 3]));
    mx2 = max3(mx2, __uint_as_float(s[c + 4]), __uint_as_float(s[c + 5]));
    mx3 = max3(mx3, __uint_as_float(s[c + 6]), __uint_as_float(s[c + 7]));
  }
  return fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
}

// p = 2^(s * k2 - m_use) for the flagged 32-column chunks among columns C0 .. C0 + 63 (zero
// elsewhere), packed as bf16 pairs into pk; returns the sum of the p's (fp32, before rounding to
// bf16).  kRest: pk holds the upper 16 bits of p and rest what they leave of it, rounded to bf16, so
// that pk + rest is p to 2^-16.
// The special-function unit takes 8 cycles per warp and exponential; everything else a pair
// needs fits under its two.
template <int C0, bool kRest>
__device__ __forceinline__ float row_exps(const uint32_t (&s)[BN], uint32_t need, float k2, float m_use,
                                          uint32_t (&pk)[32], uint32_t (&rest)[32]) {
  const uint64_t k22 = pack2(k2, k2), nm2 = pack2(-m_use, -m_use);
  uint64_t sum_a = pack2(0.f, 0.f), sum_b = pack2(0.f, 0.f);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if ((need >> (C0 / 32 + h)) & 1u) {
#pragma unroll
      for (int c = 32 * h; c < 32 * h + 32; c += 2) {
        const uint64_t x2 = fma2(pack2(__uint_as_float(s[C0 + c]), __uint_as_float(s[C0 + c + 1])), k22, nm2);
        float x0, x1;
        unpack2(x2, x0, x1);
        const float p0 = ex2(x0), p1 = ex2(x1);
        if ((c >> 1) & 1) sum_b = add2(sum_b, pack2(p0, p1)); else sum_a = add2(sum_a, pack2(p0, p1));
        if constexpr (kRest) {  // cut off instead of rounded: a byte permutation, no conversion
          const uint32_t w0 = __float_as_uint(p0), w1 = __float_as_uint(p1);
          pk[c >> 1] = __byte_perm(w0, w1, 0x7632);
          float r0, r1;
          unpack2(fma2(pack2(__uint_as_float(w0 & 0xffff0000u), __uint_as_float(w1 & 0xffff0000u)), pack2(-1.f, -1.f),
                       pack2(p0, p1)), r0, r1);
          rest[c >> 1] = pack_bf16(r0, r1);
        } else {
          pk[c >> 1] = pack_bf16(p0, p1);
        }
      }
    } else {
#pragma unroll
      for (int c = 16 * h; c < 16 * h + 16; ++c) {
        pk[c] = 0u;
        if (kRest) rest[c] = 0u;
      }
    }
  }
  float a0, a1;
  unpack2(add2(sum_a, sum_b), a0, a1);
  return a0 + a1;
}

// NQ = 1: the CTA owns one M-tile; unit u is key tile u.
// NQ = 2: the CTA owns two neighbouring M-tiles; unit u is M-tile u & 1, key tile
// u >> 1.  Every K/V tile brought into shared memory serves both, which halves the
// L2-to-SM traffic per flop.
// Unit u belongs to warpgroup u & 1 and to accumulator u & 1 either way.
template <int NQ, int HD, int NP>
__global__ void __launch_bounds__(kThreads, 1)
graph_attention_tc_kernel(const __grid_constant__ Problems<NP> problems) {
  extern __shared__ uint8_t smem_raw[];
  // an offset, not a rounded address: the compiler still knows that this is shared memory
  uint8_t* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
  using SM = Smem<NQ, HD>;
  constexpr int KS = SM::ks, VS = SM::vs, kTileBytes = SM::tile;
  constexpr int kHalves = HD / 64;    // 64-column halves of a tile
  constexpr bool kRest = HD == 64;    // P in two bf16 terms
  constexpr int kLogNQ = NQ - 1;      // key tile of unit u = u >> kLogNQ
  uint8_t* sq = smem + SM::q;
  uint8_t* sk = smem + SM::k;
  uint8_t* sv = smem + SM::v;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::bars);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;
  uint64_t* k_empty = k_full + KS;
  uint64_t* v_full = k_empty + KS;
  uint64_t* v_empty = v_full + VS;
  // one barrier per parity of the unit: no waiter may see a phase of the same parity that is not its own
  uint64_t* s_full = v_empty + VS;     // [2] scores formed
  uint64_t* s_free = s_full + 2;       // [2] ... and read
  uint64_t* p_ready = s_free + 2;      // [2] P written
  uint64_t* pv_done = p_ready + 2;     // [2] ... and consumed: their P V products are done
  uint64_t* xchg_ready = pv_done + 2;  // cluster: the others' K rings may be written
  uint64_t* xchg_full = xchg_ready + 1;  // cluster: the others' partials have arrived here
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + SM::tmem);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SM::abort_flag);
  volatile int* invited = abort_flag + 1;  // cluster: the others have been told that they may send
  int* rows = reinterpret_cast<int*>(smem + SM::rows);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // uniform to the compiler
  const int which = NP == 2 && (int)blockIdx.x >= problems.x_split ? 1 : 0;
  const Maps& maps = problems.maps[which];
  const Params& p = problems.p[which];
  const int log_cs = NQ == 1 ? p.log_cs : 0, cs = 1 << log_cs;
  const int rank = NQ == 1 ? (int)blockIdx.x & (cs - 1) : 0;  // of this CTA in its cluster
  const int unit = (((int)blockIdx.x - (which ? problems.x_split : 0)) >> log_cs) * NQ;  // the first of this CTA's M-tiles
  if (no_such_tile<NP>(p, unit)) return;
  // Set-up, by warps side by side.
  if (warp == 0) {
    // one lane per barrier: a thread's initialisations are served one after the other
    static_assert(SM::n_bars <= 64, "two rounds of lanes");
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint64_t* bar = bars + lane + 32 * h;
      // s_free and p_ready: the four warps of a softmax warpgroup arrive once each
      const bool four = bar >= s_free && bar < pv_done;
      if (bar < bars + SM::n_bars) mbar_init(bar, four ? 4u : bar == xchg_ready ? (uint32_t)max(cs - 1, 1) : 1u);
    }
    if (lane == 0) *abort_flag = *invited = 0;
    mbar_fence_init();
  } else if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
  } else if (warp == 2 && lane == 0) {
    prefetch_tensormap(&maps.q);  // the descriptors are kernel parameters
    prefetch_tensormap(p.TP1 > 0 ? &maps.kp : (p.TP > 0 ? &maps.kp2 : &maps.kb));
    prefetch_tensormap(p.TP1 > 0 ? &maps.vp : (p.TP > 0 ? &maps.vp2 : &maps.vb));
  }
  __syncwarp();
  // this CTA's rows and key tiles
  const Place place = place_of<NP>(p, unit);
  const int nl0 = place.mt * p.TNL, g = place.g, b = place.b;
  const int nl_count = min(NQ * p.TNL, p.NL - nl0);  // over all M-tiles of the CTA
  const int rows_box = p.TNL * p.group;        // rows one Q box writes
  const int n_lo = nl0 / p.L, n_hi = (nl0 + nl_count - 1) / p.L;
  const int kb_start = n_lo * p.L;
  const int TB = ((n_hi - n_lo + 1) * p.L + BN - 1) / BN;
  const int T_all = p.TP + TB;
  const int t_begin = (rank * T_all) >> log_cs;  // small numbers: cs <= 8, T_all at most a few thousand
  const int T = (((rank + 1) * T_all) >> log_cs) - t_begin;  // >= 1: cs <= T_all

  // The roles' waits, by whole warps.
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, p.spin_limit));
  };
  // Producers: the next tile of the K ring (warp 0) or of the V ring (warp 3).  Everything is counted
  // along: a division by a number the compiler does not know takes some 200 cycles.
  const bool is_k = warp == 0;
  int issued = 0, next_stage = 0;
  uint32_t round = 0;
  auto produce = [&]() -> bool {
    if (round > 0 && !wait((is_k ? k_empty : v_empty) + next_stage, (round & 1u) ^ 1u)) return false;
    uint64_t* full = (is_k ? k_full : v_full) + next_stage;
    const int t = t_begin + issued;
    // key tiles in order: first context segment, second context segment, block keys
    const int seg = t < p.TP1 ? 0 : (t < p.TP ? 1 : 2);
    const CUtensorMap* m = is_k ? (seg == 0 ? &maps.kp : seg == 1 ? &maps.kp2 : &maps.kb)
                                : (seg == 0 ? &maps.vp : seg == 1 ? &maps.vp2 : &maps.vb);
    const int key0 = seg == 0 ? t * BN : seg == 1 ? (t - p.TP1) * BN : kb_start + (t - p.TP) * BN;
    mbar_arrive_expect_tx(full, kTileBytes);
    tma_load_5d((is_k ? sk : sv) + next_stage * kTileBytes, m, full, 0, g, key0, 0, b);
    ++issued;
    if (++next_stage == (is_k ? KS : VS)) {
      next_stage = 0;
      ++round;
    }
    return true;
  };

  constexpr int kRowBytes = HD * 4;  // of an fp32 partial
  if (warp == 0) {
    // what the others will send in the epilogue: this CTA's rows, and (maximum, sum) of each
    if (cs > 1) mbar_arrive_expect_tx(xchg_full, (uint32_t)((cs - 1) * (BM >> log_cs) * (kRowBytes + 8)));
    if (!p.independent) cudaGridDependencySynchronize();
    mbar_arrive_expect_tx(q_full, (uint32_t)(NQ * kHalves) * rows_box * 128u);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {  // an M-tile beyond the last one reads as zeros
#pragma unroll
      for (int h = 0; h < kHalves; ++h)  // with fewer than 128 rows in the box the halves lie further apart than it is long
        tma_load_5d(sq + q * kTileBytes + h * kHalfBytes, &maps.q, q_full, 0, g * p.group, nl0 + q * p.TNL, h, b);
    }
    produce();
  }
  // rows of the Q tile that the TMA box does not write must be finite
  for (int i = rows_box * 8 + threadIdx.x; i < BM * 8; i += kThreads) {
    const uint4 z = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int h = 0; h < kHalves * NQ; ++h) reinterpret_cast<uint4*>(sq + h * kHalfBytes)[i] = z;
  }
  fence_proxy_async_smem();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  // all CTAs' barriers exist before any touches another's (waited for in the epilogue)
  if (cs > 1) cluster_arrive_relaxed();
  if (p.early_trigger) pdl_launch_dependents();
  // everything above is on-chip set-up (thread 0 aside); global memory is touched from here on
  if (!p.independent) cudaGridDependencySynchronize();

  const int U = T << kLogNQ;  // units of this CTA
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    if (warp == 0 || warp == 3) {
      // ----------------------------------------------------------- producers --
      while (issued < T && produce()) {
      }
      // Whoever gives up, and when: no copy is in flight into shared memory whose block has ended.
      if (is_k) mbar_wait_quiet(q_full, 0);
      const int depth = is_k ? KS : VS;
      for (int k = min(issued, depth); k > 0; --k) {
        if (--next_stage < 0) {
          next_stage = depth - 1;
          --round;
        }
        mbar_wait_quiet((is_k ? k_full : v_full) + next_stage, round & 1u);
      }
    } else if (warp == 1) {
      // ------------------------------------------------ issuer of S = Q K^T --
      constexpr uint32_t idesc = idesc_bf16_f32(BM, BN, false, false);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      const uint32_t q_lo = desc_lo_sw128(smem_u32(sq), 16);
      const uint32_t k_lo = desc_lo_sw128(smem_u32(sk), 16);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = wait(q_full, 0);
      for (int u = 0; u < U && ok; ++u) {
        if (NQ == 1 || (u & 1) == 0) ok = wait(k_full + stage, phase);
        // the scores before have been read
        if (ok && u >= 1) ok = wait(s_free + ((u - 1) & 1), (uint32_t)((u - 1) >> 1) & 1u);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t qa = q_lo + (NQ == 2 ? (uint32_t)(u & 1) * (kTileBytes >> 4) : 0u);
        const uint32_t ka = k_lo + (uint32_t)stage * (kTileBytes >> 4);
        if constexpr (HD == 128) umma_ss_k128(tmem + kColS, qa, ka, hi, idesc, 0u);
        else umma_ss_k64(tmem + kColS, qa, ka, hi, idesc, 0u);
        umma_commit(s_full + (u & 1));
        if (NQ == 1 || (u & 1)) {  // a key tile serves all M-tiles before it is released
          umma_commit(k_empty + stage);
          if (++stage == KS) { stage = 0; phase ^= 1u; }
        }
      }
    } else if (warp == 2) {
      // --------------------------------------------------- issuer of O += P V --
      constexpr uint32_t idesc = idesc_bf16_f32(BM, HD, false, true);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      const uint32_t v_lo = desc_lo_sw128(smem_u32(sv), kHalfBytes);
      int stage = 0;
      uint32_t phase = 0;
      for (int u = 0; u < U; ++u) {
        if ((NQ == 1 || (u & 1) == 0) && !wait(v_full + stage, phase)) break;
        if (!wait(p_ready + (u & 1), (uint32_t)(u >> 1) & 1u)) break;
        tc_fence_after_sync();
        umma_ts_k128(tmem + kColO + (uint32_t)(u & 1) * HD, tmem + kColP + (uint32_t)(u & 1) * 64u,
                     v_lo + (uint32_t)stage * (kTileBytes >> 4), hi, idesc, u >= 2 ? 1u : 0u);
        if constexpr (kRest)
          umma_ts_k128(tmem + kColO + (uint32_t)(u & 1) * HD, tmem + kColRest + (uint32_t)(u & 1) * 64u,
                       v_lo + (uint32_t)stage * (kTileBytes >> 4), hi, idesc, 1u);
        umma_commit(pv_done + (u & 1));
        if (NQ == 1 || (u & 1)) {
          umma_commit(v_empty + stage);
          if (++stage == VS) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else {
    // ------------------------------------------------------------- softmax --
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    const int quad = warp & 3;               // TMEM lane quadrant this warp may touch
    const int wg = (warp - 4) >> 2;
    const int r = quad * 32 + lane;          // row of the M-tile
    const int nl_tile = nl0 + (NQ == 2 ? wg * p.TNL : 0);  // first (node, position) of the rows
    const int rows_valid = max(0, min(p.TNL, p.NL - nl_tile)) * p.group;
    const int node = min(nl_tile + r / p.group, p.NL - 1) / p.L;
    const uint32_t lane_base = (uint32_t)(quad * 32);
    const float k2 = p.scale_log2;
    // key tiles every row sees whole: t < full_a, and TP1 <= t < full_b
    const int full_a = p.P / BN, full_b = p.TP1 + p.P2 / BN;
    float m_run = -INFINITY, l_run = 0.f;  // reference maximum (log2 units) and sum of this thread's accumulator
    bool ok = true;
    const uint32_t at_p = tmem_addr(tmem, lane_base, kColP + (uint32_t)wg * 64u);
    const uint32_t at_o = tmem_addr(tmem, lane_base, kColO + (uint32_t)wg * HD);
    const uint32_t at_rest = tmem_addr(tmem, lane_base, kColRest + (uint32_t)wg * 64u);
    // the P V products of unit u (one of this warpgroup's) have completed
    auto wait_pv = [&](int u) -> bool {
      const bool yes = __all_sync(0xffffffffu, mbar_wait(pv_done + wg, (uint32_t)(u >> 1) & 1u, abort_flag, p.spin_limit));
      tc_fence_after_sync();
      return yes;
    };
    // The row's place in the output, relative to the M-tile's, -1 beyond the last row: looked up
    // by whoever stores the row in the end.
    if (NQ == 2 || wg == 0)
      rows[(NQ == 2 ? wg * BM : 0) + r] = r < rows_valid ? (r / p.group * p.Hq + r % p.group) * HD : -1;
    __nv_bfloat16* out_tile = p.out + (((int64_t)b * p.NL + nl_tile) * p.Hq + (int64_t)g * p.group) * HD;
    if (cs > 1) cluster_wait();  // phase 1: the other CTAs' barriers exist
    for (int u = wg; u < U; u += 2) {
      const int j = u >> kLogNQ;
      // wait outcomes are made warp-uniform: the TMEM accesses below are warp-collective
      if (!__all_sync(0xffffffffu, mbar_wait(s_full + wg, (uint32_t)(u >> 1) & 1u, abort_flag, p.spin_limit))) {
        ok = false;
        break;
      }
      tc_fence_after_sync();
      // the last scores have been formed: the Q tile and the K ring are free for the others' partials
      if (cs > 1 && u == U - 1 && quad == 0 && lane < cs) {
        if (lane != rank) mbar_arrive_remote(map_to_cta(smem_u32(xchg_ready), (uint32_t)lane));
        else *invited = 1;
      }
      uint32_t s[BN];
      tmem_ld_x128(tmem_addr(tmem, lane_base, kColS), s);
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(s_free + wg);
      // 32-column chunks that no row of the warp sees cost nothing but zeros in P
      uint32_t chunks = 0xfu;
      const int t = t_begin + j;
      if (t >= full_a && (t < p.TP1 || t >= full_b)) {
        const Window w = visible_window(p, t, kb_start, node);
#pragma unroll
        for (int h = 0; h < BN / 32; ++h) {
          const int lo = w.lo - 32 * h, hi = w.hi - 32 * h;
          if (!__any_sync(0xffffffffu, lo < 32 && hi > 0)) chunks &= ~(1u << h);
          // bit c: column 32 h + c is visible
          const uint32_t upto = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
          const uint32_t below = lo >= 32 ? 0xffffffffu : lo <= 0 ? 0u : (1u << lo) - 1u;
          const uint32_t seen = upto & ~below;
#pragma unroll
          for (int c = 0; c < 32; ++c)
            s[32 * h + c] = (seen >> c) & 1u ? s[32 * h + c] : 0xff800000u;  // -inf
        }
      }
      const float mx = row_max(s);
      const float m_new = fmaxf(m_run, mx * k2);
      const bool need = (m_new - m_run) > kRescaleLog2;  // false when both are -inf
      if (__any_sync(0xffffffffu, need)) {
        float corr = 1.f;
        if (need) {
          corr = ex2(m_run - m_new);  // 0 for a row that had seen nothing yet
          l_run *= corr;
          m_run = m_new;
        }
        if (u >= 2) {  // the accumulator holds earlier tiles: O *= corr once their products are done
          ok = wait_pv(u - 2);
          if (!ok) break;
#pragma unroll 1
          for (uint32_t c0 = 0; c0 < HD; c0 += 32) {
            uint32_t o[32];
            tmem_ld_x32(at_o + c0, o);
#pragma unroll
            for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * corr);
            tmem_st_x32(at_o + c0, o);
          }
          tmem_wait_st();
        }
      }
      const float m_use = (m_run == -INFINITY) ? 0.f : m_run;
      uint32_t pk[32], rest[32];
      l_run += row_exps<0, kRest>(s, chunks, k2, m_use, pk, rest);
      // the products that read this P buffer last (two units ago) are done
      ok = u < 2 || wait_pv(u - 2);
      if (!ok) break;
      tmem_st_x32(at_p, pk);
      if (kRest) tmem_st_x32(at_rest, rest);
      l_run += row_exps<64, kRest>(s, chunks, k2, m_use, pk, rest);
      tmem_st_x32(at_p + 32u, pk);
      if (kRest) tmem_st_x32(at_rest + 32u, rest);
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();  // every lane's P is in tensor memory: one arrival speaks for the warp
      if (lane == 0) mbar_arrive(p_ready + wg);
    }
    // ------------------------------------------------------------ epilogue --
    // every product into this thread's accumulator has completed
    if (ok && wg < U) ok = wait_pv(U - 1 - ((U - 1 - wg) & 1));
    tc_fence_after_sync();
    // Results pass through shared memory, 16-byte chunks XOR-swizzled by row (no bank conflicts
    // either way), so that whole rows are stored at once.
    if constexpr (NQ == 2) {
      // each warpgroup owns its rows outright; its M-tile's Q tile has been read for the last time
      uint8_t* stage = sq + wg * kTileBytes;
      constexpr int kChunks = HD / 8;  // of a bf16 row
      if (ok) {
        const float inv = 1.0f / l_run;
#pragma unroll
        for (int c0 = 0; c0 < HD; c0 += 64) {
          uint32_t o[2][32];
          tmem_ld_async(at_o + (uint32_t)c0, o[0]);
          tmem_ld_async(at_o + (uint32_t)c0 + 32u, o[1]);
          tmem_wait_ld();
          tmem_loaded(o[0]);
          tmem_loaded(o[1]);
#pragma unroll
          for (int c = 0; c < 64; c += 8) {
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(o[c / 32][c % 32 + e]) * inv;
            *reinterpret_cast<uint4*>(stage + r * (HD * 2) + ((((c0 + c) / 8) ^ (r & 7)) << 4)) =
                make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
          }
        }
      }
      asm volatile("bar.sync %0, 128;" ::"r"(1 + wg) : "memory");  // the warpgroup, whatever `ok` says
      if (ok) {
        constexpr int kStep = 128 / kChunks;  // rows per pass
        const int row0 = (int)(threadIdx.x & 127) / kChunks, chunk = (int)threadIdx.x % kChunks;
#pragma unroll 8
        for (int k = 0; k < BM / kStep; ++k) {
          const int row = row0 + k * kStep, at = rows[wg * BM + row];
          const uint4 w = *reinterpret_cast<const uint4*>(stage + row * (HD * 2) + ((chunk ^ (row & 7)) << 4));
          if (at >= 0) st_global(out_tile + at + chunk * 8, w);
        }
      }
    } else {
      // The two warpgroups exchange their (reference maximum, sum) per row through shared memory
      // (the Q tile: every product has completed once both are here), and each merges one half of
      // the columns of both accumulators.
      float2* ml = reinterpret_cast<float2*>(sq);  // [2][128]
      asm volatile("bar.sync 1, 256;" ::: "memory");  // all eight softmax warps, whatever `ok` says
      ml[wg * BM + r] = make_float2(m_run, l_run);
      tc_fence_before_sync();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      tc_fence_after_sync();
      const float2 ml_a = ml[r], ml_b = ml[BM + r];
      const float m_all = fmaxf(ml_a.x, ml_b.x);
      // an accumulator whose tiles held no visible key of this row is left out
      const bool has_a = ml_a.x != -INFINITY, has_b = ml_b.x != -INFINITY;
      const float w_a = has_a ? ex2(ml_a.x - m_all) : 0.f;
      const float w_b = has_b ? ex2(ml_b.x - m_all) : 0.f;
      const float l_all = w_a * ml_a.y + w_b * ml_b.y;
      const int tid = (int)threadIdx.x - 128;  // among the softmax warps
      // Rows rank R .. rank R + R - 1 are finished here, R = 128 / cs.  With cs > 1 the other key
      // tiles went to the other CTAs of the cluster: every CTA leaves its partial of all rows in
      // its own shared memory (V ring) and copies the others' shares, each one piece, into their K
      // rings (idle since their last scores).  Hand-over by mbarriers: xchg_ready = "my buffers
      // are free" (sent from the tile loop by every other CTA), xchg_full = "your partials have
      // landed", completed by the byte counts of the copies.
      const int R = BM >> log_cs;
      float2* ml_mine = ml + 2 * BM;  // [128] of this CTA's partial
      float2* ml_recv = ml + 3 * BM;  // [cs][R] of this CTA's rows, its own among them
      float* weight = reinterpret_cast<float*>(ml + 4 * BM);  // [cs][R] what a slice's partial counts
      if (ok) {
        // half of the columns of the two accumulators, merged against m_all
        constexpr int W = HD / 4;
        uint32_t oa[2][W], ob[2][W];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t c0 = (uint32_t)(wg * (HD / 2) + h * W);
          tmem_ld_async(tmem_addr(tmem, lane_base, kColO + c0), oa[h]);
          tmem_ld_async(tmem_addr(tmem, lane_base, kColO + HD + c0), ob[h]);
        }
        tmem_wait_ld();
        const float f = cs == 1 ? 1.0f / l_all : 1.0f;
        const float f_a = w_a * f, f_b = w_b * f;
        const bool both = __all_sync(0xffffffffu, has_a && has_b);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_loaded(oa[h]);
          tmem_loaded(ob[h]);
          if (!both) {  // rare: an accumulator that was never written may hold anything
#pragma unroll
            for (int c = 0; c < W; ++c) {
              if (!has_a) oa[h][c] = 0u;
              if (!has_b) ob[h][c] = 0u;
            }
          }
          const int c0 = wg * (HD / 2) + h * W;
#pragma unroll
          for (int c = 0; c < W; c += 4) {
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              o[e] = fmaf(__uint_as_float(oa[h][c + e]), f_a, __uint_as_float(ob[h][c + e]) * f_b);
            *reinterpret_cast<float4*>(sv + r * kRowBytes + ((((c0 + c) / 4) ^ (r & 7)) << 4)) =
                make_float4(o[0], o[1], o[2], o[3]);
          }
        }
        if (wg == 0) {
          ml_mine[r] = make_float2(m_all, l_all);
          if (r / R == rank) ml_recv[r] = make_float2(m_all, l_all);
        }
      }
      if (cs > 1) fence_proxy_async_smem();  // the copies read what was just written
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (cs > 1) {
        if (ok && warp == 4) {
          if (mbar_wait_cluster(xchg_ready, 0, abort_flag, p.spin_limit) && lane < cs && lane != rank) {
            const uint32_t bar = map_to_cta(smem_u32(xchg_full), (uint32_t)lane);
            bulk_copy_to_cta(map_to_cta(smem_u32(sk), (uint32_t)lane) + (uint32_t)(rank * R * kRowBytes),
                             smem_u32(sv) + (uint32_t)(lane * R * kRowBytes), (uint32_t)(R * kRowBytes), bar);
            bulk_copy_to_cta(map_to_cta(smem_u32(ml_recv + rank * R), (uint32_t)lane), smem_u32(ml_mine + lane * R),
                             (uint32_t)(R * 8), bar);
          }
        }
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait_cluster(xchg_full, 0, abort_flag, p.spin_limit));
        // winding down: nobody sends before all have been told that they may; where this CTA has done
        // so, what may be on its way here lands before its shared memory goes
        if (!ok && warp == 4 && *invited) mbar_wait_quiet(xchg_full, 0);
        cluster_arrive();  // phase 2: what this CTA was sent has landed
        if (ok && tid < R) {
          float m = -INFINITY, l = 0.f;
          for (int k = 0; k < cs; ++k) m = fmaxf(m, ml_recv[k * R + tid].x);
          for (int k = 0; k < cs; ++k) {  // a slice that held no key the row sees: ex2(-inf) = 0
            const float2 part = ml_recv[k * R + tid];
            const float f = ex2(part.x - m);
            weight[k * R + tid] = f;
            l = fmaf(f, part.y, l);
          }
          const float inv = 1.0f / l;
          for (int k = 0; k < cs; ++k) weight[k * R + tid] *= inv;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
      }
      if (ok) {
        constexpr int kQuads = HD / 4;       // 16-byte chunks of an fp32 row
        constexpr int kStep = 256 / kQuads;  // rows per pass
        const int row0 = tid / kQuads, c = tid % kQuads;
        auto pack4 = [](float a, float b, float e, float f) { return make_uint2(pack_bf16(a, b), pack_bf16(e, f)); };
        if (cs == 1) {
#pragma unroll 8
          for (int k = 0; k < BM / kStep; ++k) {
            const int row = row0 + k * kStep, at = rows[row];
            const float4 q4 = *reinterpret_cast<const float4*>(sv + row * kRowBytes + ((c ^ (row & 7)) << 4));
            if (at >= 0) st_global(out_tile + at + c * 4, pack4(q4.x, q4.y, q4.z, q4.w));
          }
        } else {
          constexpr int kRows = 2;  // rows at a time
          for (int r0 = row0; r0 < R; r0 += kRows * kStep) {
            float o[kRows][4] = {};
            for (int k = 0; k < cs; ++k) {
              const uint8_t* part = k == rank ? sv + rank * R * kRowBytes : sk + k * R * kRowBytes;
#pragma unroll
              for (int e = 0; e < kRows; ++e) {
                const int rr = min(r0 + e * kStep, R - 1);  // R is a multiple of 8: rows keep their swizzle
                const float4 q4 = *reinterpret_cast<const float4*>(part + rr * kRowBytes + ((c ^ (rr & 7)) << 4));
                const float f = weight[k * R + rr];
                o[e][0] = fmaf(q4.x, f, o[e][0]);
                o[e][1] = fmaf(q4.y, f, o[e][1]);
                o[e][2] = fmaf(q4.z, f, o[e][2]);
                o[e][3] = fmaf(q4.w, f, o[e][3]);
              }
            }
#pragma unroll
            for (int e = 0; e < kRows; ++e) {
              const int rr = r0 + e * kStep, at = rr < R ? rows[rank * R + rr] : -1;
              if (at >= 0) st_global(out_tile + at + c * 4, pack4(o[e][0], o[e][1], o[e][2], o[e][3]));
            }
          }
        }
      }
    }  // NQ == 1
  }

  if (cs > 1) {
    // No CTA of the cluster leaves while another may still write into its shared memory, read
    // from it or arrive on its barriers: a second phase of the cluster barrier (the softmax warps
    // have arrived on it in the epilogue).
    if (warp < 4) {
      cluster_wait();  // phase 1
      cluster_arrive();
    }
    cluster_wait();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (p.independent) cudaGridDependencySynchronize();  // complete no sooner than the kernel before
  if (threadIdx.x == 0 && *abort_flag && p.status) atomicOr(p.status, SPIFFY_DEV_TIMEOUT);
}

// ------------------------------------------------------------------ host ----
// What one problem's descriptor and segment lengths amount to.
struct Shape {
  int group, TNL, NL, MT, TP1, TP;
  int T;  // key tiles of an M-tile, at least
};
Shape shape_of(const spiffy_attn_desc& d, const AttnContext& ctx, const AttnContext& ctx2, bool pair) {
  Shape s;
  s.group = d.n_q_heads / d.n_kv_heads;
  s.TNL = pair ? 2 * (BM / 2 / s.group) : BM / s.group;
  s.NL = d.n_nodes * d.block_len;
  s.MT = (s.NL + s.TNL - 1) / s.TNL;
  s.TP1 = (ctx.len + BN - 1) / BN;
  s.TP = s.TP1 + (ctx2.len + BN - 1) / BN;
  s.T = s.TP + (d.block_len + BN - 1) / BN;
  return s;
}

struct Plan {
  int nq;     // M-tiles per CTA
  int cs;     // CTAs of a cluster that share an M-tile's key tiles (nq = 1)
  bool pair;  // a pair of CTAs per M-tile instead (attention_pair.cu)
  // nq = 2: rounds that are full; what is left goes into a second launch, with one M-tile per CTA or
  // pair.  0: one launch.
  int full_rounds;
  bool rest_by_pairs;
};

template <int NP>
using Kernel = void (*)(Problems<NP>);
template <int NP>
Kernel<NP> kernel_of(int hd, int nq) {
  if constexpr (NP == 2)  // the full-sequence call takes head dimension 128 only
    return nq == 2 ? graph_attention_tc_kernel<2, 128, 2> : graph_attention_tc_kernel<1, 128, 2>;
  else
    return hd == 128 ? (nq == 2 ? graph_attention_tc_kernel<2, 128, 1> : graph_attention_tc_kernel<1, 128, 1>)
                     : (nq == 2 ? graph_attention_tc_kernel<2, 64, 1> : graph_attention_tc_kernel<1, 64, 1>);
}

// Clusters of `cs` CTAs that the current device can hold at once (a GPU cluster's SMs are no
// multiple of 8 everywhere, so this is less than SMs / cs).  Asked for once per device and size.
int resident_clusters(int hd, int cs) {
  static std::atomic<int> known[64][2][4];
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return 0;
  std::atomic<int>& slot = known[device][hd == 128][cs == 2 ? 1 : cs == 4 ? 2 : 3];
  int n = slot.load(std::memory_order_relaxed);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel_of<1>(hd, 1), &cfg) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    if (n < 1) n = -1;
    slot.store(n, std::memory_order_relaxed);
  }
  return n;
}

// One or two M-tiles per CTA, and how many CTAs share the key tiles of an M-tile:
// whatever a model of the kernel's time finds cheapest.  A round of CTAs (each holds its
// SM) takes 6.6 us plus 0.88 per key tile with one M-tile, 8 us plus 1.75 with two; at head
// dimension 64, where the second product has two terms, 4.9 and 0.93, 6 and 1.8.  Handing the
// partials around a cluster costs about 2 us (1.5 with rows half as long), so that a second
// CTA pays from about six key tiles.  (16 x 32 positions x 32 heads, one M-tile: 11.0, 21.8 and 36.0 us
// over 512, 2048 and 4096 keys; 32 x 32 positions, two: 16.6, 37.3 and 68.2.)
// A pair of CTAs per M-tile (at most 64 query heads on a key/value head) takes 5 us and 0.45 per key tile, at
// head dimension 64 3.7 and 0.69, a round: 8 x 32 positions x 32 heads over 512 + 32 keys 7.3 and 7.1 us (one
// CTA a tile 9.7 and 9.3), 64 x 4 x 32 heads on 8 over 2048 12.4 (clusters of two 15.6), 3 x 100 positions x
// 24 heads of 64 on 8 over 777 9.2 (10.4).  One round only pays: 2 x 11 x 24 x 16 heads over 450 13.9 (10.3),
// and with more key tiles than some 20 (8) clusters of eight are sooner done.
// A call of several rounds whose last one half fills the SMs or less does that one in half the time by a
// second launch, with one M-tile per CTA or pair: 4 x 32 x 32 positions x 32 heads over 4096 keys, three
// rounds and 136 M-tiles instead of four rounds, 253 -> 243 us (289 -> 278 under the power limit, which
// gives an idle SM's share to the others); 2 x 44 x 32 positions x 32 heads on 16 over 1000 62.9 -> 57.5.
// `tiles` counts the M-tiles of all problems of the launch, `doubles` the CTAs that take two
// of them, `pair_tiles` the pairs (0: not possible); T is the key tiles of the longer problem.
// `may_split`: the call may be two launches; `same_tiles`: a pair's M-tiles are one CTA's.
// `held`: SMs that the end of a decision beside this call holds as its CTAs move in, one a sequence.  A call
// whose one round needs them as well ends 3 to 4 us later, and plans of fewer CTAs are another 2 us sooner
// done beside a decision than their costs say (kLate in all).  2 x 32 positions x 74 heads, 74 pairs, with a
// decision of 32000 entries: over 100 keys 11.8 us (73 heads 8.7), with one M-tile per CTA 9.2; over 512
// 13.8 and 12.6; over 1000 18.0 and 17.9, where the line is.  8 x 32 x 74 heads, 148 CTAs of one M-tile: over 100
// keys 16.4, two M-tiles per CTA 13.9; over 512 19.7 and 20.2, left at one.  Measured for one, two and four
// sequences, at head dimension 64, and with a graph too large for the fused tail (146 x 32 x 2 heads 27.2 -> 22.3).
Plan make_plan(int64_t tiles, int64_t doubles, int64_t pair_tiles, int T, int hd, bool may_split, bool same_tiles,
               int held) {
  const int sms = sm_count();
  const float one0 = hd == 128 ? 6.6f : 4.9f, one = hd == 128 ? 0.88f : 0.93f;
  const float two0 = hd == 128 ? 8.0f : 6.0f, two = hd == 128 ? 1.75f : 1.8f;
  const float pair = hd == 128 ? 5.0f + 0.45f * (float)T : 3.7f + 0.69f * (float)T;
  const float kLate = hd == 128 ? 5.5f : 4.0f;
  auto rounds = [&](int64_t ctas) { return (float)((ctas + sms - 1) / sms); };
  if (sms <= 0) return {2, 1, false, 0, false};
  struct Choice {
    Plan plan;
    int64_t ctas;
    float cost;
  };
  // The cheapest plan of at most `most` CTAs.
  auto cheapest = [&](int64_t most) {
    Choice c = {{2, 1, false, 0, false}, 0, INFINITY};
    auto consider = [&](const Plan& pl, int64_t ctas, float a_round) {
      const float cost = rounds(ctas) * a_round;
      if (ctas <= most && cost < c.cost) c = {pl, ctas, cost};
    };
    consider({2, 1, false, 0, false}, doubles, two0 + two * (float)T);
    if (pair_tiles > 0) consider({1, 1, true, 0, false}, 2 * pair_tiles, pair);
    for (int cs = 1; cs <= 8 && cs <= T; cs *= 2) {
      // clusters only where all of them run at once
      if (cs > 1 && (tiles * cs > sms || tiles > resident_clusters(hd, cs))) continue;
      const float exchange = cs == 1 ? 0.f : (hd == 128 ? 1.9f : 1.4f) + 0.07f * (float)cs;
      consider({1, cs, false, 0, false}, tiles * cs, one0 + exchange + one * (float)((T + cs - 1) / cs));
    }
    return c;
  };
  Choice best = cheapest(INT64_MAX);
  if (best.ctas <= sms && best.ctas > sms - held) {
    const Choice fewer = cheapest(sms - held);
    if (fewer.cost < best.cost + kLate) best = fewer;
  }
  // A last round that half fills the SMs or less is done in half the time with one M-tile per CTA.
  const int64_t full = doubles / sms, left = doubles - full * sms;
  if (may_split && full > 0 && left > 0 && 2 * left <= sms) {
    const bool by_pairs = pair_tiles > 0 && same_tiles && 4 * left <= sms;
    const float rest = by_pairs ? pair : one0 + one * (float)T;
    if ((float)full * (two0 + two * (float)T) + rest < best.cost) best.plan = {2, 1, false, (int)full, by_pairs};
  }
  return best.plan;
}

bool make_problem(const spiffy_attn_desc& d, const Shape& sh, const AttnProblem& a, Maps* m, Params* p, const Plan& pl,
                  int32_t* dev_status) {
  const int halves = d.head_dim / 64;
  const int ctas = pl.pair ? 2 : 1;  // of a pair, each reads half of the rows, of the keys of K and of the columns of V
  const int64_t bs = a.ctx.batch_stride_rows, bs2 = a.ctx2.batch_stride_rows;
  auto keys = [&](CUtensorMap* map, const void* base, int64_t rows, int64_t stride, bool is_v) {
    if (is_v && pl.pair)
      return make_tile_map(map, base, d.n_kv_heads, rows, d.batch, 1, BN, 1, stride, 2, d.head_dim / 2);
    return make_tile_map(map, base, d.n_kv_heads, rows, d.batch, 1, BN / ctas, halves, stride, halves);
  };
  bool ok = make_tile_map(&m->q, a.q, d.n_q_heads, sh.NL, d.batch, sh.group, sh.TNL / ctas, 1, 0, halves);
  ok = ok && keys(&m->kb, a.kb, sh.NL, 0, false) && keys(&m->vb, a.vb, sh.NL, 0, true);
  if (a.ctx.len > 0) {
    ok = ok && keys(&m->kp, a.ctx.k, a.ctx.len, bs, false) && keys(&m->vp, a.ctx.v, a.ctx.len, bs, true);
  } else {  // never dereferenced: the segment has no tile
    m->kp = m->kb;
    m->vp = m->vb;
  }
  if (a.ctx2.len > 0) {
    ok = ok && keys(&m->kp2, a.ctx2.k, a.ctx2.len, bs2, false) && keys(&m->vp2, a.ctx2.v, a.ctx2.len, bs2, true);
  } else {
    m->kp2 = m->kb;
    m->vp2 = m->vb;
  }
  p->B = d.batch; p->N = d.n_nodes; p->L = d.block_len; p->P = a.ctx.len; p->P2 = a.ctx2.len;
  p->Hq = d.n_q_heads; p->Hkv = d.n_kv_heads; p->group = sh.group;
  p->TNL = sh.TNL; p->NL = sh.NL; p->TP1 = sh.TP1; p->TP = sh.TP; p->log_cs = pl.cs == 8 ? 3 : pl.cs / 2;
  const float scale = d.scale != 0.f ? d.scale : 1.0f / sqrtf((float)d.head_dim);
  p->scale_log2 = scale * kLog2e;
  p->out = static_cast<__nv_bfloat16*>(a.out);
  p->status = dev_status;
  p->spin_limit = mbar_poll_limit();
  p->early_trigger = (d.kernel & SPIFFY_ATTN_EARLY_DEPENDENTS) ? 1 : 0;
  p->independent = (d.kernel & SPIFFY_ATTN_INDEPENDENT) ? 1 : 0;
  return ok;
}

// One launch: of the whole call (grid.x = 0: as many CTAs as it takes), or of `grid.x` CTAs from
// M-tile `first` on.  `flags` come on top of the caller's.
template <int NP>
spiffy_status launch_part(const spiffy_attn_desc* const (&d)[NP], const AttnProblem* const (&a)[NP], const Shape (&sh)[NP],
                          const Plan& pl, dim3 grid, int first, int slots, int flags, int32_t* dev_status,
                          cudaStream_t stream) {
  Problems<NP> pr;
  unsigned x = 0;
  for (int i = 0; i < NP; ++i) {
    Params& p = pr.p[i];
    if (!make_problem(*d[i], sh[i], *a[i], &pr.maps[i], &p, pl, dev_status)) return SPIFFY_ECUDA;
    p.first = first;
    p.slots = slots;
    if (flags & SPIFFY_ATTN_EARLY_DEPENDENTS) p.early_trigger = 1;
    if (flags & SPIFFY_ATTN_INDEPENDENT) p.independent = 1;
    if (i == 1) pr.x_split = (int)x;
    x += pl.pair ? 2 * sh[i].MT : (sh[i].MT + pl.nq - 1) / pl.nq * pl.cs;
  }
  if (grid.x == 0) grid.x = x;
  if (pl.pair) return launch_attention_pair<NP>(pr, d[0]->head_dim, grid, stream);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;  // only when asked for
  attr[1].val.clusterDim.x = (unsigned)pl.cs;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pl.cs > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel_of<NP>(d[0]->head_dim, pl.nq), pr);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

template <int NP>
spiffy_status launch(const spiffy_attn_desc* const (&d)[NP], const AttnProblem* const (&a)[NP], int32_t* dev_status,
                     cudaStream_t stream) {
  const int hd = d[0]->head_dim;
  static std::atomic<bool> smem_allowed[4][64];
  for (int nq = 1; nq <= 2; ++nq)
    if (!allow_smem(kernel_of<NP>(hd, nq), kSmemBytes, smem_allowed[(hd == 128 ? 0 : 2) + nq - 1]))
      return SPIFFY_ECUDA;
  if constexpr (NP == 2) {  // make_plan asks about the one-problem kernel
    static std::atomic<bool> allowed[64];
    if (!allow_smem(kernel_of<1>(hd, 1), kSmemBytes, allowed)) return SPIFFY_ECUDA;
  }
  const int64_t bg = (int64_t)d[0]->batch * d[0]->n_kv_heads;
  Shape sh[NP], by_pairs[NP];
  int64_t tiles = 0, doubles = 0, pair_tiles = 0;
  const bool pairs_can = d[0]->n_q_heads / d[0]->n_kv_heads <= BM / 2;
  int T = 0;
  for (int i = 0; i < NP; ++i) {
    sh[i] = shape_of(*d[i], a[i]->ctx, a[i]->ctx2, false);
    tiles += bg * sh[i].MT;
    doubles += bg * ((sh[i].MT + 1) / 2);
    if (pairs_can) {
      by_pairs[i] = shape_of(*d[i], a[i]->ctx, a[i]->ctx2, true);
      pair_tiles += bg * by_pairs[i].MT;
    }
    T = sh[i].T > T ? sh[i].T : T;
  }
  const bool split = NP == 1 && bg * (sh[0].MT + 1) < (1 << 30);
  const int held = (d[0]->kernel & SPIFFY_ATTN_INDEPENDENT) ? d[0]->batch : 0;
  const Plan pl = make_plan(tiles, doubles, pair_tiles, T, hd, split, by_pairs[0].TNL == sh[0].TNL, held);
  const dim3 grid(0, (unsigned)d[0]->n_kv_heads, (unsigned)d[0]->batch);
  if (pl.full_rounds == 0) return launch_part(d, a, pl.pair ? by_pairs : sh, pl, grid, 0, 0, 0, dev_status, stream);
  // Full rounds first, which let the rest begin as they end; the rest reads nothing of theirs, and is
  // complete no sooner.
  const int slots = (sh[0].MT + 1) / 2 * 2, first = pl.full_rounds * sm_count() * 2;
  const int rest = (int)bg * slots - first;
  const spiffy_status st = launch_part(d, a, sh, pl, dim3((unsigned)first / 2), 0, slots, SPIFFY_ATTN_EARLY_DEPENDENTS,
                                       dev_status, stream);
  if (st != SPIFFY_OK) return st;
  const Plan one = {1, 1, pl.rest_by_pairs, 0, false};
  return launch_part(d, a, one.pair ? by_pairs : sh, one, dim3((unsigned)(one.pair ? 2 * rest : rest)), first, slots,
                     SPIFFY_ATTN_INDEPENDENT, dev_status, stream);
}

}  // namespace

bool attention_tc_supported(const spiffy_attn_desc& d) {
  if (d.dtype != SPIFFY_BF16 || (d.head_dim != 128 && d.head_dim != 64)) return false;
  const int group = d.n_q_heads / d.n_kv_heads;
  if (group > BM) return false;
  if ((int64_t)d.batch * d.n_kv_heads > 65535) return false;
  return true;
}

spiffy_status launch_attention_tc(const spiffy_attn_desc& d, const AttnProblem& a, int32_t* dev_status,
                                  cudaStream_t stream) {
  return launch<1>({&d}, {&a}, dev_status, stream);
}

spiffy_status launch_attention_tc_dual(const spiffy_attn_desc& d0, const AttnProblem& a0, const spiffy_attn_desc& d1,
                                       const AttnProblem& a1, int32_t* dev_status, cudaStream_t stream) {
  return launch<2>({&d0, &d1}, {&a0, &a1}, dev_status, stream);
}

}  // namespace spiffy
