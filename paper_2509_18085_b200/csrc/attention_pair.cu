// Packed draft-graph attention by pairs of CTAs: bf16, head dimension 128 or 64, calls whose key
// tiles need no splitting over more CTAs.  The mathematics, the order of the key tiles and the
// mask are those of attention_tc.cu; what differs is who holds what.
//
// The two CTAs of a cluster work on one M-tile of 128 rows with cta_group::2 products of
// M = 128: each holds 64 of the rows (as many (node, position) pairs as fit, times the query
// heads of the group), and of every key tile half of the keys of K and half of the columns of
// V, which the products of both read.  So a CTA takes in 32 KB per key tile instead of 64, a
// call fills twice as many SMs with the same M-tiles, and there is no partial result to
// exchange: a row's scores, sums and output stay in its CTA.
//
// A score tile has row r (of 64) in TMEM lane r for its first 64 keys and in lane 64 + r for
// the others, 64 columns each; the output likewise, by halves of the head dimension.  Two
// threads therefore share a row.  They need one reference maximum and exchange their halves'
// maxima through shared memory, one barrier of two warps per key tile; each adds up its own
// half's weights, and the halves are added in the end.
//
// P goes through shared memory (an A operand of this shape would have to be in tensor memory
// twice), over the K tile that its scores came from, which nobody reads any more.  A stage of
// the ring is therefore K and V together, free again when P V is done.
// At head dimension 64 P is two terms (attention_tc.cu says why), four times a K tile, and has a
// place of its own for each warpgroup; a CTA's half of V is 32 columns, rows of 64 bytes.
//
//   warp 0, 3   TMA producers of Q and K, and of V (both CTAs; bytes count on the leader's barriers)
//   warp 1      tensor memory; the leader's issues S = Q K^T
//   warp 2      the leader's issues O += P V
//   warps 4-19  four softmax warpgroups, which take the key tiles in turn into accumulators of
//               their own and merge them once at the end: a tile's way from scores to P is some
//               2300 cycles, most of them waiting, its exponentials alone 512
//
// A call this short is a chain of latencies, 8 x 32 positions x 32 heads over 512 + 32 keys (five key
// tiles, all loads at once): set-up 1000 cycles, first scores 2300 behind the wait for the kernel
// before, last P 4700 later, merge and output 2000.  What it took to get there: 12.8 us with two
// warpgroups and barriers' arrivals across the pair with release semantics at cluster scope (500
// cycles and more each); 9.5 without; 9.1 four warpgroups; 8.1 issuing warps converged instead of one
// lane; 7.2 set-up side by side by warps, no division in the producers' loops; 7.3 with arrivals and waits
// across the pair at cluster scope again, but the order they give confined to shared memory (fences with
// sync_restrict; unconfined 7.5, and 14.1 instead of 12.5 over 17 key tiles).  The kernel
// of attention_tc.cu took 10.3 then (9.7 now).  Per further key tile 0.45 us (0.88 there).  At head
// dimension 64 7.2 us (9.3 there) and 0.69 (0.93).  Tried and dropped: two
// CTAs of two warpgroups on an SM (10.6), references other than the maximum (nothing to exchange at
// the first tile, 0.5 us; but the largest weight is then no longer exact, and the error 4 % larger).
//
// Every wait is bounded; a wait that gives up raises SPIFFY_DEV_TIMEOUT in the caller's status
// word, and the pair winds down without touching its output.
#include "attention_tc.cuh"

namespace spiffy {
namespace {

constexpr int NW = 4;  // softmax warpgroups, behind the one with the producers and the issuers
constexpr int kThreads = 128 * (1 + NW), kSoftmax = 128 * NW;
// 96 registers a thread at launch; the softmax warps take over what the others do not need.
constexpr int kRegsIssue = 32, kRegsSoftmax = 104;
static_assert(kRegsIssue + NW * kRegsSoftmax <= (1 + NW) * 96, "within what the block was launched with");
constexpr int kRows = 64;           // of a CTA
constexpr int kHalf = kRows * 128;  // 64 rows of 128 bytes
constexpr int kMaxStages = 6;
// Tensor memory: warpgroup w has its scores at 64 w and its accumulator at 256 + (head dimension / 2) w.
constexpr uint32_t kTmemCols = 512, kColS = 0, kColO = 64 * NW;
// Shared memory: Q | P of each warpgroup, where it does not go over K | the ring, stage s: K at 2 s, V at
// 2 s + 1 | Tail.
template <int HD>
struct Smem {
  static constexpr int tile = kRows * HD * 2;               // a CTA's share of Q, K or V
  static constexpr int p = HD == 64 ? 4 * kHalf : 0;        // two terms of 128 keys
  static constexpr int stages = HD == 64 ? 5 : kMaxStages;
  static constexpr int ring = tile + NW * p;
  static constexpr int tail = ring + 2 * stages * tile;
};

struct Bars {
  uint64_t q_full;
  uint64_t s_done, pv_all;  // the issuers' last products have completed
  uint64_t s_full[NW];      // by warpgroup: scores formed (both CTAs)
  uint64_t s_free[NW];      // ... and read (leader)
  uint64_t p_ready[NW];     // P written (leader)
  uint64_t pv_done[NW];     // ... and used (both)
  uint64_t k_full[kMaxStages], v_full[kMaxStages];  // both CTAs' halves have landed (leader)
  uint64_t stage_free[kMaxStages];               // (both)
};
struct Tail {  // behind the tiles in shared memory
  Bars bars;
  float maxima[2][NW][2][kRows];  // of a row's halves, by parity of the warpgroup's turn
  float2 partials[NW][2][kRows];  // reference maximum and sum of a row's halves
  int rows[kRows];                // where a row is stored, relative to the CTA's first; -1: nowhere
  uint32_t tmem;
  int abort_flag;
  int issued_k, issued_v;         // by this CTA's producers
};
template <int HD>
constexpr int kSmemBytes = Smem<HD>::tail + (int)sizeof(Tail);
// (two CTAs must not share an SM: each holds all of its tensor memory until it exits)
static_assert(kSmemBytes<64> <= 227 * 1024 && kSmemBytes<128> <= 227 * 1024 && kSmemBytes<64> > 114 * 1024, "one CTA");

// Is `mine` true for any thread of the two warps that meet at this barrier?
__device__ __forceinline__ bool any_of_two_warps(int barrier, bool mine) {
  uint32_t any;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.u32 p, %2, 0;\n"
      "barrier.cta.red.or.pred q, %1, 64, p;\n"
      "selp.u32 %0, 1, 0, q;\n"
      "}\n"
      : "=r"(any)
      : "r"(barrier), "r"((uint32_t)mine)
      : "memory");
  return any != 0;
}
constexpr int kBarSoftmax = 1, kBarProducers = 2, kBarTwoWarps = 3;  // 3 .. 10
constexpr int kHeadStart = 2;  // K tiles that are asked for before the first V tile

template <int HD, int NP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
graph_attention_pair_kernel(const __grid_constant__ Problems<NP> problems) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int which = NP == 2 && (int)blockIdx.x >= problems.x_split ? 1 : 0;
  const Maps& maps = problems.maps[which];
  const Params& p = problems.p[which];
  using SM = Smem<HD>;
  constexpr int kTile = SM::tile, kStages = SM::stages, kHalves = HD / 64;
  constexpr bool kRest = HD == 64;  // P in two bf16 terms, as in attention_tc.cu
  constexpr int kColsO = HD / 2;    // columns of an accumulator: half of the head dimension
  uint8_t* sq = smem;
  uint8_t* ring = smem + SM::ring;
  Tail& tail = *reinterpret_cast<Tail*>(smem + SM::tail);
  Bars& bars = tail.bars;
  volatile int* abort_flag = &tail.abort_flag;

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // uniform to the compiler
  const int rank = (int)(blockIdx.x & 1);  // x_split is even
  const int unit = ((int)blockIdx.x - (which ? problems.x_split : 0)) >> 1;
  if (no_such_tile<NP>(p, unit)) return;  // both CTAs
  // Set-up, by warps side by side: what comes before the first copy is on the path of a call whose
  // CTAs find no room beside the call before.
  if (warp == 1) {
    tmem_alloc_pair(&tail.tmem, kTmemCols);
  } else if (warp == 0) {
    // one lane per barrier: a thread's initialisations are served one after the other
    constexpr int kBars = (int)(sizeof(Bars) / 8);
    static_assert(kBars <= 64, "two rounds of lanes");
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint64_t* bar = reinterpret_cast<uint64_t*>(&bars) + lane + 32 * h;
      // the four warps of a softmax warpgroup, in both CTAs, arrive once each
      const bool eight = bar >= bars.s_free && bar < bars.pv_done;
      if (lane + 32 * h < kBars) mbar_init(bar, eight ? 8u : 1u);
    }
    if (lane == 0) tail.abort_flag = tail.issued_k = tail.issued_v = 0;
    mbar_fence_init();
  } else if (warp == 2) {
    if (lane == 0) {
      prefetch_tensormap(&maps.q);  // the descriptors are kernel parameters
      prefetch_tensormap(p.TP1 > 0 ? &maps.kp : (p.TP > 0 ? &maps.kp2 : &maps.kb));
      prefetch_tensormap(p.TP1 > 0 ? &maps.vp : (p.TP > 0 ? &maps.vp2 : &maps.vb));
    }
  }
  tc_fence_before_sync();
  __syncwarp();
  cluster_arrive_relaxed();  // this warp's part is done: both CTAs' barriers and tensor memory exist when all are here

  // the pair's rows and key tiles
  const Place place = place_of<NP>(p, unit);
  const int nl0 = place.mt * p.TNL, g = place.g, b = place.b;
  const int nl_count = min(p.TNL, p.NL - nl0);
  const int tnl = p.TNL >> 1;          // of this CTA
  const int nl_cta = nl0 + rank * tnl;
  const int rows_box = tnl * p.group;  // rows a Q box writes
  const int n_lo = nl0 / p.L, n_hi = (nl0 + nl_count - 1) / p.L;
  const int kb_start = n_lo * p.L;
  const int T = p.TP + ((n_hi - n_lo + 1) * p.L + BN - 1) / BN;
  // rows of the Q tile that the TMA box does not write must be finite
  for (int i = rows_box * 8 + threadIdx.x; i < kRows * 8; i += kThreads) {
    const uint4 z = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int h = 0; h < kHalves; ++h) reinterpret_cast<uint4*>(sq + h * kHalf)[i] = z;
  }
  fence_proxy_async_smem();
  __syncthreads();
  cluster_wait();
  tc_fence_after_sync();
  const uint32_t tmem = tail.tmem;
  // Ahead of the wait, so that what follows a call of few CTAs sets itself up beside it: no kernel that reads
  // without waiting itself comes directly behind this one (launch_pdl, common.cuh).
  if (p.early_trigger) pdl_launch_dependents();
  // everything above is on-chip set-up; global memory is touched from here on, behind a wait in each role

  // This thread waits for and touches nothing more that the other CTA has a part in.  A CTA that has
  // given up tells the other one, so that both know.
  auto leave = [&]() {
    tc_fence_before_sync();
    __syncwarp();
    if (*abort_flag) {
      st_cta(map_to_cta(smem_u32(&tail.abort_flag), (uint32_t)(rank ^ 1)), 1u);
      fence_cluster();
    }
    cluster_arrive_relaxed();
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    // whole warps up to the elected lane's instruction (sm100_ptx.cuh)
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      return __all_sync(0xffffffffu, mbar_wait_pair(bar, parity, abort_flag, p.spin_limit));
    };
    if (!p.independent) cudaGridDependencySynchronize();
    if (warp == 0 || warp == 3) {
      // ----------------------------------------- producers: Q and K, and V --
      const bool is_k = warp == 0;
      if (is_k) {
        const uint32_t bar = map_to_cta(smem_u32(&bars.q_full), 0);
        if (rank == 0) mbar_arrive_expect_tx(&bars.q_full, 2u * kHalves * rows_box * 128u);
#pragma unroll
        for (int h = 0; h < kHalves; ++h)  // rows beyond the last one read as zeros
          tma_load_5d_pair(sq + h * kHalf, &maps.q, bar, 0, g * p.group, nl_cta, h, b);
      }
      // Key tiles in order: first context segment, second context segment, block keys.  Everything is
      // counted along: a division by a number the compiler does not know takes longer than the rest.
      const CUtensorMap* m = is_k ? &maps.kp : &maps.vp;
      uint64_t* full = is_k ? bars.k_full : bars.v_full;
      const uint32_t full_leader = map_to_cta(smem_u32(full), 0);
      uint8_t* dst = ring + (is_k ? 0 : kTile);
      const int half = is_k ? 0 : rank;   // of the columns of V; both of K's ...
      int key0 = is_k ? 64 * rank : 0;    // ... for half of the keys
      int stage = 0, t = 0;
      uint32_t phase = 1;
      if (!is_k) asm volatile("barrier.cta.sync %0, 64;" ::"n"(kBarProducers) : "memory");  // the first scores need Q and K alone
      for (; t < T; ++t, key0 += BN) {
        if (is_k && t == kHeadStart) asm volatile("barrier.cta.arrive %0, 64;" ::"n"(kBarProducers) : "memory");
        if (t == p.TP1) {
          m = is_k ? &maps.kp2 : &maps.vp2;
          key0 -= t * BN;
        }
        if (t == p.TP) {
          m = is_k ? &maps.kb : &maps.vb;
          key0 += kb_start - (t - p.TP1) * BN;
        }
        if (t >= kStages && !wait(&bars.stage_free[stage], phase)) break;
        if (rank == 0) mbar_arrive_expect_tx(full + stage, 2 * kTile);
        tma_load_5d_pair(dst + stage * 2 * kTile, m, full_leader + 8u * stage, 0, g, key0, half, b);
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (is_k && t <= kHeadStart) asm volatile("barrier.cta.arrive %0, 64;" ::"n"(kBarProducers) : "memory");
      if (lane == 0) (is_k ? tail.issued_k : tail.issued_v) = t;
      fence_cluster();  // read by the leader where the pair gives up
    } else if (warp == 1 && rank == 0) {
      // ------------------------------------------------ issuer of S = Q K^T --
      constexpr uint32_t idesc = idesc_bf16_f32(BM, BN, false, false);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      const uint32_t q_lo = desc_lo_sw128(smem_u32(sq), 16);
      const uint32_t k_lo = desc_lo_sw128(smem_u32(ring), 16);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = wait(&bars.q_full, 0);
      for (int t = 0; t < T && ok; ++t) {
        ok = wait(&bars.k_full[stage], phase);
        // the scores before these have been read
        if (ok && t >= NW) ok = wait(&bars.s_free[t % NW], (uint32_t)(t / NW - 1) & 1u);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t d = tmem + kColS + (uint32_t)(t % NW) * 64u, k_at = k_lo + (uint32_t)stage * (2 * kTile >> 4);
        if constexpr (HD == 128) umma_pair_kk_k128(d, q_lo, k_at, hi, idesc, 0u);
        else umma_pair_kk_k64(d, q_lo, k_at, hi, hi, idesc, 0u);
        umma_commit_both(&bars.s_full[t % NW]);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      umma_commit_pair(&bars.s_done);
      mbar_wait_quiet(&bars.s_done, 0);
    } else if (warp == 2 && rank == 0) {
      // --------------------------------------------------- issuer of O += P V --
      constexpr uint32_t idesc = idesc_bf16_f32(BM, HD, false, true);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      const uint32_t p_lo = desc_lo_sw128(smem_u32(kRest ? smem + kTile : ring), 16);
      const uint32_t v_lo = desc_lo_sw128(smem_u32(ring + kTile), kHalf);
      int stage = 0;
      uint32_t phase = 0;
      for (int t = 0; t < T; ++t) {
        if (!wait(&bars.v_full[stage], phase)) break;
        if (!wait(&bars.p_ready[t % NW], (uint32_t)(t / NW) & 1u)) break;
        tc_fence_after_sync();
        const uint32_t d = tmem + kColO + (uint32_t)(t % NW) * kColsO, v_at = v_lo + (uint32_t)stage * (2 * kTile >> 4);
        if constexpr (kRest) {
          constexpr uint32_t v_hi = desc_hi_sw64(512);
          const uint32_t p_at = p_lo + (uint32_t)(t % NW) * (SM::p >> 4);
          umma_pair_kn32_k128(d, p_at, v_at, hi, v_hi, idesc, t >= NW ? 1u : 0u);
          umma_pair_kn32_k128(d, p_at + (SM::p / 2 >> 4), v_at, hi, v_hi, idesc, 1u);
        } else {
          umma_pair_kn_k128(d, p_lo + (uint32_t)stage * (2 * kTile >> 4), v_at, hi, idesc, t >= NW ? 1u : 0u);
        }
        umma_commit_both(&bars.pv_done[t % NW]);
        if (t + kStages < T) umma_commit_both(&bars.stage_free[stage]);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      umma_commit_pair(&bars.pv_all);
      mbar_wait_quiet(&bars.pv_all, 0);
    }
    leave();
  } else {
    // ------------------------------------------------------------- softmax --
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    if (!p.independent) cudaGridDependencySynchronize();
    const int quad = warp & 3;  // TMEM lane quadrant this warp may touch
    const int wg = (warp - 4) >> 2;
    const int row = (quad & 1) * 32 + lane, half = quad >> 1;  // half: of a tile's keys, and of the columns of O
    const int meet = kBarTwoWarps + 2 * wg + (quad & 1);       // with the warp of the other half
    const int rows_valid = max(0, min(tnl, p.NL - nl_cta)) * p.group;
    const int node = min(nl_cta + row / p.group, p.NL - 1) / p.L;
    const uint32_t lane_base = (uint32_t)(quad * 32);
    const float k2 = p.scale_log2;
    // key tiles every row sees whole: t < full_a, and TP1 <= t < full_b
    const int full_a = p.P / BN, full_b = p.TP1 + p.P2 / BN;
    float m_run = -INFINITY, l_run = 0.f;  // the row's reference maximum (log2 units), this half's sum
    int turn = 0;
    bool ok = true;
    const uint32_t at_s = tmem_addr(tmem, lane_base, kColS + (uint32_t)wg * 64u);
    const uint32_t at_o = tmem_addr(tmem, lane_base, kColO + (uint32_t)wg * kColsO);
    const uint32_t s_free = map_to_cta(smem_u32(&bars.s_free[wg]), 0), p_ready = map_to_cta(smem_u32(&bars.p_ready[wg]), 0);
    // the P V products of key tile t (one of this warpgroup's) have completed
    auto wait_pv = [&](int t) -> bool {
      const bool yes =
          __all_sync(0xffffffffu, mbar_wait_pair(&bars.pv_done[wg], (uint32_t)(t / NW) & 1u, abort_flag, p.spin_limit));
      tc_fence_after_sync();
      return yes;
    };
    if (wg == 0 && half == 0)
      tail.rows[row] = row < rows_valid ? (row / p.group * p.Hq + row % p.group) * HD : -1;
    int stage = wg;
    for (int t = wg; t < T; t += NW) {
      // Wait outcomes are made warp-uniform: the TMEM accesses below are warp-collective.  A warp that
      // has given up still meets the other one of its rows, so that both leave together.
      bool good =
          __all_sync(0xffffffffu, ok && mbar_wait_pair(&bars.s_full[wg], (uint32_t)(t / NW) & 1u, abort_flag, p.spin_limit));
      uint32_t s[2][32];
      uint32_t chunks = 3u;  // 32-column chunks that no row of the warp sees cost nothing but zeros in P
      float mx = -INFINITY;
      if (good) {
        tc_fence_after_sync();
        tmem_ld_async(at_s, s[0]);
        tmem_ld_async(at_s + 32u, s[1]);
        // the accumulator's last products: waited for tile by tile, never two phases at once
        if (t >= NW) good = wait_pv(t - NW);
        tmem_wait_ld();
        tmem_loaded(s[0]);
        tmem_loaded(s[1]);
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0 && t + NW < T) mbar_arrive_remote_relaxed(s_free);
        if (t >= full_a && (t < p.TP1 || t >= full_b)) {
          const Window w = visible_window(p, t, kb_start, node);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int lo = w.lo - 64 * half - 32 * h, hi = w.hi - 64 * half - 32 * h;
            if (!__any_sync(0xffffffffu, lo < 32 && hi > 0)) chunks &= ~(1u << h);
            // bit c: column 32 h + c of this half is visible
            const uint32_t upto = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
            const uint32_t below = lo >= 32 ? 0xffffffffu : lo <= 0 ? 0u : (1u << lo) - 1u;
            const uint32_t seen = upto & ~below;
#pragma unroll
            for (int c = 0; c < 32; ++c) s[h][c] = (seen >> c) & 1u ? s[h][c] : 0xff800000u;  // -inf
          }
        }
        float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
          m0 = max3(m0, __uint_as_float(s[0][c]), __uint_as_float(s[0][c + 1]));
          m1 = max3(m1, __uint_as_float(s[1][c]), __uint_as_float(s[1][c + 1]));
        }
        mx = fmaxf(m0, m1) * k2;
      }
      // over K, read for the last time, or where the products that read it last are done
      uint8_t* p_row = (kRest ? smem + kTile + wg * SM::p : ring + 2 * stage * kTile) + half * kHalf + row * 128;
      stage += NW;
      if (stage >= kStages) stage -= kStages;
      // The two halves of a row agree on its maximum (by turns in two places, so that nobody writes
      // where the other may still read); a warp that has given up takes the other one along.
      float(*maxima)[kRows] = tail.maxima[turn][wg];
      turn ^= 1;
      maxima[half][row] = mx;
      if (any_of_two_warps(meet, !good)) {
        ok = false;
        break;
      }
      const float m_new = max3(m_run, mx, maxima[half ^ 1][row]);
      const bool need = (m_new - m_run) > kRescaleLog2;  // false when both are -inf
      if (__any_sync(0xffffffffu, need)) {
        float corr = 1.f;
        if (need) {
          corr = ex2(m_run - m_new);  // 0 for a row that had seen nothing yet
          l_run *= corr;
          m_run = m_new;
        }
        if (t >= NW) {  // the accumulator holds earlier tiles, whose products are done
#pragma unroll 1
          for (uint32_t c0 = 0; c0 < kColsO; c0 += 16) {
            uint32_t o[16];
            tmem_ld_async(at_o + c0, o);
            tmem_wait_ld();
            tmem_loaded(o);
#pragma unroll
            for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * corr);
            tmem_st_x16(at_o + c0, o);
          }
          tmem_wait_st();
          tc_fence_before_sync();
        }
      }
      const float m_use = (m_run == -INFINITY) ? 0.f : m_run;
      const uint64_t k22 = pack2(k2, k2), nm2 = pack2(-m_use, -m_use);
      uint64_t sum_a = pack2(0.f, 0.f), sum_b = pack2(0.f, 0.f);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        auto store = [&](int c, const uint32_t (&pk)[4], const uint32_t (&rest)[4]) {
          uint8_t* at = p_row + (((4 * h + c / 8) ^ (row & 7)) << 4);
          *reinterpret_cast<uint4*>(at) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          if constexpr (kRest) *reinterpret_cast<uint4*>(at + SM::p / 2) = make_uint4(rest[0], rest[1], rest[2], rest[3]);
        };
        if ((chunks >> h) & 1u) {
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            uint32_t pk[4], rest[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint64_t x2 =
                  fma2(pack2(__uint_as_float(s[h][c + 2 * e]), __uint_as_float(s[h][c + 2 * e + 1])), k22, nm2);
              float x0, x1;
              unpack2(x2, x0, x1);
              const float p0 = ex2(x0), p1 = ex2(x1);
              if (e & 1) sum_b = add2(sum_b, pack2(p0, p1)); else sum_a = add2(sum_a, pack2(p0, p1));
              if constexpr (kRest) {  // cut off instead of rounded: a byte permutation, no conversion
                const uint32_t w0 = __float_as_uint(p0), w1 = __float_as_uint(p1);
                pk[e] = __byte_perm(w0, w1, 0x7632);
                float r0, r1;
                unpack2(fma2(pack2(__uint_as_float(w0 & 0xffff0000u), __uint_as_float(w1 & 0xffff0000u)), pack2(-1.f, -1.f),
                             pack2(p0, p1)), r0, r1);
                rest[e] = pack_bf16(r0, r1);
              } else {
                pk[e] = pack_bf16(p0, p1);
                rest[e] = 0u;
              }
            }
            store(c, pk, rest);
          }
        } else {
          const uint32_t zero[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int c = 0; c < 32; c += 8) store(c, zero, zero);
        }
      }
      float a0, a1;
      unpack2(add2(sum_a, sum_b), a0, a1);
      l_run += a0 + a1;
      fence_proxy_async_smem();
      __syncwarp();  // every lane's P is in shared memory: one arrival speaks for the warp
      if (lane == 0) mbar_arrive_remote_own(p_ready);
    }
    // ------------------------------------------------------------ epilogue --
    // every product into this warpgroup's accumulator has completed
    if (ok && wg < T) ok = wait_pv(T - 1 - (T - 1 - wg) % NW);
    // The warpgroups exchange (reference, sum) through shared memory, and each merges its share of this
    // half's columns.
    tail.partials[wg][half][row] = make_float2(m_run, l_run);
    tc_fence_before_sync();
    asm volatile("bar.sync %0, %1;" ::"n"(kBarSoftmax), "n"(kSoftmax) : "memory");  // all of them, whatever `ok` says
    tc_fence_after_sync();
    constexpr int kCols = kColsO / NW;
    uint32_t o[NW][kCols];
    if (ok) {
#pragma unroll
      for (int w = 0; w < NW; ++w) tmem_ld_async(tmem_addr(tmem, lane_base, kColO + (uint32_t)(kColsO * w + wg * kCols)), o[w]);
      tmem_wait_ld();
#pragma unroll
      for (int w = 0; w < NW; ++w) tmem_loaded(o[w]);
    }
    leave();
    if (ok) {
      float m_all = -INFINITY, weight[NW], sum[NW], l_all = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float2 lo = tail.partials[w][0][row], hi = tail.partials[w][1][row];
        weight[w] = lo.x;  // -inf: no key that this row sees among its tiles, or no tile
        sum[w] = lo.y + hi.y;
        m_all = fmaxf(m_all, weight[w]);
      }
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        weight[w] = ex2(weight[w] - m_all);
        l_all = fmaf(weight[w], sum[w], l_all);
        if (w >= T) {  // an accumulator that was never written may hold anything
#pragma unroll
          for (int c = 0; c < kCols; ++c) o[w][c] = 0u;
        }
      }
      const float inv = 1.0f / l_all;
#pragma unroll
      for (int w = 0; w < NW; ++w) weight[w] *= inv;
      uint8_t* out_row = sq + row * (HD * 2);  // results pass through the Q tile, so that whole rows are stored at once
#pragma unroll
      for (int c = 0; c < kCols; c += 8) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float x = __uint_as_float(o[0][c + 2 * e]) * weight[0], y = __uint_as_float(o[0][c + 2 * e + 1]) * weight[0];
#pragma unroll
          for (int w = 1; w < NW; ++w) {
            x = fmaf(__uint_as_float(o[w][c + 2 * e]), weight[w], x);
            y = fmaf(__uint_as_float(o[w][c + 2 * e + 1]), weight[w], y);
          }
          pk[e] = pack_bf16(x, y);
        }
        *reinterpret_cast<uint4*>(out_row + (((half * (kColsO / 8) + (wg * kCols + c) / 8) ^ (row & 7)) << 4)) =
            make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    asm volatile("bar.sync %0, %1;" ::"n"(kBarSoftmax), "n"(kSoftmax) : "memory");
    if (!*abort_flag) {
      constexpr int kChunks = HD / 8, kStep = kSoftmax / kChunks;  // 16-byte chunks of a row, rows per pass
      const int tid = (int)threadIdx.x - 128, row0 = tid / kChunks, chunk = tid % kChunks;
      __nv_bfloat16* out = p.out + (((int64_t)b * p.NL + nl_cta) * p.Hq + (int64_t)g * p.group) * HD + chunk * 8;
#pragma unroll
      for (int k = 0; k < kRows / kStep; ++k) {
        const int r = row0 + kStep * k, at = tail.rows[r];
        const uint4 w = *reinterpret_cast<const uint4*>(sq + r * (HD * 2) + ((chunk ^ (r & 7)) << 4));
        if (at >= 0) st_global(out + at, w);
      }
    }
  }

  // Neither CTA leaves while the other's products, arrivals or copies may still touch it.
  cluster_wait();
  tc_fence_after_sync();
  if (*abort_flag) {
    // copies that nobody has waited for: all of them count on the leader's barriers
    if (rank == 0 && warp == 0) {
      mbar_wait_quiet(&bars.q_full, 0);
      for (int kv = 0; kv < 2; ++kv) {
        uint64_t* full = kv ? bars.v_full : bars.k_full;
        const int mine = kv ? tail.issued_v : tail.issued_k;
        const int theirs = (int)ld_cta(map_to_cta(smem_u32(kv ? &tail.issued_v : &tail.issued_k), 1));
        const int n = max(mine, theirs);
        for (int t = max(0, n - kStages); t < n; ++t) {
          if (t >= mine) mbar_arrive_expect_tx(full + t % kStages, kTile);  // the other's half alone is on its way
          mbar_wait_quiet(full + t % kStages, (uint32_t)(t / kStages) & 1u);
        }
      }
    }
    cluster_arrive();
    cluster_wait();
  }
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
  if (p.independent) cudaGridDependencySynchronize();  // complete no sooner than the kernel before
  if (threadIdx.x == 0 && *abort_flag && p.status) atomicOr(p.status, SPIFFY_DEV_TIMEOUT);
}

}  // namespace

template <int NP>
spiffy_status launch_attention_pair(const Problems<NP>& pr, int head_dim, dim3 grid, cudaStream_t stream) {
  static std::atomic<bool> allowed[2][64];
  auto run = [&](auto kernel, int smem, std::atomic<bool>(&done)[64]) {
    if (!allow_smem(kernel, smem, done)) return SPIFFY_ECUDA;
    const cudaError_t e = launch_pdl(kernel, grid, dim3(kThreads), (size_t)smem, stream, pr);
    count_launch();
    return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
  };
  if constexpr (NP == 1)  // the full-sequence call takes head dimension 128 only
    if (head_dim == 64) return run(graph_attention_pair_kernel<64, NP>, kSmemBytes<64>, allowed[0]);
  return run(graph_attention_pair_kernel<128, NP>, kSmemBytes<128>, allowed[1]);
}
template spiffy_status launch_attention_pair<1>(const Problems<1>&, int, dim3, cudaStream_t);
template spiffy_status launch_attention_pair<2>(const Problems<2>&, int, dim3, cudaStream_t);

}  // namespace spiffy
