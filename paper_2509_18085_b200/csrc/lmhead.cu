// The decision step fused into the output projection: logits = H W^T are formed
// tile by tile in tensor memory and reduced there to (maximum, sum of
// exponentials, arg-max) per row, so that the [rows x vocabulary] logits are
// never written to memory (Algorithm 1, steps 1-2, on the distribution of
// Sec. 3.1 before it is materialised).
//
// H: [rows][hidden] bf16 hidden states of the B*N*L positions,
// W: [vocabulary][hidden] bf16 output embedding.
//
//   lmhead_gather_kernel   copies the hidden states of the still-masked positions,
//                          the only ones the decision needs, one after another;
//                          left out when there are few positions anyhow
//   lmhead_reduce_kernel   D[vocabulary, position] = W H^T.  The vocabulary is the M
//                          side of the products and the masked positions are N, so
//                          that the work follows their number in steps of 16 (up to
//                          256 at a time; beyond that, passes that read W again).  A
//                          CTA owns a contiguous share of the vocabulary, cut into
//                          tiles of 256 entries, and runs the K loop over `hidden`
//                          in chunks of 64:
//     warp 0      TMA producer: per chunk 256 rows of W and the positions' rows
//                 of H into a ring
//     warp 1      allocates tensor memory and issues tcgen05.mma, M = 128,
//                 two M-tiles per chunk
//     warps 4-11  one thread per vocabulary entry (TMEM lane): for every position
//                 (column) the warp's 32 entries are reduced across lanes
//
// Bound: the weights, read once (1.04 GB, 159 us at the measured copy rate, for
// 126464 x 4096).  What an SM takes in is 32 KB of W and 128 bytes per position per
// chunk, and 48.7 bytes per clock is what TMA delivers: with 256 positions as M and
// a vocabulary tile of 224 as N, as it was, that came to 1232 cycles per chunk and
// 238-277 us per call; with 166 masked positions as N to about 1110 per 256 entries.
// The reduction across lanes takes 6.6 us a tile there, and tensor memory has no room
// for a second accumulator pair: the epilogue empties the first into registers (192 a
// thread, which is why its warps take the others' share) and gives it back, so that
// the next tile's products run meanwhile: 234 -> 214 us with 164 masked positions, in
// runs of tens of milliseconds.  With the producer and the issuer as converged warps, and two or three
// TMA instructions a chunk where there were eight, 193 us in such runs (209 before on that board), and
// 210 us called back to back for seconds, which draws the board's power limit (228 before).  A ring of
// its own for the weights, four chunks deep beside three of H, with a producer each: 222.
//
// Each CTA leaves one partial result per position; the decision's finalize kernel
// merges them (in a fixed order) and applies the unmasking rule.  Every wait is
// bounded; a wait that gives up raises SPIFFY_DEV_TIMEOUT.
#include <math.h>

#include "common.cuh"
#include "decide_core.cuh"
#include "sm100_ptx.cuh"
#include "tma_map.cuh"

namespace spiffy {
namespace {

using namespace sm100;

constexpr int kLmThreads = 384;
constexpr int kGatherThreads = 128;
constexpr int kPass = 256;              // positions per pass
// Up to this many positions are taken as they are, masked or not: they cost less time as columns
// (their part of what an SM takes in stays below the weights' third) than the launch that packs.
constexpr int kDirectRows = 128;
constexpr int kBox = 32;                // rows of W and H are loaded in boxes of 32, 64, 128 or 256
constexpr int kBoxSizes = 4;
constexpr int kTileV = 256;             // vocabulary entries per tile: two M-tiles
constexpr int kRing = 200 * 1024;
constexpr int kMaxStages = 12;          // at least three: 64 KB per stage at 256 positions
constexpr int kHeld = 6;                // blocks of 32 columns that the epilogue holds in registers
constexpr int kRegsIssue = 40, kRegsEpilogue = 232;
static_assert(kRegsIssue + 2 * kRegsEpilogue <= 3 * 168, "within what the block was launched with");
constexpr uint32_t kLmTmemCols = 512;

// Running reduction of one column over one warp's vocabulary entries.
struct ColumnState {
  float m[8][kPass];  // [warp][column] maximum
  float s[8][kPass];  // sum of exp(x - m)
  int idx[8][kPass];  // lowest entry attaining m
};
constexpr int kLmBars = 2 * kMaxStages + 4;
constexpr int kLmSmem = kRing + (int)sizeof(ColumnState) + 8 * kLmBars + 16 + 1024;

struct LmParams {
  int hidden, vocab;
  int rows;              // positions, when all of them are taken in their own order ...
  const int* list;       // ... which is when this is null: [0] number of masked positions, [1 + i] row of the i-th
  Partial* partials;     // [rows][gridDim.x]
  int32_t* status;       // [B], may be null
  int n_status;
  int clear_status;      // the status words arrive with arbitrary contents (without a list only)
  uint32_t spin_limit;   // polls of one mbarrier wait
};

struct LmMaps {
  CUtensorMap w[kBoxSizes], h[kBoxSizes];  // [i]: boxes of 32 << i rows, 64 columns
};

// grid = rows.  Block r copies row r, if its position is masked, behind the masked rows before it.
__global__ void __launch_bounds__(kGatherThreads)
lmhead_gather_kernel(const uint4* __restrict__ h, int row_vecs, const int32_t* __restrict__ tokens, int mask_id,
                     uint4* __restrict__ packed, int* __restrict__ list, StatusClear clear) {
  cudaGridDependencySynchronize();
  pdl_launch_dependents();
  const int row = blockIdx.x, tid = threadIdx.x;
  const bool last = row + 1 == (int)gridDim.x;
  if (tid == kGatherThreads - 1 && row < clear.batch) clear.run(row);
  const bool masked = tokens[row] == mask_id;
  if (!masked && !last) return;
  int before = 0;
  for (int i = tid; i < row; i += kGatherThreads) before += tokens[i] == mask_id;
  before = __reduce_add_sync(0xffffffffu, before);
  __shared__ int part[kGatherThreads / 32];
  if ((tid & 31) == 0) part[tid >> 5] = before;
  __syncthreads();
  before = 0;
#pragma unroll
  for (int w = 0; w < kGatherThreads / 32; ++w) before += part[w];
  if (tid == 0) {
    if (masked) list[1 + before] = row;
    if (last) list[0] = before + (masked ? 1 : 0);
  }
  if (!masked) return;
  for (int i = tid; i < row_vecs; i += kGatherThreads)
    packed[(int64_t)before * row_vecs + i] = h[(int64_t)row * row_vecs + i];
}

// Reduction across the 32 lanes of 32 columns at once: lane i ends with column i.  At each step a
// lane gives away the half of the columns that is not its own: 31 exchanges instead of 160.
template <typename Op>
__device__ __forceinline__ float reduce_columns(uint32_t (&v)[32], int lane, Op op) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < off; ++i) {
      const uint32_t give = upper ? v[i] : v[i + off];
      const uint32_t keep = upper ? v[i + off] : v[i];
      v[i] = __float_as_uint(op(__uint_as_float(keep), __uint_as_float(__shfl_xor_sync(0xffffffffu, give, off))));
    }
  }
  return __uint_as_float(v[0]);
}

// Adds 32 columns (state column `at` belongs to this lane), one of them per register and one
// vocabulary entry (v0 + lane) per lane, to the state of warp `ew`.  Uses x up.
__device__ __forceinline__ void add_columns(ColumnState& state, int ew, int at, uint32_t (&x)[32], int v0,
                                            bool valid, int lane) {
  uint32_t f[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    if (!valid) x[c] = 0xff800000u;  // -inf
    f[c] = x[c];
  }
  // lane c: the maximum of column c over the warp's entries
  const float cm = reduce_columns(f, lane, [](float a, float b) { return fmaxf(a, b); });
  const float m_old = state.m[ew][at];
  const bool better = cm > m_old;  // strictly: tiles come in ascending token order
  const float m_new = better ? cm : m_old;
  const unsigned improved = __ballot_sync(0xffffffffu, better);
  if (improved) {  // the lowest entry that attains the new maximum: rare after the first tiles
    int found = 0;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      if ((improved >> c) & 1u) {
        const unsigned who = __ballot_sync(0xffffffffu, __uint_as_float(x[c]) == __shfl_sync(0xffffffffu, cm, c));
        if (lane == c) found = __ffs(who) - 1;
      }
    }
    if (better) {
      state.m[ew][at] = m_new;
      state.idx[ew][at] = v0 + found;
    }
  }
  const float ref = m_new == -INFINITY ? 0.f : m_new * kLog2e;
#pragma unroll
  for (int c = 0; c < 32; ++c)
    x[c] = __float_as_uint(ex2(fmaf(__uint_as_float(x[c]), kLog2e, -__shfl_sync(0xffffffffu, ref, c))));
  const float cs = reduce_columns(x, lane, [](float a, float b) { return a + b; });
  state.s[ew][at] = fmaf(state.s[ew][at], better ? ex2((m_old - m_new) * kLog2e) : 1.f, cs);
}

__global__ void __launch_bounds__(kLmThreads, 1)
lmhead_reduce_kernel(const __grid_constant__ LmMaps maps, const LmParams p) {
  extern __shared__ uint8_t lm_smem_raw[];
  uint8_t* smem = lm_smem_raw + ((0u - smem_u32(lm_smem_raw)) & 1023u);
  ColumnState& state = *reinterpret_cast<ColumnState*>(smem + kRing);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kRing + sizeof(ColumnState));
  uint64_t* full = bars;
  uint64_t* empty = full + kMaxStages;
  uint64_t* acc_full = empty + kMaxStages;  // [2] an accumulator pair holds a finished tile
  uint64_t* acc_empty = acc_full + 2;       // [2] ... and has been read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kLmBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // uniform to the compiler
  // this CTA's share of the vocabulary, in steps of 32 entries
  const int64_t units = (p.vocab + kBox - 1) / kBox;
  const int v_begin = (int)(units * blockIdx.x / gridDim.x) * kBox;
  const int v_end = (int)(units * (blockIdx.x + 1) / gridDim.x) * kBox;
  const int tiles = (v_end - v_begin + kTileV - 1) / kTileV;
  const int kc_count = p.hidden / 64;

  if (threadIdx.x == 0) {
    prefetch_tensormap(&maps.w[kBoxSizes - 1]);
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(acc_full + i, 1); mbar_init(acc_empty + i, 8); }  // the epilogue warps
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, kLmTmemCols);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  cudaGridDependencySynchronize();  // the packed rows (and everything before them) are visible

  const int count = p.list ? *reinterpret_cast<const volatile int*>(p.list) : p.rows;
  if (p.clear_status && blockIdx.x == 0 && threadIdx.x == 0 && p.status)
    for (int b = 0; b < p.n_status; ++b) p.status[b] = 0;
  const int passes = (count + kPass - 1) / kPass;
  auto positions = [&](int pass) { return min(kPass, count - pass * kPass); };
  auto boxes = [&](int pass) { return (positions(pass) + kBox - 1) / kBox; };
  // The ring is cut for the longest tile of this CTA and the first pass, the one with the most
  // positions: a CTA whose share of the vocabulary is a short tile has more chunks in flight.
  const int w_bytes = min(kTileV, v_end - v_begin) * 128;
  const int stage_bytes = w_bytes + (passes > 0 ? boxes(0) : 0) * kBox * 128;
  // (the products read whole M-tiles, so the last stage is followed by as much of the ring)
  const int reach = w_bytes > 128 * 128 ? kTileV * 128 : 128 * 128;
  const int stages = min(kMaxStages, min(kRing / stage_bytes, (kRing - reach) / stage_bytes + 1));
  // accumulator pairs that fit tensor memory: two (columns 0 and 256 on) up to 128 positions
  const int bufs = count <= 128 ? 2 : 1;
  const uint32_t acc_step = bufs == 2 ? 128u : 256u;  // columns between the accumulators of a pair

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    // whole warps up to the elected lane's instruction (sm100_ptx.cuh)
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, p.spin_limit));
    };
    if (warp == 0) {
      // ---------------------------------------------------------- producer --
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0, used = 0;  // `used`: stages that hold a copy this thread has issued
      for (int pass = 0; pass < passes && ok; ++pass) {
        const int nb = boxes(pass);
        for (int i = 0; i < tiles && ok; ++i) {
          const int v0 = v_begin + i * kTileV, rows = min(kTileV, v_end - v0);
          for (int kc = 0; kc < kc_count; ++kc) {
            if (!wait(empty + stage, phase ^ 1u)) { ok = false; break; }
            uint8_t* dst = smem + stage * stage_bytes;
            mbar_arrive_expect_tx(full + stage, (uint32_t)(rows + nb * kBox) * 128u);
            used |= 1u << stage;
            // as few instructions as the rows' number has binary digits: each takes its warp 85 to 105 cycles, some 200 among others
            auto load = [&](const CUtensorMap* m, uint8_t* to, int row, int n) {
#pragma unroll
              for (int s = kBoxSizes - 1; s >= 0; --s) {
                if (n < (kBox << s)) continue;
                tma_load_4d(to, m + s, full + stage, (kc & 1) * 64, kc >> 1, row, 0);
                to += kBox * 128 << s;
                row += kBox << s;
                n -= kBox << s;
              }
            };
            load(maps.w, dst, v0, rows);
            load(maps.h, dst + w_bytes, pass * kPass, nb * kBox);
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
        }
      }
      // Whoever gives up, and when: no copy is in flight into shared memory whose block has ended.
      for (int q = 0; q < kMaxStages; ++q)
        if ((used >> q) & 1u)
          for (uint32_t s = 0; s < kSpinLimit; ++s)
            if (mbar_try_wait(full + q, q < stage ? phase : phase ^ 1u)) break;
    } else if (warp == 1) {
      // -------------------------------------------------------- MMA issuer --
      constexpr uint32_t hi = desc_hi_sw128(1024);
      bool ok = true;
      int stage = 0, g = 0;
      uint32_t phase = 0;
      for (int pass = 0; pass < passes && ok; ++pass) {
        const int n16 = (positions(pass) + 15) / 16 * 16;
        const uint32_t idesc = idesc_bf16_f32(128, n16, false, false);
        for (int i = 0; i < tiles && ok; ++i, ++g) {
          const int m_tiles = v_end - (v_begin + i * kTileV) > 128 ? 2 : 1;
          const int buf = bufs == 2 ? g & 1 : 0;
          const uint32_t round = (uint32_t)(bufs == 2 ? g >> 1 : g);
          ok = wait(acc_empty + buf, (round & 1u) ^ 1u);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t d = tmem + (uint32_t)buf * 256u;
          for (int kc = 0; kc < kc_count; ++kc) {
            if (!wait(full + stage, phase)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t w_lo = desc_lo_sw128(smem_u32(smem + stage * stage_bytes), 16);
            const uint32_t h_lo = w_lo + ((uint32_t)w_bytes >> 4);
            for (int t = 0; t < m_tiles; ++t)
              umma_ss_k64(d + (uint32_t)t * acc_step, w_lo + (uint32_t)t * (128 * 128 >> 4), h_lo, hi, idesc, kc > 0 ? 1u : 0u);
            umma_commit(empty + stage);  // the stage is free once these products have read it
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
          if (ok) umma_commit(acc_full + buf);
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue --
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
    const int quad = warp & 3, ew = warp - 4;
    const int t = ew >> 2;  // M-tile of this warp
    bool ok = true;
    int g = 0;
    for (int pass = 0; pass < passes && ok; ++pass) {
      const int nb = boxes(pass);
      for (int c = lane; c < nb * 32; c += 32) {
        state.m[ew][c] = -INFINITY;
        state.s[ew][c] = 0.f;
        state.idx[ew][c] = 0x7fffffff;
      }
      __syncwarp();
      for (int i = 0; i < tiles && ok; ++i, ++g) {
        const int buf = bufs == 2 ? g & 1 : 0;
        const uint32_t round = (uint32_t)(bufs == 2 ? g >> 1 : g);
        ok = __all_sync(0xffffffffu, mbar_wait(acc_full + buf, round & 1u, abort_flag, p.spin_limit));
        if (!ok) break;
        tc_fence_after_sync();
        const int v0 = v_begin + i * kTileV + t * 128 + quad * 32;  // first vocabulary entry of this warp
        const bool live = v0 < v_end && v0 < p.vocab;
        const bool valid = v0 + lane < p.vocab;
        const uint32_t acc = tmem_addr(tmem, (uint32_t)quad * 32u, (uint32_t)buf * 256u + (uint32_t)t * acc_step);
        // What the issuer waits for is emptied into registers and given back before any of the
        // arithmetic, which then runs under the next tile's products.  Behind the last tile, or with a
        // second pair, nothing waits: there the loop takes all of it, whose few instructions are
        // fetched sooner (3 us less at a single tile).
        const int q0 = bufs == 2 || (i + 1 == tiles && pass + 1 == passes) ? 0 : kHeld;
        uint32_t x[kHeld][32];
        if (live) {
#pragma unroll 1
          for (int q = q0; q < nb; ++q) {
            tmem_ld_x32(acc + (uint32_t)q * 32u, x[0]);
            add_columns(state, ew, q * 32 + lane, x[0], v0, valid, lane);
          }
          if (q0 == kHeld) {
#pragma unroll
            for (int q = 0; q < kHeld; ++q)
              if (q < nb) tmem_ld_async(acc + (uint32_t)q * 32u, x[q]);
            tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < kHeld; ++q) tmem_loaded(x[q]);
          }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + buf);
        if (live && q0 == kHeld) {
#pragma unroll
          for (int q = 0; q < kHeld; ++q)
            if (q < nb) add_columns(state, ew, q * 32 + lane, x[q], v0, valid, lane);
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");  // every warp's columns, whatever `ok` says
      const int c = (int)threadIdx.x - 128;
      if (ok && c < positions(pass)) {
        float m = -INFINITY, sum = 0.f;
        int idx = 0x7fffffff;
#pragma unroll 1
        for (int w = 0; w < 8; ++w) merge(m, sum, idx, state.m[w][c], state.s[w][c], state.idx[w][c]);
        // NaN logits never win a comparison: report them through the maximum
        if (!(sum == sum)) m = sum;
        const int at = pass * kPass + c, row = p.list ? p.list[1 + at] : at;
        p.partials[(int64_t)row * gridDim.x + blockIdx.x] = Partial{m, sum, idx, 0};
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kLmTmemCols);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status)
    for (int b = 0; b < p.n_status; ++b) atomicOr(p.status + b, SPIFFY_DEV_TIMEOUT);
}

size_t up256(size_t n) { return (n + 255) / 256 * 256; }
size_t partial_bytes(const spiffy_decide_desc& d, int grid) {
  return up256((size_t)d.batch * d.n_nodes * d.block_len * (size_t)grid * sizeof(Partial));
}
size_t list_bytes(const spiffy_decide_desc& d) { return up256(((size_t)d.batch * d.n_nodes * d.block_len + 1) * sizeof(int)); }

}  // namespace

// One CTA per SM, or fewer for a vocabulary of fewer than 32 entries each.
int lmhead_grid(const spiffy_decide_desc& d) {
  const int n = sm_count();
  const int units = (d.vocab + kBox - 1) / kBox;
  return units < n ? units : n;
}

// partial results | list of masked rows | their hidden states
size_t lmhead_workspace_bytes(const spiffy_decide_desc& d, int hidden, int grid) {
  return partial_bytes(d, grid) + list_bytes(d) + (size_t)d.batch * d.n_nodes * d.block_len * (size_t)hidden * 2;
}

spiffy_status launch_lmhead_decide(const spiffy_decide_desc& d, int hidden, const void* hstates,
                                   const void* weight, const int32_t* block_tokens, float* conf,
                                   int32_t* top_tok, uint64_t* unmask_bits, int32_t* n_unmask,
                                   int32_t* dev_status, void* ws, bool fresh, cudaStream_t stream) {
  const int rows = d.batch * d.n_nodes * d.block_len;
  const int grid = lmhead_grid(d);
  if (grid <= 0) return SPIFFY_ECUDA;
  char* at = static_cast<char*>(ws);
  int* list = reinterpret_cast<int*>(at + partial_bytes(d, grid));
  uint4* packed = reinterpret_cast<uint4*>(at + partial_bytes(d, grid) + list_bytes(d));
  LmMaps maps;
  const bool pack = rows > kDirectRows;
  for (int i = 0; i < kBoxSizes; ++i)
    if (!make_map(&maps.w[i], weight, hidden / 128, d.vocab, 1, 1, kBox << i) ||
        !make_map(&maps.h[i], pack ? static_cast<const void*>(packed) : hstates, hidden / 128, rows, 1, 1, kBox << i))
      return SPIFFY_ECUDA;
  static std::atomic<bool> smem_allowed[64];
  if (!allow_smem(lmhead_reduce_kernel, kLmSmem, smem_allowed)) return SPIFFY_ECUDA;
  cudaError_t e = cudaSuccess;
  if (pack) {
    e = launch_pdl(lmhead_gather_kernel, dim3(rows), dim3(kGatherThreads), (size_t)0, stream,
                   static_cast<const uint4*>(hstates), hidden / 8, block_tokens, (int)d.mask_token_id,
                   packed, list, status_clear(d, fresh, dev_status, nullptr));
    count_launch();
    if (e != cudaSuccess) return SPIFFY_ECUDA;
  }
  LmParams p;
  p.hidden = hidden;
  p.vocab = d.vocab;
  p.rows = rows;
  p.list = pack ? list : nullptr;
  p.clear_status = !pack && fresh ? 1 : 0;
  p.partials = static_cast<Partial*>(ws);
  p.status = dev_status;
  p.n_status = d.batch;
  p.spin_limit = mbar_poll_limit();
  e = launch_pdl(lmhead_reduce_kernel, dim3(grid), dim3(kLmThreads), (size_t)kLmSmem, stream, maps, p);
  count_launch();
  if (e != cudaSuccess) return SPIFFY_ECUDA;
  return launch_decide_finalize(d, ws, grid, block_tokens, conf, top_tok, unmask_bits, n_unmask, dev_status,
                                stream);
}

}  // namespace spiffy
