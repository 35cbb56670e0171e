// Lazy chain evaluation of Algorithm 1: the decision (steps 1-4) is computed
// only for the nodes the walk (step 5) actually reaches.
//
// The eager path reduces the logits of every node of the draft graph; only the
// 1 + n_accepted nodes on the accepted path are ever used.  Here one
// cooperative kernel works level by level.  For every sequence b that is still
// walking:
//   R  the reducing CTAs of b take the vocabulary slices of the masked rows of b's
//      current node (the HBM-bound part, 1/N of the eager traffic
//      per level); a slice's result carries the level;
//   T  CTA b waits until all slices carry it, merges them, applies the unmasking
//      rule, forms the next state, looks for the child that equals it (the graph
//      of b sits in its shared memory) and publishes the new current node, its
//      masked positions and the level in one word, for which the reducers wait.
// Sequences never wait for one another.  The arithmetic is the code the eager
// kernels use (decide_core.cuh), so the results on the path have the same bits.
//
// Waiting: a wait for level k of sequence b depends only on work of levels
// < k, or of level k's R phase, so there is no cycle; the launch is cooperative
// (all CTAs resident); every wait is bounded, and when one runs out the kernel
// sets SPIFFY_DEV_TIMEOUT, tells the others through the header and returns.
// The host zeroes header, words and slices before the launch.
//
// Bound: a chain of trips through L2 and HBM, level after level.  What passes
// between the CTAs is therefore the data itself, 16 bytes at a time in one access
// with the level in it, instead of data, fence, counter and a load behind the
// counter: per level two trips each way became one, and the reducers no longer
// look the tokens up.  The time follows the levels of the slowest sequence, about 10 us
// each behind 12 us of set-up (4 x 32 x 32 positions, 126464 entries, bf16: 42-43 us where
// two drafts are accepted, 53 where three, 74 where five; with 1.13 levels on average 24.0,
// 29.3 before the slices carried their level).
#include "common.cuh"
#include "decide_core.cuh"
#include "walk_core.cuh"

namespace spiffy {
namespace {

struct LazyHeader {
  int timeout;  // a bounded wait ran out somewhere
  int pad[3];
};

// Where a sequence stands.
struct __align__(16) LazyWord {
  int level;        // levels whose tail has finished; 0x7fffffff: the walk has ended
  int node;
  uint64_t masked;  // still-masked positions of the node
};

struct LazyParams {
  const void* logits;
  int64_t row_stride, chunk;
  int B, N, L, V, splits, mask_id, rule, top_s;
  FastDiv by_splits;
  float tau;
  const int32_t* block_tokens;
  const int32_t* parent_off;
  const int32_t* parent_idx;
  int parent_cap;
  float* conf;
  int32_t* top_tok;
  uint64_t* unmask_bits;
  int32_t* n_unmask;
  int32_t* decide_status;
  int32_t* accepted_node;
  int32_t* n_accepted;
  int32_t* path;
  int32_t* next_block;
  int32_t* walk_status;
  Partial* partials;   // [B][L][splits]
  LazyHeader* header;
  LazyWord* words;     // [B]
  int clear_status;    // the status words arrive with arbitrary contents
  int stage_graph;     // the sequence's states and parent lists fit shared memory
  int stage_slices;    // ... and so do the slices of one node
  unsigned wait_spins;   // polls of one wait before it gives up
  int lost_slices;       // test hook: sequence 0 expects slices that never come
};


// One access each: 16 aligned bytes that belong together.
__device__ __forceinline__ LazyWord load_word(const LazyWord* p) {
  uint64_t a, b;
  asm volatile("{\n.reg .b128 t;\nld.relaxed.gpu.global.b128 t, [%2];\nmov.b128 {%0, %1}, t;\n}"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
  return LazyWord{(int)(uint32_t)a, (int)(uint32_t)(a >> 32), b};
}
__device__ __forceinline__ void store_word(LazyWord* p, const LazyWord& w) {
  store16(p, (uint64_t)(uint32_t)w.level | (uint64_t)(uint32_t)w.node << 32, w.masked);
}

// True while polling may go on; gives up after `limit` polls here, or once another wait has.
__device__ __forceinline__ bool keep_polling(unsigned& polls, LazyHeader* h, unsigned limit) {
  if (++polls > limit || ((polls & 7u) == 0 && *reinterpret_cast<volatile int*>(&h->timeout))) {
    h->timeout = 1;
    return false;
  }
  __nanosleep(32);
  return true;
}

template <typename T>
__global__ void __launch_bounds__(kReduceThreads, 6)  // at most 80 registers (bf16 79): six CTAs per SM
decide_walk_lazy_kernel(const LazyParams p) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b_own = blockIdx.x < p.B ? (int)blockIdx.x : -1;  // the sequence whose tail this CTA runs
  const int N = p.N, L = p.L;
  __shared__ float s_conf[64];
  __shared__ int32_t s_top[64], s_next[64];
  __shared__ uint64_t s_bits, s_mask;
  __shared__ LazyWord s_word;
  __shared__ int s_found, s_bad;
  extern __shared__ __align__(16) unsigned char lazy_smem[];
  // the slices of the own sequence's current node: [L][splits], staged when they fit
  Partial* s_part = reinterpret_cast<Partial*>(lazy_smem);
  // the graph of the own sequence: [states N*L | off N+1 | idx cap], staged when it fits
  const int32_t* g_state = nullptr;
  const int32_t* g_off = nullptr;
  const int32_t* g_idx = nullptr;
  if (b_own >= 0) {
    g_state = p.block_tokens + (int64_t)b_own * N * L;
    g_off = p.parent_off + (int64_t)b_own * (N + 1);
    g_idx = p.parent_idx + (int64_t)b_own * p.parent_cap;
    if (p.stage_graph) {
      int32_t* s_state = reinterpret_cast<int32_t*>(s_part + (p.stage_slices ? L * p.splits : 0));
      int32_t* s_off = s_state + N * L;
      int32_t* s_idx = s_off + (N + 1);
      auto copy4 = [](void* dst, const void* src) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(dst)),
                     "l"(src)
                     : "memory");
      };
      for (int i = tid; i < N * L; i += kReduceThreads) copy4(s_state + i, g_state + i);
      for (int i = tid; i <= N; i += kReduceThreads) copy4(s_off + i, g_off + i);
      for (int i = tid; i < p.parent_cap; i += kReduceThreads) copy4(s_idx + i, g_idx + i);
      g_state = s_state;
      g_off = s_off;
      g_idx = s_idx;  // waited for before the first tail phase
    }
    for (int i = tid; i < N; i += kReduceThreads) {
      p.path[(int64_t)b_own * N + i] = i == 0 ? 0 : -1;
      p.n_unmask[(int64_t)b_own * N + i] = -1;  // not evaluated (yet)
    }
  }
  if (tid == 0) {
    s_bad = 0;
    if (b_own >= 0 && p.clear_status) {  // only this CTA touches its sequence's words
      if (p.decide_status) p.decide_status[b_own] = 0;
      if (p.walk_status) p.walk_status[b_own] = 0;
    }
  }
  int own_node = b_own >= 0 ? 0 : -1;  // uniform over the CTA
  int own_hops = 0;
  uint64_t own_mask = 0;  // still-masked positions of own_node, from level 1 on
  bool failed = false;
  // CTA b runs the tail of sequence b and, where there are others, nothing else; the others divide
  // the sequences among them, so that none of them waits for one on behalf of another.
  const bool apart = (int)gridDim.x > p.B;
  const int reducers = apart ? (int)gridDim.x - p.B : (int)gridDim.x;
  const int r = apart ? (int)blockIdx.x - p.B : (int)blockIdx.x;
  const bool many = reducers >= p.B;  // several CTAs per sequence, else several sequences per CTA
  const int step_b = many ? p.B : reducers;
  for (int level = 0; level < N && !failed; ++level) {
    bool alive = false;
    // R: this CTA's slices of the current nodes
    for (int b = many ? r % p.B : r; r >= 0 && b < p.B; b += step_b) {
      __syncthreads();  // s_word is free
      if (level == 0) {
        if (warp == 0) {
          const int32_t* st = p.block_tokens + (int64_t)b * N * L;
          uint64_t masked = 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int l = lane + 32 * h;
            masked |= (uint64_t)__ballot_sync(0xffffffffu, l < L && st[min(l, L - 1)] == p.mask_id) << (32 * h);
          }
          if (lane == 0) s_word = LazyWord{0, 0, masked};
        }
      } else if (b != b_own && tid == 0) {
        LazyWord w;
        unsigned polls = 0;
        while ((w = load_word(p.words + b)).level < level)
          if (!keep_polling(polls, p.header, p.wait_spins)) break;
        s_word = w;
      }
      __syncthreads();
      const LazyWord w = level > 0 && b == b_own ? LazyWord{level, own_node, own_mask} : s_word;
      if (w.level < level) {
        failed = true;
        break;
      }
      if (w.node < 0) continue;  // this sequence's walk has ended
      alive = true;
      // the slices of the masked rows; the others are never read
      const int items = __popcll(w.masked) * p.splits;
      const int stride = many ? (reducers - b + p.B - 1) / p.B : 1;
      for (int i = many ? r / p.B : 0; i < items; i += stride) {
        uint64_t left = w.masked;
        const int nth = p.by_splits.div(i), split = i - nth * p.splits;
        for (int k = nth; k > 0; --k) left &= left - 1;
        const int l = __ffsll((long long)left) - 1;
        const int64_t row = ((int64_t)b * N + w.node) * L + l;
        reduce_slice(static_cast<const T*>(p.logits) + row * p.row_stride, p.V, p.chunk, split,
                     p.partials + ((int64_t)b * L + l) * p.splits + split, kLog2e, level + 1);
        __syncthreads();  // the reduce's shared scratch is reused by the next item
      }
    }
    if (failed) break;
    // T: the own sequence
    if (own_node >= 0) {
      alive = true;
      const int b = b_own, node = own_node;
      if (level == 0) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
      }
      const int32_t* state = g_state + node * L;
      // slices of this level: those of every still-masked row of the node
      bool ok_wait = true;
      {
        const Partial* from = p.partials + (int64_t)b * L * p.splits;
        const int tag = b == 0 && p.lost_slices != 0 ? -1 : level + 1;
        unsigned polls = 0;
        for (int i = tid; i < L * p.splits && ok_wait; i += kReduceThreads) {
          if (state[p.by_splits.div(i)] != p.mask_id) continue;
          LazyWord w;  // 16 bytes, the tag last
          while ((int)((w = load_word(reinterpret_cast<const LazyWord*>(from + i))).masked >> 32) != tag)
            if (!(ok_wait = keep_polling(polls, p.header, p.wait_spins))) break;
          if (p.stage_slices) reinterpret_cast<LazyWord*>(s_part)[i] = w;
        }
      }
      if (__syncthreads_or(!ok_wait)) {
        failed = true;
        break;
      }
      {
        const int r = tid >> 1, sub = tid & 1, l = min(r, L - 1);
        const int32_t st = state[l];
        float conf;
        int32_t tok;
        const bool ok = p.stage_slices ? finalize_row<2, true>(s_part + l * p.splits, p.splits, sub, st, p.mask_id, conf, tok)
                                       : finalize_row<2>(p.partials + ((int64_t)b * L + l) * p.splits, p.splits, sub, st,
                                                         p.mask_id, conf, tok);
        if (sub == 0 && r < L) {
          const int64_t row = ((int64_t)b * N + node) * L + l;
          p.conf[row] = conf;
          p.top_tok[row] = tok;
          s_conf[l] = conf;
          s_top[l] = tok;
          if (!ok && p.decide_status) atomicOr(p.decide_status + b, SPIFFY_DEV_NONFINITE);
        }
      }
      __syncthreads();
      if (warp == 0) {
        const uint64_t bits = unmask_rule(s_conf, state, L, p.mask_id, p.rule, p.top_s, p.tau, lane);
        if (lane == 0) {
          p.unmask_bits[(int64_t)b * N + node] = bits;
          p.n_unmask[(int64_t)b * N + node] = __popcll(bits);
          s_bits = bits;
          s_found = kNoLink;
        }
      }
      __syncthreads();
      const uint64_t bits = s_bits;
      if (tid < L) s_next[tid] = ((bits >> tid) & 1ull) ? s_top[tid] : state[tid];
      if (warp == 0) {  // positions the next state still masks
        uint64_t left = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = lane + 32 * h;
          const bool m = l < L && (((bits >> l) & 1ull) ? s_top[l] : state[l]) == p.mask_id;
          left |= (uint64_t)__ballot_sync(0xffffffffu, m) << (32 * h);
        }
        if (lane == 0) s_mask = left;
      }
      __syncthreads();
      const bool may_go_on = bits != 0 && own_hops < N - 1;
      if (may_go_on) {
        // the first node (ascending) that lists `node` as a parent and equals its next state
        bool bad = false;
        for (int m = node + 1 + warp; m < N; m += kReduceThreads / 32) {
          const int e0 = g_off[m], e1 = g_off[m + 1];
          if (e0 < 0 || e1 < e0 || e1 > p.parent_cap) {  // malformed offsets
            bad = true;
            continue;
          }
          bool is_child = false;
          for (int e = e0 + lane; e < e1; e += 32) {
            const int q = g_idx[e];
            if (q < 0 || q >= m) bad = true;  // ignored entry
            is_child |= q == node;
          }
          if (!__any_sync(0xffffffffu, is_child)) continue;
          const int32_t* sm = g_state + m * L;
          bool eq = true;
          if (lane < L) eq &= sm[lane] == s_next[lane];
          if (lane + 32 < L) eq &= sm[lane + 32] == s_next[lane + 32];
          if (__all_sync(0xffffffffu, eq) && lane == 0) atomicMin(&s_found, m);
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) s_bad = 1;
      }
      __syncthreads();
      const int found = may_go_on ? s_found : kNoLink;
      if (found != kNoLink) {  // accepted: its distribution replaces the target's
        own_hops += 1;
        own_node = found;
        if (tid == 0) p.path[(int64_t)b * N + own_hops] = found;
      } else {  // the walk ends on `node`
        if (tid < L) p.next_block[(int64_t)b * L + tid] = s_next[tid];
        if (tid == 0) {
          p.accepted_node[b] = node;
          p.n_accepted[b] = own_hops;
          if (s_bad && p.walk_status) atomicOr(p.walk_status + b, SPIFFY_DEV_BADGRAPH);
        }
        own_node = -1;
      }
      own_mask = s_mask;
      if (tid == 0)  // what the reducers of b wait for
        store_word(p.words + b, LazyWord{own_node < 0 ? 0x7fffffff : level + 1, own_node, own_mask});
      __syncthreads();
    }
    if (!alive) return;  // every sequence this CTA works for has ended
  }
  // a bounded wait ran out (here or in another CTA): say so on the sequence this CTA owns
  if (*reinterpret_cast<volatile int*>(&p.header->timeout) && b_own >= 0 && tid == 0) {
    if (p.decide_status) atomicOr(p.decide_status + b_own, SPIFFY_DEV_TIMEOUT);
    if (p.walk_status) atomicOr(p.walk_status + b_own, SPIFFY_DEV_TIMEOUT);
  }
}

size_t lazy_graph_bytes(const spiffy_decide_desc& d, int parent_cap) {
  return ((size_t)d.n_nodes * d.block_len + d.n_nodes + 1 + parent_cap) * 4;
}

// CTAs that can be resident at once on the current device (cooperative launch limit).
template <typename T>
int resident_ctas(size_t smem) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, decide_walk_lazy_kernel<T>,
                                                    kReduceThreads, smem) != cudaSuccess)
    return 0;
  return per_sm * sm_count();
}

}  // namespace

size_t decide_lazy_workspace_bytes(const spiffy_decide_desc& d) {
  const size_t partials = (size_t)d.batch * d.block_len * decide_splits(d, nullptr) * sizeof(Partial);
  // slices | header | words[B], all zeroed by every call
  return partials + sizeof(LazyHeader) + (size_t)d.batch * sizeof(LazyWord);
}

spiffy_status launch_decide_walk_lazy(const spiffy_decide_desc& d, const void* logits,
                                      const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                      uint64_t* unmask_bits, int32_t* n_unmask,
                                      int32_t* decide_status, const int32_t* parent_off,
                                      const int32_t* parent_idx, int32_t parent_cap,
                                      int32_t* accepted_node, int32_t* n_accepted, int32_t* path,
                                      int32_t* next_block, int32_t* walk_status, void* ws,
                                      bool fresh, cudaStream_t stream) {
  const bool bf16 = d.logits_dtype == SPIFFY_BF16;
  const size_t graph = lazy_graph_bytes(d, parent_cap);
  const int stage_graph = graph <= 16 * 1024;  // beyond that it would cost resident CTAs
  const size_t slices = (size_t)d.block_len * decide_splits(d, nullptr) * sizeof(Partial);
  const int stage_slices = slices <= 20 * 1024;
  const size_t smem = (stage_graph ? graph : 0) + (stage_slices ? slices : 0);
  const int resident = bf16 ? resident_ctas<__nv_bfloat16>(smem) : resident_ctas<float>(smem);
  if (resident <= 0) return SPIFFY_ECUDA;
  if (d.batch > resident) return SPIFFY_EUNSUPPORTED;  // one resident CTA per sequence runs its tail
  LazyParams p;
  p.logits = logits;
  p.row_stride = d.row_stride;
  p.splits = decide_splits(d, &p.chunk);
  p.by_splits = FastDiv::by(p.splits);
  p.B = d.batch;
  p.N = d.n_nodes;
  p.L = d.block_len;
  p.V = d.vocab;
  p.mask_id = d.mask_token_id;
  p.rule = d.rule;
  p.top_s = d.top_s;
  p.tau = d.threshold;
  p.block_tokens = block_tokens;
  p.parent_off = parent_off;
  p.parent_idx = parent_idx;
  p.parent_cap = parent_cap;
  p.conf = conf;
  p.top_tok = top_tok;
  p.unmask_bits = unmask_bits;
  p.n_unmask = n_unmask;
  p.decide_status = decide_status;
  p.accepted_node = accepted_node;
  p.n_accepted = n_accepted;
  p.path = path;
  p.next_block = next_block;
  p.walk_status = walk_status;
  const size_t partial_bytes = (size_t)d.batch * d.block_len * p.splits * sizeof(Partial);
  p.partials = static_cast<Partial*>(ws);
  p.header = reinterpret_cast<LazyHeader*>(static_cast<char*>(ws) + partial_bytes);
  p.words = reinterpret_cast<LazyWord*>(p.header + 1);
  p.clear_status = fresh ? 1 : 0;
  p.stage_graph = stage_graph;
  p.stage_slices = stage_slices;
  p.wait_spins = flag_poll_limit();
  p.lost_slices = lazy_extra_arrivals();
  const int64_t items = (int64_t)d.batch * d.block_len * p.splits;
  int grid = (int)(items + d.batch < resident ? items + d.batch : resident);
  if (cudaMemsetAsync(ws, 0, decide_lazy_workspace_bytes(d), stream) != cudaSuccess)
    return SPIFFY_ECUDA;
  void* args[] = {&p};
  const void* fn = bf16 ? (const void*)decide_walk_lazy_kernel<__nv_bfloat16>
                        : (const void*)decide_walk_lazy_kernel<float>;
  const cudaError_t e =
      cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kReduceThreads), args, smem, stream);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

}  // namespace spiffy
