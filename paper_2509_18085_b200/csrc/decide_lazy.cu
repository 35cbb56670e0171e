// Lazy chain evaluation of Algorithm 1: the decision (steps 1-4) is computed
// only for the nodes the walk (step 5) actually reaches.
//
// The eager path reduces the logits of every node of the draft graph; only the
// 1 + n_accepted nodes on the accepted path are ever used.  Here two kernels work
// level by level:
//   lazy_root_kernel   the slices of the true blocks' masked rows, as the eager reduce takes
//                      them, and the workspace cleared for what follows;
//   lazy_walk_kernel   CTA b, the tail of sequence b: waits until all slices of b's current
//                      node are there, merges them, applies the unmasking rule, forms the
//                      next state, looks for the child that equals it and publishes that
//                      node, its masked positions and the level in one word.  The other
//                      CTAs, each with a sequence of its own, reduce: the current node's
//                      slices, and while the tail works on those, the slices of the node
//                      that will probably be next.
// Sequences never wait for one another.  The arithmetic is the code the eager
// kernels use (decide_core.cuh), so the results on the path have the same bits.
//
// The guess is the first node that lists the current one as a parent: the graph is built from the
// likeliest successors in front.  A slice belongs to its node, whoever asked for it and when; a
// wrong guess leaves slices that nobody reads.  Reducers look at the word between two slices and
// drop a guess that it refutes.
//
// Waiting: the tail waits for slices, reducers out of guesses for the word.  No residency of other
// CTAs is needed for an end: a tail that has looked for its slices often enough, or has no
// reducers, reduces the missing ones itself, and a reducer that has looked at the word often
// enough leaves.  A tail whose own wait runs out even so sets SPIFFY_DEV_TIMEOUT, ends its
// sequence's walk in the word and returns.
//
// Bound: a chain of trips through L2 and HBM, level after level.  What passes between the CTAs
// is the data itself, 16 bytes in one access with its mark in it.  4 x 32 x 32 positions, 126464
// entries, bf16, CUDA graph, by the drafts that the deepest of the four accepts (one cooperative kernel
// behind a memset, reducers waiting for every node: 12 us and 10 a level, so 42, 53 and 74 us for two,
// three and five): 28 us for one, 33 two, 38 three, 44 five; 1 x 16 x 32 x 152064 12.3 for none, then
// 5 each.  Guesses more than one level ahead of the word cost more than they gave (32, 36, 39 and 42;
// none accepted 16.4 for 12.3).
// What guessing is worth depends on the guess: reducers look up from a wrong one after the slice at hand, or the next.
// Without guesses / right / wrong / the one kernel from before, us, two drafts accepted: 1 x 8 x 32 x 126464 19.1 13.3
// 20.3 25.1, 4 x 32 x 32 x 126464 35.7 28.7 41.8 38.5, 64 x 8 x 16 x 64000 74.9 69.8 85.3 75.1; none accepted, 4 x 32 x
// 32, 14.0, 20.0 and 16.6.  One slice of a guess per reducer and then the word waited for: 31.5 for the 28.7, 38.1 for
// 41.8, 17.3 for 20.0.  On drafted graphs of 4 x 32 x 32, one new token in five wrong, 16 of them on average: 32.6; with
// one slice 34.5, with none 39.7, before 46.6.
#include "common.cuh"
#include "decide_core.cuh"
#include "walk_core.cuh"

namespace spiffy {
namespace {

// Where a sequence stands.
struct __align__(16) LazyWord {
  int level;        // levels whose tail has finished; kEnded: the walk has ended
  int node;
  uint64_t masked;  // still-masked positions of the node
};
constexpr int kEnded = 0x7fffffff;
constexpr int kPresent = 1;     // mark of a slice that has been written
constexpr int kWalkCtas = 6;    // of the walk kernel per SM: 80 registers, 208 bytes spilled; five of 96 spill as much, 1 to 2 % slower
constexpr unsigned kPollsABatch = 64, kPollsToHelp = 1u << 12;

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
  Partial* partials;   // [B][N][L][splits]
  LazyWord* words;     // [B]
  StatusClear clear;   // the status words arrive with arbitrary contents
  int stage_graph;     // a sequence's states and parent lists fit shared memory
  unsigned wait_spins; // polls of one wait before it gives up
  int lost_slices;     // test hook: sequence 0 expects slices that never come
};

__device__ __forceinline__ LazyWord load_word(const LazyWord* p) {
  const int4 w = load16(p);
  return LazyWord{w.x, w.y, (uint64_t)(uint32_t)w.z | (uint64_t)(uint32_t)w.w << 32};
}
__device__ __forceinline__ void store_word(LazyWord* p, const LazyWord& w) {
  store16(p, (uint64_t)(uint32_t)w.level | (uint64_t)(uint32_t)w.node << 32, w.masked);
}

// grid = (splits, B * L): slices of the true blocks' rows.  The CTA of slice s of row (b, l) clears the
// marks of slice s of row l of b's other nodes.
template <typename T>
__global__ void __launch_bounds__(kReduceThreads, 9)
lazy_root_kernel(const __grid_constant__ LazyParams p) {
  const int s = blockIdx.x, b = (int)blockIdx.y / p.L, l = (int)blockIdx.y - b * p.L;
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();  // inputs written by earlier kernels are visible, outputs and workspace free
#endif
  const int64_t row = (int64_t)b * p.N * p.L + l;
  const int32_t token = p.block_tokens[row];
  for (int n = 1 + threadIdx.x; n < p.N; n += kReduceThreads)
    *reinterpret_cast<int4*>(p.partials + (row + (int64_t)n * p.L) * p.splits + s) = make_int4(0, 0, 0, 0);
  if (s == 0 && l == 0 && threadIdx.x == kReduceThreads - 1) {
    p.words[b] = LazyWord{0, 0, 0};
    if (p.clear.batch) p.clear.run(b);
  }
  if (token != p.mask_id) return;  // already unmasked: never read
#if __CUDA_ARCH__ >= 900
  pdl_launch_dependents();  // the walk kernel gets the graph, and its first guesses, on the way
#endif
  reduce_slice(static_cast<const T*>(p.logits) + row * p.row_stride, p.V, p.chunk, s, p.partials + row * p.splits + s,
               kLog2e, kPresent);
}

// What both roles know about a sequence's graph.
struct Graph {
  const int32_t* state;  // [N][L]; of reducers the tokens in global memory
  const int32_t* off;
  const int32_t* idx;
};

// Item i of a node: a slice of one of its masked rows; the others are never read.
struct Item {
  int64_t row;
  int split;
};
__device__ __forceinline__ Item item_of(const LazyParams& p, int node, uint64_t masked, int i) {
  const int nth = p.by_splits.div(i);
  for (int k = nth; k > 0; --k) masked &= masked - 1;
  return Item{(int64_t)node * p.L + __ffsll((long long)masked) - 1, i - nth * p.splits};
}

// A tail's own way to the slices of its node that are not there.
template <typename T>
__device__ __noinline__ void reduce_missing(const LazyParams& p, const T* logits, Partial* slices, int node, uint64_t masked) {
  const int items = __popcll(masked) * p.splits;
  for (int i = 0; i < items; ++i) {
    const Item it = item_of(p, node, masked, i);
    Partial* out = slices + it.row * p.splits + it.split;
    if (__syncthreads_or(threadIdx.x == 0 && load16(out).w != kPresent))
      reduce_slice(logits + it.row * p.row_stride, p.V, p.chunk, it.split, out, kLog2e, kPresent);
  }
  __syncthreads();
}

// The rows of a node whose slices are `from`: merged, by `kLanes` threads a row (all bits the same whatever
// their number).  False for the whole CTA: some slices are not there.
template <int kLanes>
__device__ __forceinline__ bool merge_rows(const LazyParams& p, int b, int node, const int32_t* state, int tag,
                                           float* s_conf, int32_t* s_top) {
  const int tid = threadIdx.x, r = tid / kLanes, sub = tid % kLanes, l = min(r, p.L - 1);
  const int32_t st = state[l];
  const int64_t row = ((int64_t)b * p.N + node) * p.L + l;
  float conf;
  int32_t tok;
  TaggedSlices from{tag, kPollsABatch};
  const bool ok = finalize_row<kLanes>(p.partials + row * p.splits, p.splits, sub, st, p.mask_id, conf, tok, from);
  if (__syncthreads_or(from.missing)) return false;
  if (sub == 0 && r < p.L) {
    s_conf[l] = conf;
    s_top[l] = tok;
    p.conf[row] = conf;
    p.top_tok[row] = tok;
    if (!ok && p.decide_status) atomicOr(p.decide_status + b, SPIFFY_DEV_NONFINITE);
  }
  __syncthreads();
  return true;
}

// grid: B tails, then reducers, sequence r % B for reducer r; dynamic shared memory: the graph, when staged.
template <typename T>
__global__ void __launch_bounds__(kReduceThreads, kWalkCtas)
lazy_walk_kernel(const __grid_constant__ LazyParams p) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = p.N, L = p.L, B = p.B;
  const bool is_tail = (int)blockIdx.x < B;
  const int r = (int)blockIdx.x - B, reducers = (int)gridDim.x - B;
  const int b = is_tail ? (int)blockIdx.x : r % B;
  __shared__ uint32_t s_kids[kTableNodes][2];  // which nodes list this one as a parent, a bit each
  __shared__ uint32_t s_hash[kTableNodes];    // of its state
  __shared__ uint64_t s_masked[kTableNodes];  // its still-masked positions
  __shared__ int s_guess[kTableNodes];        // reducers: the node taken up at each level
  __shared__ LazyWord s_word;
  __shared__ int s_bad;
  extern __shared__ __align__(16) unsigned char lazy_smem[];
  // The graph and the tokens were complete before the root kernel let this one start (it waits first).
  Graph g = {p.block_tokens + (int64_t)b * N * L, p.parent_off + (int64_t)b * (N + 1), p.parent_idx + (int64_t)b * p.parent_cap};
  const int32_t* tokens = g.state;
  const bool table = N <= kTableNodes;
  if (p.stage_graph && (is_tail || table)) {
    int32_t* s_off = reinterpret_cast<int32_t*>(lazy_smem);
    int32_t* s_idx = s_off + (N + 1);
    int32_t* s_state = s_idx + p.parent_cap;
    auto copy4 = [](void* dst, const void* src) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    };
    for (int i = tid; i <= N; i += kReduceThreads) copy4(s_off + i, g.off + i);
    for (int i = tid; i < p.parent_cap; i += kReduceThreads) copy4(s_idx + i, g.idx + i);
    g.off = s_off;
    g.idx = s_idx;
    if (is_tail) {
      for (int i = tid; i < N * L; i += kReduceThreads) copy4(s_state + i, g.state + i);
      g.state = s_state;
    }
  }
  if (tid == 0) s_bad = 0;
  if (table) {
    if (tid < kTableNodes) s_kids[tid][0] = s_kids[tid][1] = 0u;
#pragma unroll 4
    for (int n = warp; n < N; n += kReduceThreads / 32) {
      int32_t state[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) state[h] = lane + 32 * h < L ? tokens[n * L + lane + 32 * h] : 0;
      const uint64_t masked = masked_of(state, L, p.mask_id, lane);
      const uint32_t hash = hash_of(state, lane);
      if (lane == 0) {
        s_masked[n] = masked;
        s_hash[n] = hash;
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (table) {
    for (int m = 1 + warp; m < N; m += kReduceThreads / 32)
      if (!enter_parents(s_kids, g.off, g.idx, p.parent_cap, m, lane)) s_bad = 1;
    __syncthreads();
  }
  Partial* const slices = p.partials + (int64_t)b * N * L * p.splits;
  const T* const logits = static_cast<const T*>(p.logits) + (int64_t)b * N * L * p.row_stride;

  if (!is_tail) {
    // ---------------------------------------------------------- reducers --
    const int rank = r / B, stride = (reducers - b + B - 1) / B;
    auto likely = [&](int n) {
      if (!table || n < 0) return -1;
      const uint32_t lo = s_kids[n][0], hi = s_kids[n][1];
      return lo ? __ffs(lo) - 1 : hi ? __ffs(hi) + 31 : -1;
    };
    bool waited = false;
    auto wait_root = [&]() {
#if __CUDA_ARCH__ >= 900
      if (!waited) {
        cudaGridDependencySynchronize();  // the root's slices and the cleared marks and words
        pdl_launch_dependents();
      }
#endif
      waited = true;
    };
    LazyWord w = {0, 0, 0};    // the last one seen
    int level = 1, taken = 0;  // the level worked at; those of s_guess
    int node = likely(0);
    uint64_t masked = node >= 0 ? s_masked[node] : 0;
    // the word says something that was not acted upon
    auto news = [&](const LazyWord& x) {
      return x.level != kEnded && (x.level > taken || (table && x.level > 0 && s_guess[x.level] != x.node));
    };
    for (;;) {
      if (node < 0 || level > w.level + 1) {  // no guess, or one too far ahead: wait for the word
        wait_root();
        const int enough = node < 0 ? kEnded : level - 1;
        if (tid == 0) {
          unsigned polls = 0;
          LazyWord x = load_word(p.words + b);
          while (x.level < enough && !news(x) && ++polls <= p.wait_spins) {
            __nanosleep(32);
            x = load_word(p.words + b);
          }
          s_word = x;
        }
        __syncthreads();
        w = s_word;
        const bool other = news(w);
        __syncthreads();  // s_word and s_guess are read
        if (w.level == kEnded || (!other && w.level < enough)) return;
        if (other) {
          level = w.level;
          node = w.node;
          masked = w.masked;
        }
      }
      // `node` is taken up at `level`
      if (tid == 0 && level < kTableNodes) s_guess[level] = node;
      taken = level;
      bool dropped = false;
      const int items = __popcll(masked) * p.splits;
      for (int i = rank; i < items; i += stride) {
        LazyWord peek = w;
        if (tid == 0 && waited) peek = load_word(p.words + b);  // on its way beside the slice
        const Item it = item_of(p, node, masked, i);
        Partial* out = slices + it.row * p.splits + it.split;
        const T* row = logits + it.row * p.row_stride;
        const Partial q = reduce_slice(row, p.V, p.chunk, it.split, static_cast<Partial*>(nullptr));
        wait_root();  // a first guess is read, not written, while the root is at work
        if (tid == 0) {
          store16(out, (uint64_t)__float_as_uint(q.m) | (uint64_t)__float_as_uint(q.s) << 32,
                  (uint64_t)(uint32_t)q.idx | (uint64_t)(uint32_t)kPresent << 32);
          s_word = peek;
        }
        __syncthreads();  // the word; the reduce's shared scratch
        w = s_word;
        if (w.level == kEnded) return;
        if (news(w)) {
          dropped = true;
          level = w.level;
          node = w.node;
          masked = w.masked;
          break;
        }
      }
      __syncthreads();
      if (dropped) continue;
      ++level;
      node = likely(node);
      if (level >= kTableNodes) node = -1;
      masked = node >= 0 ? s_masked[node] : 0;
    }
  }

  // ---------------------------------------------------------------- tail --
  __shared__ float s_conf[64];
  __shared__ int32_t s_top[64], s_next[64];
  __shared__ int s_found;
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();
  pdl_launch_dependents();
#endif
  for (int i = tid; i < N; i += kReduceThreads) {
    p.path[(int64_t)b * N + i] = i == 0 ? 0 : -1;
    p.n_unmask[(int64_t)b * N + i] = -1;  // not evaluated (yet)
  }
  const int tag = b == 0 && p.lost_slices != 0 ? -1 : kPresent;
  int node = 0, hops = 0;
  bool looked = false;  // for children: the parent lists were read
  for (;;) {
    const int32_t* state = g.state + node * L;
    // slices of this node's still-masked rows
    unsigned polls = 0;
    bool there, helped = false;
    while (!(there = L <= 16   ? merge_rows<8>(p, b, node, state, tag, s_conf, s_top)
                     : L <= 32 ? merge_rows<4>(p, b, node, state, tag, s_conf, s_top)
                               : merge_rows<2>(p, b, node, state, tag, s_conf, s_top))) {
      polls += kPollsABatch;
      if (polls > p.wait_spins) break;
      if (!helped && (b >= reducers || polls > kPollsToHelp)) {
        helped = true;
        const int32_t mine[2] = {lane < L ? state[lane] : 0, lane + 32 < L ? state[lane + 32] : 0};
        reduce_missing(p, logits, slices, node, masked_of(mine, L, p.mask_id, lane));
      }
    }
    if (!there) {  // a bounded wait ran out: the walk ends here, in the word too
      if (tid == 0) {
        store_word(p.words + b, LazyWord{kEnded, -1, 0});
        if (p.decide_status) atomicOr(p.decide_status + b, SPIFFY_DEV_TIMEOUT);
        if (p.walk_status) atomicOr(p.walk_status + b, SPIFFY_DEV_TIMEOUT);
      }
      return;
    }
    if (warp == 0) {
      const uint64_t bits = unmask_rule(s_conf, state, L, p.mask_id, p.rule, p.top_s, p.tau, lane);
      const bool go_on = bits != 0 && hops < N - 1;
      int32_t next[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int l = lane + 32 * h;
        next[h] = l < L ? (((bits >> l) & 1ull) ? s_top[l] : state[l]) : 0;
        if (l < L) s_next[l] = next[h];
      }
      const uint64_t left = masked_of(next, L, p.mask_id, lane);
      int found = kNoLink;
      // the first node (ascending) that lists `node` as a parent and equals its next state
      if (table && go_on) found = child_of(s_kids[node], s_hash, g.state, next, N, L, lane);
      if (lane == 0) {
        s_found = found;
        s_word = LazyWord{go_on, 0, left};
        if (table)  // what the reducers of b wait for
          store_word(p.words + b, found == kNoLink ? LazyWord{kEnded, -1, 0} : LazyWord{hops + 1, found, left});
        p.unmask_bits[(int64_t)b * N + node] = bits;
        p.n_unmask[(int64_t)b * N + node] = __popcll(bits);
      }
    }
    __syncthreads();
    const bool go_on = s_word.level != 0;
    looked |= go_on;
    if (!table) {
      if (go_on) {
        bool bad = false;
        for (int m = node + 1 + warp; m < N; m += kReduceThreads / 32) {
          const int e0 = g.off[m], e1 = g.off[m + 1];
          if (e0 < 0 || e1 < e0 || e1 > p.parent_cap) {  // malformed offsets
            bad = true;
            continue;
          }
          bool is_child = false;
          for (int e = e0 + lane; e < e1; e += 32) {
            const int q = g.idx[e];
            if (q < 0 || q >= m) bad = true;  // ignored entry
            is_child |= q == node;
          }
          if (!__any_sync(0xffffffffu, is_child)) continue;
          const int32_t* sm = g.state + m * L;
          const bool eq = (lane >= L || sm[lane] == s_next[lane]) && (lane + 32 >= L || sm[lane + 32] == s_next[lane + 32]);
          if (__all_sync(0xffffffffu, eq) && lane == 0) atomicMin(&s_found, m);
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) s_bad = 1;
      }
      __syncthreads();
      if (tid == 0)
        store_word(p.words + b, s_found == kNoLink ? LazyWord{kEnded, -1, 0} : LazyWord{hops + 1, s_found, s_word.masked});
    }
    const int found = s_found;
    if (found == kNoLink) break;
    hops += 1;  // accepted: its distribution replaces the target's
    node = found;
    if (tid == 0) p.path[(int64_t)b * N + hops] = found;
    __syncthreads();  // s_found, s_conf and s_top are read
  }
  // the walk ends on `node`
  if (tid < L) p.next_block[(int64_t)b * L + tid] = s_next[tid];
  if (tid == 0) {
    p.accepted_node[b] = node;
    p.n_accepted[b] = hops;
    if (looked && s_bad && p.walk_status) atomicOr(p.walk_status + b, SPIFFY_DEV_BADGRAPH);
  }
}

size_t lazy_graph_bytes(const spiffy_decide_desc& d, int parent_cap) {
  return ((size_t)d.n_nodes * d.block_len + d.n_nodes + 1 + parent_cap) * 4;
}

size_t lazy_partial_bytes(const spiffy_decide_desc& d) {
  return (size_t)d.batch * d.n_nodes * d.block_len * decide_splits(d, nullptr) * sizeof(Partial);
}

}  // namespace

size_t decide_lazy_workspace_bytes(const spiffy_decide_desc& d) {
  return lazy_partial_bytes(d) + (size_t)d.batch * sizeof(LazyWord);  // slices | words[B]
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
  const int stage_graph = graph <= 32 * 1024;  // kWalkCtas of them fit an SM
  const int most = kWalkCtas * sm_count();
  if (most <= 0) return SPIFFY_ECUDA;
  if (d.batch > most) return SPIFFY_EUNSUPPORTED;
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
  p.partials = static_cast<Partial*>(ws);
  p.words = reinterpret_cast<LazyWord*>(static_cast<char*>(ws) + lazy_partial_bytes(d));
  p.clear = status_clear(d, fresh, decide_status, walk_status);
  p.stage_graph = stage_graph;
  p.wait_spins = flag_poll_limit();
  p.lost_slices = lazy_extra_arrivals();
  const dim3 root(p.splits, d.batch * d.block_len);
  cudaError_t e = bf16 ? launch_pdl(lazy_root_kernel<__nv_bfloat16>, root, dim3(kReduceThreads), (size_t)0, stream, p)
                       : launch_pdl(lazy_root_kernel<float>, root, dim3(kReduceThreads), (size_t)0, stream, p);
  count_launch();
  if (e != cudaSuccess) return SPIFFY_ECUDA;
  const int64_t items = d.n_nodes > 1 ? (int64_t)d.batch * d.block_len * p.splits : 0;
  const dim3 grid((unsigned)(items + d.batch < most ? items + d.batch : most));
  const size_t smem = stage_graph ? graph : 0;
  e = bf16 ? launch_pdl(lazy_walk_kernel<__nv_bfloat16>, grid, dim3(kReduceThreads), smem, stream, p)
           : launch_pdl(lazy_walk_kernel<float>, grid, dim3(kReduceThreads), smem, stream, p);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

}  // namespace spiffy
