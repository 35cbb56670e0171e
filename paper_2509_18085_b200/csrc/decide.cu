// Decision kernels: steps 1-4 of Algorithm 1 (the function Next() of App. A)
// evaluated for every node of the draft graph, and their fusion with step 5.
//
//   decide_reduce_kernel    streams the logits rows of still-masked positions
//                           once (the HBM-bound part): per (row, vocabulary
//                           slice) the maximum, the sum of exponentials and the
//                           lowest index that attains the maximum
//   decide_finalize_kernel  per node: merges the slices in a fixed order, turns
//                           them into (confidence, top token) and applies the
//                           unmasking rule of Sec. 3.1
//   decide_tail_kernel      per sequence, for small graphs: the finalize step
//                           of all its nodes and the acceptance walk (step 5)
//                           in one CTA, resident before the reduce ends
//
// The arithmetic shared with the other decision kernels is in decide_core.cuh,
// the walk in walk_core.cuh.
#include "common.cuh"
#include "decide_core.cuh"
#include "sm100_ptx.cuh"
#include "walk_core.cuh"

namespace spiffy {
namespace {

// grid = (splits, B*N*L); one CTA reduces one vocabulary slice of one row.
// kIndependent: the kernel before this one, which may still run, writes none of its inputs and has
// let it start only when all others were complete (SPIFFY_INDEPENDENT).  A kernel of its own: the
// token from L2 instead of L1, the wait at the end and the way to it cost the plain one 3 to 4 % of
// the call, and the status words cleared ahead of the token's load, for which every CTA waits first,
// another 1 to 2 % (256 rows x 126464 with 164 masked: 13.0 us with all that, 12.4 so; 512 rows x
// 152064 with 348 masked: 24.6 and 23.4).
// What bounds it beside the bytes is instructions issued, and CTAs in flight to cover one another's
// chains: the search for the maximum's index by the threads that hold it alone, their vote through one
// atomic, a maximum by one instruction a warp, and with the registers that saves nine CTAs per SM
// (56 registers; eight before, with 64): 4096 rows x 126464 with 2596 masked 121 -> 108.5 us (6.05
// TB/s), 512 x 152064 with 322 masked 27.3 -> 25.3 with the walk, 256 x 126464 with 142 13.8 -> 13.1.
// Tried and dropped: ten CTAs (113.6), slices in shared memory by asynchronous copies with ten or
// twelve CTAs (120), runs of slices per CTA, the next one's loads under this one's end (111 to 120, and
// 3 us more at 256 rows) or in a second set of registers (150).
template <typename T, bool kIndependent>
__global__ void __launch_bounds__(kReduceThreads, 9)  // 56 registers: nine CTAs per SM
decide_reduce_kernel(const T* __restrict__ logits, int64_t row_stride, int V,
                     int64_t chunk, int splits,
                     const int32_t* __restrict__ block_tokens, int mask_id,
                     Partial* __restrict__ partials, int early_trigger, StatusClear clear) {
#if __CUDA_ARCH__ >= 900
  if (!kIndependent) cudaGridDependencySynchronize();  // inputs written by earlier kernels are visible
#endif
  const int row = blockIdx.y;
  const int32_t token = kIndependent ? __ldcg(block_tokens + row) : block_tokens[row];
  if (blockIdx.x == 0 && threadIdx.x == kReduceThreads - 1 && row < clear.batch) clear.run(row);
  if (!kIndependent && token != mask_id) return;  // already unmasked: never read
  // kIndependent: this grid is complete, for all that wait for it, no sooner than the one before it
  const bool waits = kIndependent && blockIdx.x + 1 == gridDim.x && blockIdx.y + 1 == gridDim.y;
#if __CUDA_ARCH__ >= 900
  // The one-CTA-per-sequence tail kernel may take its SM while this grid still runs (it waits there for
  // this grid to finish): its launch latency is hidden.  A CTA that has nothing to read says the same by
  // ending; triggering first costs the grid 0.5 ns for each of them, much of the call where few rows are
  // still masked (one in twenty of 256 rows x 126464: 9.7 us, 8.2 so; of 512 x 152064, 9728 CTAs, beside an
  // attention of 28 heads 25.6 and 21.5).
  if (early_trigger && (token == mask_id || waits)) pdl_launch_dependents();
#endif
  if (token == mask_id)
    reduce_slice(logits + (int64_t)row * row_stride, V, chunk, (int)blockIdx.x,
                 partials + (int64_t)row * splits + blockIdx.x);
#if __CUDA_ARCH__ >= 900
  if (waits) cudaGridDependencySynchronize();
#endif
}

// grid = B*N nodes, 512 threads: eight threads per position merge the slices of
// its row, then warp 0 applies the rule.
// kAtOnce: slices of a thread on their way at a time; a further trip is 0.4 us or more.  Ten for the output
// projection with more than 32 slices a row (148: 0.5 to 1.3 us a call, 4 x 32 positions x 1024 x 32000 31.6 -> 30.3,
// 8 x 32 x 4096 x 126464 193.0 -> 192.0).  Else four: one trip for the 32 slices of 131072 fp32 or 262144 bf16 entries.
// With four, four CTAs to an SM at 32 registers: 100 nodes x 8 rows of one slice 6.6 us a call, with three (35
// registers) 7.2; 200 x 2 5.1 and 5.6.  With ten, as many registers as it likes, 62: 1 x 4 x 8 positions x 512 x 16000
// 11.0 us, at 40 registers 12.2.
constexpr int kFinalizeThreads = 512;
template <int kAtOnce>
__global__ void __launch_bounds__(kFinalizeThreads, kAtOnce > 4 ? 1 : 4)
decide_finalize_kernel(const Partial* __restrict__ partials, int splits, int N,
                       int L, const int32_t* __restrict__ block_tokens,
                       int mask_id, int rule, int top_s, float tau,
                       float* __restrict__ conf_out, int32_t* __restrict__ tok_out,
                       uint64_t* __restrict__ bits_out,
                       int32_t* __restrict__ n_unmask_out,
                       int32_t* __restrict__ dev_status) {
#if __CUDA_ARCH__ >= 900
  pdl_launch_dependents();
  cudaGridDependencySynchronize();  // the reduce kernel's partials are visible
#endif
  const int node = blockIdx.x;
  const int pos = threadIdx.x >> 3, sub = threadIdx.x & 7;
  __shared__ float sconf[64];
  {
    const int row = node * L + min(pos, L - 1);
    // the token and the partials are read together (one trip to memory); the
    // partials of an unmasked row were never written and are ignored
    const int32_t state = block_tokens[row];
    float conf;
    int32_t tok;
    const bool ok = finalize_row<8, CompleteSlices, kAtOnce>(partials + (int64_t)row * splits, splits, sub, state, mask_id,
                                                             conf, tok, CompleteSlices{});
    if (sub == 0 && pos < L) {
      conf_out[row] = conf;
      tok_out[row] = tok;
      sconf[pos] = conf;
      if (!ok && dev_status) atomicOr(dev_status + node / N, SPIFFY_DEV_NONFINITE);
    }
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const uint64_t bits = unmask_rule(sconf, block_tokens + (int64_t)node * L, L, mask_id, rule, top_s,
                                    tau, threadIdx.x);
  if (threadIdx.x == 0) {
    bits_out[node] = bits;
    n_unmask_out[node] = __popcll(bits);
  }
}

// Decision tail and acceptance walk of one sequence in one CTA (Algorithm 1,
// steps 1-5 after the vocabulary reduce): up to eight threads per row merge the
// slices, then one warp per node applies the rule and looks for the child that
// equals the node's next state, and warp 0 walks.  The graph (states, parent
// lists) does not depend on the reduce kernel; ahead of the wait it is copied to
// shared memory and, for up to kTableNodes nodes, made a table of children with
// hashes of the states, which saves a step of its own for the links.
// grid = B, kTailThreads threads or fewer, dynamic shared memory tail_smem_bytes().
// Bound: a chain of short steps.  Behind the wait, 3 x 100 rows x 7 slices, two positions a node: 2640 cycles
// for the merge, 1640 for the rule, 1020 for links and 1010 for the chase when the rule ranked positions one
// by one and links were a step of their own with an exchange through atomics; 2040, 2110 for rule and links,
// 770 now (the decision behind an attention of that shape 18.3 -> 17.6 us, 4 x 8 rows of one slice 9.1 -> 8.6).
// 48 registers: with 56 and more, fewer reduce CTAs stay on the SM that the tail moves in on, and it comes
// later (16 x 32 rows x 19 slices with an attention beside them 30.9 us, 30.8 so, 31.0 with 64).
constexpr int kTailThreads = 1024;
struct TailArgs {
  int splits, N, L, mask_id, rule, top_s;
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
};
// A sequence's tail, by all threads of a CTA; `memory`: tail_smem_bytes().  kHold: the results stay in shared
// memory until publish().
template <bool kHold>
class Tail {
 public:
  __device__ __forceinline__ Tail(const TailArgs& a, int b, unsigned char* memory)
      : a(a), b(b), rows(a.N * a.L), warp(threadIdx.x >> 5), lane(threadIdx.x & 31), warps(blockDim.x >> 5),
        table(a.N <= kTableNodes) {
    bits = reinterpret_cast<uint64_t*>(memory);
    state = reinterpret_cast<int32_t*>(bits + a.N);
    top = state + rows;
    conf = reinterpret_cast<float*>(top + rows);
    off = reinterpret_cast<int32_t*>(conf + rows);
    idx = off + (a.N + 1);
    link = idx + a.parent_cap;
    __shared__ uint32_t s_kids[kTableNodes][2];
    __shared__ uint32_t s_hash[kTableNodes];
    __shared__ int32_t s_flags[kHold ? 4 : 1];
    kids = s_kids;
    hash = s_hash;
    flags = s_flags;
  }
  // The graph on its way to shared memory.  kNow: read at L2, by a kernel that does not wait for the one before it.
  template <bool kNow>
  __device__ __forceinline__ void fetch() {
    auto copy4 = [](void* dst, const void* src) {
      if constexpr (kNow) {
        *static_cast<int32_t*>(dst) = __ldcg(static_cast<const int32_t*>(src));
        return;
      }
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(dst)),
                   "l"(src)
                   : "memory");
    };
    const int32_t* from_state = a.block_tokens + (int64_t)b * rows;
    const int32_t* from_off = a.parent_off + (int64_t)b * (a.N + 1);
    const int32_t* from_idx = a.parent_idx + (int64_t)b * a.parent_cap;
    const int tid = threadIdx.x, step = blockDim.x;
    for (int i = tid; i < rows; i += step) copy4(state + i, from_state + i);
    for (int i = tid; i <= a.N; i += step) copy4(off + i, from_off + i);
    for (int i = tid; i < a.parent_cap; i += step) copy4(idx + i, from_idx + i);
    for (int i = tid; i < a.N; i += step) link[i] = kNoLink;
    for (int i = tid; i < 2 * kTableNodes; i += step) (&kids[0][0])[i] = 0u;
    if (kHold && tid < 2) flags[tid] = 0;
  }
  // ... has arrived: children and hashes, complete behind the next barrier of the CTA.
  __device__ __forceinline__ void arrived() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (!table) return;
#pragma unroll 1
    for (int n = warp; n < a.N; n += warps) {
      const int32_t mine[2] = {lane < a.L ? state[n * a.L + lane] : 0, lane + 32 < a.L ? state[n * a.L + lane + 32] : 0};
      const uint32_t h = hash_of(mine, lane);
      if (lane == 0) hash[n] = h;
      if (n > 0) good &= enter_parents(kids, off, idx, a.parent_cap, n, lane);
    }
  }
  // Steps 1 and 2: kLanes threads a row merge its slices, `splits` from partials + row * splits on.
  template <int kLanes, class Source>
  __device__ __forceinline__ void merge_rows(const Partial* partials, Source source) {
    const int sub = threadIdx.x & (kLanes - 1), step = blockDim.x / kLanes;
    for (int base = 0; base < rows; base += step) {
      const int r = base + threadIdx.x / kLanes;
      const int row = min(r, rows - 1);
      float c;
      int32_t tok;
      const bool ok = finalize_row<kLanes>(partials + (int64_t)row * a.splits, a.splits, sub, state[row], a.mask_id, c, tok,
                                           source);
      if (sub == 0 && r < rows) {
        if (!kHold) {
          a.conf[(int64_t)b * rows + row] = c;
          a.top_tok[(int64_t)b * rows + row] = tok;
        }
        conf[row] = c;
        top[row] = tok;
        if (!ok) report(0, a.decide_status, SPIFFY_DEV_NONFINITE);
      }
    }
  }
  // Steps 3 to 5.
  __device__ __forceinline__ void walk() {
    const int N = a.N, L = a.L;
    __syncthreads();
#pragma unroll 1
    for (int node = warp; node < N; node += warps) {
      const uint64_t take = unmask_rule(conf + node * L, state + node * L, L, a.mask_id, a.rule, a.top_s, a.tau, lane);
      int child = kNoLink;
      if (table && take != 0) {  // a node with nothing to unmask ends the walk
        int32_t next[2];         // the node's next state
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = lane + 32 * h;
          next[h] = l < L ? walk_next_token(state, top, take, node, L, l) : 0;
        }
        child = child_of(kids[node], hash, state, next, N, L, lane);
      }
      if (lane == 0) {
        if (!kHold) {
          a.unmask_bits[(int64_t)b * N + node] = take;
          a.n_unmask[(int64_t)b * N + node] = __popcll(take);
        }
        bits[node] = take;
        if (table) link[node] = child;
      }
    }
    if (!table) {
      __syncthreads();
      good = !walk_link_children(N, L, a.parent_cap, state, top, off, idx, bits, link, warp, warps, lane);
    }
    if (!good) report(1, a.walk_status, SPIFFY_DEV_BADGRAPH);
    __syncthreads();
    if (warp != 0) return;
    if (kHold) {
      int hops;
      const int end = walk_follow(N, link, link, lane, hops);
      if (lane == 0) flags[2] = end, flags[3] = hops;
    } else {
      walk_chase(N, L, state, top, bits, link, a.path + (int64_t)b * N, a.next_block + (int64_t)b * L, a.accepted_node + b,
                 a.n_accepted + b, lane);
    }
  }
  // kHold, 256 threads, up to 64 rows: the results to where they belong once the kernel before is complete, whose
  // memory that may have been.  What a thread writes is in its registers by then (4 x 16 rows of one slice beside an
  // attention over 500 keys 20.0 us; read from shared memory behind the wait 21.3, written ahead of it 19.9).
  __device__ __forceinline__ void publish(bool fresh) {
    __syncthreads();
    const int N = a.N, L = a.L, part = (int)threadIdx.x / 64, i = (int)threadIdx.x % 64, end = flags[2], hops = flags[3];
    int32_t *one = nullptr, *two = nullptr;
    int32_t first = 0, second = 0;
    uint64_t set = 0;
    if (part == 0) {
      if (i < rows) one = reinterpret_cast<int32_t*>(a.conf) + b * rows + i, first = __float_as_int(conf[i]);
      if (i == 0) two = a.accepted_node + b, second = end;
      if (i == 1) two = a.n_accepted + b, second = hops;
    } else if (part == 1) {
      if (i < rows) one = a.top_tok + b * rows + i, first = top[i];
      if (i < 2) two = i == 0 ? a.decide_status : a.walk_status, second = flags[i];
      if (two) two += b;
      if (!fresh && second == 0) two = nullptr;
    } else if (part == 2) {
      if (i < N) one = a.n_unmask + b * N + i, set = bits[i], first = __popcll(set);
    } else {
      if (i < N) one = a.path + b * N + i, first = i <= hops ? link[i] : -1;
      if (i < L) two = a.next_block + b * L + i, second = walk_next_token(state, top, bits[end], end, L, i);
    }
#if __CUDA_ARCH__ >= 900
    cudaGridDependencySynchronize();
    pdl_launch_dependents();
#endif
    if (one) *one = first;
    if (part == 2 && i < N) a.unmask_bits[b * N + i] = set;
    if (two) {
      if (part == 1 && !fresh) atomicOr(two, second);
      else *two = second;
    }
  }
  int32_t* state;

 private:
  const TailArgs& a;
  const int b, rows, warp, lane, warps;
  const bool table;
  bool good = true;  // no malformed offset or entry met
  int32_t* flags;    // kHold: status bits of the decision and of the walk, the node it ends on, the hops
  __device__ __forceinline__ void report(int which, int32_t* status, int32_t flag) {
    if (kHold) atomicOr(flags + which, flag);
    else if (status) atomicOr(status + b, flag);
  }
  uint64_t* bits;
  int32_t *top, *off, *idx;
  float* conf;
  int* link;
  uint32_t (*kids)[2];
  uint32_t* hash;
};

template <int kLanes>  // threads per row: all N * L rows are merged in one pass when there are kLanes * N * L threads
__global__ void __launch_bounds__(kTailThreads + 256, 1)  // 48 registers
decide_tail_kernel(const Partial* __restrict__ partials, int splits, int N, int L,
                   const int32_t* __restrict__ block_tokens, int mask_id, int rule, int top_s,
                   float tau, float* __restrict__ conf_out, int32_t* __restrict__ tok_out,
                   uint64_t* __restrict__ bits_out, int32_t* __restrict__ n_unmask_out,
                   int32_t* __restrict__ decide_status,
                   const int32_t* __restrict__ parent_off, const int32_t* __restrict__ parent_idx,
                   int parent_cap, int32_t* __restrict__ accepted_node,
                   int32_t* __restrict__ n_accepted, int32_t* __restrict__ path,
                   int32_t* __restrict__ next_block, int32_t* __restrict__ walk_status, int early_trigger) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
#if __CUDA_ARCH__ >= 900
  if (early_trigger) pdl_launch_dependents();  // an independent kernel comes next, and takes the SMs the reduce leaves
#endif
  const TailArgs a = {splits, N, L, mask_id, rule, top_s, tau, block_tokens, parent_off, parent_idx, parent_cap, conf_out,
                      tok_out, bits_out, n_unmask_out, decide_status, accepted_node, n_accepted, path, next_block, walk_status};
  Tail<false> tail(a, (int)blockIdx.x, tail_smem);
  tail.template fetch<false>();
  tail.arrived();
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();  // the reduce kernel's partials are visible
  pdl_launch_dependents();          // only now: this CTA was resident during the reduce, the next kernel's need not be
#endif
  tail.template merge_rows<kLanes>(partials + (int64_t)blockIdx.x * N * L * splits, CompleteSlices{});
  tail.walk();
}

// The same for few slices beside a CUDA-core attention (SPIFFY_INDEPENDENT), reduce included: a cluster of
// kSmallCtas CTAs per sequence, whose groups of kReduceThreads threads take the slices of masked rows in turn;
// the partial results go straight into the shared memory of the first CTA, which does the rest, writes its
// results once the attention is complete and keeps them in shared memory until then.  One launch
// instead of two, and no partial result waits for a kernel to end and another to read it from L2.  Bound: the
// launch, a trip for the tokens and one for each round of slices, the steps of the tail.  Two groups a CTA: larger
// ones find no room beside an attention that fills the machine (2 x 32 positions x 32 heads over 4000 keys
// 127.2 us, with four groups 133.9, without this kernel 130.1; 4 x 2 x 8 positions x 12 heads over 300 10.8, 14.8
// and 13.7), and the smallest gain nothing by them (4 x 8 rows of one slice 6.3, 6.2 and 9.2; all with the results
// written ahead of the wait).
constexpr int kSmallCtas = 8, kSmallGroups = 2, kSmallRows = 64;
template <typename T>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallGroups* kReduceThreads)
decide_small_kernel(const __grid_constant__ TailArgs a, const T* __restrict__ logits, int64_t row_stride, int V,
                    int64_t chunk, int next, int fresh) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ int16_t list[kSmallRows];  // the masked rows
  __shared__ int n_masked;
  const int b = (int)blockIdx.x / kSmallCtas, rank = (int)blockIdx.x % kSmallCtas, tid = threadIdx.x;
  const int rows = a.N * a.L, group = tid / kReduceThreads;
  sm100::cluster_arrive_relaxed();  // the first CTA is there when all are
#if __CUDA_ARCH__ >= 900
  if (next) pdl_launch_dependents();
#endif
  if (tid < 32) {
    int32_t token[kSmallRows / 32];
    int n = 0;
#pragma unroll
    for (int h = 0; h < kSmallRows / 32; ++h)  // all on their way at once
      token[h] = 32 * h < rows ? __ldcg(a.block_tokens + (int64_t)b * rows + min(tid + 32 * h, rows - 1)) : 0;
#pragma unroll
    for (int h = 0; h < kSmallRows / 32; ++h) {
      const bool masked = tid + 32 * h < rows && token[h] == a.mask_id;
      const unsigned vote = __ballot_sync(0xffffffffu, masked);
      if (masked) list[n + __popc(vote & ((1u << tid) - 1u))] = (int16_t)(tid + 32 * h);
      n += __popc(vote);
    }
    if (tid == 0) n_masked = n;
  }
  Partial* slots = reinterpret_cast<Partial*>(tail_smem);
  Tail<true> tail(a, b, tail_smem + (size_t)rows * a.splits * sizeof(Partial));
  if (rank == 0) tail.template fetch<true>();
  __syncthreads();
  // the first CTA, which has the graph to prepare, comes last
  const int items = n_masked * a.splits, first = (rank + kSmallCtas - 1) % kSmallCtas * kSmallGroups + group;
  const uint32_t leader = sm100::map_to_cta(sm100::smem_u32(slots), 0);
  bool all_here = false;
  for (int i = first; i < items; i += kSmallCtas * kSmallGroups) {
    const int nth = i / a.splits, split = i - nth * a.splits, row = list[nth];
    const Partial r = reduce_slice<T, kSmallGroups>(logits + ((int64_t)b * rows + row) * row_stride, V, chunk, split,
                                               static_cast<Partial*>(nullptr));
    if (!all_here) sm100::cluster_wait();
    all_here = true;
    if (tid % kReduceThreads == 0)
      asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(leader + (uint32_t)(row * a.splits + split) * 16u),
                   "r"(__float_as_uint(r.m)), "r"(__float_as_uint(r.s)), "r"((uint32_t)r.idx), "r"(0u)
                   : "memory");
  }
  if (!all_here) sm100::cluster_wait();
  sm100::cluster_arrive();
  if (rank != 0) return;
  tail.arrived();
  sm100::cluster_wait();  // every slice is here
  tail.template merge_rows<4>(slots, SharedSlices{});
  tail.walk();
  tail.publish(fresh);
}

size_t tail_smem_bytes(const spiffy_decide_desc& d, int parent_cap) {
  return (size_t)d.n_nodes * 8 +
         ((size_t)3 * d.n_nodes * d.block_len + 2 * d.n_nodes + 1 + parent_cap) * 4;
}

}  // namespace

int decide_splits(const spiffy_decide_desc& d, int64_t* chunk_elems) {
  // A slice is at most what one CTA holds in registers: kReduceThreads * kUnroll
  // vectors of 16 bytes (8192 bf16 or 4096 fp32 logits); slices start on
  // 16-byte boundaries.
  const int64_t epv = d.logits_dtype == SPIFFY_BF16 ? 8 : 4;
  const int64_t most = (int64_t)kReduceThreads * kUnroll * epv;
  const int64_t splits = (d.vocab + most - 1) / most;
  // equal slices, rounded up to whole vectors
  int64_t chunk = (d.vocab + splits - 1) / splits;
  chunk = (chunk + epv - 1) / epv * epv;
  if (chunk_elems) *chunk_elems = chunk;
  return (int)(splits < 1 ? 1 : splits);
}

size_t decide_workspace_bytes(const spiffy_decide_desc& d) {
  const int64_t rows = (int64_t)d.batch * d.n_nodes * d.block_len;
  return (size_t)rows * decide_splits(d, nullptr) * sizeof(Partial);
}

namespace {

spiffy_status launch_reduce(const spiffy_decide_desc& d, const void* logits,
                            const int32_t* block_tokens, Partial* partials, int splits,
                            int64_t chunk, int early_trigger, bool independent, StatusClear clear,
                            cudaStream_t stream) {
  const int rows = d.batch * d.n_nodes * d.block_len;
  const dim3 grid(splits, rows);
  auto run = [&](auto* typed, auto plain, auto beside) {
    return launch_pdl(independent ? beside : plain, grid, dim3(kReduceThreads), (size_t)0, stream, typed,
                      (int64_t)d.row_stride, (int)d.vocab, chunk, splits, block_tokens, (int)d.mask_token_id,
                      partials, early_trigger, clear);
  };
  const cudaError_t e = d.logits_dtype == SPIFFY_BF16
                            ? run(static_cast<const __nv_bfloat16*>(logits), decide_reduce_kernel<__nv_bfloat16, false>,
                                  decide_reduce_kernel<__nv_bfloat16, true>)
                            : run(static_cast<const float*>(logits), decide_reduce_kernel<float, false>,
                                  decide_reduce_kernel<float, true>);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

spiffy_status decide_only(const spiffy_decide_desc& d, const void* logits,
                          const int32_t* block_tokens, float* conf,
                          int32_t* top_tok, uint64_t* unmask_bits,
                          int32_t* n_unmask, int32_t* dev_status, void* ws, bool fresh, bool independent,
                          bool next, cudaStream_t stream) {
  int64_t chunk = 0;
  const int splits = decide_splits(d, &chunk);
  Partial* partials = static_cast<Partial*>(ws);
  // `next`: an independent kernel comes after this call and takes the SMs the reduce leaves; the
  // small kernels in between trigger as soon as they are resident, so it is the reduce that lets it in.
  const spiffy_status st = launch_reduce(d, logits, block_tokens, partials, splits, chunk, next, independent,
                                         status_clear(d, fresh, dev_status, nullptr), stream);
  if (st != SPIFFY_OK) return st;
  // The finalize kernel's launch overlaps the tail of the reduce kernel; it
  // waits on the device (cudaGridDependencySynchronize) for the partials.
  const Partial* cpart = partials;
  const cudaError_t e =
      launch_pdl(decide_finalize_kernel<4>, dim3(d.batch * d.n_nodes), dim3(kFinalizeThreads), (size_t)0,
                 stream, cpart, splits, (int)d.n_nodes, (int)d.block_len, block_tokens,
                 (int)d.mask_token_id, (int)d.rule, (int)d.top_s, d.threshold, conf, top_tok,
                 unmask_bits, n_unmask, dev_status);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

}  // namespace

spiffy_status launch_decide(const spiffy_decide_desc& d, const void* logits, const int32_t* block_tokens,
                            float* conf, int32_t* top_tok, uint64_t* unmask_bits, int32_t* n_unmask,
                            int32_t* dev_status, void* ws, bool fresh, cudaStream_t stream) {
  return decide_only(d, logits, block_tokens, conf, top_tok, unmask_bits, n_unmask, dev_status, ws, fresh, false,
                     false, stream);
}

// The finalize kernel alone, on partial results another kernel produced
// (`splits` per row, in the layout of this file's reduce kernel).
spiffy_status launch_decide_finalize(const spiffy_decide_desc& d, const void* partials, int splits,
                                     const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                     uint64_t* unmask_bits, int32_t* n_unmask, int32_t* dev_status,
                                     cudaStream_t stream) {
  const Partial* cpart = static_cast<const Partial*>(partials);
  const cudaError_t e =
      launch_pdl(splits > 32 ? decide_finalize_kernel<10> : decide_finalize_kernel<4>, dim3(d.batch * d.n_nodes), dim3(kFinalizeThreads), (size_t)0,
                 stream, cpart, splits, (int)d.n_nodes, (int)d.block_len, block_tokens,
                 (int)d.mask_token_id, (int)d.rule, (int)d.top_s, d.threshold, conf, top_tok,
                 unmask_bits, n_unmask, dev_status);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

// Decision and walk in one call.  Small graphs (at most kTailRows rows per sequence, arrays within the
// default shared-memory limit) take the fused tail: two launches instead of three.  Larger ones keep
// one finalize CTA per node, which spreads the merging over more SMs, and so do those with more partial
// results than one SM merges as fast, whatever part of them is of rows still masked.  Tail and kernels,
// us, with 5, 40 and 95 % of the rows masked:
//   512 rows x  4 slices  7.7  9.0    9.2 10.3   11.0 12.1
//   512 x  8, 4096 in all 8.7  9.2   11.3 12.1   16.4 16.5     256 x 16  8.2  8.2   11.8 11.8   15.9 15.9
//   512 x  9              9.2  9.2   13.3 12.8   18.1 17.7     256 x 19  9.5  9.0   13.2 12.5   18.5 17.8
//   512 x 19             14.4 13.1   21.5 18.8   31.4 29.0     4 x 512 x 19  30.6 28.0  51.7 49.2  99.3 96.4
// Beside a CUDA-core attention (`independent`; 512 rows of fp32, 40 % masked) the line lies there too:
// x 8 25.1 and 26.1, x 10 26.6 and 26.2, x 31 37.9 and 33.7; where the attention is by far the longer
// one (170 us) 1 us either way.  Where an attention follows beside the decision (`next`) the merging
// runs under it, on one SM instead of many that the attention waits for: the tail, whatever there is to
// merge (16 x 32 positions x 28 heads, x 19: 21.5 and 21.5, 27.0 and 27.7, 36.9 and 37.3).
constexpr int kTailRows = 512, kTailPartials = 4096;
// The tail's threads: a warp per node and four threads a row, 256 at least.  At 48 registers 1024 of them take most of
// an SM, where a CUDA-core attention beside the decision lets no such CTA in until it ends: the steps, us, with 1024
// and so: 9 sequences x 4 x 8 rows over 500 keys x 8 heads 65.3 48.9, 32 x 2 x 4 over 300 45.9 34.8; before a
// tensor-core attention 30 x 4 x 8 over 100 13.1 10.8; by itself 4 x 8 of 1024 entries 5.4 4.6, 16 x 8 x 8 7.9 7.1.  Fewer
// than a warp per node are slower (64 x 2 7.4, with 512 8.2).
// With more sequences than SMs several smaller ones to an SM, us with 256, 512 and 1024: 600 sequences x 64 rows of one
// slice 61.4 66.6 74.8, 2000 x 32 106.5 119.3 145.9, 300 x 128 64.4 66.8 71.3, 200 x 256 88.5 87.6 91.2, 150 x 432 117.2
// 111.4 113.6.
int tail_threads(int batch, int N, int rows) {
  const int most = batch <= sm_count() ? kTailThreads : rows <= kTailThreads / 8 ? kTailThreads / 4 : kTailThreads / 2;
  int threads = kTailThreads / 4;
  while (threads < most && (threads < 32 * N || threads < 4 * rows)) threads *= 2;
  return threads;
}
constexpr size_t kTailSmem = 48 * 1024 - 1024;  // what the kernel declares itself comes on top
// Beside a CUDA-core attention (`independent`) up to kSmallSlices slices a sequence take one launch of a cluster.
// fp32, the step with one launch and with two, us: 4 x 8 rows of one slice 6.7 and 8.4, 4 x 16 over 500 keys 20.0
// and 21.5, 2 x 32 over 4000 keys x 32 heads 125.2 and 127.3, 4 x 2 x 32 so 492 and 495, 2 x 8 x 8 over 4000 x 16
// 76.3 and 78.5, 3 x 8 of two 7.1 and 8.0; beyond, 3 x 8 rows of five slices 10.2 and 8.5, 8 x 32 of one 19.4 and 12.3.
// (12 sequences of 8 x 8 over 300 keys 55.5 and 57.4: the line for the batch could lie higher.)
// A decision in front of an attention or by itself is no sooner done in one launch (bf16, 4 x 8 rows of one
// slice 7.2 and 7.2 us with the attention, 4 x 16 9.3 and 7.3).
constexpr int kSmallSlices = 64, kSmallBatch = 8;
spiffy_status launch_decide_walk(const spiffy_decide_desc& d, const void* logits,
                                 const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                 uint64_t* unmask_bits, int32_t* n_unmask,
                                 int32_t* decide_status, const int32_t* parent_off,
                                 const int32_t* parent_idx, int32_t parent_cap,
                                 int32_t* accepted_node, int32_t* n_accepted, int32_t* path,
                                 int32_t* next_block, int32_t* walk_status, void* ws,
                                 bool fresh, bool independent, bool next, cudaStream_t stream) {
  const size_t smem = tail_smem_bytes(d, parent_cap);
  const int64_t rows_of_one = (int64_t)d.n_nodes * d.block_len;
  int64_t chunk = 0;
  const int splits = decide_splits(d, &chunk);
  if (rows_of_one > kTailRows || smem > kTailSmem || (!next && rows_of_one * splits > kTailPartials)) {
    const spiffy_status st = decide_only(d, logits, block_tokens, conf, top_tok, unmask_bits,
                                         n_unmask, decide_status, ws, fresh, independent, next, stream);
    if (st != SPIFFY_OK) return st;
    return launch_walk(d, block_tokens, parent_off, parent_idx, parent_cap, top_tok, unmask_bits,
                       accepted_node, n_accepted, path, next_block, walk_status, fresh, stream);
  }
  const size_t small_smem = smem + (size_t)rows_of_one * splits * sizeof(Partial);
  if (independent && rows_of_one <= kSmallRows && rows_of_one * splits <= kSmallSlices && small_smem <= kTailSmem &&
      d.batch <= kSmallBatch) {
    const TailArgs a = {splits, (int)d.n_nodes, (int)d.block_len, (int)d.mask_token_id, (int)d.rule, (int)d.top_s,
                        d.threshold, block_tokens, parent_off, parent_idx, (int)parent_cap, conf, top_tok, unmask_bits,
                        n_unmask, decide_status, accepted_node, n_accepted, path, next_block, walk_status};
    auto run = [&](auto kernel, auto* typed) {
      return launch_pdl(kernel, dim3(kSmallCtas * d.batch), dim3(kSmallGroups * kReduceThreads), small_smem, stream, a, typed,
                        (int64_t)d.row_stride, (int)d.vocab, chunk, (int)next, (int)fresh);
    };
    const cudaError_t e = d.logits_dtype == SPIFFY_BF16
                              ? run(decide_small_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16*>(logits))
                              : run(decide_small_kernel<float>, static_cast<const float*>(logits));
    count_launch();
    return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
  }
  Partial* partials = static_cast<Partial*>(ws);
  const spiffy_status st = launch_reduce(d, logits, block_tokens, partials, splits, chunk, 1, independent,
                                         status_clear(d, fresh, decide_status, walk_status), stream);
  if (st != SPIFFY_OK) return st;
  const Partial* cpart = partials;
  const int rows = d.n_nodes * d.block_len, threads = tail_threads(d.batch, d.n_nodes, rows);
  auto launch = [&](auto kernel) {
    return launch_pdl(kernel, dim3(d.batch), dim3(threads), smem, stream, cpart, splits,
                      (int)d.n_nodes, (int)d.block_len, block_tokens, (int)d.mask_token_id,
                      (int)d.rule, (int)d.top_s, d.threshold, conf, top_tok, unmask_bits, n_unmask,
                      decide_status, parent_off, parent_idx, (int)parent_cap, accepted_node,
                      n_accepted, path, next_block, walk_status, (int)next);
  };
  const cudaError_t e = rows <= threads / 8   ? launch(decide_tail_kernel<8>)
                        : rows <= threads / 4 ? launch(decide_tail_kernel<4>)
                                              : launch(decide_tail_kernel<2>);
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

}  // namespace spiffy
