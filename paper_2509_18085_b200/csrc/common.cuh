// Internal helpers shared by the kernels of libspiffy (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "fast_div.cuh"
#include "spiffy.h"

namespace spiffy {

constexpr float kLog2e = 1.4426950408889634f;

// 2^x on the special-function unit (approximate, denormals flushed).
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Two fp32 lanes in one 64-bit register: Blackwell issues their multiply-add and
// their add as one instruction each (for loops bound by instruction issue).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// 128-bit streaming load: read-only path, no L1 allocation (data used once).
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Stores to global memory that order nothing else: a store through a pointer whose
// address space the compiler cannot tell would hold up the shared-memory loads of
// the next turn of a loop.
__device__ __forceinline__ void st_global(void* p, uint2 v) {
  asm volatile("st.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(v.x), "r"(v.y));
}
__device__ __forceinline__ void st_global(void* p, uint4 v) {
  asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
}

// Multiprocessors of the current device, 0 when it cannot be asked.  Safe with several threads.
int sm_count();

// Every launch of the library goes through this counter (spiffy_launch_count).
void count_launch(int n = 1);

// Poll limits of the bounded device-side waits, read at launch.  The defaults
// (about a fraction of a second) change only through spiffy_set_wait_limits,
// which exists so that the give-up paths can be exercised.
uint32_t mbar_poll_limit();   // polls of one mbarrier wait (tensor-core kernels)
uint32_t flag_poll_limit();   // polls of one wait on a global-memory word (lazy call)
int32_t lazy_extra_arrivals();  // not 0: sequence 0's tail waits for results that cannot come

// Entry points implemented in the kernel files; all validated by the caller.
// `fresh`: the call's first kernel clears the status words (SPIFFY_FRESH_STATUS);
// the descriptors arrive without that flag.
spiffy_status launch_decide(const spiffy_decide_desc& d, const void* logits,
                            const int32_t* block_tokens, float* conf,
                            int32_t* top_tok, uint64_t* unmask_bits,
                            int32_t* n_unmask, int32_t* dev_status, void* ws,
                            bool fresh,
                            cudaStream_t stream);
size_t decide_workspace_bytes(const spiffy_decide_desc& d);
int decide_splits(const spiffy_decide_desc& d, int64_t* chunk_elems);

// Does the walk copy a sequence's graph to shared memory, reading every list once?  (The fused
// tail does for all such sizes: at 512 rows its arrays take 2 KB more than the walk's, of 48 KB.)
bool walk_stages_graph(const spiffy_decide_desc& d, int32_t parent_cap);
spiffy_status launch_walk(const spiffy_decide_desc& d,
                          const int32_t* block_tokens,
                          const int32_t* parent_off, const int32_t* parent_idx,
                          int32_t parent_cap, const int32_t* top_tok,
                          const uint64_t* unmask_bits, int32_t* accepted_node,
                          int32_t* n_accepted, int32_t* path,
                          int32_t* next_block, int32_t* dev_status,
                          bool fresh,
                            cudaStream_t stream);

spiffy_status launch_decide_walk(const spiffy_decide_desc& d, const void* logits,
                                 const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                 uint64_t* unmask_bits, int32_t* n_unmask,
                                 int32_t* decide_status, const int32_t* parent_off,
                                 const int32_t* parent_idx, int32_t parent_cap,
                                 int32_t* accepted_node, int32_t* n_accepted, int32_t* path,
                                 int32_t* next_block, int32_t* walk_status, void* ws,
                                 bool fresh, bool independent, bool next, cudaStream_t stream);

size_t decide_lazy_workspace_bytes(const spiffy_decide_desc& d);
spiffy_status launch_decide_walk_lazy(const spiffy_decide_desc& d, const void* logits,
                                      const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                      uint64_t* unmask_bits, int32_t* n_unmask,
                                      int32_t* decide_status, const int32_t* parent_off,
                                      const int32_t* parent_idx, int32_t parent_cap,
                                      int32_t* accepted_node, int32_t* n_accepted, int32_t* path,
                                      int32_t* next_block, int32_t* walk_status, void* ws,
                                      bool fresh,
                            cudaStream_t stream);

spiffy_status launch_stage_masked_rows(const void* src, void* dst, int64_t row_bytes,
                                       const int32_t* tokens, int32_t mask_id, int64_t n_rows,
                                       cudaStream_t stream);

size_t decide_sampled_workspace_bytes(const spiffy_decide_desc& d);
spiffy_status launch_decide_sampled(const spiffy_decide_desc& d, float temperature, uint64_t seed,
                                    const void* logits, const int32_t* block_tokens, float* conf,
                                    int32_t* top_tok, uint64_t* unmask_bits, int32_t* n_unmask,
                                    int32_t* dev_status, void* ws, bool fresh,
                            cudaStream_t stream);

spiffy_status launch_decide_finalize(const spiffy_decide_desc& d, const void* partials, int splits,
                                     const int32_t* block_tokens, float* conf, int32_t* top_tok,
                                     uint64_t* unmask_bits, int32_t* n_unmask, int32_t* dev_status,
                                     cudaStream_t stream);
int lmhead_grid(const spiffy_decide_desc& d);
size_t lmhead_workspace_bytes(const spiffy_decide_desc& d, int hidden, int grid);
spiffy_status launch_lmhead_decide(const spiffy_decide_desc& d, int hidden, const void* hstates,
                                   const void* weight, const int32_t* block_tokens, float* conf,
                                   int32_t* top_tok, uint64_t* unmask_bits, int32_t* n_unmask,
                                   int32_t* dev_status, void* ws, bool fresh,
                            cudaStream_t stream);

spiffy_status launch_attention_simt(const spiffy_attn_desc& d, const void* q,
                                    const void* kp, const void* vp,
                                    const void* kb, const void* vb, void* out,
                                    cudaStream_t stream);

size_t draft_workspace_bytes(const spiffy_draft_desc& d);
spiffy_status launch_draft(const spiffy_draft_desc& d, const void* logits, const int32_t* state,
                           const int32_t* formula_off, const int32_t* formula_i,
                           const int32_t* formula_j, const int32_t* child_off,
                           const int32_t* child_idx, int32_t* tokens, int32_t* kept, float* score,
                           int32_t* parent_off, int32_t* parent_idx, int32_t* dev_status, void* ws,
                           bool fresh,
                            cudaStream_t stream);

// tcgen05 path: shape support query and launch.  The cached context
// comes as up to two segments of keys/values, [B][len][Hkv][d] each, whose
// sequences may lie `batch_stride_rows` rows apart (0: densely packed).
struct AttnContext {
  const void* k;
  const void* v;
  int len;
  int64_t batch_stride_rows;
};
// One attention problem's tensors: queries, two context segments, block keys/values, output.
struct AttnProblem {
  const void* q;
  AttnContext ctx, ctx2;
  const void* kb;
  const void* vb;
  void* out;
};
bool attention_tc_supported(const spiffy_attn_desc& d);
// What spiffy_graph_attention makes of a descriptor: the status it would refuse it with, and,
// for one it takes, whether that goes to the tensor-core kernel.
spiffy_status check_attention(const spiffy_attn_desc& d);
bool attention_uses_tc(const spiffy_attn_desc& d);
spiffy_status launch_attention_tc(const spiffy_attn_desc& d, const AttnProblem& a, int32_t* dev_status,
                                  cudaStream_t stream);
// Two problems of the same batch, heads and head dimension (128) in one launch.
spiffy_status launch_attention_tc_dual(const spiffy_attn_desc& d0, const AttnProblem& a0, const spiffy_attn_desc& d1,
                                       const AttnProblem& a1, int32_t* dev_status, cudaStream_t stream);

// Launch with programmatic stream serialisation: the kernel may be scheduled once every CTA
// of its predecessor in the stream has called pdl_launch_dependents() or ended.  "Waits" below
// means cudaGridDependencySynchronize(), which returns when the predecessor is complete and
// its writes are visible.  Who may start when, and why what it touches is complete:
//   - Every kernel waits, and none is complete before it has waited, so that a kernel which
//     is complete, or has been waited for, stands for all that came before it in the stream.
//   - Before its wait a kernel writes nothing in global memory and reads nothing, except:
//     (a) The walk, tail, sampled selection and rule kernels read the block's tokens, the first two
//         the parent lists as well.  Each comes behind a kernel of its own call that waited
//         before it let its dependents start (the reduces do, and the finalize kernel is
//         itself launched behind one), so whatever wrote those arrays ahead of the call is
//         complete.  spiffy_accept_walk called by itself has no such kernel in front: its
//         contract in spiffy.h puts that on the caller.
//         The lazy call's walk kernel reads all inputs of its call, logits included: it comes behind
//         the root kernel, which waited.
//     (b) The draft-build kernel reads the draft formulas, constants of the model, and the block, as the
//         top-k kernel in front of it waited before it let it start.
//     (c) The reduce under SPIFFY_INDEPENDENT and the attention under SPIFFY_ATTN_INDEPENDENT
//         read their inputs, write their outputs and wait last; the one kernel that few slices
//         take under SPIFFY_INDEPENDENT reads its inputs, waits and writes.  What precedes them is, by the
//         flags' contract, a call that touches none of these; its kernels started, in turn,
//         behind one that had waited before it triggered (the CUDA-core attention; the reduce
//         of a plain decision), so everything ahead of that call is complete.  The second launch
//         of an attention in two does the same behind the first, which touches other rows of the
//         output and has waited before it triggered, or is itself under the flag.
//   - Triggering early is safe for what follows for the same reasons; where it pays is a
//     matter of measurement and said at each kernel.
template <typename... Args>
cudaError_t launch_pdl(void (*kern)(Args...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// The next kernel in the stream may be launched once every CTA has come here; it still
// waits for this one to finish, and its launch latency is off the critical path.
__device__ __forceinline__ void pdl_launch_dependents() {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 900
  cudaTriggerProgrammaticLaunchCompletion();
#endif
}

// Lets `kern` use `bytes` of dynamic shared memory on the current device.  Asked
// for once per kernel and device (the attribute sticks to the kernel); `done` is
// the kernel's own table, all false at first.
template <typename Kernel>
bool allow_smem(Kernel kern, int bytes, std::atomic<bool> (&done)[64]) {
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return false;
  if (done[device].load(std::memory_order_acquire)) return true;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
  done[device].store(true, std::memory_order_release);
  return true;
}

}  // namespace spiffy
