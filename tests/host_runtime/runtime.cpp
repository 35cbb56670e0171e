// A stand-in for the CUDA runtime and for the attention kernels' launchers, so that
// the library's host code can run where there is no GPU: every call is written to a
// log, any of them can be made to fail, nothing is copied and no kernel runs.  With REAL_ATTENTION the
// launcher of the tensor-core kernels is the library's own, on a device of 148 multiprocessors.
#include <cuda.h>
#include <stdio.h>
#include <string.h>

#include <map>
#include <string>

#include "common.cuh"

namespace {

std::string g_log, g_fail;
std::map<const void*, std::string> g_kernels;
uintptr_t g_pinned_lo = 0, g_pinned_hi = 0;  // host memory that the device can read and write
intptr_t g_handles = 0x100;

cudaError_t note(const std::string& what) {
  const bool fails = !g_fail.empty() && what.compare(0, g_fail.size(), g_fail) == 0;
  g_log += what + (fails ? " FAILED\n" : "\n");
  return fails ? cudaErrorUnknown : cudaSuccess;
}
std::string on(cudaStream_t s) { return " on " + std::to_string((long)(intptr_t)s); }
std::string num(const void* p) { return std::to_string((long)(intptr_t)p); }

}  // namespace

extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_reset(const char* fail, uintptr_t pinned_lo, uintptr_t pinned_hi) {
  g_log.clear();
  g_fail = fail;
  g_pinned_lo = pinned_lo;
  g_pinned_hi = pinned_hi;
}

void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&g_handles); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_kernels[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }

cudaError_t cudaGetDevice(int* device) { *device = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr, int) { *value = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(g_handles += 1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)(g_handles += 1); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return note("record " + num(e) + on(s)); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return note("wait " + num(e) + on(s)); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return note("sync" + on(s)); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) { return note("memset" + on(s)); }
cudaError_t cudaMemcpyAsync(void*, const void* src, size_t bytes, cudaMemcpyKind, cudaStream_t s) {
  return note("memcpy" + on(s) + " from " + num(src) + " bytes " + std::to_string(bytes));
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* at, const void* p) {
  memset(at, 0, sizeof *at);
  const uintptr_t a = (uintptr_t)p;
  at->type = a >= g_pinned_lo && a < g_pinned_hi ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  at->devicePointer = at->hostPointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
// as a B200 answers for thread blocks that hold a multiprocessor each
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  const unsigned size = c->attrs[0].val.clusterDim.x;
  *n = size == 2 ? 74 : size == 4 ? 33 : 15;
  return cudaSuccess;
}
static CUresult encode_tiled(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** f, unsigned long long, cudaDriverEntryPointQueryResult*) {
  *f = reinterpret_cast<void*>(encode_tiled);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) { return note("launch " + g_kernels[f] + on(s)); }
// The arguments that decide what a kernel may read and when, by position.
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  const std::string& name = g_kernels[f];
  auto i = [&](int k) { return std::to_string(*static_cast<int*>(args[k])); };
  auto p = [&](int k) { return num(*static_cast<void**>(args[k])); };
  std::string more;
  if (name.find("decide_reduce_kernel") != std::string::npos) more = " early " + i(8);
  if (name.find("accept_walk_kernel") != std::string::npos) more = " lists " + p(3) + " staged " + i(13);
  if (name.find("decide_tail_kernel") != std::string::npos) more = " threads " + std::to_string(c->blockDim.x) + " lists " + p(14) + " early " + i(22);
  if (name.find("draft_build_kernel") != std::string::npos) more = " threads " + std::to_string(c->blockDim.x);
  if (name.find("graph_attention") != std::string::npos) {
    unsigned cluster = 1;
    for (unsigned k = 0; k < c->numAttrs; ++k)
      if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[k].val.clusterDim.x;
    more = " blocks " + std::to_string((long)c->gridDim.x * c->gridDim.y * c->gridDim.z) + " cluster " + std::to_string(cluster);
  }
  return note("launch " + name + on(c->stream) + more);
}
}  // extern "C"

namespace spiffy {
#ifdef REAL_ATTENTION
spiffy_status launch_attention_simt(const spiffy_attn_desc&, const void*, const void*, const void*, const void*,
                                    const void*, void*, cudaStream_t) { return SPIFFY_ECUDA; }
#else
bool attention_tc_supported(const spiffy_attn_desc& d) { return d.dtype == SPIFFY_BF16; }
spiffy_status launch_attention_tc(const spiffy_attn_desc& d, const AttnProblem&, int32_t*, cudaStream_t s) {
  return note("launch attention" + on(s) + " independent " + std::to_string((d.kernel & SPIFFY_ATTN_INDEPENDENT) != 0)) ==
                 cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}
spiffy_status launch_attention_simt(const spiffy_attn_desc& d, const void*, const void*, const void*, const void*,
                                    const void*, void*, cudaStream_t s) {
  return launch_attention_tc(d, AttnProblem{}, nullptr, s);
}
spiffy_status launch_attention_tc_dual(const spiffy_attn_desc&, const AttnProblem&, const spiffy_attn_desc&,
                                       const AttnProblem&, int32_t*, cudaStream_t) { return SPIFFY_ECUDA; }
#endif
// calls that no test here makes
size_t decide_lazy_workspace_bytes(const spiffy_decide_desc&) { return 0; }
spiffy_status launch_decide_walk_lazy(const spiffy_decide_desc&, const void*, const int32_t*, float*, int32_t*, uint64_t*,
                                      int32_t*, int32_t*, const int32_t*, const int32_t*, int32_t, int32_t*, int32_t*,
                                      int32_t*, int32_t*, int32_t*, void*, bool, cudaStream_t) { return SPIFFY_ECUDA; }
size_t decide_sampled_workspace_bytes(const spiffy_decide_desc&) { return 0; }
spiffy_status launch_decide_sampled(const spiffy_decide_desc&, float, uint64_t, const void*, const int32_t*, float*,
                                    int32_t*, uint64_t*, int32_t*, int32_t*, void*, bool, cudaStream_t) { return SPIFFY_ECUDA; }
int lmhead_grid(const spiffy_decide_desc&) { return 0; }
size_t lmhead_workspace_bytes(const spiffy_decide_desc&, int, int) { return 0; }
spiffy_status launch_lmhead_decide(const spiffy_decide_desc&, int, const void*, const void*, const int32_t*, float*,
                                   int32_t*, uint64_t*, int32_t*, int32_t*, void*, bool, cudaStream_t) { return SPIFFY_ECUDA; }
#ifdef REAL_ATTENTION
size_t draft_workspace_bytes(const spiffy_draft_desc&) { return 0; }
spiffy_status launch_draft(const spiffy_draft_desc&, const void*, const int32_t*, const int32_t*, const int32_t*,
                           const int32_t*, const int32_t*, const int32_t*, int32_t*, int32_t*, float*, int32_t*, int32_t*,
                           int32_t*, void*, bool, cudaStream_t) { return SPIFFY_ECUDA; }
#endif
}  // namespace spiffy
