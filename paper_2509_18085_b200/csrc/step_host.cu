// spiffy_verify_step_host: one whole verification step (Sec. 4.3 packed
// attention for one layer, then Algorithm 1 steps 1-5) for a caller whose
// tensors sit in HOST memory.  The call stages the inputs on the device, runs the
// three kernels of the step and brings the verdict back; see include/spiffy.h.
//
// The attention's inputs go through the copy engine on a helper stream of the
// library, and the attention follows them there.  Meanwhile, on the caller's
// stream, the decision reads the logits rows of still-masked positions, each once,
// straight out of the pinned host buffer, and the parent lists likewise: its work
// is hidden under the transfer.  Staging those rows first, by a kernel that copied
// them, and running both halves after the last byte took 3 to 8 us more
// (146 against 142 at 18 x 16 positions, 1155 against 1150 us at the LLaDA-8B shape,
// where the bus is the bound).
// Where the parent lists are not pinned, or too long for the walk to keep on chip,
// that is still the way; logits that are not pinned are copied whole.
#include <mutex>

#include "common.cuh"

namespace spiffy {
namespace {

constexpr size_t kAlign = 256;
constexpr size_t kDirectNodes = 8192;  // nodes up to which the walk keeps its links in shared memory
size_t up(size_t n) { return (n + kAlign - 1) / kAlign * kAlign; }

struct Layout {
  size_t q, kp, vp, kb, vb, logits, tokens, poff, pidx;       // inputs
  size_t qn, pn, bn;                                          // bytes of q, of a prefix tensor, of a block tensor
  size_t attn_out, conf, top_tok, bits, n_unmask;             // intermediate results
  size_t accepted, n_accepted, path, next_block;              // verdict
  size_t status;                                              // [attention | decision[B] | walk[B]]
  size_t attn_ws, decide_ws, total;
};

Layout layout_of(const spiffy_step_desc& s) {
  const spiffy_attn_desc& a = s.attn;
  const spiffy_decide_desc& d = s.decide;
  const size_t e = a.dtype == SPIFFY_BF16 ? 2 : 4, le = d.logits_dtype == SPIFFY_BF16 ? 2 : 4;
  const size_t B = a.batch, N = a.n_nodes, L = a.block_len;
  Layout l;
  l.qn = B * N * L * a.n_q_heads * a.head_dim * e;
  l.pn = B * (size_t)a.prefix_len * a.n_kv_heads * a.head_dim * e;
  l.bn = B * N * L * a.n_kv_heads * a.head_dim * e;
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o += up(bytes); return at; };
  l.q = take(l.qn); l.kp = take(l.pn); l.vp = take(l.pn); l.kb = take(l.bn); l.vb = take(l.bn);
  l.logits = take(B * N * L * (size_t)d.row_stride * le);
  l.tokens = take(B * N * L * 4);
  l.poff = take(B * (N + 1) * 4);
  l.pidx = take(B * (size_t)s.parent_cap * 4);
  l.attn_out = take(l.qn);
  l.conf = take(B * N * L * 4); l.top_tok = take(B * N * L * 4);
  l.bits = take(B * N * 8); l.n_unmask = take(B * N * 4);
  l.accepted = take(B * 4); l.n_accepted = take(B * 4); l.path = take(B * N * 4); l.next_block = take(B * L * 4);
  l.status = take((1 + 2 * B) * 4);
  l.attn_ws = take(spiffy_graph_attention_workspace(&a));
  l.decide_ws = take(spiffy_unmask_decide_workspace(&d));
  l.total = o;
  return l;
}

// The descriptor without the flags of the component calls: the step orders its own calls and
// clears all its status words.
spiffy_step_desc plain(const spiffy_step_desc& desc) {
  spiffy_step_desc s = desc;
  s.decide.logits_dtype &= ~(SPIFFY_FRESH_STATUS | SPIFFY_INDEPENDENT | SPIFFY_INDEPENDENT_NEXT);
  s.attn.kernel &= ~(SPIFFY_ATTN_EARLY_DEPENDENTS | SPIFFY_ATTN_INDEPENDENT);
  return s;
}

spiffy_status check(const spiffy_step_desc* s) {
  if (!s) return SPIFFY_EINVAL;
  if (s->attn.batch != s->decide.batch || s->attn.n_nodes != s->decide.n_nodes ||
      s->attn.block_len != s->decide.block_len || s->parent_cap < 1)
    return SPIFFY_EINVAL;
  if (s->attn.block_len > 64) return SPIFFY_EUNSUPPORTED;
  // all that the component calls would refuse: nothing is enqueued for a call that fails
  if (spiffy_unmask_decide_workspace(&s->decide) == 0) return SPIFFY_EINVAL;
  return check_attention(s->attn);
}

// One helper stream and two events per device, created at the first call there.
struct Helper {
  cudaStream_t stream = nullptr;
  cudaEvent_t start = nullptr, done = nullptr;
};
std::mutex g_mutex;
Helper g_helper[64];

spiffy_status helper_for_current_device(Helper** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPIFFY_ECUDA;
  std::lock_guard<std::mutex> lock(g_mutex);
  Helper& h = g_helper[dev];
  if (!h.stream) {
    if (cudaStreamCreateWithFlags(&h.stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h.start, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h.done, cudaEventDisableTiming) != cudaSuccess)
      return SPIFFY_ECUDA;
  }
  *out = &h;
  return SPIFFY_OK;
}

bool device_can_read(const void* host_ptr) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, host_ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeHost || at.type == cudaMemoryTypeManaged || at.type == cudaMemoryTypeDevice;
}
bool device_can_write(const void* host_ptr) {  // at the same address
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, host_ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeHost && at.devicePointer == host_ptr;
}

}  // namespace
}  // namespace spiffy

using namespace spiffy;

extern "C" {

size_t spiffy_verify_step_host_workspace(const spiffy_step_desc* desc) {
  if (check(desc) != SPIFFY_OK) return 0;
  return layout_of(plain(*desc)).total;
}

spiffy_status spiffy_verify_step_host(const spiffy_step_desc* desc, const void* q, const void* k_prefix,
                                      const void* v_prefix, const void* k_block, const void* v_block,
                                      const void* logits, const int32_t* block_tokens,
                                      const int32_t* parent_off, const int32_t* parent_idx,
                                      int32_t* accepted_node, int32_t* n_accepted, int32_t* path,
                                      int32_t* next_block, int32_t* status, void* device_workspace,
                                      size_t workspace_bytes, void* cuda_stream) {
  spiffy_status st = check(desc);
  if (st != SPIFFY_OK) return st;
  spiffy_step_desc s = plain(*desc);
  if (!q || !k_block || !v_block || !logits || !block_tokens || !parent_off || !parent_idx ||
      !accepted_node || !n_accepted || !path || !next_block || !status)
    return SPIFFY_EINVAL;
  if (s.attn.prefix_len > 0 && (!k_prefix || !v_prefix)) return SPIFFY_EINVAL;
  const Layout l = layout_of(s);
  if (!device_workspace || workspace_bytes < l.total ||
      (reinterpret_cast<uintptr_t>(device_workspace) & (kAlign - 1)) != 0)
    return SPIFFY_EWORKSPACE;
  Helper* h = nullptr;
  st = helper_for_current_device(&h);
  if (st != SPIFFY_OK) return st;

  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  char* ws = static_cast<char*>(device_workspace);
  const size_t B = s.attn.batch, N = s.attn.n_nodes, L = s.attn.block_len;
  const size_t le = s.decide.logits_dtype == SPIFFY_BF16 ? 2 : 4;
  const size_t rows = B * N * L;
  bool ok = true;
  // (by 16-byte loads: rows that do not start on such a boundary are copied by the runtime)
  const bool readable = device_can_read(logits) && rows <= 65535 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
  // the decision reads logits and parent lists where they are, the lists once
  const bool in_place = readable && walk_stages_graph(s.decide, s.parent_cap) && device_can_write(logits) &&
                        device_can_write(parent_off) && device_can_write(parent_idx);
  auto h2d = [&](size_t at, const void* src, size_t bytes, cudaStream_t on) {
    if (bytes) ok = ok && cudaMemcpyAsync(ws + at, src, bytes, cudaMemcpyHostToDevice, on) == cudaSuccess;
  };
  // the status words are OR-ed into by the kernels: [attention | decision per sequence | walk per sequence]
  ok = ok && cudaMemsetAsync(ws + l.status, 0, (1 + 2 * B) * 4, stream) == cudaSuccess;
  // the staging buffers are free once earlier work on the caller's stream is done
  ok = ok && cudaEventRecord(h->start, stream) == cudaSuccess;
  ok = ok && cudaStreamWaitEvent(h->stream, h->start, 0) == cudaSuccess;
  h2d(l.tokens, block_tokens, rows * 4, stream);
  h2d(l.q, q, l.qn, h->stream);
  h2d(l.kp, k_prefix, l.pn, h->stream);
  h2d(l.vp, v_prefix, l.pn, h->stream);
  h2d(l.kb, k_block, l.bn, h->stream);
  h2d(l.vb, v_block, l.bn, h->stream);
  int32_t* dev_status = reinterpret_cast<int32_t*>(ws + l.status);
  auto attention = [&](int flags, cudaStream_t on) {
    spiffy_attn_desc a = s.attn;
    a.kernel |= flags;
    return spiffy_graph_attention(&a, ws + l.q, s.attn.prefix_len ? ws + l.kp : nullptr,
                                  s.attn.prefix_len ? ws + l.vp : nullptr, ws + l.kb, ws + l.vb, ws + l.attn_out,
                                  dev_status, ws + l.attn_ws, l.decide_ws - l.attn_ws, on);
  };
  // From here on work is in flight on both streams, one of which the caller cannot see: whatever
  // fails, the caller's arrays and workspace are at rest when it is told.
  auto leave = [&](spiffy_status why) {
    cudaStreamSynchronize(h->stream);
    cudaStreamSynchronize(stream);
    return why;
  };
  if (in_place) {
    if (ok) st = attention(0, h->stream);
    if (st != SPIFFY_OK) return leave(st);
  } else {
    h2d(l.poff, parent_off, B * (N + 1) * 4, h->stream);
    h2d(l.pidx, parent_idx, B * (size_t)s.parent_cap * 4, h->stream);
  }
  ok = ok && cudaEventRecord(h->done, h->stream) == cudaSuccess;
  if (!ok) return leave(SPIFFY_ECUDA);
  if (!in_place) {
    // logits: only the rows of still-masked positions cross the bus
    const size_t row_bytes = (size_t)s.decide.row_stride * le;
    if (readable) {
      st = launch_stage_masked_rows(logits, ws + l.logits, (int64_t)row_bytes,
                                    reinterpret_cast<const int32_t*>(ws + l.tokens), s.decide.mask_token_id,
                                    (int64_t)rows, stream);
      if (st != SPIFFY_OK) return leave(st);
    } else {  // pageable memory: the runtime stages it; all rows go
      h2d(l.logits, logits, rows * row_bytes, stream);
    }
    ok = ok && cudaStreamWaitEvent(stream, h->done, 0) == cudaSuccess;
    if (!ok) return leave(SPIFFY_ECUDA);
  }
  // The verdict goes straight to the caller's arrays where the device can write them (a copy each
  // otherwise, about 2 us): the walk writes each word once and, with its links in shared memory,
  // reads none back.
  struct Out {
    int32_t* host;
    size_t at, bytes;
    bool direct;
    int32_t* device(char* ws) const { return direct ? host : reinterpret_cast<int32_t*>(ws + at); }
  } outs[4] = {{accepted_node, l.accepted, B * 4, false},
               {n_accepted, l.n_accepted, B * 4, false},
               {path, l.path, B * N * 4, false},
               {next_block, l.next_block, B * L * 4, false}};
  for (Out& o : outs) o.direct = N <= kDirectNodes && device_can_write(o.host);
  // Behind the staging the two run side by side on the tensor-core kernel, the attention second;
  // else one after the other.
  const bool second = !in_place && attention_uses_tc(s.attn);
  if (!second && !in_place) st = attention(0, stream);
  if (st != SPIFFY_OK) return leave(st);
  if (second) s.decide.logits_dtype |= SPIFFY_INDEPENDENT_NEXT;
  st = spiffy_decide_walk(&s.decide, in_place ? logits : ws + l.logits,
                          reinterpret_cast<const int32_t*>(ws + l.tokens),
                          in_place ? parent_off : reinterpret_cast<const int32_t*>(ws + l.poff),
                          in_place ? parent_idx : reinterpret_cast<const int32_t*>(ws + l.pidx), s.parent_cap,
                          reinterpret_cast<float*>(ws + l.conf), reinterpret_cast<int32_t*>(ws + l.top_tok),
                          reinterpret_cast<uint64_t*>(ws + l.bits), reinterpret_cast<int32_t*>(ws + l.n_unmask),
                          dev_status + 1, outs[0].device(ws), outs[1].device(ws), outs[2].device(ws),
                          outs[3].device(ws), dev_status + 1 + B, ws + l.decide_ws, l.total - l.decide_ws, stream);
  if (st == SPIFFY_OK && second) st = attention(SPIFFY_ATTN_INDEPENDENT, stream);
  if (st != SPIFFY_OK) return leave(st);
  if (in_place) ok = ok && cudaStreamWaitEvent(stream, h->done, 0) == cudaSuccess;
  auto d2h = [&](void* dst, size_t at, size_t bytes) {
    ok = ok && cudaMemcpyAsync(dst, ws + at, bytes, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
  };
  for (const Out& o : outs)
    if (!o.direct) d2h(o.host, o.at, o.bytes);
  d2h(status, l.status, (1 + 2 * B) * 4);
  ok = ok && cudaStreamSynchronize(stream) == cudaSuccess;
  return ok ? SPIFFY_OK : leave(SPIFFY_ECUDA);
}

}  // extern "C"
