// Python binding of the C ABI: torch tensors in, descriptors and device pointers
// out, one C call, results back.  Marshalling only -- every step of the path runs
// in the library's kernels.
//
// It is native because the calls are short: at the small shapes one step of the
// path takes 10-20 us on the device, while marshalling the same calls through
// ctypes took 13-17 us of interpreter time per call (32 us per step, 77 us when
// the outputs were allocated as well), so the host was what bounded them.  Here a
// call's outputs come out of one allocation (the small arrays of a decision and a
// walk are views of it), and outputs made here are not cleared by kernels of
// their own: SPIFFY_FRESH_STATUS has the call's first kernel do it.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>
#include <optional>
#include <utility>
#include <vector>

#include "spiffy.h"

namespace {

PyObject* g_error_class = nullptr;     // SpiffyError(status, where)
PyObject* g_decision_class = nullptr;  // Decision(conf, top_tok, unmask_bits, n_unmask, dev_status)
PyObject* g_walk_class = nullptr;      // Walk(accepted_node, n_accepted, path, next_block, dev_status)
PyObject* g_drafts_class = nullptr;    // Drafts(tokens, kept, score, parent_off, parent_idx, dev_status)

// An exception has been set with PyErr_*: unwinds to the entry point.
struct PyError {};

[[noreturn]] void fail(PyObject* type, const char* fmt, const char* name, const char* more = "") {
  PyErr_Format(type, fmt, name, more);
  throw PyError{};
}

const char* dtype_name(at::ScalarType t) {
  switch (t) {
    case at::kFloat: return "torch.float32";
    case at::kBFloat16: return "torch.bfloat16";
    case at::kInt: return "torch.int32";
    case at::kLong: return "torch.int64";
    default: return c10::toString(t);
  }
}

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a torch.Tensor%s", name);
  return THPVariable_Unpack(o);
}

constexpr at::ScalarType kAnyType = at::ScalarType::Undefined;

void* device_ptr(const at::Tensor& t, const char* name, at::ScalarType dtype) {
  if (!t.is_cuda()) fail(PyExc_ValueError, "%s must live on a CUDA device (no CPU path exists)%s", name);
  if (!t.is_contiguous()) fail(PyExc_ValueError, "%s must be contiguous%s", name);
  if (dtype != kAnyType && t.scalar_type() != dtype)
  {
    PyErr_Format(PyExc_TypeError, "%s must be %s, got %s", name, dtype_name(dtype), dtype_name(t.scalar_type()));
    throw PyError{};
  }
  return t.data_ptr();
}

// None is a null pointer.
void* device_ptr(PyObject* o, const char* name, at::ScalarType dtype) {
  return o == Py_None ? nullptr : device_ptr(tensor(o, name), name, dtype);
}

int dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return SPIFFY_F32;
  if (t.scalar_type() == at::kBFloat16) return SPIFFY_BF16;
  fail(PyExc_TypeError, "unsupported dtype %s%s", dtype_name(t.scalar_type()));
}

long long as_int(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyError{};
  return v;
}

double as_float(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyError{};
  return v;
}

// The stream of a call.  None: the current stream of the current device; else an object with a
// cuda_stream attribute, which is then the current stream for as long as the call's results and
// scratch are allocated and cleared: the allocator hands memory out, and takes it back, in the order
// of the stream that was current.
class CallStream {
 public:
  CallStream(PyObject* o, const at::Tensor& like) {
    if (o == Py_None) {
      ptr_ = c10::cuda::getCurrentCUDAStream().stream();
      return;
    }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw PyError{};
    ptr_ = static_cast<cudaStream_t>(PyLong_AsVoidPtr(h));
    Py_DECREF(h);
    if (!ptr_ && PyErr_Occurred()) throw PyError{};
    if (!like.is_cuda()) return;  // refused further down
    // cudaStreamLegacy is the default stream by another name
    const cudaStream_t named = ptr_ == cudaStreamLegacy ? nullptr : ptr_;
    guard_.emplace(c10::cuda::getStreamFromExternal(named, like.device().index()));
  }
  void* get() const { return ptr_; }

 private:
  cudaStream_t ptr_ = nullptr;
  std::optional<c10::cuda::CUDAStreamGuard> guard_;
};

// One call into the library, without the interpreter lock: a launch waits when the stream's queue is
// full, and other Python threads have their own work.  All it needs has been read by now.
template <typename F, typename... Args>
int unlocked(F f, Args... args) {
  PyThreadState* const held = PyEval_SaveThread();
  const int status = f(args...);
  PyEval_RestoreThread(held);
  return status;
}

void check(int status, const char* where) {
  if (status == SPIFFY_OK) return;
  PyObject* e = PyObject_CallFunction(g_error_class, "is", status, where);
  if (e) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  }
  throw PyError{};
}

// A call's scratch: the caller's, or allocated for the call (in the order of the
// call's stream, so that it may go back to the allocator when the call returns).
struct Scratch {
  at::Tensor own;
  void* ptr = nullptr;
  size_t bytes = 0;
  Scratch(PyObject* given, size_t need, const at::Tensor& like, bool always) {
    if (given != Py_None) {
      const at::Tensor& t = tensor(given, "workspace");
      ptr = device_ptr(t, "workspace", kAnyType);
      bytes = (size_t)t.numel() * t.element_size();
    } else if (need > 0 || always) {
      own = at::empty({(int64_t)(need > 16 ? need : 16)}, like.options().dtype(at::kByte));
      ptr = device_ptr(own, "workspace", kAnyType);
      bytes = (size_t)own.numel();
    }
  }
};

// Small output arrays as views of one allocation, each on a 64-byte boundary.
class Carver {
 public:
  Carver(size_t bytes, const at::Tensor& like)
      : blob_(at::empty({(int64_t)bytes}, like.options().dtype(at::kByte))) {}
  static size_t room(int64_t n, size_t elem) { return ((size_t)n * elem + 63) / 64 * 64; }
  PyObject* take(at::IntArrayRef sizes, at::ScalarType type) {
    const size_t elem = c10::elementSize(type);
    at::Tensor t = at::detail::make_tensor<c10::TensorImpl>(
        c10::Storage(blob_.storage()), c10::DispatchKeySet(c10::DispatchKey::CUDA), c10::scalarTypeToTypeMeta(type));
    c10::TensorImpl* impl = t.unsafeGetTensorImpl();
    impl->set_storage_offset((int64_t)(at_ / elem));
    impl->set_sizes_contiguous(sizes);
    at_ += room(t.numel(), elem);
    PyObject* o = THPVariable_Wrap(std::move(t));
    if (!o) throw PyError{};
    return o;
  }

 private:
  at::Tensor blob_;
  size_t at_ = 0;
};

// A new reference, released on unwinding.
struct Ref {
  PyObject* o;
  explicit Ref(PyObject* p = nullptr) : o(p) {}
  Ref(const Ref&) = delete;
  ~Ref() { Py_XDECREF(o); }
  PyObject* release() {
    PyObject* p = o;
    o = nullptr;
    return p;
  }
};

PyObject* make(PyObject* cls, PyObject* const* fields, Py_ssize_t n) {
  PyObject* o = PyObject_Vectorcall(cls, fields, (size_t)n, nullptr);
  for (Py_ssize_t i = 0; i < n; ++i) Py_DECREF(fields[i]);
  if (!o) throw PyError{};
  return o;
}

size_t decision_room(int64_t B, int64_t N, int64_t L) {
  return 2 * Carver::room(B * N * L, 4) + Carver::room(B * N, 8) + Carver::room(B * N, 4) + Carver::room(B, 4);
}
PyObject* new_decision(Carver& c, int64_t B, int64_t N, int64_t L) {
  PyObject* f[5] = {c.take({B, N, L}, at::kFloat), c.take({B, N, L}, at::kInt), c.take({B, N}, at::kLong),
                    c.take({B, N}, at::kInt), c.take({B}, at::kInt)};
  return make(g_decision_class, f, 5);
}
size_t walk_room(int64_t B, int64_t N, int64_t L) {
  return 3 * Carver::room(B, 4) + Carver::room(B * N, 4) + Carver::room(B * L, 4);
}
PyObject* new_walk(Carver& c, int64_t B, int64_t N, int64_t L) {
  PyObject* f[5] = {c.take({B}, at::kInt), c.take({B}, at::kInt), c.take({B, N}, at::kInt), c.take({B, L}, at::kInt),
                    c.take({B}, at::kInt)};
  return make(g_walk_class, f, 5);
}

void* field_ptr(PyObject* o, PyObject* attr, const char* name, at::ScalarType dtype) {
  Ref f(PyObject_GetAttr(o, attr));
  if (!f.o) throw PyError{};
  return device_ptr(f.o, name, dtype);  // the object keeps the tensor
}

// Interned attribute names.
struct Names {
  PyObject *conf, *top_tok, *unmask_bits, *n_unmask, *dev_status, *accepted_node, *n_accepted, *path, *next_block;
  PyObject *tokens, *kept, *score, *parent_off, *parent_idx, *formula_off, *formula_i, *formula_j, *child_off,
      *child_idx;
} g_names;

struct DecisionPtrs {
  float* conf;
  int32_t* top_tok;
  uint64_t* bits;
  int32_t* n_unmask;
  int32_t* status;
  DecisionPtrs(PyObject* d, const char* status_name)
      : conf((float*)field_ptr(d, g_names.conf, "conf", at::kFloat)),
        top_tok((int32_t*)field_ptr(d, g_names.top_tok, "top_tok", at::kInt)),
        bits((uint64_t*)field_ptr(d, g_names.unmask_bits, "unmask_bits", at::kLong)),
        n_unmask((int32_t*)field_ptr(d, g_names.n_unmask, "n_unmask", at::kInt)),
        status((int32_t*)field_ptr(d, g_names.dev_status, status_name, at::kInt)) {}
};
struct WalkPtrs {
  int32_t *accepted_node, *n_accepted, *path, *next_block, *status;
  WalkPtrs(PyObject* w, const char* status_name)
      : accepted_node((int32_t*)field_ptr(w, g_names.accepted_node, "accepted_node", at::kInt)),
        n_accepted((int32_t*)field_ptr(w, g_names.n_accepted, "n_accepted", at::kInt)),
        path((int32_t*)field_ptr(w, g_names.path, "path", at::kInt)),
        next_block((int32_t*)field_ptr(w, g_names.next_block, "next_block", at::kInt)),
        status((int32_t*)field_ptr(w, g_names.dev_status, status_name, at::kInt)) {}
};

// ------------------------------------------------------------ attention ----
spiffy_attn_desc attn_desc(const at::Tensor& q, PyObject* k_prefix, const at::Tensor& k_block, double scale,
                           long long kernel) {
  if (q.dim() != 5 || k_block.dim() != 5) fail(PyExc_ValueError, "%s must be [B,N,L,H,d]%s", "q and k_block");
  spiffy_attn_desc d;
  d.batch = (int32_t)q.size(0);
  d.n_nodes = (int32_t)q.size(1);
  d.block_len = (int32_t)q.size(2);
  d.prefix_len = 0;
  if (k_prefix != Py_None) {
    const at::Tensor& kp = tensor(k_prefix, "k_prefix");
    if (kp.dim() != 4) fail(PyExc_ValueError, "%s must be [B,P,Hkv,d]%s", "k_prefix");
    d.prefix_len = (int32_t)kp.size(1);
  }
  d.n_q_heads = (int32_t)q.size(3);
  d.n_kv_heads = (int32_t)k_block.size(3);
  d.head_dim = (int32_t)q.size(4);
  d.dtype = dtype_code(q);
  d.scale = (float)scale;
  d.kernel = (int32_t)kernel;
  return d;
}

// The caller's output, or one like `like`; a new reference in `o`.
const at::Tensor& output_like(PyObject* given, const at::Tensor& like, const char* name, Ref* o) {
  if (given != Py_None) {
    Py_INCREF(given);
    o->o = given;
  } else {
    o->o = THPVariable_Wrap(at::empty(like.sizes(), like.options()));
    if (!o->o) throw PyError{};
  }
  return tensor(o->o, name);
}

// q, k_prefix, v_prefix, k_block, v_block, out, scale, kernel, dev_status, workspace, stream
PyObject* graph_attention(PyObject* const* a) {
  const at::Tensor& q = tensor(a[0], "q");
  const spiffy_attn_desc d = attn_desc(q, a[1], tensor(a[3], "k_block"), as_float(a[6]), as_int(a[7]));
  const at::ScalarType t = q.scalar_type();
  const void* qp = device_ptr(q, "q", kAnyType);
  const void* kp = device_ptr(a[1], "k_prefix", t);
  const void* vp = device_ptr(a[2], "v_prefix", t);
  const void* kb = device_ptr(a[3], "k_block", t);
  const void* vb = device_ptr(a[4], "v_block", t);
  const CallStream stream(a[10], q);
  Ref out;
  void* op = device_ptr(output_like(a[5], q, "out", &out), "out", t);
  int32_t* status = (int32_t*)device_ptr(a[8], "dev_status", at::kInt);
  const Scratch ws(a[9], a[9] == Py_None ? spiffy_graph_attention_workspace(&d) : 0, q, false);
  check(unlocked(spiffy_graph_attention, &d, qp, kp, vp, kb, vb, op, status, ws.ptr, ws.bytes, stream.get()),
        "spiffy_graph_attention");
  return out.release();
}

// q_nodes, q_suffix, k_prefix, v_prefix, k_suffix, v_suffix, k_block, v_block, scale, kernel, out_nodes,
// out_suffix, dev_status, workspace, stream
PyObject* full_sequence_attention(PyObject* const* a) {
  const at::Tensor& q = tensor(a[0], "q_nodes");
  const at::Tensor& qs = tensor(a[1], "q_suffix");
  const spiffy_attn_desc d = attn_desc(q, a[2], tensor(a[6], "k_block"), as_float(a[8]), as_int(a[9]));
  if (qs.dim() != 4) fail(PyExc_ValueError, "%s must be [B,S,Hq,d]%s", "q_suffix");
  const int32_t S = (int32_t)qs.size(1);
  const at::ScalarType t = q.scalar_type();
  const void* qp = device_ptr(q, "q_nodes", kAnyType);
  const void* qsp = device_ptr(qs, "q_suffix", t);
  static const char* const names[] = {"k_prefix", "v_prefix", "k_suffix", "v_suffix", "k_block", "v_block"};
  const void* kv[6];
  for (int i = 0; i < 6; ++i) kv[i] = device_ptr(a[2 + i], names[i], t);
  const CallStream stream(a[14], q);
  Ref on, os;
  void* onp = device_ptr(output_like(a[10], q, "out_nodes", &on), "out_nodes", t);
  void* osp = device_ptr(output_like(a[11], qs, "out_suffix", &os), "out_suffix", t);
  int32_t* status = (int32_t*)device_ptr(a[12], "dev_status", at::kInt);
  const Scratch ws(a[13], a[13] == Py_None ? spiffy_full_sequence_attention_workspace(&d, S) : 0, q, false);
  check(unlocked(spiffy_full_sequence_attention, &d, S, qp, qsp, kv[0], kv[1], kv[2], kv[3], kv[4], kv[5], onp, osp,
                 status, ws.ptr, ws.bytes, stream.get()),
        "spiffy_full_sequence_attention");
  PyObject* r = PyTuple_Pack(2, on.o, os.o);
  if (!r) throw PyError{};
  return r;
}

// ------------------------------------------------------------- decision ----
// logits [B,N,L,V] (rows may be a strided view of a wider buffer)
const void* logits_ptr(const at::Tensor& t) {
  if (!t.is_cuda()) fail(PyExc_ValueError, "%s must live on a CUDA device (no CPU path exists)%s", "logits");
  if (t.stride(-1) != 1) fail(PyExc_ValueError, "%s rows must be dense%s", "logits");
  if (t.dim() == 4) {
    const int64_t N = t.size(1), L = t.size(2), rs = t.stride(2);
    if ((N > 1 && t.stride(1) != L * rs) || (t.size(0) > 1 && t.stride(0) != N * L * rs))
      fail(PyExc_ValueError, "%s rows must be equally spaced%s", "logits");
  }
  return t.data_ptr();
}

// block_tokens, mask id, rule, top_s, threshold = a[0 .. 4]
spiffy_decide_desc decide_desc(const at::Tensor& logits, const at::Tensor& tokens, PyObject* const* a) {
  if (tokens.dim() != 3) fail(PyExc_ValueError, "%s must be [B,N,L]%s", "block_tokens");
  if (logits.dim() < 1) fail(PyExc_ValueError, "%s must be [B,N,L,V]%s", "logits");
  spiffy_decide_desc d;
  d.batch = (int32_t)tokens.size(0);
  d.n_nodes = (int32_t)tokens.size(1);
  d.block_len = (int32_t)tokens.size(2);
  d.vocab = (int32_t)logits.size(-1);
  d.logits_dtype = dtype_code(logits);
  d.row_stride = logits.dim() >= 2 ? logits.stride(-2) : logits.size(-1);
  d.mask_token_id = (int32_t)as_int(a[0]);
  d.rule = (int32_t)as_int(a[1]);
  d.top_s = (int32_t)as_int(a[2]);
  d.threshold = (float)as_float(a[3]);
  return d;
}

// The caller's decision, or a new one whose status words the call clears itself.
PyObject* decision_for(PyObject* given, spiffy_decide_desc* d, const at::Tensor& like) {
  if (given != Py_None) {
    Py_INCREF(given);
    return given;
  }
  d->logits_dtype |= SPIFFY_FRESH_STATUS;
  Carver c(decision_room(d->batch, d->n_nodes, d->block_len), like);
  return new_decision(c, d->batch, d->n_nodes, d->block_len);
}

// logits, block_tokens, mask_token_id, rule, top_s, threshold, out, workspace, stream
PyObject* unmask_decide(PyObject* const* a) {
  const at::Tensor& logits = tensor(a[0], "logits");
  const at::Tensor& tokens = tensor(a[1], "block_tokens");
  spiffy_decide_desc d = decide_desc(logits, tokens, a + 2);
  const void* lp = logits_ptr(logits);
  const int32_t* tp = (const int32_t*)device_ptr(tokens, "block_tokens", at::kInt);
  const CallStream stream(a[8], logits);
  Ref out(decision_for(a[6], &d, logits));
  const DecisionPtrs p(out.o, "dev_status");
  const Scratch ws(a[7], a[7] == Py_None ? spiffy_unmask_decide_workspace(&d) : 0, logits, true);
  check(unlocked(spiffy_unmask_decide, &d, lp, tp, p.conf, p.top_tok, p.bits, p.n_unmask, p.status, ws.ptr, ws.bytes,
                 stream.get()),
        "spiffy_unmask_decide");
  return out.release();
}

// logits, block_tokens, mask_token_id, rule, top_s, threshold, temperature, seed, out, workspace, stream
PyObject* unmask_decide_sampled(PyObject* const* a) {
  const at::Tensor& logits = tensor(a[0], "logits");
  const at::Tensor& tokens = tensor(a[1], "block_tokens");
  spiffy_decide_desc d = decide_desc(logits, tokens, a + 2);
  spiffy_sample_desc s;
  s.temperature = (float)as_float(a[6]);
  s.reserved = 0;
  s.seed = PyLong_AsUnsignedLongLongMask(a[7]);
  if (PyErr_Occurred()) throw PyError{};
  const void* lp = logits_ptr(logits);
  const int32_t* tp = (const int32_t*)device_ptr(tokens, "block_tokens", at::kInt);
  const CallStream stream(a[10], logits);
  Ref out(decision_for(a[8], &d, logits));
  const DecisionPtrs p(out.o, "dev_status");
  const Scratch ws(a[9], a[9] == Py_None ? spiffy_unmask_decide_sampled_workspace(&d) : 0, logits, true);
  check(unlocked(spiffy_unmask_decide_sampled, &d, &s, lp, tp, p.conf, p.top_tok, p.bits, p.n_unmask, p.status, ws.ptr,
                 ws.bytes, stream.get()),
        "spiffy_unmask_decide_sampled");
  return out.release();
}

// hidden_states, weight, block_tokens, mask_token_id, rule, top_s, threshold, out, workspace, stream
PyObject* lmhead_decide(PyObject* const* a) {
  const at::Tensor& h = tensor(a[0], "hidden_states");
  const at::Tensor& w = tensor(a[1], "weight");
  const at::Tensor& tokens = tensor(a[2], "block_tokens");
  if (tokens.dim() != 3) fail(PyExc_ValueError, "%s must be [B,N,L]%s", "block_tokens");
  if (h.scalar_type() != at::kBFloat16 || w.scalar_type() != at::kBFloat16)
    fail(PyExc_ValueError, "%s must be bf16%s", "hidden_states and weight");
  const int64_t H = h.dim() > 0 ? h.size(-1) : 0;
  if (h.dim() != 4 || h.size(0) != tokens.size(0) || h.size(1) != tokens.size(1) || h.size(2) != tokens.size(2) ||
      w.dim() != 2 || w.size(1) != H)
    fail(PyExc_ValueError, "%s must be [B,N,L,H] and weight [V,H]%s", "hidden_states");
  if (!h.is_contiguous() || !w.is_contiguous())
    fail(PyExc_ValueError, "%s must be contiguous%s", "hidden_states and weight");
  spiffy_decide_desc d;
  d.batch = (int32_t)tokens.size(0);
  d.n_nodes = (int32_t)tokens.size(1);
  d.block_len = (int32_t)tokens.size(2);
  d.vocab = (int32_t)w.size(0);
  d.logits_dtype = SPIFFY_BF16;
  d.row_stride = d.vocab;
  d.mask_token_id = (int32_t)as_int(a[3]);
  d.rule = (int32_t)as_int(a[4]);
  d.top_s = (int32_t)as_int(a[5]);
  d.threshold = (float)as_float(a[6]);
  const void* hp = device_ptr(h, "hidden_states", kAnyType);
  const void* wp = device_ptr(w, "weight", kAnyType);
  const int32_t* tp = (const int32_t*)device_ptr(tokens, "block_tokens", at::kInt);
  const CallStream stream(a[9], h);
  Ref out(decision_for(a[7], &d, h));
  const DecisionPtrs p(out.o, "dev_status");
  const Scratch ws(a[8], a[8] == Py_None ? spiffy_lmhead_decide_workspace(&d, (int32_t)H) : 0, h, true);
  check(unlocked(spiffy_lmhead_decide, &d, (int32_t)H, hp, wp, tp, p.conf, p.top_tok, p.bits, p.n_unmask, p.status,
                 ws.ptr, ws.bytes, stream.get()),
        "spiffy_lmhead_decide");
  return out.release();
}

// ----------------------------------------------------------------- walk ----
int32_t parent_cap(const at::Tensor& off, const at::Tensor& idx, int64_t B, int64_t N) {
  if (off.dim() != 2 || off.size(0) != B || off.size(1) != N + 1 || idx.dim() != 2 || idx.size(0) != B)
    fail(PyExc_ValueError, "%s must be [B,N+1] and parent_idx [B,cap]%s", "parent_off");
  return (int32_t)idx.size(1);
}

// block_tokens, parent_off, parent_idx, top_tok, unmask_bits, out, stream
PyObject* accept_walk(PyObject* const* a) {
  const at::Tensor& tokens = tensor(a[0], "block_tokens");
  const at::Tensor& off = tensor(a[1], "parent_off");
  const at::Tensor& idx = tensor(a[2], "parent_idx");
  if (tokens.dim() != 3) fail(PyExc_ValueError, "%s must be [B,N,L]%s", "block_tokens");
  spiffy_decide_desc d = {};
  d.batch = (int32_t)tokens.size(0);
  d.n_nodes = (int32_t)tokens.size(1);
  d.block_len = (int32_t)tokens.size(2);
  d.top_s = 1;
  const int32_t cap = parent_cap(off, idx, d.batch, d.n_nodes);
  const int32_t* tp = (const int32_t*)device_ptr(tokens, "block_tokens", at::kInt);
  const int32_t* op = (const int32_t*)device_ptr(off, "parent_off", at::kInt);
  const int32_t* ip = (const int32_t*)device_ptr(idx, "parent_idx", at::kInt);
  const int32_t* top = (const int32_t*)device_ptr(a[3], "top_tok", at::kInt);
  const uint64_t* bits = (const uint64_t*)device_ptr(a[4], "unmask_bits", at::kLong);
  const CallStream stream(a[6], tokens);
  Ref out;
  if (a[5] != Py_None) {
    Py_INCREF(a[5]);
    out.o = a[5];
  } else {
    d.logits_dtype |= SPIFFY_FRESH_STATUS;
    Carver c(walk_room(d.batch, d.n_nodes, d.block_len), tokens);
    out.o = new_walk(c, d.batch, d.n_nodes, d.block_len);
  }
  const WalkPtrs w(out.o, "dev_status");
  check(unlocked(spiffy_accept_walk, &d, tp, op, ip, cap, top, bits, w.accepted_node, w.n_accepted, w.path, w.next_block,
                 w.status, stream.get()),
        "spiffy_accept_walk");
  return out.release();
}

// logits, block_tokens, mask_token_id, rule, top_s, threshold, parent_off, parent_idx, decision, walk, workspace,
// stream, lazy, flags
PyObject* decide_walk(PyObject* const* a) {
  const at::Tensor& logits = tensor(a[0], "logits");
  const at::Tensor& tokens = tensor(a[1], "block_tokens");
  const at::Tensor& off = tensor(a[6], "parent_off");
  const at::Tensor& idx = tensor(a[7], "parent_idx");
  spiffy_decide_desc d = decide_desc(logits, tokens, a + 2);
  const int64_t B = d.batch, N = d.n_nodes, L = d.block_len;
  const int32_t cap = parent_cap(off, idx, B, N);
  const int lazy = PyObject_IsTrue(a[12]);
  const long flags = PyLong_AsLong(a[13]);
  if (lazy < 0 || (flags == -1 && PyErr_Occurred())) throw PyError{};
  d.logits_dtype |= (int32_t)flags & (SPIFFY_INDEPENDENT | SPIFFY_INDEPENDENT_NEXT);
  const void* lp = logits_ptr(logits);
  const int32_t* tp = (const int32_t*)device_ptr(tokens, "block_tokens", at::kInt);
  const int32_t* op = (const int32_t*)device_ptr(off, "parent_off", at::kInt);
  const int32_t* ip = (const int32_t*)device_ptr(idx, "parent_idx", at::kInt);
  const CallStream stream(a[11], logits);
  Ref dec, walk;
  if (a[8] == Py_None && a[9] == Py_None) {
    d.logits_dtype |= SPIFFY_FRESH_STATUS;
    Carver c(decision_room(B, N, L) + walk_room(B, N, L), logits);
    dec.o = new_decision(c, B, N, L);
    walk.o = new_walk(c, B, N, L);
  } else {
    // one of the two is the caller's and keeps its status bits: the other one's words are cleared here
    if (a[8] != Py_None) {
      Py_INCREF(a[8]);
      dec.o = a[8];
    } else {
      Carver c(decision_room(B, N, L), logits);
      dec.o = new_decision(c, B, N, L);
    }
    if (a[9] != Py_None) {
      Py_INCREF(a[9]);
      walk.o = a[9];
    } else {
      Carver c(walk_room(B, N, L), logits);
      walk.o = new_walk(c, B, N, L);
    }
    for (PyObject* o : {a[8] == Py_None ? dec.o : nullptr, a[9] == Py_None ? walk.o : nullptr})
      if (o) {
        Ref s(PyObject_GetAttr(o, g_names.dev_status));
        if (!s.o) throw PyError{};
        tensor(s.o, "dev_status").zero_();
      }
  }
  const DecisionPtrs p(dec.o, "decide_status");
  const WalkPtrs w(walk.o, "walk_status");
  const size_t need = a[10] != Py_None ? 0
                      : lazy           ? spiffy_decide_walk_lazy_workspace(&d)
                                       : spiffy_unmask_decide_workspace(&d);
  const Scratch ws(a[10], need, logits, true);
  check(unlocked(lazy ? spiffy_decide_walk_lazy : spiffy_decide_walk, &d, lp, tp, op, ip, cap, p.conf, p.top_tok, p.bits,
                 p.n_unmask, p.status, w.accepted_node, w.n_accepted, w.path, w.next_block, w.status, ws.ptr, ws.bytes,
                 stream.get()),
        lazy ? "spiffy_decide_walk_lazy" : "spiffy_decide_walk");
  PyObject* r = PyTuple_Pack(2, dec.o, walk.o);
  if (!r) throw PyError{};
  return r;
}

// ------------------------------------------------------------- drafting ----
// logits, state, mask_token_id, graph, budget, top_k, parent_cap, out, workspace, stream
PyObject* draft_blocks(PyObject* const* a) {
  const at::Tensor& logits = tensor(a[0], "logits");
  const at::Tensor& state = tensor(a[1], "state");
  if (state.dim() != 2 || logits.dim() < 2) fail(PyExc_ValueError, "%s must be [B,L,V] and state [B,L]%s", "logits");
  const int64_t B = state.size(0), L = state.size(1);
  spiffy_draft_desc d;
  d.batch = (int32_t)B;
  d.block_len = (int32_t)L;
  d.vocab = (int32_t)logits.size(-1);
  d.logits_dtype = dtype_code(logits);
  d.row_stride = logits.stride(-2);
  if (B > 1 && logits.stride(0) != L * d.row_stride) fail(PyExc_ValueError, "%s rows must be equally spaced%s", "logits");
  d.mask_token_id = (int32_t)as_int(a[2]);
  d.budget = (int32_t)as_int(a[4]);
  d.top_k = (int32_t)as_int(a[5]);
  const int64_t cap = as_int(a[6]);
  const int64_t all = ((int64_t)d.budget + 1) * d.budget / 2;  // every kept draft a parent of every later one
  d.parent_cap = (int32_t)(cap ? cap : (all > 4 ? all : 4));
  if (logits.dim() == 4) logits_ptr(logits);
  if (!logits.is_cuda()) fail(PyExc_ValueError, "%s must live on a CUDA device (no CPU path exists)%s", "logits");
  const int32_t* sp = (const int32_t*)device_ptr(state, "state", at::kInt);
  PyObject* g = a[3];
  Ref foff(PyObject_GetAttr(g, g_names.formula_off));
  if (!foff.o) throw PyError{};
  const int32_t* fo = (const int32_t*)device_ptr(foff.o, "formula_off", at::kInt);
  d.n_formulas = (int32_t)tensor(foff.o, "formula_off").numel() - 1;
  const int32_t* fi = (const int32_t*)field_ptr(g, g_names.formula_i, "formula_i", at::kInt);
  const int32_t* fj = (const int32_t*)field_ptr(g, g_names.formula_j, "formula_j", at::kInt);
  const int32_t* co = (const int32_t*)field_ptr(g, g_names.child_off, "child_off", at::kInt);
  const int32_t* ci = (const int32_t*)field_ptr(g, g_names.child_idx, "child_idx", at::kInt);
  const CallStream stream(a[9], logits);
  Ref out;
  if (a[7] != Py_None) {
    Py_INCREF(a[7]);
    out.o = a[7];
  } else {
    d.logits_dtype |= SPIFFY_FRESH_STATUS;
    const int64_t n = d.budget > 0 ? d.budget : 0, D = d.n_formulas;
    const int64_t pc = d.parent_cap > 0 ? d.parent_cap : 0;
    Carver c(Carver::room(B * (n + 1) * L, 4) + Carver::room(B * n, 4) + Carver::room(B * D, 4) +
                 Carver::room(B * (n + 2), 4) + Carver::room(B * pc, 4) + Carver::room(B, 4),
             logits);
    PyObject* f[6] = {c.take({B, n + 1, L}, at::kInt), c.take({B, n}, at::kInt),  c.take({B, D}, at::kFloat),
                      c.take({B, n + 2}, at::kInt),    c.take({B, pc}, at::kInt), c.take({B}, at::kInt)};
    out.o = make(g_drafts_class, f, 6);
  }
  int32_t* tokens = (int32_t*)field_ptr(out.o, g_names.tokens, "tokens", at::kInt);
  int32_t* kept = (int32_t*)field_ptr(out.o, g_names.kept, "kept", at::kInt);
  float* score = (float*)field_ptr(out.o, g_names.score, "score", at::kFloat);
  int32_t* poff = (int32_t*)field_ptr(out.o, g_names.parent_off, "parent_off", at::kInt);
  int32_t* pidx = (int32_t*)field_ptr(out.o, g_names.parent_idx, "parent_idx", at::kInt);
  int32_t* status = (int32_t*)field_ptr(out.o, g_names.dev_status, "dev_status", at::kInt);
  const Scratch ws(a[8], a[8] == Py_None ? spiffy_draft_blocks_workspace(&d) : 0, logits, true);
  check(unlocked(spiffy_draft_blocks, &d, logits.data_ptr(), sp, fo, fi, fj, co, ci, tokens, kept, score, poff, pidx,
                 status, ws.ptr, ws.bytes, stream.get()),
        "spiffy_draft_blocks");
  return out.release();
}

// --------------------------------------------------------------- module ----
template <PyObject* (*F)(PyObject* const*), Py_ssize_t N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (const PyError&) {
  } catch (const std::exception& e) {  // an allocation that failed, say
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

// classes(SpiffyError, Decision, Walk, Drafts): what errors and results are made of
PyObject* set_classes(PyObject* const* a) {
  PyObject** slots[4] = {&g_error_class, &g_decision_class, &g_walk_class, &g_drafts_class};
  for (int i = 0; i < 4; ++i) {
    Py_INCREF(a[i]);
    Py_XDECREF(*slots[i]);
    *slots[i] = a[i];
  }
  Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject* const*), Py_ssize_t N>
constexpr PyMethodDef method(const char* name) {
  return PyMethodDef{name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<F, N>)), METH_FASTCALL,
                     nullptr};
}

PyMethodDef g_methods[] = {
    method<set_classes, 4>("set_classes"),
    method<graph_attention, 11>("graph_attention"),
    method<full_sequence_attention, 15>("full_sequence_attention"),
    method<unmask_decide, 9>("unmask_decide"),
    method<unmask_decide_sampled, 11>("unmask_decide_sampled"),
    method<lmhead_decide, 10>("lmhead_decide"),
    method<accept_walk, 7>("accept_walk"),
    method<decide_walk, 14>("decide_walk"),
    method<draft_blocks, 10>("draft_blocks"),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
  const std::pair<PyObject**, const char*> names[] = {
      {&g_names.conf, "conf"},           {&g_names.top_tok, "top_tok"},
      {&g_names.unmask_bits, "unmask_bits"}, {&g_names.n_unmask, "n_unmask"},
      {&g_names.dev_status, "dev_status"},   {&g_names.accepted_node, "accepted_node"},
      {&g_names.n_accepted, "n_accepted"},   {&g_names.path, "path"},
      {&g_names.next_block, "next_block"},   {&g_names.tokens, "tokens"},
      {&g_names.kept, "kept"},               {&g_names.score, "score"},
      {&g_names.parent_off, "parent_off"},   {&g_names.parent_idx, "parent_idx"},
      {&g_names.formula_off, "formula_off"}, {&g_names.formula_i, "formula_i"},
      {&g_names.formula_j, "formula_j"},     {&g_names.child_off, "child_off"},
      {&g_names.child_idx, "child_idx"}};
  for (const auto& n : names)
    if (!(*n.first = PyUnicode_InternFromString(n.second))) return nullptr;
  return PyModule_Create(&g_module);
}
