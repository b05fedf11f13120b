// Argument marshalling of the Selector classes in native code: checks the tensors a caller hands over, fills the C
// structures of spf.h and makes the library calls of one prompt (or one batch of prompts) in a row.
//
// Why not in Python: with a tensor per layer, the checks and the ctypes conversions took 75 to 120 us a prompt (500 us for a
// batch of eight), several times what the kernels of a short prompt take; here they take 2 to 3 us.
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>

#include <string>
#include <vector>

#include "spf.h"

namespace {

struct PyFailure {};   // a Python exception is set

[[noreturn]] void raise(PyObject* type, const std::string& text) {
  PyErr_SetString(type, text.c_str());
  throw PyFailure{};
}

// New reference, released at the end of the scope.
struct Ref {
  PyObject* p;
  explicit Ref(PyObject* p_) : p(p_) {
    if (p == nullptr) throw PyFailure{};
  }
  Ref(Ref&& o) noexcept : p(o.p) { o.p = nullptr; }
  Ref(const Ref&) = delete;
  ~Ref() { Py_XDECREF(p); }
};

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + " must be a CUDA tensor");
  return THPVariable_Unpack(o);
}

const char* dtype_name(at::ScalarType t) {
  switch (t) {
    case at::kBFloat16: return "torch.bfloat16";
    case at::kFloat: return "torch.float32";
    case at::kInt: return "torch.int32";
    case at::kLong: return "torch.int64";
    default: return "torch.uint8";
  }
}

const at::Tensor& device_tensor(PyObject* o, at::ScalarType dtype, const char* name) {
  const at::Tensor& t = tensor(o, name);
  if (!t.is_cuda() || t.scalar_type() != dtype)
    raise(PyExc_TypeError, std::string(name) + " must be a CUDA tensor of dtype " + dtype_name(dtype));
  return t;
}

// Attribute names, interned once.
struct Names {
  PyObject *importance, *lse, *chunk_scores, *kept, *out_ids, *out_pos, *tok_spans, *char_spans, *counts, *dev_status, *workspace, *chunk,
      *pool_kernel, *softmax_scale, *pool_edge_rule, *force_first, *force_last, *max_tokens, *slots, *q, *k, *token_ids, *char_start,
      *char_end, *n_tokens;
};
Names N;

Ref attr(PyObject* o, PyObject* name) { return Ref(PyObject_GetAttr(o, name)); }
// A reference of its own: the attribute may be computed, or be replaced by another thread during the call.
at::Tensor attr_tensor(PyObject* o, PyObject* name, at::ScalarType dtype, const char* what) {
  return device_tensor(attr(o, name).p, dtype, what);
}
// The same for a buffer that may be None: an undefined tensor.
at::Tensor attr_tensor_or_none(PyObject* o, PyObject* name, at::ScalarType dtype, const char* what) {
  const Ref value = attr(o, name);
  return value.p == Py_None ? at::Tensor() : device_tensor(value.p, dtype, what);
}
int64_t attr_int(PyObject* o, PyObject* name) {
  const int64_t v = PyLong_AsLongLong(attr(o, name).p);
  if (v == -1 && PyErr_Occurred()) throw PyFailure{};
  return v;
}
double attr_float(PyObject* o, PyObject* name) {
  const double v = PyFloat_AsDouble(attr(o, name).p);
  if (v == -1.0 && PyErr_Occurred()) throw PyFailure{};
  return v;
}
bool attr_true(PyObject* o, PyObject* name) {
  const int v = PyObject_IsTrue(attr(o, name).p);
  if (v < 0) throw PyFailure{};
  return v != 0;
}

enum Kind { kPlain = 0, kPaged = 1, kFp8 = 2 };

// One prompt's scoring inputs in the form of its kind.  `held` keeps the tensors behind the pointers until the kernels are
// enqueued: what the caller handed over may be temporary (a property that casts, a sequence that makes its items), and memory
// given back before that could be the workspace's, or the next prompt's, when the kernels run.
struct Inputs {
  std::vector<at::Tensor> held;
  std::vector<const void*> layers;
  int64_t n = 0;
  const void *q = nullptr, *aux = nullptr;     // aux: block table or key scales
  int64_t stride_head = 0, stride_tok = 0, pool_blocks = 0;
  int block_tokens = 0;
};

// Checks q and the layers' key tensors; the first prompt of a call fixes the shape.  `n_paged`: tokens of a paged prompt.
void read_inputs(Kind kind, PyObject* q_obj, PyObject* layers_obj, PyObject* aux_obj, int64_t n_paged, double scale, bool first,
                 spf_shape* shape, Inputs* in) {
  const at::Tensor& q = device_tensor(q_obj, at::kBFloat16, "q");
  if (q.dim() != 4) raise(PyExc_ValueError, "q must be [L, Hq, m, d]");
  if (PyIter_Check(layers_obj)) raise(PyExc_TypeError, "the key tensors must be a sequence");   // an iterator is used up by one look
  Ref layers(PySequence_Fast(layers_obj, "the key tensors must be a sequence"));
  const Py_ssize_t count = PySequence_Fast_GET_SIZE(layers.p);
  PyObject** items = PySequence_Fast_ITEMS(layers.p);
  const at::ScalarType dtype = kind == kFp8 ? at::kByte : at::kBFloat16;
  if (count < 1) raise(PyExc_ValueError, "k_layers must hold one tensor per layer");
  const at::Tensor& k0 = device_tensor(items[0], dtype, "k_layers[l]");
  const int64_t dims = kind == kPaged ? 4 : 3;
  if (k0.dim() != dims) raise(PyExc_ValueError, "a key tensor has the wrong number of dimensions");
  const int64_t hkv = kind == kPaged ? k0.size(1) : k0.size(0);
  if (first) {
    shape->n_layers = (int32_t)q.size(0);
    shape->n_q_heads = (int32_t)q.size(1);
    shape->n_lookahead = (int32_t)q.size(2);
    shape->head_dim = (int32_t)q.size(3);
    shape->n_kv_heads = (int32_t)hkv;
    shape->softmax_scale = (float)scale;
  }
  if (q.size(0) != shape->n_layers || q.size(1) != shape->n_q_heads || q.size(2) != shape->n_lookahead || q.size(3) != shape->head_dim ||
      !q.is_contiguous())
    raise(PyExc_ValueError, "q must be contiguous [L, Hq, m, d], the same shape for all prompts");
  if (count != shape->n_layers) raise(PyExc_ValueError, "k_layers must hold one tensor per layer");
  in->layers.resize((size_t)count);
  in->held.reserve((size_t)count + 2);
  in->held.push_back(q);
  for (Py_ssize_t l = 0; l < count; ++l) {
    const at::Tensor& kl = device_tensor(items[l], dtype, "k_layers[l]");
    in->held.push_back(kl);
    bool fine = kl.dim() == dims && kl.sizes() == k0.sizes() && kl.size(dims - 1) == shape->head_dim && hkv == shape->n_kv_heads;
    if (kind == kPaged) fine = fine && kl.is_contiguous();
    else fine = fine && kl.stride(2) == 1 && kl.strides() == k0.strides();
    if (!fine)
      raise(PyExc_ValueError, kind == kPaged ? "every pool must be contiguous bf16 [n_pool_blocks, Hkv, block_tokens, d]"
                                             : "every k_layers[l] must be [Hkv, N, d] with a contiguous last dim and equal strides");
    in->layers[(size_t)l] = kl.data_ptr();
  }
  in->q = q.data_ptr();
  if (kind == kPaged) {
    const at::Tensor& table = device_tensor(aux_obj, at::kInt, "block_table");
    in->n = n_paged;
    in->block_tokens = (int)k0.size(2);
    in->pool_blocks = k0.size(0);
    if (!table.is_contiguous()) raise(PyExc_ValueError, "one contiguous pool per layer, contiguous q and block_table");
    if (in->block_tokens < 1 || table.numel() < (in->n + in->block_tokens - 1) / in->block_tokens)
      raise(PyExc_ValueError, "block_table or importance has the wrong size");
    in->aux = table.data_ptr();
    in->held.push_back(table);
  } else {
    in->n = k0.size(1);
    in->stride_head = k0.stride(0);
    in->stride_tok = k0.stride(1);
    if (kind == kFp8) {
      const at::Tensor& scales = device_tensor(aux_obj, at::kFloat, "k_scale");
      if (scales.numel() != (int64_t)shape->n_layers * hkv || !scales.is_contiguous())
        raise(PyExc_ValueError, "k_scale must be contiguous fp32 [L, Hkv] and importance fp32 [N]");
      in->aux = scales.data_ptr();
      in->held.push_back(scales);
    }
  }
}

// What a Selector brings for one prompt, and the prompt's token arrays (`held`: as in Inputs).
struct Buffers {
  std::vector<at::Tensor> held;
  at::Tensor importance, lse, scores;      // trimmed to the prompt, for the result
  float *importance_ptr, *scores_ptr, *lse_ptr;
  int32_t *kept, *out_ids, *out_pos, *tok_spans, *char_spans;
  int64_t* counts;
  const int32_t *ids, *char_start, *char_end;
  int64_t n_chunks, k;
};

void read_buffers(PyObject* slot, const spf_shape& shape, int64_t n, int64_t chunk, double keep, bool force_first, bool force_last,
                  PyObject* ids, PyObject* char_start, PyObject* char_end, Buffers* b) {
  const int64_t max_tokens = attr_int(slot, N.max_tokens);
  if (n > max_tokens)
    raise(PyExc_ValueError, "prompt has " + std::to_string(n) + " tokens, selector was sized for " + std::to_string(max_tokens));
  if (chunk < 1 || chunk > INT32_MAX || n < 0) raise(PyExc_ValueError, "chunk must be in [1, 2^31) and n_tokens not negative");
  b->n_chunks = (n + chunk - 1) / chunk;
  b->k = spf_keep_count(b->n_chunks, keep);
  if (force_first || force_last) b->k = std::max(b->k, (int64_t)(force_first ? 1 : 0) + (force_last && (b->n_chunks > 1 || !force_first) ? 1 : 0));
  const at::Tensor importance = attr_tensor(slot, N.importance, at::kFloat, "importance");
  const at::Tensor lse = attr_tensor(slot, N.lse, at::kFloat, "lse");
  const at::Tensor scores = attr_tensor(slot, N.chunk_scores, at::kFloat, "chunk_scores");
  if (importance.numel() < n || !importance.is_contiguous()) raise(PyExc_ValueError, "importance must be contiguous fp32 [N]");
  if (lse.numel() != (int64_t)shape.n_layers * shape.n_q_heads * shape.n_lookahead || !lse.is_contiguous())
    raise(PyExc_ValueError, "lse must be contiguous fp32 [L, Hq, m]");
  const at::Tensor kept = attr_tensor(slot, N.kept, at::kInt, "kept_chunks");
  const at::Tensor out_ids = attr_tensor(slot, N.out_ids, at::kInt, "out_ids");
  const at::Tensor out_pos = attr_tensor_or_none(slot, N.out_pos, at::kInt, "out_pos");
  const at::Tensor tok = attr_tensor(slot, N.tok_spans, at::kInt, "out_tok_spans");
  const at::Tensor ch = attr_tensor(slot, N.char_spans, at::kInt, "out_char_spans");
  const at::Tensor counts = attr_tensor(slot, N.counts, at::kLong, "out_counts");
  const at::Tensor& i = device_tensor(ids, at::kInt, "token_ids");
  const at::Tensor& cs = device_tensor(char_start, at::kInt, "char_start");
  const at::Tensor& ce = device_tensor(char_end, at::kInt, "char_end");
  const int64_t need = std::min(b->k * chunk, n);
  if (scores.numel() < b->n_chunks || kept.numel() < b->k || out_ids.numel() < need || (out_pos.defined() && out_pos.numel() < need) || tok.numel() < 2 * b->k ||
      ch.numel() < 2 * b->k || counts.numel() < 2 || std::min(std::min(i.numel(), cs.numel()), ce.numel()) < n)
    raise(PyExc_ValueError, "a buffer is smaller than include/spf.h requires");
  b->importance = importance.narrow(0, 0, n);
  b->scores = scores.narrow(0, 0, b->n_chunks);
  b->lse = lse.view({shape.n_layers, shape.n_q_heads, shape.n_lookahead});
  b->importance_ptr = importance.data_ptr<float>();
  b->scores_ptr = scores.data_ptr<float>();
  b->lse_ptr = lse.data_ptr<float>();
  b->kept = kept.data_ptr<int32_t>();
  b->out_ids = out_ids.data_ptr<int32_t>();
  b->out_pos = out_pos.defined() ? out_pos.data_ptr<int32_t>() : nullptr;
  b->tok_spans = tok.data_ptr<int32_t>();
  b->char_spans = ch.data_ptr<int32_t>();
  b->counts = counts.data_ptr<int64_t>();
  b->ids = i.data_ptr<int32_t>();
  b->char_start = cs.data_ptr<int32_t>();
  b->char_end = ce.data_ptr<int32_t>();
  b->held = {importance, lse, scores, kept, out_ids, out_pos, tok, ch, counts, i, cs, ce};
}

spf_path_item path_item(const Buffers& b, int64_t n) {
  return spf_path_item{b.importance_ptr, n, b.scores_ptr, b.k, b.ids, b.char_start, b.char_end, b.kept, b.out_ids, b.out_pos, b.tok_spans, b.char_spans,
                       b.counts};
}

// The selector's workspace, grown where it is too small.
at::Tensor workspace_of(PyObject* selector, size_t need, const at::Tensor& like) {
  Ref now = attr(selector, N.workspace);
  if (now.p != Py_None) {
    const at::Tensor& t = tensor(now.p, "workspace");
    if ((size_t)t.numel() * t.element_size() >= need) return t;
  }
  at::Tensor t = at::empty({(int64_t)need}, like.options().dtype(at::kByte));
  Ref wrapped(THPVariable_Wrap(t));
  if (PyObject_SetAttr(selector, N.workspace, wrapped.p) != 0) throw PyFailure{};
  return t;
}

void* stream_of(PyObject* stream) {
  if (stream == Py_None) return c10::cuda::getCurrentCUDAStream(c10::cuda::current_device()).stream();
  Ref handle(PyObject_GetAttrString(stream, "cuda_stream"));
  void* p = PyLong_AsVoidPtr(handle.p);
  if (p == nullptr && PyErr_Occurred()) throw PyFailure{};
  return p;
}

PyObject* result_tuple(int32_t status, const char* where, const Buffers* b, size_t n) {
  Ref list(PyList_New((Py_ssize_t)n));
  for (size_t i = 0; i < n; ++i) {
    Ref importance(THPVariable_Wrap(b[i].importance)), lse(THPVariable_Wrap(b[i].lse)), scores(THPVariable_Wrap(b[i].scores));
    PyObject* t = Py_BuildValue("(OOOL)", importance.p, lse.p, scores.p, (long long)b[i].k);
    if (t == nullptr) throw PyFailure{};
    PyList_SET_ITEM(list.p, (Py_ssize_t)i, t);
  }
  return Py_BuildValue("(isO)", (int)status, where, list.p);
}

// select(selector, kind, q, layers, aux, n_paged, token_ids, char_start, char_end, keep, stream)
//   -> (status, failing call, [(importance, lse, chunk_scores, k)])
PyObject* select_one(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  try {
    if (n_args != 11) raise(PyExc_TypeError, "select takes 11 arguments");
    PyObject* selector = args[0];
    const Kind kind = (Kind)PyLong_AsLong(args[1]);
    const int64_t n_paged = PyLong_AsLongLong(args[5]);
    const double keep = PyFloat_AsDouble(args[9]);
    if (PyErr_Occurred()) throw PyFailure{};
    spf_shape shape{};
    Inputs in;
    read_inputs(kind, args[2], args[3], args[4], n_paged, attr_float(selector, N.softmax_scale), true, &shape, &in);
    const int64_t chunk = attr_int(selector, N.chunk);
    const int32_t pool = (int32_t)attr_int(selector, N.pool_kernel);
    const int32_t edge = (int32_t)attr_int(selector, N.pool_edge_rule);
    const bool force_first = attr_true(selector, N.force_first), force_last = attr_true(selector, N.force_last);
    Buffers b;
    read_buffers(selector, shape, in.n, chunk, keep, force_first, force_last, args[6], args[7], args[8], &b);
    const at::Tensor dev_status = attr_tensor_or_none(selector, N.dev_status, at::kInt, "dev_status");
    int32_t* status = dev_status.defined() ? dev_status.data_ptr<int32_t>() : nullptr;
    void* stream = stream_of(args[10]);

    spf_prompt plain{in.n, in.layers.data(), in.stride_head, in.stride_tok, in.q, b.importance_ptr, b.lse_ptr};
    spf_paged_prompt paged{in.n, in.layers.data(), in.pool_blocks, in.block_tokens, static_cast<const int32_t*>(in.aux), in.q, b.importance_ptr, b.lse_ptr};
    spf_fp8_prompt fp8{in.n, in.layers.data(), in.stride_head, in.stride_tok, static_cast<const float*>(in.aux), in.q, b.importance_ptr, b.lse_ptr};
    const size_t need = kind == kPlain ? spf_score_workspace_bytes(&shape, &plain, 1)
                        : kind == kPaged ? spf_score_paged_workspace_bytes(&shape, &paged, 1)
                                         : spf_score_fp8_workspace_bytes(&shape, &fp8, 1);
    if (need == 0) return result_tuple(SPF_ERR_INVALID_ARG, "spf_score_workspace_bytes", nullptr, 0);
    const at::Tensor ws = workspace_of(selector, need, b.importance);
    const size_t ws_bytes = (size_t)ws.numel() * ws.element_size();
    void* ws_ptr = ws.data_ptr();

    int32_t st;
    const char* where;
    Py_BEGIN_ALLOW_THREADS;
    where = kind == kPlain ? "spf_score" : kind == kPaged ? "spf_score_paged" : "spf_score_fp8";
    st = kind == kPlain ? spf_score(&shape, &plain, 1, ws_ptr, ws_bytes, status, stream)
         : kind == kPaged ? spf_score_paged(&shape, &paged, 1, ws_ptr, ws_bytes, status, stream)
                          : spf_score_fp8(&shape, &fp8, 1, ws_ptr, ws_bytes, status, stream);
    if (st == SPF_OK) {
      where = "spf_pool_select_compact";
      const spf_path_item item = path_item(b, in.n);
      st = spf_pool_select_compact(&item, 1, pool, (int32_t)chunk, edge, force_first, force_last, stream);
    }
    Py_END_ALLOW_THREADS;
    return result_tuple(st, where, &b, 1);
  } catch (const PyFailure&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// select_batch(batch selector, prompts, keep, stream) -> (status, failing call, [(importance, lse, chunk_scores, k)])
PyObject* select_batch(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  try {
    if (n_args != 4) raise(PyExc_TypeError, "select_batch takes 4 arguments");
    PyObject* selector = args[0];
    Ref prompts(PySequence_Fast(args[1], "prompts must be a sequence"));
    const double keep = PyFloat_AsDouble(args[2]);
    if (PyErr_Occurred()) throw PyFailure{};
    const size_t count = (size_t)PySequence_Fast_GET_SIZE(prompts.p);
    Ref slots(attr(selector, N.slots));
    Ref slot_items(PySequence_Fast(slots.p, "slots must be a sequence"));
    if (count > (size_t)PySequence_Fast_GET_SIZE(slot_items.p)) raise(PyExc_ValueError, "more prompts than slots");
    if (count == 0) raise(PyExc_IndexError, "no prompts");
    const int64_t chunk = attr_int(selector, N.chunk);
    const int32_t pool = (int32_t)attr_int(selector, N.pool_kernel);
    const double scale = attr_float(selector, N.softmax_scale);
    spf_shape shape{};
    std::vector<Inputs> in(count);
    std::vector<Buffers> b(count);
    std::vector<spf_prompt> p(count);
    std::vector<spf_path_item> items(count);
    for (size_t i = 0; i < count; ++i) {
      PyObject* prompt = PySequence_Fast_GET_ITEM(prompts.p, (Py_ssize_t)i);
      Ref q(attr(prompt, N.q)), k(attr(prompt, N.k));
      read_inputs(kPlain, q.p, k.p, nullptr, 0, scale, i == 0, &shape, &in[i]);
      const int64_t n = attr_int(prompt, N.n_tokens);
      if (n != in[i].n) raise(PyExc_ValueError, "importance must be contiguous fp32 [N]");
      Ref ids(attr(prompt, N.token_ids)), cs(attr(prompt, N.char_start)), ce(attr(prompt, N.char_end));
      read_buffers(PySequence_Fast_GET_ITEM(slot_items.p, (Py_ssize_t)i), shape, n, chunk, keep, false, false, ids.p, cs.p, ce.p, &b[i]);
      p[i] = spf_prompt{n, in[i].layers.data(), in[i].stride_head, in[i].stride_tok, in[i].q, b[i].importance_ptr, b[i].lse_ptr};
      items[i] = path_item(b[i], n);
    }
    const at::Tensor dev_status = attr_tensor_or_none(selector, N.dev_status, at::kInt, "dev_status");
    int32_t* status = dev_status.defined() ? dev_status.data_ptr<int32_t>() : nullptr;
    void* stream = stream_of(args[3]);
    const size_t need = spf_score_workspace_bytes(&shape, p.data(), (int32_t)count);
    if (need == 0) return result_tuple(SPF_ERR_INVALID_ARG, "spf_score_workspace_bytes", nullptr, 0);
    const at::Tensor ws = workspace_of(selector, need, b[0].importance);
    const size_t ws_bytes = (size_t)ws.numel() * ws.element_size();
    void* ws_ptr = ws.data_ptr();
    int32_t st;
    const char* where;
    Py_BEGIN_ALLOW_THREADS;
    where = "spf_score";
    st = spf_score(&shape, p.data(), (int32_t)count, ws_ptr, ws_bytes, status, stream);
    if (st == SPF_OK) {
      where = "spf_pool_select_compact";
      st = spf_pool_select_compact(items.data(), (int32_t)count, pool, (int32_t)chunk, 0, 0, 0, stream);
    }
    Py_END_ALLOW_THREADS;
    return result_tuple(st, where, b.data(), count);
  } catch (const PyFailure&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

const at::Tensor& host_tensor(PyObject* o, at::ScalarType dtype, const char* name) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() && t.scalar_type() == dtype && t.is_contiguous()) return t;
  }
  raise(PyExc_TypeError, std::string(name) + " must be a contiguous host tensor of dtype " + dtype_name(dtype));
}

// compress_host(q, layers, token_ids, char_start, char_end, chunk, pool_kernel, keep, arena, out_ids, out_pos, tok_spans, char_spans,
//               counts, softmax_scale, stream) -> status
PyObject* compress_host(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  try {
    if (n_args != 16) raise(PyExc_TypeError, "compress_host takes 16 arguments");
    const at::Tensor& q = host_tensor(args[0], at::kBFloat16, "q");
    if (q.dim() != 4) raise(PyExc_ValueError, "q must be [L, Hq, m, d]");
    Ref layers(PySequence_Fast(args[1], "k_layers must be a sequence"));
    const Py_ssize_t count = PySequence_Fast_GET_SIZE(layers.p);
    if (count < 1) raise(PyExc_ValueError, "k_layers must hold one tensor per layer");
    std::vector<const void*> ptrs((size_t)count);
    int64_t hkv = 0, n = 0;
    for (Py_ssize_t l = 0; l < count; ++l) {
      const at::Tensor& k = host_tensor(PySequence_Fast_GET_ITEM(layers.p, l), at::kBFloat16, "k_layers[l]");
      if (l == 0 && k.dim() == 3) {
        hkv = k.size(0);
        n = k.size(1);
      }
      if (k.dim() != 3 || k.size(0) != hkv || k.size(1) != n || k.size(2) != q.size(3))
        raise(PyExc_ValueError, "every k_layers[l] must be [Hkv, N, d]");
      ptrs[(size_t)l] = k.data_ptr();
    }
    const at::Tensor& ids = host_tensor(args[2], at::kInt, "token_ids");
    const at::Tensor& cs = host_tensor(args[3], at::kInt, "char_start");
    const at::Tensor& ce = host_tensor(args[4], at::kInt, "char_end");
    spf_select_params params{};
    params.chunk = (int32_t)PyLong_AsLong(args[5]);
    params.pool_kernel = (int32_t)PyLong_AsLong(args[6]);
    params.keep_ratio = PyFloat_AsDouble(args[7]);
    const double scale = PyFloat_AsDouble(args[14]);
    if (PyErr_Occurred()) throw PyFailure{};
    const at::Tensor& arena = tensor(args[8], "arena");
    if (!arena.is_cuda()) raise(PyExc_TypeError, "arena must be a CUDA tensor");
    const at::Tensor& out_ids = host_tensor(args[9], at::kInt, "out_ids");
    const at::Tensor* out_pos = args[10] == Py_None ? nullptr : &host_tensor(args[10], at::kInt, "out_pos");
    const at::Tensor& tok = host_tensor(args[11], at::kInt, "out_tok_spans");
    const at::Tensor& ch = host_tensor(args[12], at::kInt, "out_char_spans");
    const at::Tensor& counts = host_tensor(args[13], at::kLong, "out_counts");
    if (params.chunk >= 1) {
      const int64_t k = spf_keep_count((n + params.chunk - 1) / params.chunk, params.keep_ratio), need = std::min(k * params.chunk, n);
      if (count != q.size(0) || std::min(std::min(ids.numel(), cs.numel()), ce.numel()) < n || out_ids.numel() < need ||
          (out_pos != nullptr && out_pos->numel() < need) || tok.numel() < 2 * k || ch.numel() < 2 * k || counts.numel() < 2)
        raise(PyExc_ValueError, "a buffer is smaller than include/spf.h requires");
    }
    const spf_shape shape{(int32_t)q.size(0), (int32_t)q.size(1), (int32_t)hkv, (int32_t)q.size(3), (int32_t)q.size(2), (float)scale};
    void* stream = stream_of(args[15]);
    void* arena_ptr = arena.data_ptr();
    const size_t arena_bytes = (size_t)arena.numel() * arena.element_size();
    int32_t st;
    Py_BEGIN_ALLOW_THREADS;
    st = spf_compress_host(&shape, n, ptrs.data(), q.data_ptr(), ids.data_ptr<int32_t>(), cs.data_ptr<int32_t>(), ce.data_ptr<int32_t>(), &params,
                           arena_ptr, arena_bytes, out_ids.data_ptr<int32_t>(), out_pos != nullptr ? out_pos->data_ptr<int32_t>() : nullptr,
                           tok.data_ptr<int32_t>(), ch.data_ptr<int32_t>(), counts.data_ptr<int64_t>(), stream);
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(st);
  } catch (const PyFailure&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef kMethods[] = {
    {"select", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(select_one)), METH_FASTCALL, "The path for one prompt."},
    {"select_batch", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(select_batch)), METH_FASTCALL, "The path for a batch of prompts."},
    {"compress_host", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(compress_host)), METH_FASTCALL, "The path for one prompt in host tensors."},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Native marshalling of the Selector classes.", -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
#define SPF_NAME(x) N.x = PyUnicode_InternFromString(#x)
  SPF_NAME(importance); SPF_NAME(lse); SPF_NAME(chunk_scores); SPF_NAME(kept); SPF_NAME(out_ids); SPF_NAME(out_pos); SPF_NAME(tok_spans);
  SPF_NAME(char_spans); SPF_NAME(counts); SPF_NAME(dev_status); SPF_NAME(workspace); SPF_NAME(chunk); SPF_NAME(pool_kernel);
  SPF_NAME(softmax_scale); SPF_NAME(pool_edge_rule); SPF_NAME(force_first); SPF_NAME(force_last); SPF_NAME(max_tokens); SPF_NAME(slots);
  SPF_NAME(q); SPF_NAME(k); SPF_NAME(token_ids); SPF_NAME(char_start); SPF_NAME(char_end); SPF_NAME(n_tokens);
#undef SPF_NAME
  return PyModule_Create(&kModule);
}
