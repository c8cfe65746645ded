// Argument marshalling of the Python binding's per-layer calls, in native code: shape descriptor, output and workspace
// tensors, stream, call.  The Python functions of the same names (__init__.py) keep the interface and raise the errors;
// what is here is what they would otherwise do object by object.  No tensor data is touched.
//
// Why: a small call is bound by the host.  fwd() over 2 heads of 2,048 tokens spends 12.5 us on the device and took 16.3 us
// of host time: 5.2 in the library (two launches, three tensor maps), the rest in ctypes conversions, a Shape object, a
// workspace query and the tuples of sizes and strides behind each check.  Now 8.1, and the call takes what the device takes:
// 16.5 -> 12.6 us; selection + forward of 3 heads of 1,200 tokens 36.4 -> 19.0.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstring>
#include <initializer_list>

#include "../../include/sparkattn.h"

namespace {

// Entry points of the library that the Python side has loaded (bind()).
struct Library {
  decltype(&sparkattn_workspace_bytes) workspace_bytes;
  decltype(&sparkattn_select) select;
  decltype(&sparkattn_select_window) select_window;
  decltype(&sparkattn_select_padded) select_padded;
  decltype(&sparkattn_select_pooled) select_pooled;
  decltype(&sparkattn_quant_fp8) quant_fp8;
  decltype(&sparkattn_quant_fp8_pooled) quant_fp8_pooled;
  decltype(&sparkattn_quant_fp8_per_token) quant_fp8_per_token;
  decltype(&sparkattn_fwd) fwd;
  decltype(&sparkattn_fwd_window) fwd_window;
  decltype(&sparkattn_fwd_padded) fwd_padded;
  decltype(&sparkattn_gather_tokens) gather_tokens;
  decltype(&sparkattn_comp_workspace_bytes) comp_workspace_bytes;
  decltype(&sparkattn_comp_state) comp_state;
  decltype(&sparkattn_comp_apply) comp_apply;
  decltype(&sparkattn_fwd_gated_workspace_bytes) fwd_gated_workspace_bytes;
  decltype(&sparkattn_fwd_gated) fwd_gated;
};
Library g_lib{};

// A stream's handle, or the current stream of the current device, asked for when the call is made.
struct Stream {
  void* handle = nullptr;
  bool given = false;
  operator void*() const { return given ? handle : c10::cuda::getCurrentCUDAStream().stream(); }
};

// The arguments of one call, taken in order; the first one of a wrong kind raises.
class Args {
 public:
  Args(PyObject* const* args, Py_ssize_t n) : args_(args), n_(n) {}
  void expect(Py_ssize_t n) const { TORCH_CHECK_TYPE(n_ == n, "expected ", n, " arguments, got ", n_); }
  at::Tensor tensor() {
    PyObject* o = next();
    TORCH_CHECK_TYPE(THPVariable_Check(o), "expected a tensor, got ", Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
  }
  at::Tensor optional_tensor() {      // undefined for None
    if (args_[at_] == Py_None) { ++at_; return at::Tensor(); }
    return tensor();
  }
  int64_t integer() {
    const long long v = PyLong_AsLongLong(next());
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
  }
  int32_t i32() {
    const int64_t v = integer();
    TORCH_CHECK_VALUE(v == (int32_t)v, v, " does not fit 32 bits");
    return (int32_t)v;
  }
  float number() {
    const double v = PyFloat_AsDouble(next());
    if (v == -1.0 && PyErr_Occurred()) throw python_error();
    return (float)v;
  }
  bool truth() {
    const int v = PyObject_IsTrue(next());
    if (v < 0) throw python_error();
    return v != 0;
  }
  Stream stream() {
    if (args_[at_] == Py_None) { ++at_; return {}; }
    return {(void*)(intptr_t)integer(), true};
  }

 private:
  PyObject* next() { return args_[at_++]; }
  PyObject* const* args_;
  Py_ssize_t n_, at_ = 0;
};

sparkattn_shape_t make_shape(const at::Tensor& x, int32_t block, float softmax_scale = 0.0f) {
  TORCH_CHECK_VALUE(x.dim() == 4 && x.stride(3) == 1, "expected a [B, H, N, d] tensor with a contiguous last dimension");
  sparkattn_shape_t s{};
  s.struct_size = sizeof(s);
  s.version = SPARKATTN_VERSION;
  s.B = (int32_t)x.size(0); s.H = (int32_t)x.size(1); s.N = (int32_t)x.size(2); s.d = (int32_t)x.size(3);
  s.block = block;
  s.stride_b = x.stride(0); s.stride_h = x.stride(1); s.stride_n = x.stride(2);
  s.softmax_scale = softmax_scale;
  return s;
}

void same_layout(const at::Tensor& a, const at::Tensor& b) {
  TORCH_CHECK_VALUE(a.sizes() == b.sizes() && a.strides() == b.strides(), "tensors of one call must share shape and strides");
}

void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }
int32_t* iptr(const at::Tensor& t) { return static_cast<int32_t*>(ptr(t)); }
float* fptr(const at::Tensor& t) { return static_cast<float*>(ptr(t)); }
at::TensorOptions on(const at::Tensor& x, at::ScalarType type) { return at::TensorOptions().dtype(type).device(x.device()); }
// Token blocks of a head.  Outputs are sized with it before the library has looked at the shape: a block size below 1,
// which the library refuses, has none.
int64_t blocks(const sparkattn_shape_t& s) { return s.block < 1 ? 0 : ((int64_t)s.N + s.block - 1) / s.block; }

// The caller's workspace, or a new one; undefined when the library does not serve the shape.
at::Tensor workspace_for(at::Tensor given, const sparkattn_shape_t& s, int32_t which, int32_t k, const at::Tensor& x) {
  if (given.defined()) return given;
  const size_t n = g_lib.workspace_bytes(&s, which, k);
  return n == 0 ? at::Tensor() : at::empty({(int64_t)n}, on(x, at::kByte));
}

PyObject* result(int rc, std::initializer_list<at::Tensor> tensors) {
  PyObject* t = PyTuple_New((Py_ssize_t)tensors.size() + 1);
  if (t == nullptr) throw python_error();
  PyTuple_SET_ITEM(t, 0, PyLong_FromLong(rc));
  Py_ssize_t i = 1;
  for (const at::Tensor& x : tensors) {
    if (x.defined()) {
      PyTuple_SET_ITEM(t, i++, THPVariable_Wrap(x));
    } else {
      Py_INCREF(Py_None);
      PyTuple_SET_ITEM(t, i++, Py_None);
    }
  }
  return t;
}
// workspace_for() found no workspace: what the Python side raises for the query that returned 0
constexpr int kNoWorkspace = 1;

// select(q, k, block, topk, kept_idx, kept_cnt, workspace, stream, frame_tokens, window, block_valid) -> rc, kept_idx, kept_cnt
PyObject* select(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(11);
  const at::Tensor q = a.tensor(), k = a.tensor();
  const int32_t block = a.i32(), topk = a.i32();
  at::Tensor idx = a.optional_tensor(), cnt = a.optional_tensor(), ws = a.optional_tensor();
  const Stream stream = a.stream();
  const int32_t frame_tokens = a.i32(), window = a.i32();
  const at::Tensor valid = a.optional_tensor();
  same_layout(q, k);
  const sparkattn_shape_t s = make_shape(q, block);
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    if (!idx.defined()) idx = at::empty({s.B, s.H, blocks(s), std::max(topk, 1)}, on(q, at::kInt));
    if (!cnt.defined()) cnt = at::empty({s.B, s.H, blocks(s)}, on(q, at::kInt));
    ws = workspace_for(ws, s, 0, topk, q);
    if (!ws.defined()) rc = kNoWorkspace;
    else if (valid.defined())
      rc = g_lib.select_padded(&s, ptr(q), ptr(k), topk, iptr(valid), iptr(idx), iptr(cnt), ptr(ws), (size_t)ws.numel(), stream);
    else if (frame_tokens > 0)
      rc = g_lib.select_window(&s, ptr(q), ptr(k), topk, frame_tokens, window, iptr(idx), iptr(cnt), ptr(ws), (size_t)ws.numel(), stream);
    else
      rc = g_lib.select(&s, ptr(q), ptr(k), topk, iptr(idx), iptr(cnt), ptr(ws), (size_t)ws.numel(), stream);
  }
  return result(rc, {idx, cnt});
  END_HANDLE_TH_ERRORS
}

// select_pooled(ref, block, topk, workspace, kept_idx, kept_cnt, stream) -> rc, kept_idx, kept_cnt
PyObject* select_pooled(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(7);
  const at::Tensor ref = a.tensor();
  const int32_t block = a.i32(), topk = a.i32();
  const at::Tensor ws = a.tensor();
  at::Tensor idx = a.optional_tensor(), cnt = a.optional_tensor();
  const Stream stream = a.stream();
  const sparkattn_shape_t s = make_shape(ref, block);
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    if (!idx.defined()) idx = at::empty({s.B, s.H, blocks(s), std::max(topk, 1)}, on(ref, at::kInt));
    if (!cnt.defined()) cnt = at::empty({s.B, s.H, blocks(s)}, on(ref, at::kInt));
    rc = g_lib.select_pooled(&s, topk, iptr(idx), iptr(cnt), ptr(ws), (size_t)ws.numel(), stream);
  }
  return result(rc, {idx, cnt});
  END_HANDLE_TH_ERRORS
}

// What the three quantisation calls share: codes (laid out like x) and scales [B, H, per_head] where the caller brings none.
template <typename Call>
PyObject* quantise(const at::Tensor& x, const sparkattn_shape_t& s, int64_t per_head, at::Tensor codes, at::Tensor scales, Call call) {
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    if (!codes.defined()) codes = at::empty_strided(x.sizes(), x.strides(), on(x, at::kByte));
    if (!scales.defined()) scales = at::empty({s.B, s.H, per_head}, on(x, at::kFloat));
    rc = call(&s, ptr(x), static_cast<uint8_t*>(ptr(codes)), fptr(scales));
  }
  return result(rc, {codes, scales});
}

// quant_fp8(x, block, codes, scales, stream) -> rc, codes, scales
PyObject* quant_fp8(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(5);
  const at::Tensor x = a.tensor();
  const sparkattn_shape_t s = make_shape(x, a.i32());
  const at::Tensor codes = a.optional_tensor(), scales = a.optional_tensor();
  const Stream stream = a.stream();
  return quantise(x, s, blocks(s), codes, scales, [&](auto... to) { return g_lib.quant_fp8(to..., 0, stream); });
  END_HANDLE_TH_ERRORS
}

// quant_fp8_pooled(x, block, key side, select workspace, codes, scales, stream) -> rc, codes, scales
PyObject* quant_fp8_pooled(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(7);
  const at::Tensor x = a.tensor();
  const sparkattn_shape_t s = make_shape(x, a.i32());
  const bool key_side = a.truth();
  const at::Tensor ws = a.tensor(), codes = a.optional_tensor(), scales = a.optional_tensor();
  const Stream stream = a.stream();
  return quantise(x, s, blocks(s), codes, scales,
                  [&](auto... to) { return g_lib.quant_fp8_pooled(to..., key_side, ptr(ws), (size_t)ws.numel(), stream); });
  END_HANDLE_TH_ERRORS
}

// quant_fp8_per_token(x, codes, scales, stream) -> rc, codes, scales
PyObject* quant_fp8_per_token(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(4);
  const at::Tensor x = a.tensor();
  const sparkattn_shape_t s = make_shape(x, x.size(-1) == 64 ? 64 : 128);
  const at::Tensor codes = a.optional_tensor(), scales = a.optional_tensor();
  const Stream stream = a.stream();
  return quantise(x, s, s.N, codes, scales, [&](auto... to) { return g_lib.quant_fp8_per_token(to..., stream); });
  END_HANDLE_TH_ERRORS
}

// fwd(q, k, v, kept_idx, kept_cnt, block, dtype, q_scale, k_scale, v_scale, softmax_scale, out, return_lse, workspace, stream,
// frame_tokens, window, block_valid) -> rc, out, lse, workspace
PyObject* fwd(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(18);
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), idx = a.tensor(), cnt = a.optional_tensor();
  const int32_t block = a.i32(), dtype = a.i32();
  const at::Tensor sq = a.optional_tensor(), sk = a.optional_tensor(), sv = a.optional_tensor();
  const float softmax_scale = a.number();
  at::Tensor out = a.optional_tensor(), lse;
  const bool return_lse = a.truth();
  at::Tensor ws = a.optional_tensor();
  const Stream stream = a.stream();
  const int32_t frame_tokens = a.i32(), window = a.i32();
  const at::Tensor valid = a.optional_tensor();
  same_layout(q, k);
  same_layout(q, v);
  const sparkattn_shape_t s = make_shape(q, block, softmax_scale);
  const int32_t kmax = (int32_t)idx.size(-1);
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    if (!out.defined()) out = at::empty_strided(q.sizes(), q.strides(), on(q, at::kBFloat16));
    if (return_lse) lse = at::empty({s.B, s.H, s.N}, on(q, at::kFloat));
    ws = workspace_for(ws, s, 1, kmax, q);
    const size_t bytes = ws.defined() ? (size_t)ws.numel() : 0;
    if (!ws.defined()) rc = kNoWorkspace;
    else if (valid.defined())
      rc = g_lib.fwd_padded(&s, dtype, ptr(q), ptr(k), ptr(v), fptr(sq), fptr(sk), fptr(sv), iptr(idx), iptr(cnt), kmax, iptr(valid),
                            ptr(out), fptr(lse), ptr(ws), bytes, stream);
    else if (frame_tokens > 0)
      rc = g_lib.fwd_window(&s, dtype, ptr(q), ptr(k), ptr(v), fptr(sq), fptr(sk), fptr(sv), iptr(idx), iptr(cnt), kmax, frame_tokens,
                            window, ptr(out), fptr(lse), ptr(ws), bytes, stream);
    else
      rc = g_lib.fwd(&s, dtype, ptr(q), ptr(k), ptr(v), fptr(sq), fptr(sk), fptr(sv), iptr(idx), iptr(cnt), kmax, ptr(out), fptr(lse),
                     ptr(ws), bytes, stream);
  }
  return result(rc, {out, lse, ws});
  END_HANDLE_TH_ERRORS
}

// gather_tokens(x, index, out, workspace, stream) -> rc, out, workspace
PyObject* gather_tokens(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(5);
  const at::Tensor x = a.tensor(), index = a.tensor();
  at::Tensor out = a.optional_tensor(), ws = a.optional_tensor();
  const Stream stream = a.stream();
  const int32_t block = x.size(-1) == 64 ? 64 : 128;
  TORCH_CHECK_VALUE(index.scalar_type() == at::kInt && index.dim() == 1 && index.is_contiguous(),
                    "index must be a contiguous 1-D int32 tensor");
  const sparkattn_shape_t src = make_shape(x, block);
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    if (!out.defined()) out = at::empty({src.B, src.H, index.numel(), src.d}, on(x, x.scalar_type()));
    const sparkattn_shape_t dst = make_shape(out, block);
    if (!ws.defined()) ws = at::empty({256}, on(x, at::kByte));
    rc = g_lib.gather_tokens(&src, ptr(x), &dst, iptr(index), ptr(out), ptr(ws), (size_t)ws.numel(), stream);
  }
  return result(rc, {out, ws});
  END_HANDLE_TH_ERRORS
}

// What the calls of the compensation branch share: the grid and the rotary tables.
struct Rope {
  int32_t grid[3];
  at::Tensor axis, freq;
  explicit Rope(Args& a) {
    for (int32_t& g : grid) g = a.i32();
    axis = a.tensor();
    freq = a.tensor();
    TORCH_CHECK_VALUE(axis.numel() == freq.numel(), "rope axis and frequency tables must have rank/2 entries each");
  }
  // The library reads the tables on the host.  A copy from the device waits for the stream's earlier work, so this is
  // called without the interpreter lock.
  void to_host() {
    axis = axis.detach().to(at::kCPU, at::kInt).contiguous();
    freq = freq.detach().to(at::kCPU, at::kFloat).contiguous();
  }
};
bool is_contiguous(const at::Tensor& t, at::IntArrayRef sizes) { return t.is_contiguous() && t.sizes() == sizes; }
int32_t check_projection(const at::Tensor& p, const sparkattn_shape_t& s, const char* what) {
  TORCH_CHECK_VALUE(p.dim() == 3 && is_contiguous(p, {s.H, p.size(1), s.d}), what, " must be contiguous [H, rank, d]");
  return (int32_t)p.size(1);
}
void check_gate_operands(const at::Tensor& state, const at::Tensor& gate, const sparkattn_shape_t& s, int32_t rank) {
  TORCH_CHECK_VALUE(is_contiguous(state, {s.B, s.H, rank, s.d}) && state.scalar_type() == at::kFloat,
                    "state must be contiguous fp32 [B, H, rank, d]");
  TORCH_CHECK_VALUE(is_contiguous(gate, {s.B, s.H, s.N}) && gate.scalar_type() == at::kFloat, "gate must be contiguous fp32 [B, H, N]");
}
at::Tensor at_least_256(size_t bytes, const at::Tensor& x) { return at::empty({(int64_t)std::max(bytes, (size_t)256)}, on(x, at::kByte)); }

// comp_state(k, v, pk, T, Hg, Wg, axis, freq, state, workspace, stream) -> rc, state, workspace
PyObject* comp_state(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(11);
  const at::Tensor k = a.tensor(), v = a.tensor(), pk = a.tensor();
  same_layout(k, v);
  const sparkattn_shape_t s = make_shape(k, 128);
  Rope rope(a);
  const int32_t rank = check_projection(pk, s, "pk");
  at::Tensor state = a.optional_tensor(), ws = a.optional_tensor();
  const Stream stream = a.stream();
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    rope.to_host();
    if (!state.defined()) state = at::empty({s.B, s.H, rank, s.d}, on(k, at::kFloat));
    if (!ws.defined()) ws = at_least_256(g_lib.comp_workspace_bytes(&s, rope.grid), k);
    rc = g_lib.comp_state(&s, ptr(k), ptr(v), ptr(pk), rank, rope.grid, iptr(rope.axis), fptr(rope.freq), fptr(state), ptr(ws),
                          (size_t)ws.numel(), stream);
  }
  return result(rc, {state, ws});
  END_HANDLE_TH_ERRORS
}

// comp_apply(q, pq, state, gate, o_sparse, T, Hg, Wg, axis, freq, eps, out, workspace, stream) -> rc, out, workspace
PyObject* comp_apply(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(14);
  const at::Tensor q = a.tensor(), pq = a.tensor(), state = a.tensor(), gate = a.tensor(), o_sparse = a.tensor();
  same_layout(q, o_sparse);
  const sparkattn_shape_t s = make_shape(q, 128);
  Rope rope(a);
  const int32_t rank = check_projection(pq, s, "pq");
  check_gate_operands(state, gate, s, rank);
  const float eps = a.number();
  at::Tensor out = a.optional_tensor(), ws = a.optional_tensor();
  const Stream stream = a.stream();
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    rope.to_host();
    if (!out.defined()) out = at::empty_strided(q.sizes(), q.strides(), on(q, at::kBFloat16));
    if (!ws.defined()) ws = at_least_256(g_lib.comp_workspace_bytes(&s, rope.grid), q);
    rc = g_lib.comp_apply(&s, ptr(q), ptr(pq), rank, rope.grid, iptr(rope.axis), fptr(rope.freq), fptr(state), fptr(gate),
                          ptr(o_sparse), ptr(out), eps, ptr(ws), (size_t)ws.numel(), stream);
  }
  return result(rc, {out, ws});
  END_HANDLE_TH_ERRORS
}

// fwd_gated(q, k, v, kept_idx, kept_cnt, pq, state, gate, T, Hg, Wg, axis, freq, eps, softmax_scale, out, return_lse, workspace,
// stream) -> rc, out, lse, workspace
PyObject* fwd_gated(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  a.expect(19);
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), idx = a.tensor(), cnt = a.optional_tensor(), pq = a.tensor(),
                   state = a.tensor(), gate = a.tensor();
  same_layout(q, k);
  same_layout(q, v);
  Rope rope(a);
  const float eps = a.number(), softmax_scale = a.number();
  const sparkattn_shape_t s = make_shape(q, 128, softmax_scale);
  const int32_t rank = check_projection(pq, s, "pq"), kmax = (int32_t)idx.size(-1);
  check_gate_operands(state, gate, s, rank);
  at::Tensor out = a.optional_tensor(), lse;
  const bool return_lse = a.truth();
  at::Tensor ws = a.optional_tensor();
  const Stream stream = a.stream();
  int rc;
  {
    pybind11::gil_scoped_release no_gil;
    rope.to_host();
    if (!out.defined()) out = at::empty_strided(q.sizes(), q.strides(), on(q, at::kBFloat16));
    if (return_lse) lse = at::empty({s.B, s.H, s.N}, on(q, at::kFloat));
    if (!ws.defined()) ws = at_least_256(g_lib.fwd_gated_workspace_bytes(&s, kmax, rope.grid), q);
    rc = g_lib.fwd_gated(&s, ptr(q), ptr(k), ptr(v), iptr(idx), iptr(cnt), kmax, ptr(pq), rank, rope.grid, iptr(rope.axis),
                         fptr(rope.freq), fptr(state), fptr(gate), eps, ptr(out), fptr(lse), ptr(ws), (size_t)ws.numel(), stream);
  }
  return result(rc, {out, lse, ws});
  END_HANDLE_TH_ERRORS
}

// bind(address of each entry point, in the order of Library)
PyObject* bind(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(argv, n);
  constexpr Py_ssize_t kEntries = sizeof(Library) / sizeof(void*);
  a.expect(kEntries);
  void* entry[kEntries];
  for (void*& e : entry) e = reinterpret_cast<void*>((intptr_t)a.integer());
  static_assert(sizeof(entry) == sizeof(Library), "one address per entry point");
  memcpy(&g_lib, entry, sizeof(entry));
  Py_RETURN_NONE;
  END_HANDLE_TH_ERRORS
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) { return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr}; }
PyMethodDef g_methods[] = {method<bind>("bind"), method<select>("select"), method<select_pooled>("select_pooled"),
                           method<quant_fp8>("quant_fp8"), method<quant_fp8_pooled>("quant_fp8_pooled"),
                           method<quant_fp8_per_token>("quant_fp8_per_token"), method<fwd>("fwd"), method<gather_tokens>("gather_tokens"),
                           method<comp_state>("comp_state"), method<comp_apply>("comp_apply"), method<fwd_gated>("fwd_gated"), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_sparkattn", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sparkattn(void) { return PyModule_Create(&g_module); }
