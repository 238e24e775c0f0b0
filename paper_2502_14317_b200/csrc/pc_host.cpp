// Host side of hot_path() in binding.py as one call: output and workspace tensors, descriptor, launches.
//
// What bounds a short prompt through the whole path is the time between its launches: of 54 us a pass over four chunks of 256 tokens
// that keeps nothing between calls, thirteen new tensors made one by one in Python took 26 and the arguments some 6 more,
// beside 22 for the six launches and their tensor maps; the kernels need 36.  Here a new tensor takes a third of that.
//
// The library's entry points come as addresses with each call: this module holds no state.
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/core/impl/VirtualGuardImpl.h>
#include <pybind11/pybind11.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/pc.h"

namespace {

// outputs and workspaces, in the order of binding.py's _HOT_PATH_BUFFERS
enum { O, K_ROT, WIN_SCORE, WIN_LSE, SCORE, KEPT, IDX, KC, VC, POS, FG, STATUS, WS_PREFILL, WS_PAR, N_BUFFERS };
// result codes beside the library's own; with BAD_BUFFER the stage is the buffer's place
enum { NOT_INNERMOST = 1, NOT_CONTIGUOUS = 2, BAD_INPUT = 3, BAD_BUFFER = 4 };

using ws_bytes_fn = size_t (*)(const pc_prefill_desc*, int32_t, int32_t, size_t*);
using hot_path_fn = int32_t (*)(const pc_prefill_desc*, const pc_hot_path_args*, int32_t*, void*);

struct Call {
  ws_bytes_fn ws_bytes;
  hot_path_fn run;
  at::Tensor q, k, v, given, t[N_BUFFERS];
  bool has_given, made[N_BUFFERS] = {};
  int64_t C, L, Hq, Hkv, d, w, m, k_keep;
  double theta, scale;
  void* stream;
  int32_t rc, stage = 0;

  // Whether buffer i can be written as contiguous elements of that type (any type for a workspace, whose bytes are counted).
  bool writable(int i, at::ScalarType type) {
    if (t[i].scalar_type() == type && t[i].device() == q.device() && t[i].is_contiguous()) return true;
    rc = BAD_BUFFER; stage = i;
    return false;
  }
  // Buffer i is about to be dropped.  Its memory belongs to the stream it was made on; the calls that used it may have been on the present
  // one, and it is not given out again before that has come here.
  void let_go(int i) {
    if (t[i].is_cuda()) t[i].record_stream(c10::impl::VirtualGuardImpl(t[i].device().type()).getStream(t[i].device()));
  }
  // Buffer i of these sizes.  One that is there may be of an earlier call with other sizes: it serves as it is, or through a view of its
  // first elements where it has enough, and is replaced where it has not.  False: one that cannot be written.
  bool make(int i, at::IntArrayRef sizes, at::ScalarType type) {
    if (t[i].defined()) {
      if (i == O && t[i].sizes().equals(sizes) && t[i].scalar_type() == type && t[i].device() == q.device()) return true;   // any strides
      if (!writable(i, type)) return false;
      if (t[i].sizes().equals(sizes)) return true;
      int64_t n = 1;
      for (int64_t s : sizes) n *= s;
      if (n >= 0 && t[i].numel() >= n) {
        t[i] = t[i].view(-1).narrow(0, 0, n).view(sizes);
        made[i] = true;
        return true;
      }
      let_go(i);
    }
    t[i] = at::empty(sizes, at::TensorOptions().dtype(type).device(q.device()));
    return made[i] = true;
  }
  void operator()();
};

void Call::operator()() {
  // The launches go by q's sizes alone: keys and values of others would be read out of range.
  for (const at::Tensor* x : {&q, &k, &v})
    if (x->scalar_type() != at::kBFloat16 || x->device() != q.device()) { rc = BAD_INPUT; return; }
  for (const at::Tensor* x : {&k, &v})                             // (chunks beyond the queries' are not looked at)
    if (x->dim() != 4 || x->size(0) < C || x->size(1) != L || x->size(2) != Hkv || x->size(3) != d) { rc = BAD_INPUT; return; }
  if (has_given && given.device() != q.device()) { rc = BAD_INPUT; return; }
  const int64_t mk = m * k_keep;
  if (has_given) t[SCORE] = given;
  if (!(make(O, q.sizes(), at::kBFloat16) && make(K_ROT, k.sizes(), at::kBFloat16) && make(WIN_SCORE, {C, Hkv, L}, at::kFloat) &&
        make(WIN_LSE, {C, Hq, w}, at::kFloat) && (has_given || make(SCORE, {C}, at::kFloat)) && make(KEPT, {m}, at::kInt) &&
        make(IDX, {m, Hkv, k_keep}, at::kInt) && make(KC, {Hkv, mk, d}, at::kBFloat16) && make(VC, {Hkv, mk, d}, at::kBFloat16) &&
        make(POS, {Hkv, mk}, at::kInt) && make(FG, {1, w, Hq, d}, at::kBFloat16)))
    return;
  const bool clear = !t[STATUS].defined() || t[STATUS].numel() < 1;
  if (!make(STATUS, {1}, at::kInt)) return;

  pc_prefill_desc desc;
  desc.C = (int32_t)C; desc.L = (int32_t)L; desc.w = (int32_t)w; desc.Hq = (int32_t)Hq; desc.Hkv = (int32_t)Hkv; desc.d = (int32_t)d;
  desc.rope_theta = (float)theta;
  desc.softmax_scale = (float)scale;
  const at::Tensor* const in[4] = {&q, &k, &v, &t[O]};
  int64_t* const strides[4] = {desc.q_stride, desc.k_stride, desc.v_stride, desc.o_stride};
  for (int i = 0; i < 4; ++i) {
    TORCH_CHECK_INDEX(in[i]->dim() == 4, "tuple index out of range");
    if (in[i]->stride(3) != 1) { rc = NOT_INNERMOST; return; }
    for (int j = 0; j < 3; ++j) strides[i][j] = in[i]->stride(j);
  }
  for (int i : {WS_PREFILL, WS_PAR})
    if (t[i].defined() && !writable(i, t[i].scalar_type())) return;
  size_t need_par = 0;
  const size_t need = ws_bytes(&desc, (int32_t)m, (int32_t)k_keep, &need_par);
  auto scratch = [&](size_t bytes) { return at::empty({(int64_t)std::max<size_t>(bytes, 16)}, at::TensorOptions().dtype(at::kByte).device(q.device())); };
  if (!t[WS_PREFILL].defined() || (size_t)t[WS_PREFILL].numel() < need) {      // 0: a bad argument, which the call below names
    if (t[WS_PREFILL].defined()) let_go(WS_PREFILL);
    t[WS_PREFILL] = scratch(std::max(need, need_par));
    made[WS_PREFILL] = true;
  }
  if (!t[WS_PAR].defined() || (size_t)t[WS_PAR].numel() < need_par) {          // (the prefill is done with its own by then)
    if (t[WS_PAR].defined()) let_go(WS_PAR);
    t[WS_PAR] = (size_t)t[WS_PREFILL].numel() >= need_par ? t[WS_PREFILL] : scratch(need_par);
    made[WS_PAR] = true;
  }
  if (!t[K_ROT].is_contiguous() || !v.is_contiguous()) { rc = NOT_CONTIGUOUS; return; }
  // the window is the same in every chunk: take it from chunk 0
  at::Tensor window;
  const char* q_win = static_cast<const char*>(q.data_ptr()) + (L - w) * Hq * d * 2;
  if (!q.is_contiguous()) {
    window = q.as_strided({1, w, Hq, d}, q.strides(), q.storage_offset() + (L - w) * q.stride(1)).contiguous();
    q_win = static_cast<const char*>(window.data_ptr());
  }
  pc_hot_path_args a;
  a.q = q.data_ptr(); a.k = k.data_ptr(); a.v = v.data_ptr(); a.q_win = q_win;
  a.o = t[O].data_ptr(); a.k_rot = t[K_ROT].data_ptr();
  a.win_score = static_cast<float*>(t[WIN_SCORE].data_ptr()); a.win_lse = static_cast<float*>(t[WIN_LSE].data_ptr());
  a.given_score = has_given ? static_cast<const float*>(given.data_ptr()) : nullptr;
  a.chunk_score = static_cast<float*>(t[SCORE].data_ptr());
  a.kept = static_cast<int32_t*>(t[KEPT].data_ptr()); a.idx = static_cast<int32_t*>(t[IDX].data_ptr());
  a.kc = t[KC].data_ptr(); a.vc = t[VC].data_ptr(); a.pos = static_cast<int32_t*>(t[POS].data_ptr()); a.fg = t[FG].data_ptr();
  a.status_word = static_cast<int32_t*>(t[STATUS].data_ptr());
  a.ws_prefill = t[WS_PREFILL].data_ptr(); a.ws_prefill_bytes = (size_t)t[WS_PREFILL].numel();
  a.ws_parallel = t[WS_PAR].data_ptr(); a.ws_parallel_bytes = (size_t)t[WS_PAR].numel();
  a.m = (int32_t)m; a.k_keep = (int32_t)k_keep; a.n_score = (int32_t)t[SCORE].numel(); a.clear_status = clear;
  rc = run(&desc, &a, &stage, stream);
}

// hot_path(ws_bytes, run, stream, q, k, v, chunk_score or None, buffers, (C, L, Hq, Hkv, d, w, m, k_keep), rope_theta, softmax_scale)
// -> (result code, stage, buffers): those given, or new ones in the place of None and of those that are too small
PyObject* hot_path(PyObject*, PyObject* args) {
  HANDLE_TH_ERRORS
  unsigned long long ws_bytes, run, stream;
  PyObject *in[3], *given, *buffers;
  Call c;
  if (!PyArg_ParseTuple(args, "KKKOOOOO!(LLLLLLLL)dd", &ws_bytes, &run, &stream, &in[0], &in[1], &in[2], &given, &PyTuple_Type, &buffers, &c.C,
                        &c.L, &c.Hq, &c.Hkv, &c.d, &c.w, &c.m, &c.k_keep, &c.theta, &c.scale))
    return nullptr;
  if (PyTuple_GET_SIZE(buffers) != N_BUFFERS) { PyErr_SetString(PyExc_TypeError, "hot_path: wrong number of buffers"); return nullptr; }
  c.ws_bytes = reinterpret_cast<ws_bytes_fn>(static_cast<uintptr_t>(ws_bytes));
  c.run = reinterpret_cast<hot_path_fn>(static_cast<uintptr_t>(run));
  c.stream = reinterpret_cast<void*>(static_cast<uintptr_t>(stream));
  auto tensor = [](PyObject* p, at::Tensor& t) {
    if (p == Py_None) return true;
    if (!THPVariable_Check(p)) { PyErr_SetString(PyExc_TypeError, "hot_path: expected a tensor"); return false; }
    t = THPVariable_Unpack(p);
    return true;
  };
  if (!tensor(in[0], c.q) || !tensor(in[1], c.k) || !tensor(in[2], c.v) || !tensor(given, c.given)) return nullptr;
  c.has_given = given != Py_None;
  for (int i = 0; i < N_BUFFERS; ++i)
    if (!tensor(PyTuple_GET_ITEM(buffers, i), c.t[i])) return nullptr;
  {
    pybind11::gil_scoped_release release;
    c();
  }
  PyObject* const out = PyTuple_New(N_BUFFERS);
  if (out == nullptr) return nullptr;
  PyObject* ws_prefill = nullptr;
  for (int i = 0; i < N_BUFFERS; ++i) {
    PyObject* p = PyTuple_GET_ITEM(buffers, i);
    if (i == SCORE && c.has_given) p = given;
    else if (i == WS_PAR && c.made[i] && c.t[i].is_same(c.t[WS_PREFILL])) p = ws_prefill;
    else if (c.made[i]) p = nullptr;
    if (p != nullptr) Py_INCREF(p);
    else p = c.t[i].defined() ? THPVariable_Wrap(c.t[i]) : (Py_INCREF(Py_None), Py_None);
    if (p == nullptr) { Py_DECREF(out); return nullptr; }
    if (i == WS_PREFILL) ws_prefill = p;
    PyTuple_SET_ITEM(out, i, p);
  }
  return Py_BuildValue("iiN", (int)c.rc, (int)c.stage, out);
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"hot_path", hot_path, METH_VARARGS, "See binding.py."}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_pc_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pc_host() { return PyModule_Create(&module_def); }
