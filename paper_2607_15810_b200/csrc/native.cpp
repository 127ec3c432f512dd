// The binding's ordinary calls as native functions: what a call needs from its tensors is read and its outputs are allocated
// here, without a Python object per step.  A call that spends 2 to 10 us in kernels took 10 to 18 us of host time through
// ctypes and torch.empty (about 1 us per output and 2 to 3 us of argument conversion).  In a loop, us per call, ctypes / so:
// quantizer 64 x 1024 14.1 / 8.4, with a given scale 11.8 / 6.1; one-sided 64 x 512 -> 512 W16A16 10.0 / 6.7, W16A4 14.6 / 11.4;
// dense 16 x 512 -> 512 11.1 / 7.9; host time of a MoE layer's call at one token 16.4 / 12.7.
//
// Every function takes the arguments of the binding's function of that name and returns what it returns, or None for
// arguments that it does not know (tensor subclasses, other types and ranks), which the binding then handles itself.
// The library's status becomes the binding's QuadsError.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/quads.h"

namespace {

// The torch and Python whose inline code this object holds; the binding looks for it in the file before it loads it.
__attribute__((used)) const char g_tag[] = "built for " QUADS_NATIVE_TAG;

PyObject* g_error = nullptr;                               // the binding's exception class
PyObject *s_q, *s_sf, *s_gs, *s_atoms, *s_out, *s_workspace;

// A plain tensor on a CUDA device, or null.
const at::Tensor* cuda_tensor(PyObject* o) {
  if (!o || !THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.is_cuda() ? &t : nullptr;
}
// The same, or None (`*t` = null).  False: neither.
bool cuda_tensor_or_none(PyObject* o, const at::Tensor** t) {
  *t = nullptr;
  if (o == Py_None) return true;
  *t = cuda_tensor(o);
  return *t != nullptr;
}
const at::Tensor* entry(PyObject* dict, PyObject* key) { return PyDict_CheckExact(dict) ? cuda_tensor(PyDict_GetItem(dict, key)) : nullptr; }
bool small_int(PyObject* o, int32_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  const long long x = PyLong_AsLongLongAndOverflow(o, &over);
  if (over || x > INT32_MAX || x < INT32_MIN) return false;
  *v = (int32_t)x;
  return true;
}
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
at::Tensor alloc(at::IntArrayRef sizes, const at::Tensor& like, at::ScalarType type) {
  return at::empty(sizes, at::TensorOptions().dtype(type).device(like.device()));
}
at::Tensor alloc_workspace(size_t bytes, const at::Tensor& like) { return alloc({(int64_t)std::max<size_t>(bytes, 256)}, like, at::kByte); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Null, with the binding's exception set, unless `s` is QUADS_OK.
bool passed(quads_status s) {
  if (s == QUADS_OK) return true;
  PyObject* e = PyObject_CallFunction(g_error, "i", (int)s);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  return false;
}
template <typename F>
quads_status unlocked(F f) {
  quads_status s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return s;
}
PyObject* out_and_workspace(PyObject* out, PyObject* ws) {             // takes both references
  PyObject* d = out && ws ? PyDict_New() : nullptr;
  if (d && (PyDict_SetItem(d, s_out, out) < 0 || PyDict_SetItem(d, s_workspace, ws) < 0)) Py_CLEAR(d);
  Py_XDECREF(out);
  Py_XDECREF(ws);
  return d;
}
PyObject* wrapped(const at::Tensor& made, PyObject* given) {           // a new reference to the caller's object, or to a new one
  if (given != Py_None) return Py_NewRef(given);
  return THPVariable_Wrap(made);
}

// (x, gs, sf_layout, out, workspace) -> (q, sf, gs)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  int32_t layout;
  const at::Tensor *x, *gs, *ws, *given[3];
  if (n != 5 || !(x = cuda_tensor(a[0])) || !cuda_tensor_or_none(a[1], &gs) || !small_int(a[2], &layout) || !cuda_tensor_or_none(a[4], &ws))
    Py_RETURN_NONE;
  if (x->scalar_type() != at::kBFloat16 || x->dim() != 2 || x->stride(1) != 1 || (layout != QUADS_SF_LINEAR && layout != QUADS_SF_TILED))
    Py_RETURN_NONE;
  const int64_t rows = x->size(0), K = x->size(1);
  at::Tensor made[3], made_ws;
  if (a[3] == Py_None) {
    made[0] = alloc({rows, K / 2}, *x, at::kByte);
    made[1] = layout == QUADS_SF_LINEAR ? alloc({rows, K / 16}, *x, at::kByte) : alloc({(int64_t)quads_sf_tiled_bytes(rows, K)}, *x, at::kByte);
    made[2] = alloc({1}, *x, at::kFloat);
    for (int i = 0; i < 3; ++i) given[i] = &made[i];
  } else {
    if (!PyTuple_CheckExact(a[3]) || PyTuple_GET_SIZE(a[3]) != 3) Py_RETURN_NONE;
    for (int i = 0; i < 3; ++i)
      if (!(given[i] = cuda_tensor(PyTuple_GET_ITEM(a[3], i)))) Py_RETURN_NONE;
  }
  if (!ws) { made_ws = alloc_workspace(quads_quantize_workspace_bytes(), *x); ws = &made_ws; }
  const int64_t ld = rows > 1 ? x->stride(0) : std::max(K, x->stride(0));
  uint8_t *q = (uint8_t*)ptr(given[0]), *sf = (uint8_t*)ptr(given[1]);
  float* g = (float*)ptr(given[2]);
  const void *xp = ptr(x), *gp = ptr(gs);
  void *wp = ptr(ws), *st = stream();
  if (!passed(unlocked([&] { return quads_quantize_nvfp4(xp, rows, K, ld, (const float*)gp, q, sf, g, layout, wp, (size_t)ws->numel(), st); })))
    return nullptr;
  PyObject* r = PyTuple_New(3);
  for (int i = 0; r && i < 3; ++i) {
    PyObject* o = a[3] == Py_None ? THPVariable_Wrap(made[i]) : Py_NewRef(PyTuple_GET_ITEM(a[3], i));
    if (!o) Py_CLEAR(r);
    else PyTuple_SET_ITEM(r, i, o);
  }
  return r;
  END_HANDLE_TH_ERRORS
}

// One dense projection; the arguments of the tensors are in `m` already.
PyObject* run_dense(quads_moe_args& m, const at::Tensor& x, PyObject* ws_obj, const at::Tensor* ws) {
  at::Tensor out = alloc({m.T, m.N}, x, at::kBFloat16), made_ws;
  if (!ws) { made_ws = alloc_workspace(quads_moe_workspace_bytes(m.T, m.H, 0, 1, 1, m.N), x); ws = &made_ws; }
  m.out = out.data_ptr();
  m.workspace = ptr(ws);
  m.workspace_bytes = (size_t)ws->numel();
  void* st = stream();
  if (!passed(unlocked([&] { return quads_moe_w4a4_rac(&m, st); }))) return nullptr;
  return out_and_workspace(THPVariable_Wrap(out), wrapped(made_ws, ws_obj));
}
bool rows_and_width(const at::Tensor& x, quads_moe_args* m) {
  if (x.dim() != 2 || x.size(0) > INT32_MAX || x.size(1) > INT32_MAX) return false;
  m->T = (int32_t)x.size(0);
  m->H = (int32_t)x.size(1);
  m->x = x.data_ptr();
  return true;
}
bool dense_weight(PyObject* w, quads_moe_args* m) {
  const at::Tensor *q = entry(w, s_q), *sf = entry(w, s_sf), *gs = entry(w, s_gs);
  if (!q || !sf || !gs || q->dim() < 2 || q->size(-2) > INT32_MAX) return false;
  m->w13_q = (const uint8_t*)ptr(q); m->w13_sf = (const uint8_t*)ptr(sf); m->w13_gs = (const float*)ptr(gs);
  m->N = (int32_t)q->size(-2);
  return true;
}

// (x, w, nsel, a_gs, workspace) -> dict(out, workspace)
PyObject* dense(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  quads_moe_args m{};
  const at::Tensor *x, *gs, *ws;
  if (n != 5 || !(x = cuda_tensor(a[0])) || !small_int(a[2], &m.rac_nsel_13) || !cuda_tensor_or_none(a[3], &gs) || !cuda_tensor_or_none(a[4], &ws) ||
      !rows_and_width(*x, &m) || !dense_weight(a[1], &m))
    Py_RETURN_NONE;
  m.E = m.topk = 1;
  m.a13_gs = (const float*)ptr(gs);
  return run_dense(m, *x, a[4], ws);
  END_HANDLE_TH_ERRORS
}

// (x, mode, w, w_bf16, a_gs, workspace) -> dict(out, workspace)
PyObject* one_sided(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  quads_moe_args m{};
  const at::Tensor *x, *gs, *ws;
  if (n != 6 || !(x = cuda_tensor(a[0])) || !small_int(a[1], &m.operand_mode) || !cuda_tensor_or_none(a[4], &gs) || !cuda_tensor_or_none(a[5], &ws) ||
      !rows_and_width(*x, &m))
    Py_RETURN_NONE;
  if (m.operand_mode == QUADS_W4A16) {
    if (!dense_weight(a[2], &m)) Py_RETURN_NONE;
  } else if (m.operand_mode == QUADS_W16A4 || m.operand_mode == QUADS_W16A16) {
    const at::Tensor* w = cuda_tensor(a[3]);
    if (!w || w->dim() < 1 || w->size(0) > INT32_MAX) Py_RETURN_NONE;
    m.N = (int32_t)w->size(0);
    m.w13_bf16 = ptr(w);
    if (m.operand_mode == QUADS_W16A4) m.a13_gs = (const float*)ptr(gs);
  } else {
    Py_RETURN_NONE;
  }
  m.E = m.topk = 1;
  return run_dense(m, *x, a[5], ws);
  END_HANDLE_TH_ERRORS
}

// (x, logits, w13, w2, topk, nsel13, nsel2, a2_gs, a13_gs, renormalize, workspace, out) -> dict(out, workspace)
PyObject* moe(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  quads_moe_args m{};
  const at::Tensor *x, *lg, *a2, *a13, *ws, *out;
  if (n != 12 || !(x = cuda_tensor(a[0])) || !(lg = cuda_tensor(a[1])) || !small_int(a[4], &m.topk) || !small_int(a[5], &m.rac_nsel_13) ||
      !small_int(a[6], &m.rac_nsel_2) || !cuda_tensor_or_none(a[7], &a2) || !cuda_tensor_or_none(a[8], &a13) || !cuda_tensor_or_none(a[10], &ws) ||
      !cuda_tensor_or_none(a[11], &out) || !rows_and_width(*x, &m) || lg->dim() < 2 || lg->size(1) > INT32_MAX)
    Py_RETURN_NONE;
  const at::Tensor *q1 = entry(a[2], s_q), *f1 = entry(a[2], s_sf), *g1 = entry(a[2], s_gs);
  const at::Tensor *q2 = entry(a[3], s_q), *f2 = entry(a[3], s_sf), *g2 = entry(a[3], s_gs);
  if (!q1 || !f1 || !g1 || !q2 || !f2 || !g2 || q2->dim() < 3 || q2->size(2) > INT32_MAX / 2) Py_RETURN_NONE;
  const int renorm = PyObject_IsTrue(a[9]);
  if (renorm < 0) return nullptr;
  m.E = (int32_t)lg->size(1);
  m.I = (int32_t)q2->size(2) * 2;
  m.router_logits = (const float*)ptr(lg);
  m.w13_q = (const uint8_t*)ptr(q1); m.w13_sf = (const uint8_t*)ptr(f1); m.w13_gs = (const float*)ptr(g1);
  m.w2_q = (const uint8_t*)ptr(q2); m.w2_sf = (const uint8_t*)ptr(f2); m.w2_gs = (const float*)ptr(g2);
  m.a13_gs = (const float*)ptr(a13); m.a2_gs = (const float*)ptr(a2);
  m.renormalize = renorm;
  at::Tensor made_out, made_ws;
  if (!out) { made_out = alloc({m.T, m.H}, *x, at::kBFloat16); out = &made_out; }
  if (!ws) { made_ws = alloc_workspace(quads_moe_workspace_bytes(m.T, m.H, m.I, m.E, m.topk, 0), *x); ws = &made_ws; }
  m.out = ptr(out);
  m.workspace = ptr(ws);
  m.workspace_bytes = (size_t)ws->numel();
  void* st = stream();
  if (!passed(unlocked([&] { return quads_moe_w4a4_rac(&m, st); }))) return nullptr;
  return out_and_workspace(wrapped(made_out, a[11]), wrapped(made_ws, a[10]));
  END_HANDLE_TH_ERRORS
}

// (x, logits, w13, w2, topk, renormalize, workspace, out) -> dict(out, workspace)
PyObject* moe_fp8(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  quads_moe_fp8_args m{};
  const at::Tensor *x, *lg, *ws, *out;
  if (n != 8 || !(x = cuda_tensor(a[0])) || !(lg = cuda_tensor(a[1])) || !small_int(a[4], &m.topk) || !cuda_tensor_or_none(a[6], &ws) ||
      !cuda_tensor_or_none(a[7], &out) || x->dim() != 2 || x->size(0) > INT32_MAX || x->size(1) > INT32_MAX || lg->dim() < 2 ||
      lg->size(1) > INT32_MAX)
    Py_RETURN_NONE;
  const at::Tensor *q1 = entry(a[2], s_q), *t1 = entry(a[2], s_atoms), *q2 = entry(a[3], s_q), *t2 = entry(a[3], s_atoms);
  if (!q1 || !t1 || !q2 || !t2 || q2->dim() < 3 || q2->size(2) > INT32_MAX) Py_RETURN_NONE;
  const int renorm = PyObject_IsTrue(a[5]);
  if (renorm < 0) return nullptr;
  m.T = (int32_t)x->size(0); m.H = (int32_t)x->size(1); m.I = (int32_t)q2->size(2); m.E = (int32_t)lg->size(1);
  m.x = ptr(x);
  m.router_logits = (const float*)ptr(lg);
  m.w13_q = (const uint8_t*)ptr(q1); m.w13_atoms = (const uint8_t*)ptr(t1);
  m.w2_q = (const uint8_t*)ptr(q2); m.w2_atoms = (const uint8_t*)ptr(t2);
  m.renormalize = renorm;
  at::Tensor made_out, made_ws;
  if (!out) { made_out = alloc({m.T, m.H}, *x, at::kBFloat16); out = &made_out; }
  if (!ws) { made_ws = alloc_workspace(quads_moe_fp8_workspace_bytes(m.T, m.H, m.I, m.E, m.topk), *x); ws = &made_ws; }
  m.out = ptr(out);
  m.workspace = ptr(ws);
  m.workspace_bytes = (size_t)ws->numel();
  void* st = stream();
  if (!passed(unlocked([&] { return quads_moe_fp8_w8a8(&m, st); }))) return nullptr;
  return out_and_workspace(wrapped(made_out, a[7]), wrapped(made_ws, a[6]));
  END_HANDLE_TH_ERRORS
}

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_XSETREF(g_error, Py_NewRef(cls));
  Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"set_error", set_error, METH_O, "The exception class raised for a status other than QUADS_OK."},
    {"quantize_nvfp4", (PyCFunction)(void (*)(void))quantize, METH_FASTCALL, nullptr},
    {"dense_w4a4_rac", (PyCFunction)(void (*)(void))dense, METH_FASTCALL, nullptr},
    {"dense_one_sided", (PyCFunction)(void (*)(void))one_sided, METH_FASTCALL, nullptr},
    {"moe_w4a4_rac", (PyCFunction)(void (*)(void))moe, METH_FASTCALL, nullptr},
    {"moe_fp8_w8a8", (PyCFunction)(void (*)(void))moe_fp8, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  s_q = PyUnicode_InternFromString("q"); s_sf = PyUnicode_InternFromString("sf"); s_gs = PyUnicode_InternFromString("gs");
  s_atoms = PyUnicode_InternFromString("atoms"); s_out = PyUnicode_InternFromString("out");
  s_workspace = PyUnicode_InternFromString("workspace");
  if (!s_q || !s_sf || !s_gs || !s_atoms || !s_out || !s_workspace) return nullptr;
  return PyModule_Create(&g_module);
}
