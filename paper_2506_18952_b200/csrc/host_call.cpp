// The host side of a call on torch tensors, in native code: reads the tensors, fills hola_verify_args and calls the C ABI;
// makes the output tensors of a call that is given none.  What a call costs the host bounds small problems.  us, Python -> native:
// arguments filled and a call that is refused 3.5 -> 0.8, five output tensors 8.2 -> 5.1, seven 11.7 -> 7.0, beside 5 for the two
// launches; whole calls: one sequence, V = 1000 10.45 -> 9.75; three, V = 5000, fresh outputs 19.75 -> 13.2; host entry, two sequences,
// V = 10000 42.1 -> 37.4; mixed-width quantiser, 1000 x 128 50 -> 13.8.
//
// call() takes the plain forms only (torch.Tensor or Parameter objects with storage, strided, contiguous, of the types that
// the entry points know) and answers None for everything else, before it has done anything: the caller then goes the long
// way through Python, which also words the errors.
#include <Python.h>

#include <vector>

#include <ATen/ops/empty.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/hola_verify.h"

namespace {

typedef hola_status (*EntryFn)(hola_ctx*, const hola_verify_args*, void*);

// A tensor whose memory can be handed over as it is: null for anything else.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || t.layout() != at::kStrided || !t.has_storage() || t.unsafeGetTensorImpl()->is_python_dispatch() ||
      t.unsafeGetTensorImpl()->has_symbolic_sizes_strides())
    return nullptr;
  return &t;
}

// Pointer of an optional input (None: null).  False: not a form that is handled here.
bool input(PyObject* o, void** ptr, const at::Tensor** t = nullptr) {
  if (o == Py_None) return true;
  const at::Tensor* x = plain(o);
  if (!x || !x->is_contiguous()) return false;
  *ptr = x->data_ptr();
  if (t) *t = x;
  return true;
}

// Pointer of an output attribute (None: null; the library refuses it where it needs it).
bool output(PyObject* out, PyObject* name, void** ptr) {
  PyObject* o = PyObject_GetAttr(out, name);
  if (!o) { PyErr_Clear(); return false; }
  bool ok = true;
  if (o != Py_None) {
    const at::Tensor* x = plain(o);
    if (x) *ptr = x->data_ptr();
    else ok = false;
  }
  Py_DECREF(o);                                          // (the outputs object holds it)
  return ok;
}

bool integer(PyObject* o, long long* v) {
  if (!PyLong_CheckExact(o)) return false;
  *v = PyLong_AsLongLong(o);
  if (*v == -1 && PyErr_Occurred()) { PyErr_Clear(); return false; }
  return true;
}
bool int32(PyObject* o, int32_t* v) {
  long long x = 0;
  if (!integer(o, &x) || x < INT32_MIN || x > INT32_MAX) return false;
  *v = static_cast<int32_t>(x);
  return true;
}
bool address(PyObject* o, void** p) {
  if (!PyLong_CheckExact(o)) return false;
  *p = PyLong_AsVoidPtr(o);
  if (!*p && PyErr_Occurred()) { PyErr_Clear(); return false; }
  return true;
}

PyObject *n_accept, *n_next, *n_entropy, *n_logZ, *n_logits, *n_status, *n_dent;

// call(function, ctx, H, V, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, draws, flags, gate_source, fallback, w_scale,
//      a8, wmix, stream) -> status, or None where the caller has to go the long way.  wmix: address of the hola_wmix of a head of
// mixed widths, whose first buffer is W_lm then, or 0.
PyObject* call(PyObject*, PyObject* const* v, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 19) { PyErr_SetString(PyExc_TypeError, "call() takes 19 arguments"); return nullptr; }
  void *fn = nullptr, *ctx = nullptr, *stream = nullptr, *wmix = nullptr, *p = nullptr;
  hola_verify_args a = {};
  int32_t H = 0, V = 0, draws = 0;
  if (!address(v[0], &fn) || !fn || !address(v[1], &ctx) || !ctx || !int32(v[2], &H) || !int32(v[3], &V) ||
      !int32(v[11], &draws) || !int32(v[12], &a.flags) || !int32(v[13], &a.gate_source) || !int32(v[14], &a.fallback) ||
      !address(v[17], &wmix) || !address(v[18], &stream))
    Py_RETURN_NONE;
  const at::Tensor *hidden = nullptr, *W = nullptr, *q = nullptr, *scale = nullptr;
  void *ph = nullptr, *pw = nullptr, *pt = nullptr, *pq = nullptr, *pu = nullptr;
  if (!input(v[4], &ph, &hidden) || !hidden || !input(v[5], &pw, &W) || !W || !input(v[6], &pt) || !input(v[7], &pq, &q) ||
      !input(v[8], &pu))
    Py_RETURN_NONE;
  if (v[15] != Py_None) {
    scale = plain(v[15]);
    if (!scale) Py_RETURN_NONE;
  }
  const bool w8 = !wmix && W->scalar_type() == at::kChar;
  if (hidden->dim() < 2 || hidden->size(0) > INT32_MAX || hidden->size(1) > INT32_MAX || hidden->scalar_type() != at::kBFloat16 ||
      (!wmix && !w8 && W->scalar_type() != at::kBFloat16) || (w8 || wmix) != (scale != nullptr) ||
      (q && q->scalar_type() != at::kBFloat16 && q->scalar_type() != at::kFloat))
    Py_RETURN_NONE;
  if (w8) {
    if (v[16] == Py_False) a.w_dtype = HOLA_W_INT8;
    else if (v[16] == Py_True) a.w_dtype = HOLA_W8A8;
    else if (PyUnicode_CheckExact(v[16]) && PyUnicode_CompareWithASCIIString(v[16], "a16") == 0) a.w_dtype = HOLA_W8A16;
    else Py_RETURN_NONE;
    a.w_scale = static_cast<const float*>(scale->data_ptr());
  } else if (v[16] != Py_False) {
    Py_RETURN_NONE;
  } else if (wmix) {
    a.w_dtype = HOLA_W_MIXED;
    a.wmix = static_cast<const hola_wmix*>(wmix);
    a.w_scale = static_cast<const float*>(scale->data_ptr());
    pw = nullptr;
  }
  long long whole = 0;
  if (PyFloat_CheckExact(v[9])) a.tau = static_cast<float>(PyFloat_AS_DOUBLE(v[9]));
  else if (integer(v[9], &whole)) a.tau = static_cast<float>(static_cast<double>(whole));
  else Py_RETURN_NONE;
  a.B = static_cast<int32_t>(hidden->size(0));
  a.k = static_cast<int32_t>(hidden->size(1)) - 1;
  a.H = H; a.V = V;
  a.hidden = ph; a.W_lm = pw;
  if (a.k > 0) { a.draft_tok = static_cast<const int32_t*>(pt); a.draft_q = pq; }
  a.q_dtype = q && q->scalar_type() == at::kFloat ? HOLA_Q_F32 : HOLA_Q_BF16;
  a.uniforms = static_cast<const float*>(pu);
  PyObject* out = v[10];
  if (draws) {
    p = nullptr; if (!output(out, n_accept, &p)) Py_RETURN_NONE;
    a.accept_len = static_cast<int32_t*>(p);
    p = nullptr; if (!output(out, n_next, &p)) Py_RETURN_NONE;
    a.next_tok = static_cast<int32_t*>(p);
  }
  p = nullptr; if (!output(out, n_entropy, &p)) Py_RETURN_NONE;
  a.entropy = static_cast<float*>(p);
  p = nullptr; if (!output(out, n_logZ, &p)) Py_RETURN_NONE;
  a.logZ = static_cast<float*>(p);
  p = nullptr; if (!output(out, n_logits, &p)) Py_RETURN_NONE;
  a.logits_out = static_cast<float*>(p);
  p = nullptr; if (!output(out, n_status, &p)) Py_RETURN_NONE;
  a.status_word = static_cast<uint32_t*>(p);
  if (a.gate_source == HOLA_GATE_DRAFT_ENTROPY) {
    p = nullptr; if (!output(out, n_dent, &p)) Py_RETURN_NONE;
    a.draft_entropy = static_cast<float*>(p);
  }
  hola_status s;
  Py_BEGIN_ALLOW_THREADS
  s = reinterpret_cast<EntryFn>(fn)(static_cast<hola_ctx*>(ctx), &a, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
  END_HANDLE_TH_ERRORS
}

// outputs(out, device index, B, k1, V, logits wanted, draws, draft gate): the tensors that such a call fills, as attributes.
PyObject* outputs(PyObject*, PyObject* const* v, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  long long x[7];
  if (n != 8) { PyErr_SetString(PyExc_TypeError, "outputs() takes 8 arguments"); return nullptr; }
  for (int i = 0; i < 7; ++i) {                          // (what is wanted: any object, by its truth value)
    x[i] = i < 4 ? PyLong_AsLongLong(v[1 + i]) : PyObject_IsTrue(v[1 + i]);
    if (x[i] == -1 && PyErr_Occurred()) return nullptr;
  }
  const long long B = x[1], k1 = x[2], V = x[3];
  at::Tensor entropy, logZ, logits, status, accept, next, dent;
  Py_BEGIN_ALLOW_THREADS                                 // (an allocation may wait for the device, or call back)
  try {
    const auto f32 = at::TensorOptions().dtype(at::kFloat).device(at::Device(at::kCUDA, static_cast<c10::DeviceIndex>(x[0])));
    const auto i32 = f32.dtype(at::kInt);
    entropy = at::empty({B, k1}, f32);
    logZ = at::empty({B, k1}, f32);
    if (x[4]) logits = at::empty({B, k1, V}, f32);
    status = at::empty({1}, i32);
    if (x[5]) { accept = at::empty({B}, i32); next = at::empty({B}, i32); }
    if (x[6]) dent = at::empty({B, k1 - 1}, f32);
  } catch (...) {
    Py_BLOCK_THREADS
    throw;
  }
  Py_END_ALLOW_THREADS
  auto put = [&](PyObject* name, const at::Tensor& t) {
    PyObject* o = t.defined() ? THPVariable_Wrap(t) : Py_NewRef(Py_None);
    if (!o) return false;
    const int r = PyObject_SetAttr(v[0], name, o);
    Py_DECREF(o);
    return r == 0;
  };
  if (!put(n_entropy, entropy) || !put(n_logZ, logZ) || !put(n_logits, logits) || !put(n_status, status)) return nullptr;
  if (x[5] && (!put(n_accept, accept) || !put(n_next, next))) return nullptr;
  if (x[6] && !put(n_dent, dent)) return nullptr;
  Py_RETURN_NONE;
  END_HANDLE_TH_ERRORS
}

// quantize(function, W_lm, widths, struct, current device, stream) -> (status, V, H, widths, W16, W8, W4, shift4, w_scale,
// group_width, group_row), or None where the caller has to go the long way.  `struct`: a writable hola_wmix.
PyObject* quantize(PyObject*, PyObject* const* v, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6) { PyErr_SetString(PyExc_TypeError, "quantize() takes 6 arguments"); return nullptr; }
  void *fn = nullptr, *stream = nullptr;
  int32_t device = 0;
  if (!address(v[0], &fn) || !fn || !int32(v[4], &device) || !address(v[5], &stream)) Py_RETURN_NONE;
  const at::Tensor* W = plain(v[1]);
  if (!W || !W->is_cuda() || W->get_device() != device || W->dim() != 2 || W->scalar_type() != at::kBFloat16 || !W->is_contiguous())
    Py_RETURN_NONE;
  const int64_t V = W->size(0), H = W->size(1), groups = (V + 255) / 256;
  const bool list = PyList_CheckExact(v[2]);
  if (V <= 0 || groups > 2048 || H % 128 != 0 || H > INT32_MAX || (!list && !PyTuple_CheckExact(v[2])) ||
      (list ? PyList_GET_SIZE(v[2]) : PyTuple_GET_SIZE(v[2])) != groups)
    Py_RETURN_NONE;
  std::vector<uint8_t> widths(static_cast<size_t>(groups));
  int64_t rows[17] = {};
  for (int64_t g = 0; g < groups; ++g) {
    long long w = 0;
    if (!integer(list ? PyList_GET_ITEM(v[2], g) : PyTuple_GET_ITEM(v[2], g), &w) || (w != 4 && w != 8 && w != 16)) Py_RETURN_NONE;
    widths[g] = static_cast<uint8_t>(w);
    rows[w] += g + 1 < groups ? 256 : V - 256 * g;
  }
  Py_buffer buf;
  if (PyObject_GetBuffer(v[3], &buf, PyBUF_WRITABLE) != 0) { PyErr_Clear(); Py_RETURN_NONE; }
  if (buf.len != static_cast<Py_ssize_t>(sizeof(hola_wmix))) { PyBuffer_Release(&buf); Py_RETURN_NONE; }
  hola_wmix* mx = static_cast<hola_wmix*>(buf.buf);
  at::Tensor W16, W8, W4, shift4, scale, group_width, group_row;
  hola_status s = HOLA_OK;
  void* src = W->data_ptr();
  Py_BEGIN_ALLOW_THREADS
  try {
    const auto u8 = at::TensorOptions().dtype(at::kByte).device(W->device());
    if (rows[16]) W16 = at::empty({rows[16], H}, u8.dtype(at::kBFloat16));
    if (rows[8]) W8 = at::empty({rows[8], H}, u8.dtype(at::kChar));
    if (rows[4]) {
      W4 = at::empty({rows[4], H / 2}, u8);
      shift4 = at::empty({H / 128, rows[4]}, u8);
    }
    scale = at::empty({V}, u8.dtype(at::kFloat));
    group_width = at::empty({groups}, u8);
    group_row = at::empty({groups}, u8.dtype(at::kInt));
    mx->W16 = rows[16] ? W16.data_ptr() : nullptr;
    mx->W8 = rows[8] ? W8.data_ptr() : nullptr;
    mx->W4 = rows[4] ? W4.data_ptr() : nullptr;
    mx->shift4 = rows[4] ? static_cast<uint8_t*>(shift4.data_ptr()) : nullptr;
    mx->group_width = static_cast<uint8_t*>(group_width.data_ptr());
    mx->group_row = static_cast<int32_t*>(group_row.data_ptr());
    mx->rows16 = static_cast<int32_t>(rows[16]); mx->rows8 = static_cast<int32_t>(rows[8]); mx->rows4 = static_cast<int32_t>(rows[4]);
    s = reinterpret_cast<hola_status (*)(const void*, int, int, const uint8_t*, const hola_wmix*, float*, void*)>(fn)(
        src, static_cast<int>(V), static_cast<int>(H), widths.data(), mx, static_cast<float*>(scale.data_ptr()), stream);
  } catch (...) {
    Py_BLOCK_THREADS
    PyBuffer_Release(&buf);
    throw;
  }
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&buf);
  PyObject* used = PyList_New(static_cast<Py_ssize_t>(groups));          // (what was used: the caller's list may be another by now)
  if (!used) return nullptr;
  for (int64_t g = 0; g < groups; ++g) {
    PyObject* w = PyLong_FromLong(widths[g]);
    if (!w) { Py_DECREF(used); return nullptr; }
    PyList_SET_ITEM(used, g, w);
  }
  auto wrap = [](const at::Tensor& t) { return t.defined() ? THPVariable_Wrap(t) : Py_NewRef(Py_None); };
  return Py_BuildValue("iLLNNNNNNNN", static_cast<int>(s), static_cast<long long>(V), static_cast<long long>(H),
                       used, wrap(W16), wrap(W8), wrap(W4), wrap(shift4), wrap(scale), wrap(group_width),
                       wrap(group_row));
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL, nullptr},
    {"outputs", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(outputs)), METH_FASTCALL, nullptr},
    {"quantize", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(quantize)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_call(void) {
  PyObject* m = PyModule_Create(&module);
  if (!m) return nullptr;
  n_accept = PyUnicode_InternFromString("accept_len"); n_next = PyUnicode_InternFromString("next_tok");
  n_entropy = PyUnicode_InternFromString("entropy"); n_logZ = PyUnicode_InternFromString("logZ");
  n_logits = PyUnicode_InternFromString("logits"); n_status = PyUnicode_InternFromString("status");
  n_dent = PyUnicode_InternFromString("draft_entropy");
  return m;
}
