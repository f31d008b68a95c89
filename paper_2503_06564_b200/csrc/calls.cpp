// The hot entry points of libtrdq.so for plain torch tensors: what trdq.py does for a call (checks, outputs, pointers, strides, current
// stream) in one native function.  A small layer is bound by this host work, not by the GPU: through ctypes a call took about 9 us,
// 2 us of it for each output, 1.5 for the conversion of the arguments and 1 for the tensors' attributes, and a linear layer of 256 x 1024
// (two calls, 7 us on the GPU) 19.3 us, now 10.3; three calls for two ragged row segments 37.4, now 22.6.
//
// Every function returns None for arguments it does not handle: tensor subclasses, tensors of other devices or layouts, wrapped tensors
// (functorch, functional, fake), numbers that are not Python ints, an active function or dispatch mode.  The caller then goes its general
// way, which also is where wrong arguments are reported.  A status other than TRDQ_OK is returned as an int.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <limits>

#include "../../include/trdq.h"

namespace {

// Addresses in the library that trdq.py has loaded.
struct Entry {
  decltype(&trdq_rotate_quantize) rotate_quantize;
  decltype(&trdq_norm_rotate_quantize) norm_rotate_quantize;
  decltype(&trdq_rotate_quantize_asym) rotate_quantize_asym;
  decltype(&trdq_linear_act) linear_act;
  decltype(&trdq_linear_cfg) linear_cfg;
  decltype(&trdq_linear_asym) linear_asym;
  decltype(&trdq_linear_splitk_workspace) splitk_workspace;
  decltype(&trdq_linear_splitk) linear_splitk;
} entry;

bool no_modes() { return !at::impl::torch_function_mode_enabled() && !c10::impl::TorchDispatchModeTLS::any_modes_set(); }

// A strided CUDA tensor that is nothing but that.
bool plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  static const c10::DispatchKeySet ordinary = c10::DispatchKeySet({c10::DispatchKey::Dense, c10::DispatchKey::ADInplaceOrView, c10::DispatchKey::AutogradFunctionality,
                                                                   c10::DispatchKey::AutocastCUDA}) |
                                              c10::DispatchKeySet(c10::BackendComponent::CUDABit);
  return t.defined() && t.is_cuda() && (t.key_set().raw_repr() & ~ordinary.raw_repr()) == 0 && t.has_storage();
}
bool plain_or_none(PyObject* o) { return o == Py_None || plain(o); }
void* pointer(PyObject* o) { return o == Py_None ? nullptr : THPVariable_Unpack(o).data_ptr(); }

// an exact Python int that fits T
template <typename T>
bool number(PyObject* o, T* out) {
  if (!PyLong_CheckExact(o)) return false;
  int overflow = 0;
  const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
  if (overflow || v < static_cast<long long>(std::numeric_limits<T>::min()) || v > static_cast<long long>(std::numeric_limits<T>::max())) return false;
  *out = static_cast<T>(v);
  return true;
}
bool handle(PyObject* o, void** out) {
  if (!PyLong_CheckExact(o)) return false;
  *out = PyLong_AsVoidPtr(o);
  return true;
}

// X of a rotate + quantize call: two-dimensional, 16-bit elements, columns side by side
bool activations(PyObject* o, int64_t K, int32_t* M, int64_t* ldx) {
  if (!plain(o)) return false;
  const at::Tensor& x = THPVariable_Unpack(o);
  if (x.dim() != 2 || x.element_size() != 2 || x.stride(1) != 1 || x.size(0) > std::numeric_limits<int32_t>::max()) return false;
  *M = static_cast<int32_t>(x.size(0));
  *ldx = *M > 1 ? x.stride(0) : K;
  return true;
}
// codes of a linear call: the rows
bool rows(PyObject* o, int32_t* M) {
  if (!plain(o)) return false;
  const at::Tensor& c = THPVariable_Unpack(o);
  if (c.dim() < 1 || c.size(0) > std::numeric_limits<int32_t>::max()) return false;
  *M = static_cast<int32_t>(c.size(0));
  return true;
}
bool output(PyObject* o, int32_t M, int64_t N, int64_t* ld) {
  *ld = N;
  if (o == Py_None) return true;
  if (!plain(o) || THPVariable_Unpack(o).dim() < 1) return false;
  if (M > 1) *ld = THPVariable_Unpack(o).stride(0);
  return true;
}

// A new reference to `given`, or to a new tensor on the device of `like`.
PyObject* given_or_empty(PyObject* given, PyObject* like, at::IntArrayRef sizes, at::ScalarType type) {
  if (given != Py_None) {
    Py_INCREF(given);
    return given;
  }
  return THPVariable_Wrap(at::empty(sizes, THPVariable_Unpack(like).options().dtype(type)));
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Runs a library call without the GIL (as ctypes does) and returns the outputs in a tuple, or alone, or the status.
struct Outputs {
  PyObject* o[4] = {nullptr, nullptr, nullptr, nullptr};
  int n = 0;
  ~Outputs() {
    for (int i = 0; i < n; ++i) Py_DECREF(o[i]);
  }
  PyObject* add(PyObject* p) {
    if (!p) throw python_error();
    return o[n++] = p;
  }
  template <typename Call>
  PyObject* run(Call&& call, bool list = false) {
    trdq_status st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    if (st != TRDQ_OK) return PyLong_FromLong(st);
    if (n == 1) {
      Py_INCREF(o[0]);
      return o[0];
    }
    PyObject* const r = list ? PyList_New(n) : PyTuple_New(n);
    if (!r) return nullptr;
    for (int i = 0; i < n; ++i) {
      Py_INCREF(o[i]);
      if (list) {
        PyList_SET_ITEM(r, i, o[i]);
      } else {
        PyTuple_SET_ITEM(r, i, o[i]);
      }
    }
    return r;
  }
};

#define GENERAL_WAY_UNLESS(condition) \
  if (!(condition)) Py_RETURN_NONE

// (rot, K, t, X, codes, scales)
PyObject* rotate_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* rot;
  int64_t K, ldx;
  int32_t t, M;
  GENERAL_WAY_UNLESS(n == 6 && handle(a[0], &rot) && number(a[1], &K) && number(a[2], &t) && activations(a[3], K, &M, &ldx) &&
                     plain_or_none(a[4]) && plain_or_none(a[5]) && no_modes());
  Outputs out;
  void* const codes = pointer(out.add(given_or_empty(a[4], a[3], {M, K}, at::kChar)));
  void* const scales = pointer(out.add(given_or_empty(a[5], a[3], {M}, at::kFloat)));
  void* const x = pointer(a[3]);
  void* const s = stream();
  return out.run([&] { return entry.rotate_quantize(static_cast<trdq_rotation*>(rot), t, x, ldx, M, static_cast<int8_t*>(codes), static_cast<float*>(scales), s); });
  END_HANDLE_TH_ERRORS
}

// (rot, K, t, X, shift, scale, rows_per_sample, eps, codes, scales)
PyObject* norm_rotate_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* rot;
  int64_t K, ldx;
  int32_t t, M, per_sample;
  GENERAL_WAY_UNLESS(n == 10 && handle(a[0], &rot) && number(a[1], &K) && number(a[2], &t) && activations(a[3], K, &M, &ldx) &&
                     plain_or_none(a[4]) && plain_or_none(a[5]) && PyFloat_CheckExact(a[7]) && plain_or_none(a[8]) && plain_or_none(a[9]) && no_modes());
  if (a[6] == Py_None) {
    per_sample = M > 1 ? M : 1;
  } else {
    GENERAL_WAY_UNLESS(number(a[6], &per_sample));
  }
  const float eps = static_cast<float>(PyFloat_AS_DOUBLE(a[7]));
  Outputs out;
  void* const codes = pointer(out.add(given_or_empty(a[8], a[3], {M, K}, at::kChar)));
  void* const scales = pointer(out.add(given_or_empty(a[9], a[3], {M}, at::kFloat)));
  void *const x = pointer(a[3]), *const shift = pointer(a[4]), *const scale = pointer(a[5]);
  void* const s = stream();
  return out.run([&] {
    return entry.norm_rotate_quantize(static_cast<trdq_rotation*>(rot), t, x, ldx, M, shift, scale, per_sample, eps, static_cast<int8_t*>(codes),
                                      static_cast<float*>(scales), s);
  });
  END_HANDLE_TH_ERRORS
}

// (rot, K, t, X)
PyObject* rotate_quantize_asym(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* rot;
  int64_t K, ldx;
  int32_t t, M;
  GENERAL_WAY_UNLESS(n == 4 && handle(a[0], &rot) && number(a[1], &K) && number(a[2], &t) && activations(a[3], K, &M, &ldx) && no_modes());
  Outputs out;
  void* const codes = pointer(out.add(given_or_empty(Py_None, a[3], {M, K}, at::kByte)));
  void* const scales = pointer(out.add(given_or_empty(Py_None, a[3], {M}, at::kFloat)));
  void* const zero = pointer(out.add(given_or_empty(Py_None, a[3], {M}, at::kInt)));
  void* const x = pointer(a[3]);
  void* const s = stream();
  return out.run([&] {
    return entry.rotate_quantize_asym(static_cast<trdq_rotation*>(rot), t, x, ldx, M, static_cast<uint8_t*>(codes), static_cast<float*>(scales),
                                      static_cast<int32_t*>(zero), s);
  });
  END_HANDLE_TH_ERRORS
}

// (w, N, t, codes, scales, bias, out, act)
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* w;
  int64_t N, ldy;
  int32_t t, M, act;
  GENERAL_WAY_UNLESS(n == 8 && handle(a[0], &w) && number(a[1], &N) && number(a[2], &t) && rows(a[3], &M) && plain(a[4]) && plain_or_none(a[5]) &&
                     output(a[6], M, N, &ldy) && number(a[7], &act) && no_modes());
  Outputs out;
  void* const y = pointer(out.add(given_or_empty(a[6], a[3], {M, N}, at::kBFloat16)));
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const bias = pointer(a[5]);
  void* const s = stream();
  return out.run([&] {
    return entry.linear_act(static_cast<trdq_weights*>(w), t, static_cast<int8_t*>(codes), static_cast<float*>(scales), M, bias, y, ldy, act, s);
  });
  END_HANDLE_TH_ERRORS
}

// (w, N, t, codes, scales, zero_points, bias, out)
PyObject* linear_asym(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* w;
  int64_t N, ldy;
  int32_t t, M;
  GENERAL_WAY_UNLESS(n == 8 && handle(a[0], &w) && number(a[1], &N) && number(a[2], &t) && rows(a[3], &M) && plain(a[4]) && plain(a[5]) &&
                     plain_or_none(a[6]) && output(a[7], M, N, &ldy) && no_modes());
  Outputs out;
  void* const y = pointer(out.add(given_or_empty(a[7], a[3], {M, N}, at::kBFloat16)));
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const zero = pointer(a[5]), *const bias = pointer(a[6]);
  void* const s = stream();
  return out.run([&] {
    return entry.linear_asym(static_cast<trdq_weights*>(w), t, static_cast<uint8_t*>(codes), static_cast<float*>(scales), static_cast<int32_t*>(zero), M,
                             bias, y, ldy, s);
  });
  END_HANDLE_TH_ERRORS
}

// (w, N, t, codes, scales, bias, out, workspace)
PyObject* linear_splitk(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* w;
  int64_t N, ldy;
  int32_t t, M, splits = 0;
  uint64_t bytes = 0;
  GENERAL_WAY_UNLESS(n == 8 && handle(a[0], &w) && number(a[1], &N) && number(a[2], &t) && rows(a[3], &M) && plain(a[4]) && plain_or_none(a[5]) &&
                     output(a[6], M, N, &ldy) && plain_or_none(a[7]) && no_modes() &&
                     entry.splitk_workspace(static_cast<trdq_weights*>(w), M, &splits, &bytes) == TRDQ_OK);
  Outputs out;
  void* const y = pointer(out.add(given_or_empty(a[6], a[3], {M, N}, at::kBFloat16)));
  at::Tensor workspace;
  if (a[7] != Py_None) {
    workspace = THPVariable_Unpack(a[7]);
  } else if (bytes) {
    workspace = at::empty({static_cast<int64_t>(bytes)}, THPVariable_Unpack(a[3]).options().dtype(at::kByte));
  }
  void* const ws = workspace.defined() ? workspace.data_ptr() : nullptr;
  const uint64_t ws_bytes = workspace.defined() ? static_cast<uint64_t>(workspace.numel() * workspace.element_size()) : 0;
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const bias = pointer(a[5]);
  void* const s = stream();
  return out.run([&] {
    return entry.linear_splitk(static_cast<trdq_weights*>(w), t, static_cast<int8_t*>(codes), static_cast<float*>(scales), M, bias, y, ldy, ws, ws_bytes, s);
  });
  END_HANDLE_TH_ERRORS
}

// (w, N, t, (codes, codes), (scales, scales), bias): the outputs in a list
PyObject* linear_cfg(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  void* w;
  int64_t N;
  int32_t t, M[2];
  GENERAL_WAY_UNLESS(n == 6 && handle(a[0], &w) && number(a[1], &N) && number(a[2], &t) && plain_or_none(a[5]) && no_modes());
  PyObject *codes[2], *scales[2];
  auto two = [](PyObject* o, PyObject** items) {
    if (PyList_CheckExact(o) && PyList_GET_SIZE(o) == 2) {
      items[0] = PyList_GET_ITEM(o, 0);
      items[1] = PyList_GET_ITEM(o, 1);
      return true;
    }
    if (!PyTuple_CheckExact(o) || PyTuple_GET_SIZE(o) != 2) return false;
    items[0] = PyTuple_GET_ITEM(o, 0);
    items[1] = PyTuple_GET_ITEM(o, 1);
    return true;
  };
  GENERAL_WAY_UNLESS(two(a[3], codes) && two(a[4], scales) && rows(codes[0], &M[0]) && rows(codes[1], &M[1]) && plain(scales[0]) && plain(scales[1]));
  Outputs out;
  const void* c[2];
  const float* sx[2];
  void* y[2];
  int64_t ldy[2];
  for (int i = 0; i < 2; ++i) {
    const at::Tensor& cond = THPVariable_Unpack(codes[i]);
    c[i] = cond.data_ptr();
    sx[i] = static_cast<const float*>(pointer(scales[i]));
    y[i] = pointer(out.add(given_or_empty(Py_None, codes[0], {M[i], N}, at::kBFloat16)));
    ldy[i] = N;
  }
  void* const bias = pointer(a[5]);
  void* const s = stream();
  const int8_t* const c8[2] = {static_cast<const int8_t*>(c[0]), static_cast<const int8_t*>(c[1])};
  return out.run([&] { return entry.linear_cfg(static_cast<trdq_weights*>(w), t, c8, sx, M, bias, y, ldy, s); }, true);
  END_HANDLE_TH_ERRORS
}

// (addresses of the library's functions, in the order of Entry)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* address[8];
  if (n != 8) {
    PyErr_SetString(PyExc_TypeError, "eight addresses");
    return nullptr;
  }
  for (int i = 0; i < 8; ++i) {
    address[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
  }
  entry = {reinterpret_cast<decltype(entry.rotate_quantize)>(address[0]),      reinterpret_cast<decltype(entry.norm_rotate_quantize)>(address[1]),
           reinterpret_cast<decltype(entry.rotate_quantize_asym)>(address[2]), reinterpret_cast<decltype(entry.linear_act)>(address[3]),
           reinterpret_cast<decltype(entry.linear_cfg)>(address[4]),           reinterpret_cast<decltype(entry.linear_asym)>(address[5]),
           reinterpret_cast<decltype(entry.splitk_workspace)>(address[6]),     reinterpret_cast<decltype(entry.linear_splitk)>(address[7])};
  Py_RETURN_NONE;
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind),        METHOD(rotate_quantize), METHOD(norm_rotate_quantize), METHOD(rotate_quantize_asym), METHOD(linear),
                         METHOD(linear_asym), METHOD(linear_splitk),   METHOD(linear_cfg),           {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
