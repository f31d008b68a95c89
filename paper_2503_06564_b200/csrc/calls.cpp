// The hot entry points of libtrdq.so for plain torch tensors: what trdq.py does for a call (checks, outputs, pointers, strides, current
// stream) in one native function.  A small layer is bound by this host work, not by the GPU: through ctypes a call took about 9 us,
// 2 us of it for each output, 1.5 for the conversion of the arguments and 1 for the tensors' attributes, and a linear layer of 256 x 1024
// (two calls, 7 us on the GPU) 19.3 us, now 10.3; three calls for two ragged row segments 37.4, now 22.6.
//
// Every function returns None for arguments it does not handle: tensor subclasses, tensors of other devices or layouts, wrapped tensors
// (functorch, functional, fake), numbers that are not Python ints, an active function or dispatch mode (torch.set_default_device is one).  The caller
// then goes its general way, which costs what it did and 0.15 us for the question, and is where wrong arguments are reported.  A status other than
// TRDQ_OK is returned as an int.
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

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct WithoutGil {
  PyThreadState* const state = PyEval_SaveThread();
  ~WithoutGil() { PyEval_RestoreThread(state); }
};

// The outputs of a call: given by the caller or new tensors on the device of `like`.
class Outputs {
 public:
  explicit Outputs(PyObject* like) : options_(THPVariable_Unpack(like).options()) {}
  void add(PyObject* given, int32_t rows, int64_t columns, at::ScalarType type) { put(given, rows, columns, 2, type); }
  void add(PyObject* given, int32_t rows, at::ScalarType type) { put(given, rows, 0, 1, type); }

  // Makes the new ones, runs the library call (it gets the pointers) and returns the outputs in a tuple, a list or alone, or the status.  All
  // of it without the GIL: an allocation may wait for the device, and for other threads' work on it.
  template <typename Call>
  PyObject* run(Call&& call, bool list = false) {
    trdq_status st;
    {
      WithoutGil released;
      void* pointers[kMost];
      for (int i = 0; i < n_; ++i) {
        Item& o = item_[i];
        if (!o.given) o.made = at::empty(at::IntArrayRef(o.sizes, o.dims), options_.dtype(o.type));
        pointers[i] = o.given ? o.pointer : o.made.data_ptr();
      }
      st = call(pointers);
    }
    if (st != TRDQ_OK) return PyLong_FromLong(st);
    if (n_ == 1) return wrap(item_[0]);
    PyObject* const r = list ? PyList_New(n_) : PyTuple_New(n_);
    if (!r) return nullptr;
    for (int i = 0; i < n_; ++i) {
      PyObject* const o = wrap(item_[i]);
      if (!o) {
        Py_DECREF(r);
        return nullptr;
      }
      if (list) {
        PyList_SET_ITEM(r, i, o);
      } else {
        PyTuple_SET_ITEM(r, i, o);
      }
    }
    return r;
  }

 private:
  static constexpr int kMost = 3;
  struct Item {
    PyObject* given;  // borrowed from the caller's arguments
    void* pointer;    // of the given one
    int64_t sizes[2];
    int dims;
    at::ScalarType type;
    at::Tensor made;
  };
  void put(PyObject* given, int64_t rows, int64_t columns, int dims, at::ScalarType type) {
    Item& o = item_[n_++];
    o.given = given == Py_None ? nullptr : given;
    o.pointer = pointer(given);
    o.sizes[0] = rows;
    o.sizes[1] = columns;
    o.dims = dims;
    o.type = type;
  }
  static PyObject* wrap(Item& o) {
    if (!o.given) return THPVariable_Wrap(std::move(o.made));
    Py_INCREF(o.given);
    return o.given;
  }

  at::TensorOptions options_;
  Item item_[kMost];
  int n_ = 0;
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
  Outputs out(a[3]);
  out.add(a[4], M, K, at::kChar);
  out.add(a[5], M, at::kFloat);
  void* const x = pointer(a[3]);
  void* const s = stream();
  return out.run([&](void** o) { return entry.rotate_quantize(static_cast<trdq_rotation*>(rot), t, x, ldx, M, static_cast<int8_t*>(o[0]), static_cast<float*>(o[1]), s); });
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
  Outputs out(a[3]);
  out.add(a[8], M, K, at::kChar);
  out.add(a[9], M, at::kFloat);
  void *const x = pointer(a[3]), *const shift = pointer(a[4]), *const scale = pointer(a[5]);
  void* const s = stream();
  return out.run([&](void** o) {
    return entry.norm_rotate_quantize(static_cast<trdq_rotation*>(rot), t, x, ldx, M, shift, scale, per_sample, eps, static_cast<int8_t*>(o[0]),
                                      static_cast<float*>(o[1]), s);
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
  Outputs out(a[3]);
  out.add(Py_None, M, K, at::kByte);
  out.add(Py_None, M, at::kFloat);
  out.add(Py_None, M, at::kInt);
  void* const x = pointer(a[3]);
  void* const s = stream();
  return out.run([&](void** o) {
    return entry.rotate_quantize_asym(static_cast<trdq_rotation*>(rot), t, x, ldx, M, static_cast<uint8_t*>(o[0]), static_cast<float*>(o[1]),
                                      static_cast<int32_t*>(o[2]), s);
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
  Outputs out(a[3]);
  out.add(a[6], M, N, at::kBFloat16);
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const bias = pointer(a[5]);
  void* const s = stream();
  return out.run([&](void** o) {
    return entry.linear_act(static_cast<trdq_weights*>(w), t, static_cast<int8_t*>(codes), static_cast<float*>(scales), M, bias, o[0], ldy, act, s);
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
  Outputs out(a[3]);
  out.add(a[7], M, N, at::kBFloat16);
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const zero = pointer(a[5]), *const bias = pointer(a[6]);
  void* const s = stream();
  return out.run([&](void** o) {
    return entry.linear_asym(static_cast<trdq_weights*>(w), t, static_cast<uint8_t*>(codes), static_cast<float*>(scales), static_cast<int32_t*>(zero), M,
                             bias, o[0], ldy, s);
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
  Outputs out(a[3]);
  out.add(a[6], M, N, at::kBFloat16);
  void *const codes = pointer(a[3]), *const scales = pointer(a[4]), *const bias = pointer(a[5]), *const given = pointer(a[7]);
  const at::TensorOptions options = THPVariable_Unpack(a[3]).options().dtype(at::kByte);
  const bool make = a[7] == Py_None && bytes;
  if (a[7] != Py_None) bytes = static_cast<uint64_t>(THPVariable_Unpack(a[7]).numel() * THPVariable_Unpack(a[7]).element_size());
  void* const s = stream();
  return out.run([&](void** o) {
    at::Tensor made;
    if (make) made = at::empty({static_cast<int64_t>(bytes)}, options);
    return entry.linear_splitk(static_cast<trdq_weights*>(w), t, static_cast<int8_t*>(codes), static_cast<float*>(scales), M, bias, o[0], ldy,
                               make ? made.data_ptr() : given, bytes, s);
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
  Outputs out(codes[0]);
  at::Tensor held[4];  // the caller's lists may change while the GIL is released
  const int8_t* c[2];
  const float* sx[2];
  const int64_t ldy[2] = {N, N};
  for (int i = 0; i < 2; ++i) {
    held[2 * i] = THPVariable_Unpack(codes[i]);
    held[2 * i + 1] = THPVariable_Unpack(scales[i]);
    c[i] = static_cast<const int8_t*>(held[2 * i].data_ptr());
    sx[i] = static_cast<const float*>(held[2 * i + 1].data_ptr());
    out.add(Py_None, M[i], N, at::kBFloat16);
  }
  void* const bias = pointer(a[5]);
  void* const s = stream();
  return out.run([&](void** y) { return entry.linear_cfg(static_cast<trdq_weights*>(w), t, c, sx, M, bias, y, ldy, s); }, true);
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
