// The checks of binding.py's forward calls in native code, for the usual case: plain torch tensors of the right device, type,
// shape and layout.  A call returns the library's status, or -1 where anything is unusual - nothing has been launched then,
// and binding.py goes through its own checks, which say what is wrong.
//
// Of the no-allocation entry point it also takes the layer's arrays, where they are numpy's own and of the types the library reads.
//
// A small layer's kernel takes 3.4 us while Python's checks, conversions and call took 6; a group of 16 layers on one image 9
// and 20.  Here the checks of a layer take 0.2 us and those of a group 2.  The no-allocation call took the host 16.8 us, now 8, and
// takes the GPU 9.2.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <cstring>

#include "snn_conv.h"

namespace {

using LayerForward = snn_status_t (*)(snn_conv_t*, const void*, int32_t, int32_t, int32_t, void*, int32_t, int32_t, void*);
using GroupForward = snn_status_t (*)(snn_conv_group_t*, const void* const*, void* const*, int32_t, void*);
using StackForward = snn_status_t (*)(snn_conv_stack_t*, const void*, void*, int32_t, void*);
LayerForward g_layer = nullptr;
GroupForward g_group = nullptr;
StackForward g_stack = nullptr;
using StaticForward = snn_status_t (*)(const snn_conv_desc_t*, const void*, int32_t, int32_t, int32_t, void*, int32_t, void*);
StaticForward g_static = nullptr;
PyTypeObject* g_ndarray = nullptr;   // numpy.ndarray

constexpr int kUnusual = -1;

// What binding.py packs for a handle (struct format "=QQiiiiiiii"): the descriptions are bytes objects.
struct Layer {
  uint64_t handle, spare;
  int32_t device, act_type, c_act, c_out, ksize, stride, pad, unused;   // c_act: last dimension of the activations
};
// A member of a group ("=8i"), or the one input and output of a stack, after the head ("=Qii").
struct Head {
  uint64_t handle;
  int32_t device, act_type;
};
struct Member {
  int32_t n, h, w, c_act, ho, wo, c_out, unused;
};

// The tensor behind an argument that is exactly a torch.Tensor (or Parameter) of the device, dense and contiguous.
const at::Tensor* plain(PyObject* o, int device) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || t.get_device() != device || t.dim() != 4 || !t.is_contiguous() ||
      t.is_neg() || t.is_conj())
    return nullptr;
  return &t;
}
bool act_ok(const at::Tensor& t, int act_type) {
  const at::ScalarType s = t.scalar_type();
  return act_type == SNN_ACT_BIN ? s == at::kInt || s == at::kUInt32 : s == at::kHalf;
}
bool shape_is(const at::Tensor& t, int64_t a, int64_t b, int64_t c, int64_t d) {
  const auto s = t.sizes();
  return s[0] == a && s[1] == b && s[2] == c && s[3] == d;
}
bool out_ok(const at::Tensor& t, int64_t n, int64_t ho, int64_t wo, int64_t c_out, long out_type) {
  return t.scalar_type() == (out_type == SNN_OUT_F32 ? at::kFloat : at::kInt) &&
         shape_is(t, n, ho, wo, out_type == SNN_OUT_BITS ? (c_out + 31) / 32 : c_out);
}
bool small_int(PyObject* o, long* v) {
  if (!PyLong_CheckExact(o)) return false;
  int overflow = 0;
  *v = PyLong_AsLongAndOverflow(o, &overflow);
  return !overflow && *v >= 0 && *v <= 3;
}
template <class T>
const T* described(PyObject* o, size_t bytes) {
  return PyBytes_CheckExact(o) && (size_t)PyBytes_GET_SIZE(o) >= bytes ? reinterpret_cast<const T*>(PyBytes_AS_STRING(o)) : nullptr;
}
void* current_stream(int device) { return c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream(); }

template <class F>
PyObject* guarded(F f) {   // no C++ exception leaves (a tensor without storage, a device torch does not know)
  long st = kUnusual;
  try {
    st = f();
  } catch (...) {
    st = kUnusual;
  }
  return PyLong_FromLong(st);
}
template <class F>
long unlocked(F f) {
  long st;
  Py_BEGIN_ALLOW_THREADS
  st = (long)f();
  Py_END_ALLOW_THREADS
  return st;
}

// layer_forward(description, act, out, out_type, path)
PyObject* layer_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> long {
    long out_type, path;
    const Layer* d = n == 5 ? described<Layer>(a[0], sizeof(Layer)) : nullptr;
    if (!d || !g_layer || !small_int(a[3], &out_type) || !small_int(a[4], &path)) return kUnusual;
    const at::Tensor *x = plain(a[1], d->device), *y = plain(a[2], d->device);
    if (!x || !y || !act_ok(*x, d->act_type) || x->size(3) != d->c_act) return kUnusual;
    const int64_t N = x->size(0), H = x->size(1), W = x->size(2), k = d->ksize, p = d->pad, s = d->stride;
    if (N < 1 || H + 2 * p < k || W + 2 * p < k || N > INT32_MAX || H > INT32_MAX || W > INT32_MAX) return kUnusual;
    if (!out_ok(*y, N, (H + 2 * p - k) / s + 1, (W + 2 * p - k) / s + 1, d->c_out, out_type)) return kUnusual;
    const void* const act = x->data_ptr();
    void* const out = y->data_ptr();
    void* const stream = current_stream(d->device);
    return unlocked([&] {
      return g_layer(reinterpret_cast<snn_conv_t*>(d->handle), act, (int32_t)N, (int32_t)H, (int32_t)W, out, (int32_t)out_type, (int32_t)path, stream);
    });
  });
}

// group_forward(description, acts, outs, out_type)
PyObject* group_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> long {
    long out_type;
    const Head* d = n == 4 ? described<Head>(a[0], sizeof(Head) + sizeof(Member)) : nullptr;
    if (!d || !g_group || !small_int(a[3], &out_type)) return kUnusual;
    const Py_ssize_t count = (PyBytes_GET_SIZE(a[0]) - (Py_ssize_t)sizeof(Head)) / (Py_ssize_t)sizeof(Member);
    if (!PyList_CheckExact(a[1]) || !PyList_CheckExact(a[2]) || count > SNN_GROUP_MAX || PyList_GET_SIZE(a[1]) != count || PyList_GET_SIZE(a[2]) != count)
      return kUnusual;
    const Member* const m = reinterpret_cast<const Member*>(d + 1);
    const void* act[SNN_GROUP_MAX];
    void* out[SNN_GROUP_MAX];
    for (Py_ssize_t i = 0; i < count; ++i) {
      const at::Tensor *x = plain(PyList_GET_ITEM(a[1], i), d->device), *y = plain(PyList_GET_ITEM(a[2], i), d->device);
      if (!x || !y || !act_ok(*x, d->act_type) || !shape_is(*x, m[i].n, m[i].h, m[i].w, m[i].c_act) ||
          !out_ok(*y, m[i].n, m[i].ho, m[i].wo, m[i].c_out, out_type))
        return kUnusual;
      act[i] = x->data_ptr();
      out[i] = y->data_ptr();
    }
    void* const stream = current_stream(d->device);
    return unlocked([&] { return g_group(reinterpret_cast<snn_conv_group_t*>(d->handle), act, out, (int32_t)out_type, stream); });
  });
}

// stack_forward(description, act, out, out_type)
PyObject* stack_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> long {
    long out_type;
    const Head* d = n == 4 ? described<Head>(a[0], sizeof(Head) + sizeof(Member)) : nullptr;
    if (!d || !g_stack || !small_int(a[3], &out_type)) return kUnusual;
    const Member* const m = reinterpret_cast<const Member*>(d + 1);
    const at::Tensor *x = plain(a[1], d->device), *y = plain(a[2], d->device);
    if (!x || !y || !act_ok(*x, d->act_type) || !shape_is(*x, m->n, m->h, m->w, m->c_act) ||
        !out_ok(*y, m->n, m->ho, m->wo, m->c_out, out_type))
      return kUnusual;
    const void* const act = x->data_ptr();
    void* const out = y->data_ptr();
    void* const stream = current_stream(d->device);
    return unlocked([&] { return g_stack(reinterpret_cast<snn_conv_stack_t*>(d->handle), act, out, (int32_t)out_type, stream); });
  });
}

// An argument that is exactly a numpy array, dense in C order, of elements of one format; released with the object.
struct Array {
  Py_buffer view{};
  bool held = false;
  ~Array() {
    if (held) PyBuffer_Release(&view);
  }
  bool take(PyObject* o, const char* format) {
    if (!g_ndarray || Py_TYPE(o) != g_ndarray) return false;
    if (PyObject_GetBuffer(o, &view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) {
      PyErr_Clear();
      return false;
    }
    held = true;
    return view.format && strcmp(view.format, format) == 0;
  }
  int64_t size() const { return (int64_t)(view.len / view.itemsize); }
};
bool int_between(PyObject* o, long low, long high, int32_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  int overflow = 0;
  const long x = PyLong_AsLongAndOverflow(o, &overflow);
  *v = (int32_t)x;
  return !overflow && x >= low && x <= high;
}

// static_forward(c_in, c_out, tau, codebook, idx_packed, alpha, act, out, stride, pad, out_type, device)
PyObject* static_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> long {
    snn_conv_desc_t d{};
    int32_t out_type = 0;
    if (n != 12 || !g_static || !int_between(a[0], 1, SNN_STATIC_MAX_CHANNELS, &d.c_in) || !int_between(a[1], 1, SNN_STATIC_MAX_CHANNELS, &d.c_out) ||
        !int_between(a[2], 1, 9, &d.tau) || !int_between(a[8], 1, 2, &d.stride) || !int_between(a[9], 0, 1, &d.pad) ||
        !int_between(a[10], SNN_OUT_F32, SNN_OUT_I32, &out_type) || !int_between(a[11], 0, 1023, &d.device))
      return kUnusual;
    const at::Tensor *x = plain(a[6], d.device), *y = plain(a[7], d.device);
    if (!x || !y || !act_ok(*x, SNN_ACT_BIN) || x->size(3) != (d.c_in + 31) / 32) return kUnusual;
    const int64_t N = x->size(0), H = x->size(1), W = x->size(2), p = d.pad, s = d.stride;
    if (N < 1 || H + 2 * p < 3 || W + 2 * p < 3 || N > INT32_MAX || H > INT32_MAX || W > INT32_MAX) return kUnusual;
    if (!out_ok(*y, N, (H + 2 * p - 3) / s + 1, (W + 2 * p - 3) / s + 1, d.c_out, out_type)) return kUnusual;
    Array codebook, stream, alpha;
    if (!codebook.take(a[3], "H") || !stream.take(a[4], "B") || !alpha.take(a[5], "f") || codebook.size() != (1 << d.tau) || alpha.size() != d.c_out ||
        stream.size() < ((int64_t)d.c_out * d.c_in * d.tau + 7) / 8)
      return kUnusual;
    d.act_type = SNN_ACT_BIN;
    d.ksize = 3;
    d.codebook = static_cast<const uint16_t*>(codebook.view.buf);
    d.idx_packed = static_cast<const uint8_t*>(stream.view.buf);
    d.alpha = static_cast<const float*>(alpha.view.buf);
    const void* const act = x->data_ptr();
    void* const out = y->data_ptr();
    void* const cuda_stream = current_stream(d.device);
    return unlocked([&] { return g_static(&d, act, (int32_t)N, (int32_t)H, (int32_t)W, out, out_type, cuda_stream); });
  });
}

// bind_static(address of the library's entry point, numpy.ndarray)
PyObject* bind_static(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2 || !PyType_Check(a[1])) {
    PyErr_SetString(PyExc_TypeError, "bind_static takes an address and a type");
    return nullptr;
  }
  void* const p = PyLong_AsVoidPtr(a[0]);
  if (!p && PyErr_Occurred()) return nullptr;
  g_static = reinterpret_cast<StaticForward>(p);
  Py_INCREF(a[1]);
  g_ndarray = reinterpret_cast<PyTypeObject*>(a[1]);
  Py_RETURN_NONE;
}

// bind(layer, group, stack): addresses of the library's entry points
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 3) {
    PyErr_SetString(PyExc_TypeError, "bind takes three addresses");
    return nullptr;
  }
  void* p[3];
  for (int i = 0; i < 3; ++i) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (!p[i] && PyErr_Occurred()) return nullptr;
  }
  g_layer = reinterpret_cast<LayerForward>(p[0]);
  g_group = reinterpret_cast<GroupForward>(p[1]);
  g_stack = reinterpret_cast<StackForward>(p[2]);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"layer_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(layer_forward)), METH_FASTCALL, nullptr},
    {"group_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(group_forward)), METH_FASTCALL, nullptr},
    {"stack_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(stack_forward)), METH_FASTCALL, nullptr},
    {"static_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(static_forward)), METH_FASTCALL, nullptr},
    {"bind_static", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bind_static)), METH_FASTCALL, nullptr},
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bind)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_snn_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (the version of torch is asked for before any tensor is handed in: tensors are read by the layout of its headers)
PyMODINIT_FUNC PyInit__snn_fast() {
  PyObject* m = PyModule_Create(&module_def);
  if (m && PyModule_AddStringConstant(m, "TORCH_VERSION", SNN_TORCH_VERSION) < 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
