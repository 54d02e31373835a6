// Native marshalling of the force calls of the Python binding: looks the
// tensors over, takes their addresses and the current stream and calls the C
// entry point, as the ctypes path of __init__.py does in Python.
//
// What bounds a small call is the host: of the 6.2 us of cn_force with given
// outputs the kernel launch takes 2.6, the ctypes conversion of the eight
// arguments 0.7 and the Python checks 2.9; here the checks and the conversion
// take 0.3 together. Everything that is not simply right (a subclass, a wrapped or
// functional tensor, a wrong type, shape, stride or device, an eps2 that is no
// number) is declined, and the Python path then handles or refuses it as it does
// without this module.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using Force = int (*)(int64_t, const void*, int64_t, const void*, float, void*, void*, void*);
using ForceEpsI = int (*)(int64_t, const void*, int64_t, const void*, void*, void*, void*);

constexpr long kDeclined = -1;

// The tensor of `o` if it is an ordinary dense contiguous CUDA tensor on
// device `dev` of this element type with `dims` dimensions (the second, if any,
// of `cols`).
const at::Tensor* plain(PyObject* o, c10::ScalarType type, int64_t dims, int64_t cols, c10::DeviceIndex dev) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  static const uint64_t known =
      (c10::DispatchKeySet(c10::DispatchKey::CUDA) | c10::DispatchKeySet(c10::DispatchKey::AutogradCUDA) |
       c10::DispatchKeySet(c10::DispatchKey::ADInplaceOrView) | c10::DispatchKeySet(c10::DispatchKey::AutocastCUDA))
          .raw_repr();
  if (!t.defined() || (t.unsafeGetTensorImpl()->key_set().raw_repr() & ~known) != 0) return nullptr;
  if (!t.is_cuda() || t.layout() != c10::kStrided || !t.has_storage() || t.scalar_type() != type || t.dim() != dims)
    return nullptr;
  if ((dims == 2 && t.size(1) != cols) || t.get_device() != dev || !t.is_contiguous()) return nullptr;
  return &t;
}

// rows(pos_i, pos_mass_j): the i count of two record tensors, or -1
PyObject* rows(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2) return PyLong_FromLong(kDeclined);
  try {
    const c10::DeviceIndex dev = c10::cuda::current_device();
    const at::Tensor* i = plain(a[0], at::kFloat, 2, 4, dev);
    if (i && plain(a[1], at::kFloat, 2, 4, dev)) return PyLong_FromLongLong(i->size(0));
  } catch (const std::exception&) {
  }
  return PyLong_FromLong(kDeclined);
}

// The call of the entry point a[0]: a[1] True for double outputs, a[2] and
// a[3] the record tensors, then (EPS2) the softening, the outputs (the
// potential may be None) and the stream (None: PyTorch's current one). Status,
// or -1.
template <bool EPS2>
PyObject* force(PyObject*, PyObject* const* a, Py_ssize_t n) {
  constexpr int kOut = EPS2 ? 5 : 4;
  if (n != kOut + 3) return PyLong_FromLong(kDeclined);
  PyObject *const o_acc = a[kOut], *const o_pot = a[kOut + 1], *const o_stream = a[kOut + 2];
  int st = static_cast<int>(kDeclined);
  try {
    void* const entry = PyLong_AsVoidPtr(a[0]);
    const c10::ScalarType type = a[1] == Py_True ? at::kDouble : at::kFloat;
    const c10::DeviceIndex dev = c10::cuda::current_device();
    const at::Tensor* i = plain(a[2], at::kFloat, 2, 4, dev);
    const at::Tensor* j = plain(a[3], at::kFloat, 2, 4, dev);
    const at::Tensor* acc = plain(o_acc, type, 2, 3, dev);
    const at::Tensor* pot = o_pot == Py_None ? nullptr : plain(o_pot, type, 1, 0, dev);
    const bool numbers = (!EPS2 || PyFloat_Check(a[4]) || PyLong_CheckExact(a[4])) &&
                         (o_stream == Py_None || PyLong_CheckExact(o_stream));
    if (entry && i && j && acc && (pot || o_pot == Py_None) && numbers && acc->size(0) == i->size(0) &&
        (!pot || pot->size(0) == i->size(0))) {
      const float eps2 = EPS2 ? static_cast<float>(PyFloat_AsDouble(a[4])) : 0.f;
      void* const s =
          o_stream == Py_None ? c10::cuda::getCurrentCUDAStream(dev).stream() : PyLong_AsVoidPtr(o_stream);
      if (!PyErr_Occurred()) {
        const int64_t n_i = i->size(0), n_j = j->size(0);
        const void *const pi = i->data_ptr(), *const pj = j->data_ptr();
        void *const out = acc->data_ptr(), *const phi = pot ? pot->data_ptr() : nullptr;
        Py_BEGIN_ALLOW_THREADS;
        if constexpr (EPS2)
          st = reinterpret_cast<Force>(entry)(n_i, pi, n_j, pj, eps2, out, phi, s);
        else
          st = reinterpret_cast<ForceEpsI>(entry)(n_i, pi, n_j, pj, out, phi, s);
        Py_END_ALLOW_THREADS;
      }
    }
  } catch (const std::exception&) {
    st = static_cast<int>(kDeclined);
  }
  PyErr_Clear();
  return PyLong_FromLong(st);
}

template <PyObject* F(PyObject*, PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr};
}

PyMethodDef kMethods[] = {method<rows>("rows"), method<force<true>>("force"), method<force<false>>("force_eps_i"),
                          {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// torch_version: the version whose headers this was compiled with (another
// one is not used with it)
PyMODINIT_FUNC PyInit__binding() {
  PyObject* m = PyModule_Create(&kModule);
  if (m && PyModule_AddStringConstant(m, "torch_version", CN_TORCH_VERSION) < 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
