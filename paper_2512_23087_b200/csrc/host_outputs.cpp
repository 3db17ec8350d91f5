// Python helper: the per-token outputs of a call as views of one allocation.
//
// A call has up to twenty output vectors.  Sliced from three allocations through Python they took more than half of
// the 33 us that a call of dvp_forward on a few tokens spends on the host; as tensors laid directly over one
// storage they cost 5 us (16 tokens x 151 936 bf16 logits: 32.6 -> 18.3 us a call).

#include <Python.h>

#include <ATen/ATen.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

namespace {

// T elements of `type` over `storage`, starting at byte row * stride.
at::Tensor row_view(const c10::Storage &storage, c10::DispatchKeySet keys, at::ScalarType type, int64_t row,
                    int64_t stride, int64_t T) {
  auto impl = c10::make_intrusive<c10::TensorImpl>(c10::Storage(storage), keys, c10::scalarTypeToTypeMeta(type));
  impl->set_sizes_contiguous({T});
  impl->set_storage_offset(row * stride / static_cast<int64_t>(c10::elementSize(type)));
  return at::Tensor(std::move(impl));
}

// outputs(like, T, floats, counts) -> (tensors, address, stride): `floats` float32 vectors, `counts` int32 vectors
// and one uint8 vector of T elements on the device of `like`, in this order; vector i starts at address + i * stride.
PyObject *outputs(PyObject *, PyObject *const *args, Py_ssize_t n_args) {
  if (n_args != 4 || !THPVariable_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "outputs(like, T, floats, counts)");
    return nullptr;
  }
  const int64_t T = PyLong_AsLongLong(args[1]), floats = PyLong_AsLongLong(args[2]), counts = PyLong_AsLongLong(args[3]);
  if (PyErr_Occurred()) return nullptr;
  if (T < 0 || T >= (int64_t(1) << 56)) {
    PyErr_Format(PyExc_RuntimeError, "outputs: there are no vectors of %lld elements", static_cast<long long>(T));
    return nullptr;
  }
  // torch's own exception types reach Python, out-of-memory errors among them
  HANDLE_TH_ERRORS
  const int64_t rows = floats + counts + 1, stride = (T + 3) / 4 * 16;
  const at::Tensor buf =
      at::empty({rows * stride}, THPVariable_Unpack(args[0]).options().dtype(at::kByte).requires_grad(false));
  const c10::Storage &storage = buf.storage();
  const c10::DispatchKeySet keys = buf.key_set();
  THPObjectPtr tensors(PyTuple_New(rows));
  if (!tensors) return nullptr;
  for (int64_t i = 0; i < rows; ++i) {
    const at::ScalarType type = i < floats ? at::kFloat : i < floats + counts ? at::kInt : at::kByte;
    PyObject *t = THPVariable_Wrap(row_view(storage, keys, type, i, stride, T));
    if (!t) return nullptr;
    PyTuple_SET_ITEM(tensors.get(), i, t);
  }
  return Py_BuildValue("(NLL)", tensors.release(), static_cast<long long>(reinterpret_cast<uintptr_t>(buf.data_ptr())),
                       static_cast<long long>(stride));
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"outputs", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(outputs)), METH_FASTCALL,
                          "outputs(like, T, floats, counts) -> (tensors, address, stride)"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// PyInit__host: the module says what it was built for (build.py looks for the text in the file, binding.py asks the module)
extern "C" __attribute__((visibility("default"))) PyObject *PyInit__host() {
  static const char text[] = "[built for " DVP_HOST_TARGET "]";
  PyObject *m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_for", text) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
