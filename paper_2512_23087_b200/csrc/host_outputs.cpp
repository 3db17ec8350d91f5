// Python helper: the per-token outputs of a call as views of one allocation, and the marshalling of dvp_forward.
//
// A call has up to twenty output vectors.  Sliced from three allocations through Python they took more than half of
// the 33 us that a call of dvp_forward on a few tokens spends on the host; as tensors laid directly over one
// storage they cost 5 us (16 tokens x 151 936 bf16 logits: 32.6 -> 18.3 us a call).

#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include "dvp.h"

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

// ---- dvp_forward ------------------------------------------------------------------------------------------------------
// What binding.dvp_forward does beside the library's call, for results that it makes itself.  In Python its checks, packing
// and namespaces took half of a small call: 64 x 4,096 float32 with the gradient 20.7 -> 12.3 us, 16 x 151,936 bfloat16
// forward 17.3 -> 14.3 (then the device's).

// The error that Python code gets for what it passes; thrown inside HANDLE_TH_ERRORS blocks.
[[noreturn]] void refuse(PyObject *type, const char *format, const char *name = "") {
  PyErr_Format(type, format, name);
  throw python_error();
}

const at::Tensor &tensor(PyObject *o, const char *name) {
  if (!THPVariable_Check(o)) refuse(PyExc_TypeError, "%s must be a tensor", name);
  return THPVariable_Unpack(o);
}

const at::Tensor &matrix(PyObject *o, const char *name) {
  const at::Tensor &x = tensor(o, name);
  if (x.dim() != 2 || x.stride(1) != 1) refuse(PyExc_ValueError, "%s must be 2-D with unit inner stride", name);
  if (!x.is_cuda()) refuse(PyExc_ValueError, "%s must live on a CUDA device", name);
  return x;
}

int32_t dtype_code(at::ScalarType t) {
  switch (t) {
    case at::kFloat: return DVP_F32;
    case at::kBFloat16: return DVP_BF16;
    case at::kHalf: return DVP_F16;
    default: break;
  }
  PyErr_SetObject(PyExc_KeyError, reinterpret_cast<PyObject *>(torch::getTHPDtype(t)));
  throw python_error();
}

// Names that results have, and the type of results; made once.
struct Names {
  PyObject *max, *lse, *lse_safe, *logp, *logp_mp, *comp_mp, *log_cov, *count, *mask, *train, *infer, *log_ratio, *flags,
      *grad_train, *weight, *ns;
} g_names;

bool make_names() {
  const char *text[] = {"max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "log_cov", "count", "mask", "train",
                        "infer", "log_ratio", "flags", "grad_train", "weight"};
  PyObject **at = &g_names.max;
  for (const char *t : text)
    if (!(*at++ = PyUnicode_InternFromString(t))) return false;
  PyObject *types = PyImport_ImportModule("types");
  g_names.ns = types ? PyObject_GetAttrString(types, "SimpleNamespace") : nullptr;
  Py_XDECREF(types);
  return g_names.ns != nullptr;
}

void put(PyObject *dict, PyObject *name, PyObject *value) {  // takes `value`
  THPObjectPtr v(value);
  if (!v || PyDict_SetItem(dict, name, v.get()) != 0) throw python_error();
}
PyObject *none() {
  Py_INCREF(Py_None);
  return Py_None;
}
PyObject *namespace_of(PyObject *dict) {
  static PyObject *empty = PyTuple_New(0);
  PyObject *r = PyObject_Call(g_names.ns, empty, dict);
  if (!r) throw python_error();
  return r;
}

// Vectors over one storage, vector i at `base` + i * `stride`.
struct Vectors {
  at::Tensor buf;
  c10::DispatchKeySet keys;
  int64_t T, stride;
  char *base;

  Vectors(const at::Tensor &like, int64_t T_, int64_t rows) : T(T_), stride((T_ + 3) / 4 * 16) {
    buf = at::empty({rows * stride}, like.options().dtype(at::kByte).requires_grad(false));
    keys = buf.key_set();
    base = static_cast<char *>(buf.data_ptr());
  }
  template <typename P>
  PyObject *make(int64_t i, at::ScalarType type, P **address) {
    *address = reinterpret_cast<P *>(base + i * stride);
    return THPVariable_Wrap(row_view(buf.storage(), keys, type, i, stride, T));
  }
};

PyObject *side(Vectors &v, int64_t first, int64_t count_row, dvp_side_out &o) {
  THPObjectPtr d(PyDict_New());
  if (!d) throw python_error();
  const Names &n = g_names;
  put(d.get(), n.max, v.make(first, at::kFloat, &o.max));
  put(d.get(), n.lse, v.make(first + 1, at::kFloat, &o.lse));
  put(d.get(), n.lse_safe, v.make(first + 2, at::kFloat, &o.lse_safe));
  put(d.get(), n.logp, v.make(first + 3, at::kFloat, &o.logp));
  put(d.get(), n.logp_mp, v.make(first + 4, at::kFloat, &o.logp_mp));
  put(d.get(), n.comp_mp, v.make(first + 5, at::kFloat, &o.comp_mp));
  put(d.get(), n.log_cov, v.make(first + 6, at::kFloat, &o.log_cov));
  put(d.get(), n.count, v.make(count_row, at::kInt, &o.count));
  put(d.get(), n.mask, none());
  return namespace_of(d.get());
}

// forward(entry, train, ids, rho, infer, upstream, grad, grad_dtype, stream, hint, mode, mask_value, weight_kind,
// weight_lo, weight_hi) -> the result, or the library's status where that is not DVP_OK.  `entry`: the address of the
// library's dvp_forward; None for tensors and the gradient's type that are not given, and for the current stream.
PyObject *forward(PyObject *, PyObject *const *args, Py_ssize_t n_args) {
  if (n_args != 15) {
    PyErr_SetString(PyExc_TypeError, "forward takes 15 arguments");
    return nullptr;
  }
  HANDLE_TH_ERRORS
  const Names &n = g_names;
  const auto entry = reinterpret_cast<int (*)(const dvp_forward_args *)>(PyLong_AsVoidPtr(args[0]));
  const at::Tensor &train = matrix(args[1], "train_logits");
  const bool has_infer = args[4] != Py_None, has_grad = args[5] != Py_None;
  dvp_forward_args a = {};
  a.struct_size = sizeof(a);
  a.rho = PyFloat_AsDouble(args[3]);
  a.stream = args[8] == Py_None ? c10::cuda::getCurrentCUDAStream().stream() : PyLong_AsVoidPtr(args[8]);
  a.launch_hint = static_cast<uint32_t>(PyLong_AsUnsignedLong(args[9]));
  a.mode = static_cast<uint32_t>(PyLong_AsUnsignedLong(args[10]));
  a.mask_value = static_cast<float>(PyFloat_AsDouble(args[11]));
  a.weight_kind = static_cast<uint32_t>(PyLong_AsUnsignedLong(args[12]));
  a.weight_lo = static_cast<float>(PyFloat_AsDouble(args[13]));
  a.weight_hi = static_cast<float>(PyFloat_AsDouble(args[14]));
  if (PyErr_Occurred()) throw python_error();
  const bool weighted = a.weight_kind != DVP_WEIGHT_NONE;
  const int64_t T = a.T = train.size(0), V = a.V = train.size(1);
  a.ld_train = train.stride(0);
  a.train_logits = train.data_ptr();
  if (has_infer) {
    const at::Tensor &infer = matrix(args[4], "infer_logits");
    if (infer.scalar_type() != train.scalar_type() || infer.size(0) != T || infer.size(1) != V)
      refuse(PyExc_ValueError, "infer_logits must match train_logits in dtype and shape");
    a.ld_infer = infer.stride(0);
    a.infer_logits = infer.data_ptr();
  }
  const int sides = has_infer ? 2 : 1, floats = 7 * sides + has_infer + weighted;
  Vectors v(train, T, floats + sides + 1);
  THPObjectPtr d(PyDict_New());
  if (!d) throw python_error();
  put(d.get(), n.train, side(v, 0, floats, a.train));
  put(d.get(), n.infer, has_infer ? side(v, 7, floats + 1, a.infer) : none());
  put(d.get(), n.log_ratio, has_infer ? v.make(14, at::kFloat, &a.log_ratio) : none());
  put(d.get(), n.flags, v.make(floats + sides, at::kByte, &a.flags));
  at::Tensor made;
  if (has_grad) {
    const at::Tensor &upstream = tensor(args[5], "upstream");
    if (upstream.scalar_type() != at::kFloat) refuse(PyExc_TypeError, "upstream must be float32");
    a.upstream = static_cast<const float *>(upstream.data_ptr());
    PyObject *grad = args[6];
    if (grad == Py_None) {
      at::ScalarType type = train.scalar_type();
      if (args[7] != Py_None) {
        if (!THPDtype_Check(args[7])) refuse(PyExc_TypeError, "grad_dtype must be a torch.dtype");
        type = reinterpret_cast<THPDtype *>(args[7])->scalar_type;
      }
      made = at::empty({T, V}, train.options().dtype(type).requires_grad(false));
      put(d.get(), n.grad_train, THPVariable_Wrap(made));
    } else {
      made = matrix(grad, "grad_train");
      Py_INCREF(grad);
      put(d.get(), n.grad_train, grad);
    }
    a.grad_dtype = dtype_code(made.scalar_type());
    a.ld_grad = made.stride(0);
    a.grad_train = made.data_ptr();
  } else {
    put(d.get(), n.grad_train, none());
  }
  if (weighted) put(d.get(), n.weight, v.make(floats - 1, at::kFloat, &a.weight_out));
  a.logits_dtype = dtype_code(train.scalar_type());
  const at::Tensor &ids = tensor(args[2], "ids");
  if (ids.scalar_type() == at::kLong)
    a.id_dtype = DVP_ID_I64;
  else if (ids.scalar_type() == at::kInt)
    a.id_dtype = DVP_ID_I32;
  else
    refuse(PyExc_TypeError, "ids must be int64 or int32");
  a.ids = ids.data_ptr();
  THPObjectPtr result(namespace_of(d.get()));
  int status;
  Py_BEGIN_ALLOW_THREADS status = entry(&a);
  Py_END_ALLOW_THREADS if (status != DVP_OK) return PyLong_FromLong(status);
  return result.release();
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"outputs", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(outputs)), METH_FASTCALL,
                          "outputs(like, T, floats, counts) -> (tensors, address, stride)"},
                         {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL,
                          "dvp_forward's arguments in, its result or the library's status out"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// PyInit__host: the module says what it was built for (build.py looks for the text in the file, binding.py asks the module)
extern "C" __attribute__((visibility("default"))) PyObject *PyInit__host() {
  static const char text[] = "[built for " DVP_HOST_TARGET "]";
  if (!make_names()) return nullptr;
  PyObject *m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_for", text) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
