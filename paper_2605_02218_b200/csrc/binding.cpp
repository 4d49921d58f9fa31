// Native part of the Python binding (api.py) for the calls that are shorter on the device than their submission from Python:
// the checks, the result tensors, the addresses and the call into the library in one step.  The library sees addresses only,
// so every tensor is held against what the kernels will read or write of it.  Everything that is not the usual case (other
// argument types, tensors that do not fit, another device than the current one) goes back to Python, which says what is wrong
// or makes the call itself.  The library's functions are handed over as addresses by api.py, so that they come from the
// library it has loaded (bind).
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

namespace {

using CorrectFn = int (*)(int, int, int, long long, const void*, const void*, const int*, const float*, float, float*, int*,
                          float*, float*, int*, void*);
using CandidatesFn = int (*)(int, int, int, long long, const void*, const int*, const int*, int, int*, void*);
using StaticFn = int (*)(int, int, int, const void*, const int*, const void*, const int*, float*, void*);
CorrectFn g_correct = nullptr;
CandidatesFn g_candidates = nullptr;
StaticFn g_static = nullptr;

PyObject* bind(PyObject*, PyObject* args) {
  unsigned long long a = 0, b = 0, c = 0;
  if (!PyArg_ParseTuple(args, "KKK", &a, &b, &c)) return nullptr;
  g_correct = reinterpret_cast<CorrectFn>(static_cast<uintptr_t>(a));
  g_candidates = reinterpret_cast<CandidatesFn>(static_cast<uintptr_t>(b));
  g_static = reinterpret_cast<StaticFn>(static_cast<uintptr_t>(c));
  Py_RETURN_NONE;
}

// COVSPEC_F32, COVSPEC_BF16, COVSPEC_F16 (covspec.h); -1: no logit type
int dtype_code(const at::Tensor& t) {
  switch (t.scalar_type()) {
    case at::kFloat: return 0;
    case at::kBFloat16: return 1;
    case at::kHalf: return 2;
    default: return -1;
  }
}
// Dense memory of at least `least` elements of this type on the call's device.
bool fits(const at::Tensor& t, at::ScalarType type, const at::Device& dev, long long least) {
  return t.device() == dev && t.scalar_type() == type && t.is_contiguous() && t.numel() >= least;
}
// The call's tensors lie on the current device, whose stream takes the launch.
bool on_current_device(const at::Tensor& t) { return t.is_cuda() && t.device().index() == c10::cuda::current_device(); }
bool is_int(long long v) { return v >= INT_MIN && v <= INT_MAX; }
bool int_arg(PyObject* o, long long& v) {
  v = PyLong_AsLongLong(o);
  return !(v == -1 && PyErr_Occurred());
}
// The memory of a C-contiguous int32 array; released when the view goes.
struct IntArray {
  Py_buffer view{};
  bool held = false;
  bool get(PyObject* o, bool writable) {
    if (PyObject_GetBuffer(o, &view, PyBUF_C_CONTIGUOUS | (writable ? PyBUF_WRITABLE : 0))) return false;
    held = true;
    if (view.itemsize != 4) { PyErr_SetString(PyExc_TypeError, "int32 array required"); return false; }
    return true;
  }
  int* data() const { return static_cast<int*>(view.buf); }
  long long size() const { return view.len / 4; }
  ~IntArray() { if (held) PyBuffer_Release(&view); }
};
// The library's call with the interpreter lock released, as ctypes does: a launch may wait for the device's queue.
template <typename F, typename... A>
int call(F f, A... args) {
  int st = 0;
  Py_BEGIN_ALLOW_THREADS
  st = f(args...);
  Py_END_ALLOW_THREADS
  return st;
}
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// correct(z_draft, z_target, uniforms or None, gamma, drafted or None, vocab) -> (margin, gate, accept, mass, token), or the
// library's status; None where an argument is not of the usual kind.
PyObject* correct(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6 || !THPVariable_Check(a[0]) || !THPVariable_Check(a[1]) || !(a[2] == Py_None || THPVariable_Check(a[2])) ||
      !(a[4] == Py_None || THPVariable_Check(a[4])))
    Py_RETURN_NONE;
  const at::Tensor &zd = THPVariable_Unpack(a[0]), &zt = THPVariable_Unpack(a[1]);
  if (!on_current_device(zd) || zd.dim() != 2 || !zd.is_contiguous() || dtype_code(zd) < 0 || !zd.sizes().equals(zt.sizes()) ||
      !fits(zt, zd.scalar_type(), zd.device(), zd.numel()))
    Py_RETURN_NONE;
  const long long rows = zd.size(0), ld = zd.size(1);
  if ((a[2] != Py_None && !fits(THPVariable_Unpack(a[2]), at::kFloat, zd.device(), rows)) ||
      (a[4] != Py_None && !fits(THPVariable_Unpack(a[4]), at::kInt, zd.device(), rows)))
    Py_RETURN_NONE;
  const double gamma = PyFloat_AsDouble(a[3]);
  if (gamma == -1.0 && PyErr_Occurred()) return nullptr;
  long long vocab = ld;
  if (a[5] != Py_None && !int_arg(a[5], vocab)) return nullptr;
  if (!is_int(vocab) || !is_int(rows)) Py_RETURN_NONE;
  const auto f32 = zd.options().dtype(at::kFloat), i32 = zd.options().dtype(at::kInt);
  at::Tensor margin = at::empty({rows}, f32), gate = at::empty({rows}, i32), accept = at::empty({rows}, f32),
             mass = at::empty({rows}, f32), token = at::empty({rows}, i32);
  const void* drafted = a[4] == Py_None ? nullptr : THPVariable_Unpack(a[4]).data_ptr();
  const void* uniforms = a[2] == Py_None ? nullptr : THPVariable_Unpack(a[2]).data_ptr();
  const int st = call(g_correct, dtype_code(zd), (int)rows, (int)vocab, ld, zd.data_ptr(), zt.data_ptr(), static_cast<const int*>(drafted),
                           static_cast<const float*>(uniforms), (float)gamma, static_cast<float*>(margin.data_ptr()),
                           static_cast<int*>(gate.data_ptr()), static_cast<float*>(accept.data_ptr()),
                           static_cast<float*>(mass.data_ptr()), static_cast<int*>(token.data_ptr()), current_stream());
  if (st) return PyLong_FromLong(st);
  PyObject* out = PyTuple_New(5);
  if (!out) return nullptr;
  PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(std::move(margin)));
  PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(std::move(gate)));
  PyTuple_SET_ITEM(out, 2, THPVariable_Wrap(std::move(accept)));
  PyTuple_SET_ITEM(out, 3, THPVariable_Wrap(std::move(mass)));
  PyTuple_SET_ITEM(out, 4, THPVariable_Wrap(std::move(token)));
  return out;
  END_HANDLE_TH_ERRORS
}

// candidates(z_draft, fanouts: list of int, off: int32 array of rows + 1, filled in, drafted or None, vocab) -> cand, or the
// library's status; None where an argument is not of the usual kind.
PyObject* candidates(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 5 || !THPVariable_Check(a[0]) || !PyList_CheckExact(a[1]) || !(a[3] == Py_None || THPVariable_Check(a[3]))) Py_RETURN_NONE;
  const at::Tensor& z = THPVariable_Unpack(a[0]);
  if (!on_current_device(z) || z.dim() != 2 || !z.is_contiguous() || dtype_code(z) < 0) Py_RETURN_NONE;
  const long long rows = z.size(0), ld = z.size(1);
  if (a[3] != Py_None && !fits(THPVariable_Unpack(a[3]), at::kInt, z.device(), rows)) Py_RETURN_NONE;
  IntArray off;
  if (!off.get(a[2], true)) return nullptr;
  if (PyList_GET_SIZE(a[1]) != rows || off.size() != rows + 1 || rows < 1) Py_RETURN_NONE;
  long long vocab = ld, total = 0, most = 0;
  if (a[4] != Py_None && !int_arg(a[4], vocab)) return nullptr;
  if (!is_int(vocab) || !is_int(rows)) Py_RETURN_NONE;
  off.data()[0] = 0;
  for (long long r = 0; r < rows; ++r) {
    PyObject* item = PyList_GET_ITEM(a[1], r);
    if (!PyLong_CheckExact(item)) Py_RETURN_NONE;
    int overflow = 0;
    const long long f = PyLong_AsLongLongAndOverflow(item, &overflow);
    if (overflow || f < 0 || f > 0x7fffffff) Py_RETURN_NONE;
    total += f;
    if (total > 0x7fffffff) Py_RETURN_NONE;
    most = r == 0 || f > most ? f : most;
    off.data()[r + 1] = (int)total;
  }
  at::Tensor cand = at::empty({total > 0 ? total : 1}, z.options().dtype(at::kInt));
  const void* drafted = a[3] == Py_None ? nullptr : THPVariable_Unpack(a[3]).data_ptr();
  const int st = call(g_candidates, dtype_code(z), (int)rows, (int)vocab, ld, z.data_ptr(), static_cast<const int*>(drafted),
                              off.data(), (int)most, static_cast<int*>(cand.data_ptr()), current_stream());
  if (st) return PyLong_FromLong(st);
  return THPVariable_Wrap(total ? std::move(cand) : cand.slice(0, 0, 0));
  END_HANDLE_TH_ERRORS
}

// static_score(X, Q, vis, txt: int32 arrays, out) -> the library's status; None where an argument is not of the usual kind.
PyObject* static_score(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 5 || !THPVariable_Check(a[0]) || !THPVariable_Check(a[1]) || !THPVariable_Check(a[4])) Py_RETURN_NONE;
  IntArray vis, txt;
  if (!vis.get(a[2], false) || !txt.get(a[3], false)) return nullptr;
  const at::Tensor &x = THPVariable_Unpack(a[0]), &q = THPVariable_Unpack(a[1]), &out = THPVariable_Unpack(a[4]);
  const at::ScalarType type = x.scalar_type();
  if (!on_current_device(x) || (type != at::kBFloat16 && type != at::kFloat) || x.dim() != 2 || q.dim() != 2 || x.size(1) != q.size(1) ||
      !is_int(x.size(1)) || vis.size() < 2 || vis.size() != txt.size() || !is_int(vis.size()))
    Py_RETURN_NONE;
  // the library refuses offsets that do not ascend from 0, so the last ones say what is read
  const long long d = x.size(1), rows_x = vis.data()[vis.size() - 1], rows_q = txt.data()[txt.size() - 1];
  if (!fits(x, type, x.device(), rows_x * d) || !fits(q, type, x.device(), rows_q * d) || !fits(out, at::kFloat, x.device(), rows_x))
    Py_RETURN_NONE;
  const int st = call(g_static, type == at::kBFloat16 ? 1 : 0, (int)d, (int)vis.size() - 1, x.data_ptr(), vis.data(), q.data_ptr(),
                      txt.data(), static_cast<float*>(out.data_ptr()), current_stream());
  return PyLong_FromLong(st);
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, nullptr},
                         {"correct", (PyCFunction)(void (*)(void))correct, METH_FASTCALL, nullptr},
                         {"candidates", (PyCFunction)(void (*)(void))candidates, METH_FASTCALL, nullptr},
                         {"static_score", (PyCFunction)(void (*)(void))static_score, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module_def); }
