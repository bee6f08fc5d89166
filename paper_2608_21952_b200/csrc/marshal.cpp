// Argument marshalling of the Python binding (paper_2608_21952_b200/binding.py): torch tensors and ctypes structures
// to the pointers the C entry points take, the current stream, the call with the interpreter lock released.  No
// arithmetic and no checks beyond the ones a pointer needs (a contiguous CUDA tensor, the right ctypes structure).
// Why native: through ctypes a call with a dozen tensors took 9 to 13 us of host time (0.25 us per tensor for
// its type checks and address, 3.4 us for the stream object) ahead of a launch of 3 us, more than the device time of
// a decode step of one sequence (7 us for its three calls); from here a call takes 3.5 to 4 us, launch included, and
// that decode step 8.1 to 9.3 us, by the machine, instead of 29.
#include <torch/csrc/autograd/python_variable.h>

#include <c10/cuda/CUDAStream.h>

#include "../../include/ssdi8.h"

namespace {

struct BadArgument {};   // a Python exception is set

// device address of a tensor, 0 for None, or an address given as an integer
void* ptr(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
      PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
      throw BadArgument{};
    }
    return t.data_ptr();
  }
  void* p = PyLong_AsVoidPtr(o);
  if (p == nullptr && PyErr_Occurred()) throw BadArgument{};
  return p;
}
template <typename T>
T* ptr_as(PyObject* o) { return static_cast<T*>(ptr(o)); }

size_t nbytes(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "a workspace is a tensor");
    throw BadArgument{};
  }
  return THPVariable_Unpack(o).nbytes();
}

long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw BadArgument{};
  return v;
}
float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw BadArgument{};
  return (float)v;
}

// The binding's ctypes types, given once at its import (init): a structure of another type, or any other object with a
// buffer, would be read as pointers and sizes that it does not hold.  The errors are those of ctypes' byref and argtypes.
struct Types {
  PyObject *dims = nullptr, *fwd = nullptr, *layer = nullptr, *ctypes_base = nullptr, *argument_error = nullptr;
} g_types;

// the memory of a ctypes structure
struct Struct {
  Py_buffer b{};
  Struct(PyObject* o, PyObject* type, size_t bytes) {
    const auto is_a = [o](PyObject* t) { return t != nullptr && PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(t)); };
    if (!is_a(type)) {
      if (is_a(g_types.ctypes_base))
        PyErr_Format(g_types.argument_error, "expected %R instead of %R", type, reinterpret_cast<PyObject*>(Py_TYPE(o)));
      else
        PyErr_Format(PyExc_TypeError, "a ctypes structure is expected, not '%s'", Py_TYPE(o)->tp_name);
      throw BadArgument{};
    }
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw BadArgument{};
    if ((size_t)b.len < bytes) {
      PyBuffer_Release(&b);
      PyErr_SetString(PyExc_TypeError, "wrong argument structure");
      throw BadArgument{};
    }
  }
  ~Struct() { PyBuffer_Release(&b); }
  Struct(const Struct&) = delete;
  Struct& operator=(const Struct&) = delete;
};
struct DimsArg : Struct {
  explicit DimsArg(PyObject* o) : Struct(o, g_types.dims, sizeof(ssdi8_dims_t)) {}
  const ssdi8_dims_t* get() const { return static_cast<const ssdi8_dims_t*>(b.buf); }
};
struct FwdArg : Struct {
  explicit FwdArg(PyObject* o) : Struct(o, g_types.fwd, sizeof(ssdi8_fwd_args_t)) {}
  const ssdi8_fwd_args_t* get() const { return static_cast<const ssdi8_fwd_args_t*>(b.buf); }
};
struct LayerArg : Struct {
  explicit LayerArg(PyObject* o) : Struct(o, g_types.layer, sizeof(ssdi8_layer_args_t)) {}
  const ssdi8_layer_args_t* get() const { return static_cast<const ssdi8_layer_args_t*>(b.buf); }
};

// the stream of a call: the current one of the current device for None, else a torch stream object's
void* stream(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw BadArgument{};
  void* p = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (p == nullptr && PyErr_Occurred()) throw BadArgument{};
  return p;
}

// the library call with the interpreter lock released; the status code as a Python integer
template <typename F>
PyObject* call(F f) {
  ssdi8_status_t s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
}

// wraps a body that throws BadArgument (exception set) or a C++ exception of torch
template <int N, typename F>
PyObject* entry(Py_ssize_t n, F f) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", N, n);
    return nullptr;
  }
  try {
    return f();
  } catch (const BadArgument&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

#define ENTRY(NAME, N) PyObject* NAME(PyObject*, PyObject* const* a, Py_ssize_t n) { return entry<N>(n, [&]() -> PyObject*
#define END ); }

ENTRY(init, 5) {   // Dims, FwdArgs, LayerArgs, the base type of ctypes objects, ctypes.ArgumentError
  for (int i = 0; i < 5; ++i) {
    if (!PyType_Check(a[i])) {
      PyErr_SetString(PyExc_TypeError, "a type is expected");
      throw BadArgument{};
    }
    Py_INCREF(a[i]);   // (kept for the life of the process, like the module)
  }
  g_types = {a[0], a[1], a[2], a[3], a[4]};
  Py_RETURN_NONE;
} END

ENTRY(quantize_act, 8) {   // inp, R, Ch, I, scale, mode, out, stream
  const float* in = ptr_as<const float>(a[0]);
  const long long R = integer(a[1]), Ch = integer(a[2]), I = integer(a[3]);
  float* scale = ptr_as<float>(a[4]);
  const int mode = (int)integer(a[5]);
  int8_t* out = ptr_as<int8_t>(a[6]);
  void* st = stream(a[7]);
  return call([=] { return ssdi8_quantize_act(in, R, Ch, I, scale, mode, out, st); });
} END

ENTRY(quantize_entry, 13) {   // xBC, dtype, T, D, G, N, s_x, s_B, s_C, xq, Bq, Cq, stream
  const void* in = ptr(a[0]);
  const int dtype = (int)integer(a[1]);
  const long long T = integer(a[2]);
  const int D = (int)integer(a[3]), G = (int)integer(a[4]), N = (int)integer(a[5]);
  const float *sx = ptr_as<const float>(a[6]), *sB = ptr_as<const float>(a[7]), *sC = ptr_as<const float>(a[8]);
  int8_t *xq = ptr_as<int8_t>(a[9]), *Bq = ptr_as<int8_t>(a[10]), *Cq = ptr_as<int8_t>(a[11]);
  void* st = stream(a[12]);
  return call([=] { return ssdi8_quantize_entry(in, dtype, T, D, G, N, sx, sB, sC, xq, Bq, Cq, st); });
} END

ENTRY(chunk_scan_fwd, 5) {   // dims, args, workspace, flags, stream
  DimsArg d(a[0]);
  FwdArg f(a[1]);
  void* ws = ptr(a[2]);
  const size_t nb = nbytes(a[2]);
  const uint32_t flags = (uint32_t)integer(a[3]);
  void* st = stream(a[4]);
  return call([&] { return ssdi8_chunk_scan_fwd(d.get(), f.get(), flags, ws, nb, st); });
} END

ENTRY(chunk_scan_fwd_static, 4) {   // dims, args, flags, stream
  DimsArg d(a[0]);
  FwdArg f(a[1]);
  const uint32_t flags = (uint32_t)integer(a[2]);
  void* st = stream(a[3]);
  return call([&] { return ssdi8_chunk_scan_fwd_static(d.get(), f.get(), flags, st); });
} END

ENTRY(layer_fwd, 5) {   // dims, args, workspace, flags, stream
  DimsArg d(a[0]);
  LayerArg f(a[1]);
  void* ws = ptr(a[2]);
  const size_t nb = nbytes(a[2]);
  const uint32_t flags = (uint32_t)integer(a[3]);
  void* st = stream(a[4]);
  return call([&] { return ssdi8_layer_fwd(d.get(), f.get(), ws, nb, flags, st); });
} END

ENTRY(layer_fwd_host, 5) {   // dims, args, scratch, flags, stream
  DimsArg d(a[0]);
  LayerArg f(a[1]);
  void* ws = ptr(a[2]);
  const size_t nb = nbytes(a[2]);
  const uint32_t flags = (uint32_t)integer(a[3]);
  void* st = stream(a[4]);
  return call([&] { return ssdi8_layer_fwd_host(d.get(), f.get(), ws, nb, flags, st); });
} END

ENTRY(calibrate, 7) {   // dims, args, s_xs, s_cb, s_h, workspace, stream
  DimsArg d(a[0]);
  FwdArg f(a[1]);
  float *sxs = ptr_as<float>(a[2]), *scb = ptr_as<float>(a[3]), *sh = ptr_as<float>(a[4]);
  void* ws = ptr(a[5]);
  const size_t nb = nbytes(a[5]);
  void* st = stream(a[6]);
  return call([&] { return ssdi8_calibrate(d.get(), f.get(), sxs, scb, sh, ws, nb, st); });
} END

ENTRY(mean_correction, 8) {   // y_ref, y_q, R, Ch, eta, corr, workspace, stream
  const float *y = ptr_as<const float>(a[0]), *yq = ptr_as<const float>(a[1]);
  const long long R = integer(a[2]), Ch = integer(a[3]);
  const float eta = real(a[4]);
  float* corr = ptr_as<float>(a[5]);
  void* ws = ptr(a[6]);
  const size_t nb = nbytes(a[6]);
  void* st = stream(a[7]);
  return call([=] { return ssdi8_mean_correction(y, yq, R, Ch, eta, corr, ws, nb, st); });
} END

ENTRY(state_passing, 9) {   // dims, loc, gamma, init_state, prev, final_state, hq, s_h, stream
  DimsArg d(a[0]);
  const float *loc = ptr_as<const float>(a[1]), *gamma = ptr_as<const float>(a[2]), *init = ptr_as<const float>(a[3]);
  float *prev = ptr_as<float>(a[4]), *fin = ptr_as<float>(a[5]);
  int8_t* hq = ptr_as<int8_t>(a[6]);
  const float* sh = ptr_as<const float>(a[7]);
  void* st = stream(a[8]);
  return call([&] { return ssdi8_state_passing(d.get(), loc, gamma, init, prev, fin, hq, sh, st); });
} END

ENTRY(ssd_step, 14) {   // dims, xq, s_x, Bq, s_B, Cq, s_C, dt, A, D, corr, state, y, stream
  DimsArg d(a[0]);
  const int8_t* xq = ptr_as<const int8_t>(a[1]);
  const float* sx = ptr_as<const float>(a[2]);
  const int8_t* Bq = ptr_as<const int8_t>(a[3]);
  const float* sB = ptr_as<const float>(a[4]);
  const int8_t* Cq = ptr_as<const int8_t>(a[5]);
  const float* sC = ptr_as<const float>(a[6]);
  const float *dt = ptr_as<const float>(a[7]), *A = ptr_as<const float>(a[8]), *D = ptr_as<const float>(a[9]),
              *corr = ptr_as<const float>(a[10]);
  float *state = ptr_as<float>(a[11]), *y = ptr_as<float>(a[12]);
  void* st = stream(a[13]);
  return call([&] { return ssdi8_ssd_step(d.get(), xq, sx, Bq, sB, Cq, sC, dt, A, D, corr, state, y, st); });
} END

ENTRY(softplus_dt, 6) {   // dt_raw, dt_bias, rows, H, dt, stream
  const float *raw = ptr_as<const float>(a[0]), *bias = ptr_as<const float>(a[1]);
  const long long rows = integer(a[2]);
  const int H = (int)integer(a[3]);
  float* dt = ptr_as<float>(a[4]);
  void* st = stream(a[5]);
  return call([=] { return ssdi8_softplus_dt(raw, bias, rows, H, dt, st); });
} END

#undef ENTRY
#undef END

#define METHOD(NAME) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(NAME)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {METHOD(init), METHOD(quantize_act), METHOD(quantize_entry), METHOD(chunk_scan_fwd), METHOD(chunk_scan_fwd_static),
                          METHOD(layer_fwd), METHOD(layer_fwd_host), METHOD(calibrate), METHOD(mean_correction),
                          METHOD(state_passing), METHOD(ssd_step), METHOD(softplus_dt), {nullptr, nullptr, 0, nullptr}};
#undef METHOD

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  PyObject* m = PyModule_Create(&kModule);
  // the torch whose C++ classes this was compiled against: the binding compares it with the torch that is loaded
  if (m && PyModule_AddStringConstant(m, "TORCH_VERSION", SSDI8_TORCH_VERSION) != 0) Py_CLEAR(m);
  return m;
}
