// CPython side of the entry points that enqueue GPU work: argument marshalling only.
//
// A decode call is a few microseconds on the GPU, so what the host spends per call is part of its cost.  Going
// through ctypes, a kmq_linear call took 9.4 us of host time from Python (256 x 256, b = 1, M = 1, back to back), 2.1 us
// of it the launch: ctypes' conversion of 13 arguments, the Python frames around it and torch's stream object were the
// rest.  Here the arguments are read in place (vectorcall, no tuples): 3.8 us, 3.5 us without entering torch's Python
// layer for the tensors and the stream.  The GIL is released around the library call, as ctypes does.
//
// torch tensors go through torch's DLPack exchange table (a C function per tensor, and one for the current stream); what
// it does not describe, or another tensor library's object, is asked for data_ptr() instead.  Built against a torch whose
// headers do not have the table (it came with DLPack 1.3; 2.11 has it), everything is: 7.5 instead of 3.1 us a call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#if defined(__has_include)
#if __has_include(<ATen/dlpack.h>)
#include <ATen/dlpack.h>
#endif
#endif
#if defined(DLPACK_MAJOR_VERSION) && defined(DLPACK_MINOR_VERSION)
#if DLPACK_MAJOR_VERSION > 1 || (DLPACK_MAJOR_VERSION == 1 && DLPACK_MINOR_VERSION >= 3)
#define KMQ_HAVE_EXCHANGE_TABLE 1
#endif
#endif

#include <stdint.h>
#include <string.h>
#include <tuple>
#include <utility>

#include "kmq.h"

extern "C" int kmq_internal_current_device(void);   // of libkmq, beside its interface: -1 on error

namespace {

constexpr int kMaxParams = 16;

PyObject* s_data_ptr;        // interned attribute names
PyObject* s_cuda_stream;
PyObject* s_numel;
PyObject* s_element_size;
PyObject* g_error = nullptr;          // KmqError, handed over by the Python module
#ifdef KMQ_HAVE_EXCHANGE_TABLE
PyTypeObject* g_tensor_type = nullptr;               // torch.Tensor, once one was seen
const DLPackExchangeAPI* g_exchange = nullptr;       // its exchange table
bool g_cuda_ready = false;                           // torch's CUDA side is set up
#endif

// ---- one argument -> one C value; false with a Python error set ----
bool to_c(PyObject* o, int64_t* v) {
  *v = PyLong_AsLongLong(o);
  return !(*v == -1 && PyErr_Occurred());
}
bool to_c(PyObject* o, int* v) {
  const long x = PyLong_AsLong(o);
  *v = (int)x;
  return !(x == -1 && PyErr_Occurred());
}
bool to_c(PyObject* o, size_t* v) {
  *v = PyLong_AsSize_t(o);
  return !(*v == (size_t)-1 && PyErr_Occurred());
}
#ifdef KMQ_HAVE_EXCHANGE_TABLE
// Finds torch's exchange table; called with an object whose type may be torch.Tensor.
void find_exchange(PyObject* o) {
  PyTypeObject* const type = Py_TYPE(o);
  if (strcmp(type->tp_name, "Tensor") != 0) return;
  PyObject* capsule = PyObject_GetAttrString(reinterpret_cast<PyObject*>(type), "__dlpack_c_exchange_api__");
  if (capsule && PyCapsule_CheckExact(capsule)) {
    auto* table = static_cast<const DLPackExchangeAPI*>(PyCapsule_GetPointer(capsule, "dlpack_exchange_api"));
    if (table && table->header.version.major == DLPACK_MAJOR_VERSION && table->dltensor_from_py_object_no_sync &&
        table->current_work_stream) {
      Py_INCREF(type);
      g_tensor_type = type;
      g_exchange = table;
    }
  }
  Py_XDECREF(capsule);
  PyErr_Clear();
}
#endif

// None, an address, or an object with data_ptr()
bool to_address(PyObject* o, void** v) {
  if (o == Py_None) {
    *v = nullptr;
    return true;
  }
  if (PyLong_Check(o)) {
    *v = PyLong_AsVoidPtr(o);
    return *v || !PyErr_Occurred();
  }
#ifdef KMQ_HAVE_EXCHANGE_TABLE
  if (!g_tensor_type) find_exchange(o);
  if (Py_TYPE(o) == g_tensor_type) {
    DLTensor t;
    if (g_exchange->dltensor_from_py_object_no_sync(o, &t) == 0) {
      *v = static_cast<char*>(t.data) + t.byte_offset;
      return true;
    }
    PyErr_Clear();   // e.g. a type that DLPack has no name for
  }
#endif
  PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!r) return false;
  *v = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *v || !PyErr_Occurred();
}
template <class T>
bool to_c(PyObject* o, T** v) {
  void* p;
  if (!to_address(o, &p)) return false;
  *v = static_cast<T*>(p);
  return true;
}

// torch's current stream on the current device.  The first call goes through torch's public object, which also sets
// CUDA up.
bool current_stream(void** stream) {
#ifdef KMQ_HAVE_EXCHANGE_TABLE
  if (g_cuda_ready && g_exchange) {
    const int dev = kmq_internal_current_device();
    if (dev >= 0) return g_exchange->current_work_stream(kDLCUDA, dev, stream) == 0;
  }
#endif
  PyObject* cuda = PyImport_ImportModule("torch.cuda");
  PyObject* st = cuda ? PyObject_CallMethod(cuda, "current_stream", nullptr) : nullptr;
  PyObject* r = st ? PyObject_GetAttr(st, s_cuda_stream) : nullptr;
  Py_XDECREF(cuda);
  Py_XDECREF(st);
  if (!r) return false;
#ifdef KMQ_HAVE_EXCHANGE_TABLE
  g_cuda_ready = true;
#endif
  *stream = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *stream || !PyErr_Occurred();
}
bool to_stream(PyObject* o, void** stream) {
  if (!o || o == Py_None) return current_stream(stream);
  if (PyLong_Check(o)) {
    *stream = PyLong_AsVoidPtr(o);
    return *stream || !PyErr_Occurred();
  }
  PyObject* r = PyObject_GetAttr(o, s_cuda_stream);
  if (!r) return false;
  *stream = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *stream || !PyErr_Occurred();
}

// Size of a workspace tensor in bytes; 0 for None and for a bare address.
bool tensor_bytes(PyObject* o, size_t* v) {
  *v = 0;
  if (!o || o == Py_None || PyLong_Check(o)) return true;
  PyObject* n = PyObject_CallMethodNoArgs(o, s_numel);
  PyObject* e = n ? PyObject_CallMethodNoArgs(o, s_element_size) : nullptr;
  size_t a = 0, b = 0;
  const bool ok = e && to_c(n, &a) && to_c(e, &b);
  Py_XDECREF(n);
  Py_XDECREF(e);
  *v = a * b;
  return ok;
}

// ---- one entry point ----
// Python parameters in order; a name with '=' has a default: "=N" no value (None), "=<int>" that integer.  Every
// entry point takes "stream=N" and "check=1" as its last two.  `order[i]` is the Python parameter behind C argument i
// (the C stream argument is always the last one).
struct Entry {
  const char* name;
  const char* params[kMaxParams];
  int order[kMaxParams];
  const char* doc;
  // filled at import
  int n_params;
  PyObject* names[kMaxParams];
  PyObject* defaults[kMaxParams];   // nullptr: required
  int workspace, workspace_bytes;   // parameter numbers, -1 where the entry point has none
};

// The arguments of one call in parameter order (borrowed references).
bool collect(const Entry& e, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames, PyObject** slot) {
  if (nargs > e.n_params) {
    PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments", e.name, e.n_params);
    return false;
  }
  for (Py_ssize_t i = 0; i < nargs; ++i) slot[i] = args[i];
  for (int i = (int)nargs; i < e.n_params; ++i) slot[i] = nullptr;
  const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t k = 0; k < nkw; ++k) {
    PyObject* key = PyTuple_GET_ITEM(kwnames, k);
    int at = -1;
    for (int i = e.n_params - 1; i >= 0 && at < 0; --i)
      if (e.names[i] == key) at = i;
    for (int i = e.n_params - 1; i >= 0 && at < 0; --i)
      if (PyUnicode_Compare(e.names[i], key) == 0) at = i;
    if (at < 0) {
      PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", e.name, key);
      return false;
    }
    if (slot[at]) {
      PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%U'", e.name, key);
      return false;
    }
    slot[at] = args[nargs + k];
  }
  for (int i = 0; i < e.n_params; ++i) {
    if (!slot[i]) slot[i] = e.defaults[i];
    if (!slot[i]) {
      PyErr_Format(PyExc_TypeError, "%s() missing required argument '%U'", e.name, e.names[i]);
      return false;
    }
  }
  return true;
}

PyObject* finish(const Entry& e, int status, PyObject* check) {
  if (status != KMQ_OK) {
    const int raise = PyObject_IsTrue(check);
    if (raise < 0) return nullptr;
    if (raise) {
      PyObject* exc = g_error ? PyObject_CallFunction(g_error, "is", status, e.name) : nullptr;
      if (exc) {
        PyErr_SetObject(g_error, exc);
        Py_DECREF(exc);
      } else if (!PyErr_Occurred()) {
        PyErr_Format(PyExc_RuntimeError, "%s: status %d", e.name, status);
      }
      return nullptr;
    }
  }
  return PyLong_FromLong(status);
}

template <class T>
bool convert(const Entry& e, PyObject* const* slot, int param, T* v) {
  return to_c(slot[param], v);
}
template <>
bool convert<size_t>(const Entry& e, PyObject* const* slot, int param, size_t* v) {
  if (param == e.workspace_bytes && slot[param] == Py_None) return tensor_bytes(slot[e.workspace], v);
  return to_c(slot[param], v);
}

// Splits the trailing stream argument off a prototype, then converts, calls and reports.
template <class Done, class... Rest>
struct Split;
template <class... Done>
struct Split<std::tuple<Done...>, void*> {
  using Fn = kmq_status (*)(Done..., void*);
  static PyObject* run(const Entry& e, Fn fn, PyObject* const* slot) {
    return run(e, fn, slot, std::index_sequence_for<Done...>{});
  }
  template <size_t... I>
  static PyObject* run(const Entry& e, Fn fn, PyObject* const* slot, std::index_sequence<I...>) {
    std::tuple<Done...> v;
    void* stream;
    if (!(convert(e, slot, e.order[I], &std::get<I>(v)) && ...)) return nullptr;
    if (!to_stream(slot[e.n_params - 2], &stream)) return nullptr;
    kmq_status st;
    Py_BEGIN_ALLOW_THREADS;
    st = fn(std::get<I>(v)..., stream);
    Py_END_ALLOW_THREADS;
    return finish(e, st, slot[e.n_params - 1]);
  }
};
template <class... Done, class First, class Second, class... Rest>
struct Split<std::tuple<Done...>, First, Second, Rest...> : Split<std::tuple<Done..., First>, Second, Rest...> {};

template <class... A>
PyObject* call(const Entry& e, kmq_status (*fn)(A...), PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  PyObject* slot[kMaxParams];
  if (!collect(e, args, nargs, kwnames, slot)) return nullptr;
  return Split<std::tuple<>, A...>::run(e, fn, slot);
}

enum {
  kPack, kUnpack, kLinear, kLinearHost, kLinearStatic, kLinearTcgen05, kDequant, kBlockPack, kBlockLinear,
  kBlockDequant, kBlockTablePack, kBlockTableUnpack, kBlockTableLinear, kKmeansRows, kAssignPack, kQuantizeRows,
  kBlockScales, kBlockSample, kBlockAssignPack, kBlockQuantize, kProbeLaunch, kProbeRead, kEntries
};

Entry g_entry[kEntries] = {
    {"kmq_pack", {"idx", "N", "K", "bits", "packed", "layout=0", "stream=N", "check=1"}, {0, 1, 2, 3, 5, 4},
     "Centroid indices uint8 [N, K] -> packed words in `layout`."},
    {"kmq_unpack", {"packed", "N", "K", "bits", "idx", "layout=0", "stream=N", "check=1"}, {0, 1, 2, 3, 5, 4},
     "Packed words -> centroid indices uint8 [N, K]."},
    {"kmq_linear",
     {"packed", "codebooks", "x", "y", "N", "K", "bits", "M", "workspace=N", "workspace_bytes=N", "layout=0",
      "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 10, 8, 9},
     "y = x * W^T with per-row codebooks."},
    {"kmq_linear_host",
     {"packed", "codebooks", "x_host", "y_host", "N", "K", "bits", "M", "x_dev", "y_dev", "workspace=N",
      "workspace_bytes=N", "layout=0", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 12, 8, 9, 10, 11},
     "kmq_linear with activations and result in host memory; synchronises the stream."},
    {"kmq_linear_static_scratch",
     {"packed", "codebooks", "x", "y", "N", "K", "bits", "M", "layout=0", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 8},
     "kmq_linear for callers that may not allocate: scratch, where needed, is a fixed array inside the library."},
    {"kmq_linear_tcgen05", {"packed", "codebooks", "x", "y", "N", "K", "bits", "M", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7},
     "kmq_linear through the tcgen05 / tensor-memory kernel (tuned layout only)."},
    {"kmq_dequant_to_bf16", {"packed", "codebooks", "W", "N", "K", "bits", "layout=0", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6},
     "Packed words and codebooks -> dense bf16 W [N, K]."},
    {"kmq_block_pack", {"idx", "N", "K", "bits", "wq", "stream=N", "check=1"}, {0, 1, 2, 3, 4},
     "Block format: indices uint8 [N, K] -> bytes."},
    {"kmq_block_linear",
     {"wq", "scales", "codebook", "x", "y", "N", "K", "bits", "M", "scale_order=1", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 8, 9},
     "The paper's block format (shared codebook, bf16 scale per block of 64): y = x * W^T."},
    {"kmq_block_dequant_to_bf16", {"wq", "scales", "codebook", "W", "N", "K", "bits", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6},
     "Block format -> dense bf16 W [N, K]."},
    {"kmq_block_table_pack", {"wq", "scales", "N", "K", "bits", "table", "stream=N", "check=1"}, {0, 1, 2, 3, 4, 5},
     "Block format: byte layout -> table layout."},
    {"kmq_block_table_unpack", {"table", "N", "K", "bits", "wq", "scales", "stream=N", "check=1"}, {0, 1, 2, 3, 4, 5},
     "Block format: table layout -> byte layout."},
    {"kmq_block_table_linear",
     {"table", "codebook", "x", "y", "N", "K", "bits", "M", "workspace=N", "workspace_bytes=0", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 8, 9},
     "Block format through the activation table: y = x * W^T, one pass per batch row."},
    {"kmq_kmeans_rows", {"W", "N", "K", "bits", "iters", "codebooks", "centroids=N", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6},
     "Per-row 1-D Lloyd fit: W float32 [N, K] -> codebooks bf16 [N, 2^bits] (and float64 centroids if given)."},
    {"kmq_assign_pack", {"W", "codebooks", "N", "K", "bits", "layout", "packed", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6},
     "Nearest stored centroid of every weight, written as packed indices in `layout`."},
    {"kmq_quantize_rows", {"W", "N", "K", "bits", "iters", "layout", "codebooks", "packed", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7},
     "kmq_kmeans_rows, then kmq_assign_pack with the stored codebooks."},
    {"kmq_block_scales", {"W", "N", "K", "lam", "scales", "stream=N", "check=1"}, {0, 1, 2, 3, 4},
     "Block format: bf16 scale of every block of 64 weights."},
    {"kmq_block_sample", {"W", "scales", "N", "K", "samples", "out", "stream=N", "check=1"}, {0, 1, 2, 3, 4, 5},
     "Block format: strided sample of the normalised weights."},
    {"kmq_block_assign_pack", {"W", "scales", "codebook", "N", "K", "bits", "wq", "stream=N", "check=1"},
     {0, 1, 2, 3, 4, 5, 6},
     "Block format: nearest centroid of every normalised weight, packed."},
    {"kmq_block_quantize",
     {"W", "N", "K", "bits", "lam", "iters", "samples", "scales", "codebook", "wq", "sample_workspace", "stream=N",
      "check=1"},
     {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10},
     "Block format, all steps: scales, strided normalised sample, shared codebook fit, packed indices."},
    {"kmq_probe_launch", {"stream=N", "check=1"}, {}, "Enqueue the do-nothing kernel (the fixed cost of a call)."},
    {"kmq_probe_read", {"buf", "nbytes", "out", "stream=N", "check=1"}, {0, 1, 2},
     "Read `nbytes` of `buf` once with streaming loads (the read-only bandwidth ceiling)."},
};

template <int E, auto Fn>
PyObject* method(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  return call(g_entry[E], Fn, args, nargs, kwnames);
}

template <int E, auto Fn>
constexpr PyMethodDef define() {
  return {nullptr, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&method<E, Fn>)),
          METH_FASTCALL | METH_KEYWORDS, nullptr};
}

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

PyMethodDef g_methods[kEntries + 2];

bool prepare_entry(Entry& e) {
  e.workspace = e.workspace_bytes = -1;
  for (e.n_params = 0; e.n_params < kMaxParams && e.params[e.n_params]; ++e.n_params) {
    const char* p = e.params[e.n_params];
    const char* eq = strchr(p, '=');
    PyObject* name = PyUnicode_FromStringAndSize(p, eq ? eq - p : (Py_ssize_t)strlen(p));
    if (!name) return false;
    PyUnicode_InternInPlace(&name);
    e.names[e.n_params] = name;
    e.defaults[e.n_params] = nullptr;
    if (eq) {
      e.defaults[e.n_params] = eq[1] == 'N' ? Py_None : PyLong_FromLong(eq[1] - '0');
      if (!e.defaults[e.n_params]) return false;
    }
    if (PyUnicode_CompareWithASCIIString(name, "workspace") == 0) e.workspace = e.n_params;
    if (PyUnicode_CompareWithASCIIString(name, "workspace_bytes") == 0) e.workspace_bytes = e.n_params;
  }
  return true;
}

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_kmq_native", "Entry points of libkmq that enqueue GPU work.", -1,
                        g_methods};

}  // namespace

PyMODINIT_FUNC PyInit__kmq_native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  if (!s_data_ptr || !s_cuda_stream || !s_numel || !s_element_size) return nullptr;
  const PyMethodDef defs[kEntries] = {
      define<kPack, &kmq_pack>(), define<kUnpack, &kmq_unpack>(), define<kLinear, &kmq_linear>(),
      define<kLinearHost, &kmq_linear_host>(), define<kLinearStatic, &kmq_linear_static_scratch>(),
      define<kLinearTcgen05, &kmq_linear_tcgen05>(), define<kDequant, &kmq_dequant_to_bf16>(),
      define<kBlockPack, &kmq_block_pack>(), define<kBlockLinear, &kmq_block_linear>(),
      define<kBlockDequant, &kmq_block_dequant_to_bf16>(), define<kBlockTablePack, &kmq_block_table_pack>(),
      define<kBlockTableUnpack, &kmq_block_table_unpack>(), define<kBlockTableLinear, &kmq_block_table_linear>(),
      define<kKmeansRows, &kmq_kmeans_rows>(), define<kAssignPack, &kmq_assign_pack>(),
      define<kQuantizeRows, &kmq_quantize_rows>(), define<kBlockScales, &kmq_block_scales>(),
      define<kBlockSample, &kmq_block_sample>(), define<kBlockAssignPack, &kmq_block_assign_pack>(),
      define<kBlockQuantize, &kmq_block_quantize>(), define<kProbeLaunch, &kmq_probe_launch>(),
      define<kProbeRead, &kmq_probe_read>(),
  };
  for (int i = 0; i < kEntries; ++i) {
    if (!prepare_entry(g_entry[i])) return nullptr;
    g_methods[i] = defs[i];
    g_methods[i].ml_name = g_entry[i].name;
    g_methods[i].ml_doc = g_entry[i].doc;
  }
  g_methods[kEntries] = {"set_error", set_error, METH_O, "The exception class raised for a failed status."};
  g_methods[kEntries + 1] = {nullptr, nullptr, 0, nullptr};
  return PyModule_Create(&g_module);
}
