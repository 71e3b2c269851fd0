// The Python binding's call path in native code: reads the tensors of a call,
// allocates its outputs, takes the current stream and calls the C ABI
// (include/hive.h) through the address that ctypes resolved.
//
// Each function returns NotImplemented whenever an argument is not the plain
// case (a tensor subclass, an active function or dispatch mode, a wrong
// device, size or layout): the Python code of hive.py then takes the call and
// handles or refuses it, so the two agree on everything that is accepted.
//
// Why: the attribute calls of one tensor argument cost Python about 0.6 us and
// an output tensor 2.5 us, more than the kernels of a small batch take.
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>

#include <cstdint>
#include <exception>
#include <vector>

#include "hive.h"

namespace {

// A call that the Python code has to take.
struct NotPlain {};

bool modes_active() {
  return at::impl::torch_function_mode_enabled() ||
         c10::impl::TorchDispatchModeTLS::any_modes_set();
}

const at::Tensor& tensor_of(PyObject* o) {
  if (!THPVariable_CheckExact(o)) throw NotPlain();
  return THPVariable_Unpack(o);
}

// Refuses all but a contiguous CUDA tensor with >= n items of `item` bytes (or,
// with `host`, which is then set, a pinned CPU tensor).
void check_plain(const at::Tensor& t, size_t item, int64_t n, bool* host) {
  if (!t.is_cuda()) {
    if (!host || !t.device().is_cpu() || !t.is_pinned()) throw NotPlain();
    *host = true;
  }
  if (!t.has_storage() || !t.is_contiguous() || t.element_size() != item || t.numel() < n)
    throw NotPlain();
}
// Pointer of an input tensor; NULL for None.
const void* in_ptr(const at::Tensor& t, size_t item, int64_t n, bool* host = nullptr) {
  check_plain(t, item, n, host);
  return t.const_data_ptr();
}
const void* in_ptr(PyObject* o, size_t item, int64_t n, bool* host = nullptr) {
  if (!o || o == Py_None) return nullptr;
  return in_ptr(tensor_of(o), item, n, host);
}
// Pointer of an output tensor; NULL for None.  A copy-on-write tensor gets its
// own storage first, as data_ptr() gives it in Python: the kernels write it.
void* out_ptr(const at::Tensor& t, size_t item, int64_t n, bool* host = nullptr) {
  check_plain(t, item, n, host);
  return t.mutable_data_ptr();
}
void* out_ptr(PyObject* o, size_t item, int64_t n, bool* host = nullptr) {
  if (!o || o == Py_None) return nullptr;
  return out_ptr(tensor_of(o), item, n, host);
}

void* as_address(PyObject* o) {
  void* p = PyLong_AsVoidPtr(o);
  if (!p && PyErr_Occurred()) {
    PyErr_Clear();
    throw NotPlain();
  }
  return p;
}

void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
  if (!s) {
    PyErr_Clear();
    throw NotPlain();
  }
  void* p = PyLong_AsVoidPtr(s);
  Py_DECREF(s);
  if (!p && PyErr_Occurred()) {
    PyErr_Clear();
    throw NotPlain();
  }
  return p;
}

// An output argument: the caller's tensor, or one made here when `o` is True
// (required outputs: None); an optional output may also be None or False.
struct Out {
  PyObject* obj = nullptr;  // new reference
  void* ptr = nullptr;
  ~Out() { Py_XDECREF(obj); }
  PyObject* take() {
    PyObject* r = obj ? obj : Py_NewRef(Py_None);
    obj = nullptr;
    return r;
  }
  void make(int64_t n, const at::TensorOptions& opt, size_t item) {
    at::Tensor t = at::empty({n}, opt);
    ptr = out_ptr(t, item, n);
    obj = THPVariable_Wrap(std::move(t));
    if (!obj) throw NotPlain();
  }
  void init(PyObject* o, bool required, int64_t n, const at::TensorOptions& opt, size_t item) {
    if (o == (required ? Py_None : Py_True)) {
      make(n, opt, item);
    } else if (required || (o != Py_None && o != Py_False)) {
      ptr = out_ptr(o, item, n);
      obj = Py_NewRef(o);
    }
  }
};

at::TensorOptions bytes_like(const at::Tensor& t) { return t.options().dtype(at::kByte); }

// Runs one binding function body.  Nothing throws once the C ABI has been
// called, so after any exception (NotPlain, an output that could not be
// allocated) the Python code takes the call from its start and raises the
// error that PyTorch gives there, torch.OutOfMemoryError for instance.
template <class F>
PyObject* guarded(Py_ssize_t have, Py_ssize_t want, F body) {
  if (have != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  try {
    if (modes_active()) throw NotPlain();
    return body();
  } catch (const NotPlain&) {
  } catch (const std::exception&) {
  }
  PyErr_Clear();
  return Py_NewRef(Py_NotImplemented);
}

template <class F>
int without_gil(F call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = call();
  Py_END_ALLOW_THREADS
  return rc;
}

using InsertFn = int (*)(void*, const void*, const void*, uint64_t, void*, void*);
using EraseFn = int (*)(void*, const void*, uint64_t, void*, void*);
using FindFn = int (*)(void*, const void*, uint64_t, void*, void*, void*);
using ExecuteFn = int (*)(void*, const void*, const void*, const void*, uint64_t, void*, void*,
                          void*);
using MultiFn = int (*)(void*, const hive_segment*, uint32_t, void*);
using BoundsFn = int (*)(void*, uint64_t*, uint32_t);

// insert(fn, table, keys, vals, status, stream) -> (code, status)
PyObject* py_insert(PyObject*, PyObject* const* a, Py_ssize_t na) {
  return guarded(na, 6, [&]() -> PyObject* {
    const auto fn = reinterpret_cast<InsertFn>(as_address(a[0]));
    void* h = as_address(a[1]);
    const at::Tensor& keys = tensor_of(a[2]);
    const int64_t n = keys.numel();
    Out st;
    st.init(a[4], false, n, bytes_like(keys), 1);
    const void* k = in_ptr(keys, 4, n);
    const void* v = in_ptr(a[3], 4, n);
    void* s = stream_of(a[5]);
    const int rc = without_gil([&] { return fn(h, k, v, n, st.ptr, s); });
    return Py_BuildValue("(iN)", rc, st.take());
  });
}

// erase(fn, table, keys, status, stream) -> (code, status)
PyObject* py_erase(PyObject*, PyObject* const* a, Py_ssize_t na) {
  return guarded(na, 5, [&]() -> PyObject* {
    const auto fn = reinterpret_cast<EraseFn>(as_address(a[0]));
    void* h = as_address(a[1]);
    const at::Tensor& keys = tensor_of(a[2]);
    const int64_t n = keys.numel();
    Out st;
    st.init(a[3], false, n, bytes_like(keys), 1);
    const void* k = in_ptr(keys, 4, n);
    void* s = stream_of(a[4]);
    const int rc = without_gil([&] { return fn(h, k, n, st.ptr, s); });
    return Py_BuildValue("(iN)", rc, st.take());
  });
}

// find(fn, table, keys, vals_out, found, stream) -> (code, vals_out, found)
PyObject* py_find(PyObject*, PyObject* const* a, Py_ssize_t na) {
  return guarded(na, 6, [&]() -> PyObject* {
    const auto fn = reinterpret_cast<FindFn>(as_address(a[0]));
    void* h = as_address(a[1]);
    const at::Tensor& keys = tensor_of(a[2]);
    const int64_t n = keys.numel();
    const void* k = in_ptr(keys, 4, n);
    Out vo, fo;
    vo.init(a[3], true, n, keys.options(), 4);
    fo.init(a[4], false, n, bytes_like(keys), 1);
    void* s = stream_of(a[5]);
    const int rc = without_gil([&] { return fn(h, k, n, vo.ptr, fo.ptr, s); });
    return Py_BuildValue("(iNN)", rc, vo.take(), fo.take());
  });
}

// execute(fn, table, ops, keys, vals, stream) -> (code, vals_out, status)
PyObject* py_execute(PyObject*, PyObject* const* a, Py_ssize_t na) {
  return guarded(na, 6, [&]() -> PyObject* {
    const auto fn = reinterpret_cast<ExecuteFn>(as_address(a[0]));
    void* h = as_address(a[1]);
    const at::Tensor& keys = tensor_of(a[3]);
    const int64_t n = keys.numel();
    const void* k = in_ptr(keys, 4, n);
    const void* o = in_ptr(a[2], 1, n);
    const void* v = in_ptr(a[4], 4, n);
    Out vo, st;
    vo.make(n, keys.options(), 4);
    st.make(n, bytes_like(keys), 1);
    void* s = stream_of(a[5]);
    const int rc = without_gil([&] { return fn(h, o, k, v, n, vo.ptr, st.ptr, s); });
    return Py_BuildValue("(iNN)", rc, vo.take(), st.take());
  });
}

// Interned keys of a segment dict.
PyObject *k_table, *k_ops, *k_keys, *k_vals, *k_vals_out, *k_status, *k_n_insert;

// The item of a segment dict (borrowed), or nullptr when absent.
PyObject* item(PyObject* d, PyObject* key) {
  PyObject* o = PyDict_GetItemWithError(d, key);
  if (!o && PyErr_Occurred()) throw NotPlain();
  return o;
}

// References to a batch's arrays, in a list with room for `most` of them.
struct Held {
  PyObject* list;
  Py_ssize_t n = 0;
  explicit Held(Py_ssize_t most) : list(PyList_New(most)) {
    if (!list) throw NotPlain();
  }
  Held(const Held&) = delete;
  Held& operator=(const Held&) = delete;
  ~Held() { Py_XDECREF(list); }
  void add(PyObject* o) { PyList_SET_ITEM(list, n++, Py_NewRef(o)); }
  PyObject* take() {
    Py_SET_SIZE(reinterpret_cast<PyVarObject*>(list), n);  // the rest was never filled
    PyObject* r = list;
    list = nullptr;
    return r;
  }
};

// multi(fn, group, [segment dicts], stream, bounds) -> (code, arrays)
// bounds: hive_multi_bounds for a group whose batches are not waited for
// otherwise, to wait for one that works on host memory (its arrays may be
// touched when the call returns); 0 for the others.  arrays: the batch's
// tensors when bounds is given (a list), for the caller to keep while the batch
// runs.
PyObject* py_multi(PyObject*, PyObject* const* a, Py_ssize_t na) {
  return guarded(na, 5, [&]() -> PyObject* {
    const auto fn = reinterpret_cast<MultiFn>(as_address(a[0]));
    void* h = as_address(a[1]);
    const auto bounds = reinterpret_cast<BoundsFn>(as_address(a[4]));
    if (!PyList_CheckExact(a[2])) throw NotPlain();
    const Py_ssize_t n_segs = PyList_GET_SIZE(a[2]);
    std::vector<hive_segment> segs(n_segs > 0 ? n_segs : 1);
    Held held(bounds ? 5 * n_segs : 0);
    bool host = false;
    auto keep = [&](PyObject* o) {
      if (bounds && o && o != Py_None) held.add(o);
      return o;
    };
    for (Py_ssize_t i = 0; i < n_segs; ++i) {
      PyObject* d = PyList_GET_ITEM(a[2], i);
      if (!PyDict_CheckExact(d)) throw NotPlain();
      PyObject* keys_o = item(d, k_keys);
      PyObject* ops_o = item(d, k_ops);
      PyObject* table_o = item(d, k_table);
      PyObject* ins_o = item(d, k_n_insert);
      if (!keys_o || !ops_o || !table_o || !PyLong_CheckExact(table_o) ||
          (ins_o && !PyLong_CheckExact(ins_o)))
        throw NotPlain();
      const at::Tensor& keys = tensor_of(keys_o);
      const int64_t n = keys.numel();
      hive_segment& g = segs[i];
      g.table = static_cast<uint32_t>(PyLong_AsUnsignedLongMask(table_o));
      g.reserved0 = 0;
      g.n = static_cast<uint64_t>(n);
      g.n_insert = ins_o ? PyLong_AsUnsignedLongLongMask(ins_o) : g.n;
      g.ops = static_cast<const uint8_t*>(in_ptr(keep(ops_o), 1, n, &host));
      g.keys = static_cast<const uint32_t*>(in_ptr(keep(keys_o), 4, n, &host));
      g.vals = static_cast<const uint32_t*>(in_ptr(keep(item(d, k_vals)), 4, n, &host));
      g.vals_out = static_cast<uint32_t*>(out_ptr(keep(item(d, k_vals_out)), 4, n, &host));
      g.status = static_cast<uint8_t*>(out_ptr(keep(item(d, k_status)), 1, n, &host));
    }
    void* s = stream_of(a[3]);
    const int rc = without_gil([&] {
      uint64_t none = 0;
      const int e = fn(h, segs.data(), static_cast<uint32_t>(n_segs), s);
      return e == HIVE_OK && host && bounds ? bounds(h, &none, 0) : e;
    });
    return Py_BuildValue("(iN)", rc, held.take());
  });
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
  return PyMethodDef{name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)),
                     METH_FASTCALL, nullptr};
}

PyMethodDef methods[] = {method<py_insert>("insert"),   method<py_erase>("erase"),
                         method<py_find>("find"),       method<py_execute>("execute"),
                         method<py_multi>("multi"),     {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "hive_binding", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_hive_binding() {
  struct {
    PyObject** where;
    const char* name;
  } names[] = {{&k_table, "table"}, {&k_ops, "ops"},           {&k_keys, "keys"},
               {&k_vals, "vals"},   {&k_vals_out, "vals_out"}, {&k_status, "status"},
               {&k_n_insert, "n_insert"}};
  for (auto& n : names)
    if (!(*n.where = PyUnicode_InternFromString(n.name))) return nullptr;
  return PyModule_Create(&module);
}
