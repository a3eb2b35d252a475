// CPython side of the binding: the calls of an engine step, argument marshalling only.
//
// Through ctypes the marshalling cost more than the calls: 3.5 us of a lone decode row's append and 2.4 us of its
// attention, beside kernels that take 12 us together, and 0.6 us for every host-only call.  Here an argument is converted
// once: arrays through the buffer protocol, tensors through data_ptr(), the stream through torch's own accessor of the
// current one.  Every function takes the handle first and returns the status code; nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <cstring>

#include "../../include/tide.h"

namespace {

PyObject *g_data_ptr, *g_cuda_stream;                      // names
PyObject *g_get_device, *g_raw_stream, *g_as_int32;         // torch's two accessors, and what makes an int32 array of a sequence
PyObject* g_ndarray;                                        // numpy's array type

// A pointer argument: None, an address, a numpy array (the address of its first element) or something with data_ptr() (a
// tensor); arrays are held until the call has returned.  Other objects that export a buffer are not taken for pointers: a
// numpy integer, for one, may BE an address.
class Pointer {
 public:
  ~Pointer() { if (view_.obj != nullptr) PyBuffer_Release(&view_); }
  bool from(PyObject* x) {
    if (x == Py_None) return true;
    if (PyLong_Check(x)) {
      p = PyLong_AsVoidPtr(x);
      return !PyErr_Occurred();
    }
    if (PyType_Check(g_ndarray) && PyObject_TypeCheck(x, reinterpret_cast<PyTypeObject*>(g_ndarray))) return buffer(x, PyBUF_STRIDES);
    PyObject* v = PyObject_CallMethodNoArgs(x, g_data_ptr);
    if (v == nullptr) return false;
    p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
  }
  bool buffer(PyObject* x, int flags) {
    if (PyObject_GetBuffer(x, &view_, flags) != 0) return false;
    p = view_.buf;
    bytes = view_.len;
    return true;
  }
  const Py_buffer& view() const { return view_; }
  // int32 values: a contiguous buffer of that type, or whatever converts to one
  bool ints(PyObject* x) {
    if (PyObject_CheckBuffer(x) && PyObject_GetBuffer(x, &view_, PyBUF_ND | PyBUF_FORMAT) == 0) {
      if (view_.itemsize == 4 && view_.format != nullptr && view_.format[0] == 'i' && view_.format[1] == 0) {
        p = view_.buf;
        bytes = view_.len;
        return true;
      }
      PyBuffer_Release(&view_);
      view_ = Py_buffer{};
    }
    PyErr_Clear();
    PyObject* made = PyObject_CallOneArg(g_as_int32, x);
    if (made == nullptr) return false;
    const bool ok = buffer(made, PyBUF_SIMPLE);               // the view keeps the array
    Py_DECREF(made);
    return ok;
  }
  void* p = nullptr;
  Py_ssize_t bytes = 0;

 private:
  Py_buffer view_ = {};
};

bool stream_from(PyObject* x, void** out) {
  PyObject* v;
  if (x == Py_None) {
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    if (dev == nullptr) return false;
    v = PyObject_CallOneArg(g_raw_stream, dev);
    Py_DECREF(dev);
  } else if (PyLong_Check(x)) {
    v = Py_NewRef(x);
  } else {
    v = PyObject_GetAttr(x, g_cuda_stream);
  }
  if (v == nullptr) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

bool handle_from(PyObject* x, tide_kv_t** out) {
  *out = static_cast<tide_kv_t*>(PyLong_AsVoidPtr(x));
  return !PyErr_Occurred();
}
bool int_from(PyObject* x, int32_t* out) {
  *out = static_cast<int32_t>(PyLong_AsUnsignedLongMask(x));
  return !PyErr_Occurred();
}
bool float_from(PyObject* x, float* out) {
  *out = static_cast<float>(PyFloat_AsDouble(x));
  return !PyErr_Occurred();
}
bool arity(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments are wanted, got %zd", want, n);
  return false;
}
PyObject* code(int rc) { return PyLong_FromLong(rc); }
// The call itself; other Python threads run meanwhile (it may wait for a staging slot or for results).
template <typename F>
PyObject* call(F f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return code(rc);
}

// the (task_ids, indptr) pair: indptr has one entry more
struct TaskList {
  Pointer ids, indptr;
  int32_t n = 0;
  bool from(PyObject* a, PyObject* b) {
    if (!ids.ints(a) || !indptr.ints(b)) return false;
    n = static_cast<int32_t>(ids.bytes / 4);
    if (indptr.bytes == ids.bytes + 4) return true;
    PyErr_SetString(PyExc_AssertionError, "indptr has one entry more than task_ids");
    return false;
  }
};
// tide_row_t records (of ctypes or numpy), or int32 values in rows of three
struct Rows {
  Pointer rows;
  int32_t n = 0;
  bool from(PyObject* a) {
    if (rows.buffer(a, PyBUF_ND | PyBUF_FORMAT)) {
      const Py_buffer& v = rows.view();
      char kind[8] = "";
      types(v.format, kind, sizeof(kind));
      const bool records = std::strcmp(kind, "T{iii}") == 0 && v.itemsize == static_cast<Py_ssize_t>(sizeof(tide_row_t));
      const bool triples = std::strcmp(kind, "i") == 0 && v.itemsize == 4 && v.ndim == 2 && v.shape[1] == 3;
      if (records || triples) {
        n = static_cast<int32_t>(v.len / static_cast<Py_ssize_t>(sizeof(tide_row_t)));
        return true;
      }
    }
    PyErr_SetString(PyExc_TypeError, "rows are tide_row_t records or int32 values in rows of three");
    return false;
  }
  // a format without field names and native byte orders; `out` stays short of one that is too long
  static void types(const char* f, char* out, size_t cap) {
    size_t k = 0;
    for (; f != nullptr && *f != 0 && k + 1 < cap; ++f) {
      if (*f == ':') {
        for (++f; *f != 0 && *f != ':'; ++f) {}
        if (*f == 0) break;
      } else if (*f != '<' && *f != '=' && *f != '@') {
        out[k++] = *f;
      }
    }
    out[k] = 0;
  }
};
#define I32(x) static_cast<const int32_t*>((x).p)
#define ROWS(x) static_cast<const tide_row_t*>((x).rows.p)

PyObject* py_truncate(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  int32_t task, len;
  if (!arity(n, 3) || !handle_from(a[0], &kv) || !int_from(a[1], &task) || !int_from(a[2], &len)) return nullptr;
  return code(tide_kv_truncate(kv, task, len));
}
PyObject* py_prune(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  int32_t task, keep, tail;
  void* st;
  if (!arity(n, 5) || !handle_from(a[0], &kv) || !int_from(a[1], &task) || !int_from(a[2], &keep) || !int_from(a[3], &tail) || !stream_from(a[4], &st))
    return nullptr;
  return call([&] { return tide_kv_prune(kv, 0, task, keep, tail, st); });
}
PyObject* py_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  TaskList t;
  Pointer k, v;
  void* st;
  if (!arity(n, 6) || !handle_from(a[0], &kv) || !t.from(a[1], a[2]) || !k.from(a[3]) || !v.from(a[4]) || !stream_from(a[5], &st)) return nullptr;
  return call([&] { return tide_kv_append(kv, 0, t.n, I32(t.ids), I32(t.indptr), k.p, v.p, st); });
}
PyObject* py_extend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  TaskList t;
  void* st;
  if (!arity(n, 4) || !handle_from(a[0], &kv) || !t.from(a[1], a[2]) || !stream_from(a[3], &st)) return nullptr;
  return call([&] { return tide_kv_extend(kv, t.n, I32(t.ids), I32(t.indptr), st); });
}
PyObject* py_write(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  int32_t layer;
  TaskList t;
  Pointer k, v;
  void* st;
  if (!arity(n, 7) || !handle_from(a[0], &kv) || !int_from(a[1], &layer) || !t.from(a[2], a[3]) || !k.from(a[4]) || !v.from(a[5]) ||
      !stream_from(a[6], &st))
    return nullptr;
  return call([&] { return tide_kv_write(kv, layer, t.n, I32(t.ids), I32(t.indptr), k.p, v.p, st); });
}
// (handle, layer, rows, page_table, q, scale, out, lse, stream)
PyObject* py_attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  int32_t layer;
  Rows r;
  Pointer table, q, out, lse;
  float scale;
  void* st;
  if (!arity(n, 9) || !handle_from(a[0], &kv) || !int_from(a[1], &layer) || !r.from(a[2]) || !table.from(a[3]) || !q.from(a[4]) ||
      !float_from(a[5], &scale) || !out.from(a[6]) || !lse.from(a[7]) || !stream_from(a[8], &st))
    return nullptr;
  return call([&] { return tide_attend(kv, layer, r.n, ROWS(r), I32(table), q.p, scale, out.p, static_cast<float*>(lse.p), st); });
}
PyObject* py_step_begin(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  Rows r;
  void* st;
  if (!arity(n, 3) || !handle_from(a[0], &kv) || !r.from(a[1]) || !stream_from(a[2], &st)) return nullptr;
  return call([&] { return tide_step_begin(kv, r.n, ROWS(r), st); });
}
// (handle, layer, new_k, new_v, q, scale, out, lse, stream)
PyObject* py_step_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  int32_t layer;
  Pointer k, v, q, out, lse;
  float scale;
  void* st;
  if (!arity(n, 9) || !handle_from(a[0], &kv) || !int_from(a[1], &layer) || !k.from(a[2]) || !v.from(a[3]) || !q.from(a[4]) ||
      !float_from(a[5], &scale) || !out.from(a[6]) || !lse.from(a[7]) || !stream_from(a[8], &st))
    return nullptr;
  return call([&] { return tide_step_layer(kv, layer, k.p, v.p, q.p, scale, out.p, static_cast<float*>(lse.p), st); });
}
// (handle, rows, new_k, new_v, q, scale, out, lse, stream)
PyObject* py_step_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
  tide_kv_t* kv;
  Rows r;
  Pointer k, v, q, out, lse;
  float scale;
  void* st;
  if (!arity(n, 9) || !handle_from(a[0], &kv) || !r.from(a[1]) || !k.from(a[2]) || !v.from(a[3]) || !q.from(a[4]) || !float_from(a[5], &scale) ||
      !out.from(a[6]) || !lse.from(a[7]) || !stream_from(a[8], &st))
    return nullptr;
  return call([&] { return tide_step_host(kv, 0, r.n, ROWS(r), k.p, v.p, q.p, scale, out.p, static_cast<float*>(lse.p), st); });
}

// use(get_device, raw_stream, as_int32, ndarray)
PyObject* py_use(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 4)) return nullptr;
  Py_XSETREF(g_get_device, Py_NewRef(a[0]));
  Py_XSETREF(g_raw_stream, Py_NewRef(a[1]));
  Py_XSETREF(g_as_int32, Py_NewRef(a[2]));
  Py_XSETREF(g_ndarray, Py_NewRef(a[3]));
  Py_RETURN_NONE;
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(truncate), METHOD(prune),      METHOD(append),    METHOD(extend),    METHOD(write),       METHOD(attend),
                         METHOD(step_begin), METHOD(step_layer), METHOD(step_host), METHOD(use), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  g_get_device = Py_NewRef(Py_None);
  g_raw_stream = Py_NewRef(Py_None);
  g_as_int32 = Py_NewRef(Py_None);
  g_ndarray = Py_NewRef(Py_None);
  if (g_data_ptr == nullptr || g_cuda_stream == nullptr) return nullptr;
  return PyModule_Create(&module);
}
