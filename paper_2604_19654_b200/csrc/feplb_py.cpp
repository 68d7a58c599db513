// CPython module with the per-micro-batch calls of the binding: takes tensors (anything with is_contiguous() and
// data_ptr()), numpy arrays, addresses or None, and calls the C ABI with their pointers, without the GIL.  The ctypes route
// does the same in Python and costs 10 us for the 19 arguments of feplb_moe_forward, as much as the whole
// GPU work of a small batch; through this module the call overhead is about 2 us.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include <type_traits>

#include "feplb.h"

namespace {

PyObject *s_is_contiguous, *s_data_ptr, *s_ctypes, *s_data;
PyObject *s_buf[8], *s_bwd[6];      // attribute names of Buffers / BackwardBuffers, in the order of the C arguments

decltype(&feplb_moe_forward) p_forward;
decltype(&feplb_moe_backward) p_backward;
decltype(&feplb_route_topk) p_topk;
decltype(&feplb_route_hist) p_hist;
decltype(&feplb_dispatch) p_dispatch;
decltype(&feplb_combine) p_combine;

// Address of a numpy array (page-locked host memory is addressable from the GPU), which has no is_contiguous();
// the AttributeError that said so stays set for any other object.
bool array_ptr(PyObject* o, void** out) {
  PyObject *type, *value, *trace;
  PyErr_Fetch(&type, &value, &trace);
  PyObject* c = PyObject_GetAttr(o, s_ctypes);
  PyObject* d = c ? PyObject_GetAttr(c, s_data) : nullptr;
  Py_XDECREF(c);
  if (!d) {
    PyErr_Restore(type, value, trace);
    return false;
  }
  Py_XDECREF(type);
  Py_XDECREF(value);
  Py_XDECREF(trace);
  *out = PyLong_AsVoidPtr(d);
  Py_DECREF(d);
  return !PyErr_Occurred();
}

// Address of a tensor, array or int, NULL for None; false with a Python error set.
bool ptr_of(PyObject* o, void** out) {
  if (o == Py_None) { *out = nullptr; return true; }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return !(PyErr_Occurred());
  }
  PyObject* r = PyObject_CallMethodNoArgs(o, s_is_contiguous);
  if (!r) return PyErr_ExceptionMatches(PyExc_AttributeError) && array_ptr(o, out);
  const int yes = PyObject_IsTrue(r);
  Py_DECREF(r);
  if (yes <= 0) {
    if (yes == 0) PyErr_SetString(PyExc_AssertionError, "tensor is not contiguous");
    return false;
  }
  r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!r) return false;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !(PyErr_Occurred());
}

bool ptrs_of(PyObject* const* args, Py_ssize_t n, void** out) {
  for (Py_ssize_t i = 0; i < n; ++i)
    if (!ptr_of(args[i], out + i)) return false;
  return true;
}

bool attrs_of(PyObject* o, PyObject* const* names, int n, void** out) {
  for (int i = 0; i < n; ++i) {
    PyObject* a = PyObject_GetAttr(o, names[i]);
    if (!a) return false;
    const bool ok = ptr_of(a, out + i);
    Py_DECREF(a);
    if (!ok) return false;
  }
  return true;
}

bool want(Py_ssize_t n, Py_ssize_t expected, const char* what) {
  if (n == expected) return true;
  PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", what, expected, n);
  return false;
}

#define CALL(rc, expr)       \
  int rc;                    \
  Py_BEGIN_ALLOW_THREADS     \
  rc = (expr);               \
  Py_END_ALLOW_THREADS       \
  return PyLong_FromLong(rc)

// (ctx, x, topk_ids, gates, w1, w3, w2, mask, buf, plan, stream)
PyObject* moe_forward(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void *a[8], *b[8], *t[2];
  if (!want(n, 11, "moe_forward") || !ptrs_of(args, 8, a) || !attrs_of(args[8], s_buf, 8, b) || !ptrs_of(args + 9, 2, t)) return nullptr;
  CALL(rc, p_forward((feplb_ctx*)a[0], a[1], (const int32_t*)a[2], (const float*)a[3], a[4], a[5], a[6], (const uint8_t*)a[7],
                     (int32_t*)b[0], (int32_t*)b[1], b[2], b[3], b[4], (int32_t*)b[5], (int32_t*)b[6], b[7],
                     (feplb_plan_out*)t[0], t[1]));
}

// (ctx, d_out, gates, w1t, w3t, w2t, buf, bwd, dw1, dw3, dw2, accumulate, stream); of buf only x_perm, h_scratch, y_perm
// and slot_to_row
PyObject* moe_backward(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void *a[6], *b[4], *g[6], *t[3], *st;
  if (!want(n, 13, "moe_backward") || !ptrs_of(args, 6, a) || !attrs_of(args[6], s_buf + 2, 4, b) || !attrs_of(args[7], s_bwd, 6, g) ||
      !ptrs_of(args + 8, 3, t) || !ptr_of(args[12], &st))
    return nullptr;
  const long acc = PyLong_AsLong(args[11]);
  if (acc == -1 && PyErr_Occurred()) return nullptr;
  CALL(rc, p_backward((feplb_ctx*)a[0], a[1], (const float*)a[2], a[3], a[4], a[5], b[0], g[0], b[1], b[2], (const int32_t*)b[3],
                      g[1], g[2], g[3], g[4], (float*)g[5], (float*)t[0], (float*)t[1], (float*)t[2], (int32_t)acc, st));
}

// (ctx, logits, topk_ids, gates, stream)
PyObject* route_topk(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void* a[5];
  if (!want(n, 5, "route_topk") || !ptrs_of(args, 5, a)) return nullptr;
  CALL(rc, p_topk((feplb_ctx*)a[0], (const float*)a[1], (int32_t*)a[2], (float*)a[3], a[4]));
}

// (ctx, topk_ids, counts, rank_load, stream)
PyObject* route_hist(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void* a[5];
  if (!want(n, 5, "route_hist") || !ptrs_of(args, 5, a)) return nullptr;
  CALL(rc, p_hist((feplb_ctx*)a[0], (const int32_t*)a[1], (int32_t*)a[2], (int32_t*)a[3], a[4]));
}

// (ctx, x, topk_ids, counts, x_perm, slot_to_row, row_to_token, stream)
PyObject* dispatch(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void* a[8];
  if (!want(n, 8, "dispatch") || !ptrs_of(args, 8, a)) return nullptr;
  CALL(rc, p_dispatch((feplb_ctx*)a[0], a[1], (const int32_t*)a[2], (const int32_t*)a[3], a[4], (int32_t*)a[5], (int32_t*)a[6], a[7]));
}

// (ctx, y_perm, slot_to_row, gates, out, stream)
PyObject* combine(PyObject*, PyObject* const* args, Py_ssize_t n) {
  void* a[6];
  if (!want(n, 6, "combine") || !ptrs_of(args, 6, a)) return nullptr;
  CALL(rc, p_combine((feplb_ctx*)a[0], a[1], (const int32_t*)a[2], (const float*)a[3], a[4], a[5]));
}

// load(path): resolves the calls in the library at `path`.
PyObject* load(PyObject*, PyObject* arg) {
  const char* path = PyUnicode_AsUTF8(arg);
  if (!path) return nullptr;
  void* h = dlopen(path, RTLD_NOW);
  if (!h) return PyErr_Format(PyExc_OSError, "%s", dlerror());
  bool ok = true;
  auto sym = [&](auto& p, const char* name) {
    p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(dlsym(h, name));
    ok = ok && p;
  };
  sym(p_forward, "feplb_moe_forward");
  sym(p_backward, "feplb_moe_backward");
  sym(p_topk, "feplb_route_topk");
  sym(p_hist, "feplb_route_hist");
  sym(p_dispatch, "feplb_dispatch");
  sym(p_combine, "feplb_combine");
  if (!ok) return PyErr_Format(PyExc_OSError, "%s lacks an entry point", path);
  Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(moe_forward), FAST(moe_backward), FAST(route_topk), FAST(route_hist), FAST(dispatch), FAST(combine),
                         {"load", load, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_feplb_py", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__feplb_py(void) {
  const char* buf[8] = {"counts", "rank_load", "x_perm", "h_scratch", "y_perm", "slot_to_row", "row_to_token", "out"};
  const char* bwd[6] = {"ab", "d_y_perm", "d_ab", "d_x_perm", "d_x", "d_gates"};
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_ctypes = PyUnicode_InternFromString("ctypes");
  s_data = PyUnicode_InternFromString("data");
  for (int i = 0; i < 8; ++i) s_buf[i] = PyUnicode_InternFromString(buf[i]);
  for (int i = 0; i < 6; ++i) s_bwd[i] = PyUnicode_InternFromString(bwd[i]);
  return PyModule_Create(&module);
}
