/*
 * Argument marshalling of the hot calls for Python: tensors to addresses, numbers to C types, one call of the library.
 * A request of 32 layers makes 64 of these calls, and a small request takes the GPU less time than ctypes took to issue it:
 * ba_final_attend 6.6 -> 4.0 us, ba_reencode_k 4.6 -> 2.8 us a call (a kernel launch included), a small request 33.4 -> 27.5 us.
 * Nothing else happens here; the functions are those of the library that bind() is given (the handle ctypes opened), their
 * prototypes the header's.  Only the usual arguments are taken: None, an int that fits, a contiguous torch tensor, the ctypes
 * class of a structure.  With any other the whole call goes to the function bind() was given, which makes it through ctypes: what
 * is accepted, and what is raised, is decided there alone.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stdint.h>

#include "ba.h"

static PyObject *s_data_ptr, *s_is_contiguous;
static PyObject *other_way, *t_handle, *t_segments, *t_pages;   /* bind()'s: the ctypes way, c_void_p, ba_segments, ba_page_table */

/* The converters return 1, 0 (an exception is set) or this: not an argument this file takes. */
#define UNUSUAL (-1)

static int unusual_if(PyObject *exception) {
  if (!PyErr_ExceptionMatches(exception)) return 0;
  PyErr_Clear();
  return UNUSUAL;
}
static int from_int(PyObject *o, void **out) {
  *out = PyLong_AsVoidPtr(o);
  return *out == NULL && PyErr_Occurred() ? unusual_if(PyExc_OverflowError) : 1;
}
/* None -> NULL, an int -> that address, an object with is_contiguous() and data_ptr() (a torch tensor) -> its data. */
static int to_address(PyObject *o, void **out) {
  if (o == Py_None) { *out = NULL; return 1; }
  if (PyLong_Check(o)) return from_int(o, out);
  PyObject *r = PyObject_CallMethodNoArgs(o, s_is_contiguous);
  if (!r) return unusual_if(PyExc_AttributeError);
  const int yes = PyObject_IsTrue(r);
  Py_DECREF(r);
  if (yes < 0) return 0;
  if (!yes) { PyErr_SetString(PyExc_ValueError, "tensor must be contiguous"); return 0; }
  r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!r) return unusual_if(PyExc_AttributeError);
  const int k = PyLong_Check(r) ? from_int(r, out) : UNUSUAL;
  Py_DECREF(r);
  return k;
}
/* The memory of an instance of ctypes class `type`, at least `bytes` of it. */
static int to_memory(PyObject *o, PyObject *type, size_t bytes, void **out) {
  const int is = PyObject_IsInstance(o, type);
  if (is < 0) return 0;
  if (!is) return UNUSUAL;
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return 0;
  const int fits = (size_t)b.len >= bytes;
  *out = b.buf;
  PyBuffer_Release(&b);
  return fits ? 1 : UNUSUAL;
}
static int to_context(PyObject *o, ba_ctx **out) {
  void *at;
  if (o == Py_None || PyLong_Check(o)) return to_address(o, (void **)out);
  const int k = to_memory(o, t_handle, sizeof(void *), &at);
  if (k == 1) *out = *(ba_ctx **)at;
  return k;
}
static int to_int(PyObject *o, int32_t *out) {
  if (!PyLong_Check(o)) return UNUSUAL;
  int overflow;
  const long v = PyLong_AsLongAndOverflow(o, &overflow);
  if (overflow || v < INT32_MIN || v > INT32_MAX) return UNUSUAL;
  *out = (int32_t)v;
  return 1;
}
static int to_size(PyObject *o, size_t *out) {
  if (!PyLong_Check(o)) return UNUSUAL;
  *out = PyLong_AsSize_t(o);
  return *out == (size_t)-1 && PyErr_Occurred() ? unusual_if(PyExc_OverflowError) : 1;
}
/* other_way(name, arguments ...) */
static PyObject *go_other_way(const char *name, PyObject *const *args, Py_ssize_t nargs) {
  PyObject *all = PyTuple_New(nargs + 1), *n = PyUnicode_FromString(name);
  if (!all || !n) { Py_XDECREF(all); Py_XDECREF(n); return NULL; }
  PyTuple_SET_ITEM(all, 0, n);
  for (Py_ssize_t i = 0; i < nargs; ++i) PyTuple_SET_ITEM(all, i + 1, Py_NewRef(args[i]));
  PyObject *r = PyObject_Call(other_way, all, NULL);
  Py_DECREF(all);
  return r;
}

#define ARGS(name, n)                                                                                   \
  static const char function[] = #name;                                                                 \
  if (!other_way) return PyErr_Format(PyExc_RuntimeError, "no library bound");                          \
  if (nargs != (n)) return PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", (n), nargs)
#define TAKE(convert)                                                                     \
  do {                                                                                    \
    const int taken = (convert);                                                          \
    if (taken != 1) return taken == UNUSUAL ? go_other_way(function, args, nargs) : NULL; \
  } while (0)
#define P(i, v) void *v; TAKE(to_address(args[i], &v))
#define I(i, v) int32_t v; TAKE(to_int(args[i], &v))
#define CTX ba_ctx *ctx; TAKE(to_context(args[0], &ctx))
#define SEG(i, v) void *v; TAKE(to_memory(args[i], t_segments, sizeof(ba_segments), &v))
#define PAGES(i, v) void *v; TAKE(to_memory(args[i], t_pages, sizeof(ba_page_table), &v))
#define CALL(expr)                                   \
  do {                                               \
    ba_status st;                                    \
    Py_BEGIN_ALLOW_THREADS st = (expr);              \
    Py_END_ALLOW_THREADS return PyLong_FromLong(st); \
  } while (0)
#define FUNCTIONS(X) X(ba_segment) X(ba_reencode_k) X(ba_reencode_k_paged) X(ba_block_prefill) X(ba_block_prefill_bwd) \
  X(ba_final_attend) X(ba_final_attend_fused) X(ba_final_attend_paged) X(ba_final_attend_fused_paged)
#define DECLARE(f) static __typeof__(&f) p_##f;
FUNCTIONS(DECLARE)

static PyObject *m_segment(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_segment, 11); CTX; P(1, lens); P(2, nblocks); I(3, batch); I(4, n_blocks); I(5, n_tokens); I(6, mode); P(7, buf);
  size_t bytes; TAKE(to_size(args[8], &bytes));
  SEG(9, out); P(10, stream);
  CALL(p_ba_segment(ctx, lens, nblocks, batch, n_blocks, n_tokens, mode, buf, bytes, out, stream));
}
static PyObject *m_reencode_k(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_reencode_k, 10); CTX; P(1, src); P(2, off); I(3, n_src); P(4, dst); P(5, cu); P(6, delta); I(7, n_blocks); I(8, n_rows); P(9, stream);
  CALL(p_ba_reencode_k(ctx, src, off, n_src, dst, cu, delta, n_blocks, n_rows, stream));
}
static PyObject *m_reencode_k_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_reencode_k_paged, 9); CTX; P(1, pool); PAGES(2, pages); P(3, dst); P(4, cu); P(5, delta); I(6, n_blocks); I(7, n_rows); P(8, stream);
  CALL(p_ba_reencode_k_paged(ctx, pool, pages, dst, cu, delta, n_blocks, n_rows, stream));
}
static PyObject *m_block_prefill(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_block_prefill, 10); CTX; P(1, q); P(2, k); P(3, v); P(4, o); P(5, lse); SEG(6, seg); I(7, mode); I(8, out); P(9, stream);
  CALL(p_ba_block_prefill(ctx, q, k, v, o, lse, seg, mode, out, stream));
}
static PyObject *m_block_prefill_bwd(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_block_prefill_bwd, 14); CTX; P(1, q); P(2, k); P(3, v); P(4, o); P(5, lse); P(6, d_o); P(7, dq); P(8, dk); P(9, dv); SEG(10, seg); I(11, mode);
  I(12, out); P(13, stream);
  CALL(p_ba_block_prefill_bwd(ctx, q, k, v, o, lse, d_o, dq, dk, dv, seg, mode, out, stream));
}
static PyObject *m_final_attend(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_final_attend, 16); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kc); P(6, vc); I(7, n_cache); P(8, voff); I(9, n_v); P(10, o);
  P(11, lse); SEG(12, seg); I(13, mode); I(14, out); P(15, stream);
  CALL(p_ba_final_attend(ctx, q, k, v, n_final, kc, vc, n_cache, voff, n_v, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_fused(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_final_attend_fused, 17); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, ks); P(6, vs); I(7, n_src); P(8, off); I(9, n_cache); P(10, k_out);
  P(11, o); P(12, lse); SEG(13, seg); I(14, mode); I(15, out); P(16, stream);
  CALL(p_ba_final_attend_fused(ctx, q, k, v, n_final, ks, vs, n_src, off, n_cache, k_out, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_final_attend_paged, 15); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kc); I(6, n_cache); P(7, pool); PAGES(8, pages); P(9, o); P(10, lse);
  SEG(11, seg); I(12, mode); I(13, out); P(14, stream);
  CALL(p_ba_final_attend_paged(ctx, q, k, v, n_final, kc, n_cache, pool, pages, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_fused_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(ba_final_attend_fused_paged, 16); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kp); P(6, vp); PAGES(7, pages); I(8, n_cache); P(9, k_out); P(10, o);
  P(11, lse); SEG(12, seg); I(13, mode); I(14, out); P(15, stream);
  CALL(p_ba_final_attend_fused_paged(ctx, q, k, v, n_final, kp, vp, pages, n_cache, k_out, o, lse, seg, mode, out, stream));
}

/* bind(handle, other_way, c_void_p, ba_segments, ba_page_table): take the library's functions from the shared object a dlopen
 * handle names. */
static PyObject *m_bind(PyObject *self, PyObject *args) {
  PyObject *handle, *way, *handle_type, *segments, *pages;
  if (!PyArg_ParseTuple(args, "OOOOO", &handle, &way, &handle_type, &segments, &pages)) return NULL;
  void *h = PyLong_AsVoidPtr(handle);
  if (!h && PyErr_Occurred()) return NULL;
#define RESOLVE(f) \
  if (!(p_##f = (__typeof__(&f))dlsym(h, #f))) return PyErr_Format(PyExc_RuntimeError, "%s is not in the library", #f);
  FUNCTIONS(RESOLVE)
  Py_XSETREF(t_handle, Py_NewRef(handle_type));
  Py_XSETREF(t_segments, Py_NewRef(segments));
  Py_XSETREF(t_pages, Py_NewRef(pages));
  Py_XSETREF(other_way, Py_NewRef(way));
  Py_RETURN_NONE;
}

#define METHOD(n) {#n, (PyCFunction)(void (*)(void))m_##n, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {{"bind", m_bind, METH_VARARGS, NULL}, METHOD(segment), METHOD(reencode_k), METHOD(reencode_k_paged),
                                METHOD(block_prefill), METHOD(block_prefill_bwd), METHOD(final_attend), METHOD(final_attend_fused),
                                METHOD(final_attend_paged), METHOD(final_attend_fused_paged), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "ba_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit_ba_marshal(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  return s_data_ptr && s_is_contiguous ? PyModule_Create(&module) : NULL;
}
