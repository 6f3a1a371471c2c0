// Python side of the hot entry points: one C call per library call, no Python code in between.
//
// A decode call is 4 - 15 us of device work, and marshalling its 10 to 36 arguments in Python (ctypes objects, the
// stream object, channel maps as ctypes structures) cost 5 - 8 us of host time, more than the launch itself: the
// caller's thread, not the GPU, set the pace of a decoding step.  Here a call reads tensor addresses, types and the
// current stream through the C++ API of torch and goes straight to the C ABI.
//
// Every function takes the same arguments, positional or by keyword, as the table beside it says; `stream` is None
// (torch's current stream), an object with a `cuda_stream` attribute, or an integer handle.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/uniql.h"

namespace {

PyObject* g_error = nullptr;       // UniqlError(status, what)

constexpr int kMaxArgs = 40;

struct Arg { const char* name; bool required; };

// The arguments of one call in declaration order (NULL: not given).
struct Args {
  const char* fn;
  const Arg* spec;
  int n;
  PyObject* v[kMaxArgs];
  bool ok = true;

  bool fail(PyObject* exc, const char* what, int i) {
    if (ok && !PyErr_Occurred()) PyErr_Format(exc, "%s: %s (argument '%s')", fn, what, spec[i].name);
    ok = false;
    return false;
  }
  bool parse(const char* fn_, const Arg* spec_, int n_, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
    fn = fn_; spec = spec_; n = n_;
    if (nargs > n) {
      PyErr_Format(PyExc_TypeError, "%s takes at most %d arguments (%zd given)", fn, n, nargs);
      return ok = false;
    }
    for (int i = 0; i < n; ++i) v[i] = i < nargs ? args[i] : nullptr;
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
      PyObject* name = PyTuple_GET_ITEM(kwnames, k);
      int i = 0;
      while (i < n && PyUnicode_CompareWithASCIIString(name, spec[i].name) != 0) ++i;
      if (i == n || v[i]) {
        PyErr_Format(PyExc_TypeError, i == n ? "%s got an unexpected keyword argument '%U'" : "%s got multiple values for argument '%U'",
                     fn, name);
        return ok = false;
      }
      v[i] = args[nargs + k];
    }
    for (int i = 0; i < n; ++i)
      if (spec[i].required && !v[i]) return fail(PyExc_TypeError, "missing argument", i);
    return true;
  }
  bool none(int i) const { return !v[i] || v[i] == Py_None; }
  const at::Tensor* tensor(int i) {
    if (none(i)) return nullptr;
    if (!THPVariable_Check(v[i])) { fail(PyExc_TypeError, "a torch tensor or None is expected", i); return nullptr; }
    return &THPVariable_Unpack(v[i]);
  }
  // device address of a tensor that the call reads, NULL for None
  void* ptr(int i) {
    const at::Tensor* t = tensor(i);
    return t ? const_cast<void*>(t->const_data_ptr()) : nullptr;
  }
  // ... that the call writes: a tensor that shares its storage until the first write (a lazy clone) gets its own here
  void* out(int i) {
    const at::Tensor* t = tensor(i);
    return t ? t->mutable_data_ptr() : nullptr;
  }
  long long integer(int i, long long dflt = 0) {
    if (!v[i]) return dflt;
    const long long r = PyLong_AsLongLong(v[i]);
    if (r == -1 && PyErr_Occurred()) { PyErr_Clear(); fail(PyExc_TypeError, "an integer is expected", i); }
    return r;
  }
  int i32(int i, int dflt = 0) {
    const long long r = integer(i, dflt);
    if (r < INT32_MIN || r > INT32_MAX) { fail(PyExc_OverflowError, "the value does not fit 32 bits", i); return 0; }
    return (int)r;
  }
  double real(int i) {
    const double r = PyFloat_AsDouble(v[i]);
    if (r == -1.0 && PyErr_Occurred()) { PyErr_Clear(); fail(PyExc_TypeError, "a number is expected", i); }
    return r;
  }
  // uniql_dtype of an activation tensor
  int dtype(int i) {
    const at::Tensor* t = tensor(i);
    if (!t) { fail(PyExc_TypeError, "a torch tensor is expected", i); return 0; }
    if (t->scalar_type() == at::kHalf) return UNIQL_F16;
    if (t->scalar_type() == at::kBFloat16) return UNIQL_BF16;
    fail(PyExc_TypeError, "activations must be float16 or bfloat16", i);
    return 0;
  }
  void* workspace(int i, size_t* bytes) {
    *bytes = 0;
    const at::Tensor* t = tensor(i);
    if (!t) return nullptr;
    *bytes = (size_t)t->numel() * (size_t)t->element_size();
    return t->mutable_data_ptr();
  }
  void* stream(int i) {
    if (none(i)) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* o = v[i];
    PyObject* h = PyLong_Check(o) ? (Py_INCREF(o), o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!h) { PyErr_Clear(); h = PyNumber_Long(o); }
    void* p = h ? PyLong_AsVoidPtr(h) : nullptr;
    Py_XDECREF(h);
    if (PyErr_Occurred()) { PyErr_Clear(); fail(PyExc_TypeError, "a stream, a handle or None is expected", i); }
    return p;
  }
  // a sequence of (start, period, keep, count) families, NULL for None
  const uniql_chanmap* map(int i, uniql_chanmap* m) { return none(i) ? nullptr : map_of(v[i], m, i); }
  const uniql_chanmap* map_of(PyObject* o, uniql_chanmap* m, int i) {
    PyObject* seq = PySequence_Fast(o, "a sequence of families is expected");
    if (!seq) { ok = false; return nullptr; }
    const Py_ssize_t nf = PySequence_Fast_GET_SIZE(seq);
    if (nf > UNIQL_MAX_FAMILIES) PyErr_Format(PyExc_ValueError, "at most %d families", UNIQL_MAX_FAMILIES);
    m->n_fam = (int32_t)nf;
    for (Py_ssize_t f = 0; f < nf && nf <= UNIQL_MAX_FAMILIES && !PyErr_Occurred(); ++f) {
      PyObject* fam = PySequence_Fast(PySequence_Fast_GET_ITEM(seq, f), "a family is (start, period, keep, count)");
      if (!fam) break;
      if (PySequence_Fast_GET_SIZE(fam) != 4) PyErr_SetString(PyExc_ValueError, "a family is (start, period, keep, count)");
      int32_t* dst = &m->fam[f].start;
      for (int k = 0; k < 4 && !PyErr_Occurred(); ++k) dst[k] = (int32_t)PyLong_AsLong(PySequence_Fast_GET_ITEM(fam, k));
      Py_DECREF(fam);
    }
    Py_DECREF(seq);
    if (PyErr_Occurred()) { ok = false; return nullptr; }
    return m;
  }
  // host table of rotation frequencies (a sequence of numbers), NULL for None
  const double* table(int i, double* buf, int cap) {
    if (none(i)) return nullptr;
    PyObject* seq = PySequence_Fast(v[i], "a sequence of frequencies is expected");
    if (!seq) { ok = false; return nullptr; }
    const Py_ssize_t nv = PySequence_Fast_GET_SIZE(seq);
    for (Py_ssize_t k = 0; k < nv && k < cap; ++k) buf[k] = PyFloat_AsDouble(PySequence_Fast_GET_ITEM(seq, k));
    Py_DECREF(seq);
    if (PyErr_Occurred()) { ok = false; return nullptr; }
    return buf;
  }
};

PyObject* done(int status, const char* what) {
  if (status == UNIQL_OK) Py_RETURN_NONE;
  PyObject* args = Py_BuildValue("(is)", status, what);
  PyObject* e = args && g_error ? PyObject_CallObject(g_error, args) : nullptr;
  Py_XDECREF(args);
  if (e) { PyErr_SetObject(g_error, e); Py_DECREF(e); }
  return nullptr;
}

// the library call itself runs without the interpreter lock, as under ctypes (a full launch queue blocks in it)
#define DONE(call, what) ([&]() -> PyObject* { \
    int st; \
    Py_BEGIN_ALLOW_THREADS st = (call); Py_END_ALLOW_THREADS \
    return done(st, what); \
  }())
#define SIGNATURE(...) \
  static const Arg spec[] = {__VA_ARGS__}; \
  constexpr int n_spec = (int)(sizeof(spec) / sizeof(spec[0])); \
  static_assert(n_spec <= kMaxArgs, "raise kMaxArgs");
#define R(name) Arg{name, true}
#define O(name) Arg{name, false}
#define PARSE(fn) Args a; if (!a.parse(fn, spec, n_spec, args, nargs, kwnames)) return nullptr;
#define FAST(fn) PyObject* fn(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames)

typedef int (*QlinearFn)(const void*, const uint8_t*, const void*, const void*, int, int, int, int, int, void*, void*);

PyObject* qlinear_as(const char* fn, const char* what, QlinearFn call, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  SIGNATURE(R("x"), R("packed_w"), R("scales"), R("zeros"), R("M"), R("K"), R("N"), R("k_in"), R("k_out"), R("y"), O("stream"))
  PARSE(fn)
  void *x = a.ptr(0), *w = a.ptr(1), *s = a.ptr(2), *z = a.ptr(3), *y = a.out(9);
  const int M = a.i32(4), K = a.i32(5), N = a.i32(6), k_in = a.i32(7), k_out = a.i32(8);
  if (!a.ok) return nullptr;
  void* stream = a.stream(10);
  if (!a.ok) return nullptr;
  return DONE(call(x, (const uint8_t*)w, s, z, M, K, N, k_in, k_out, y, stream), what);
}
FAST(qlinear) { return qlinear_as("qlinear", "uniql_qlinear", uniql_qlinear, args, nargs, kwnames); }
FAST(qlinear_noalloc) {
  return qlinear_as("qlinear_noalloc", "uniql_qlinear_noalloc", uniql_qlinear_noalloc, args, nargs, kwnames);
}

FAST(qlinear_ex) {
  SIGNATURE(R("x"), R("ldx"), R("packed_w"), R("scales"), R("zeros"), R("bias"), R("M"), R("K"), R("N"), R("in_map"),
            R("k_in"), R("out_map"), R("k_out"), R("y"), R("ldy"), O("workspace"), O("stream"))
  PARSE("qlinear_ex")
  void *x = a.ptr(0), *w = a.ptr(2), *s = a.ptr(3), *z = a.ptr(4), *b = a.ptr(5), *y = a.out(13);
  const int ldx = a.i32(1), M = a.i32(6), K = a.i32(7), N = a.i32(8), k_in = a.i32(10), k_out = a.i32(12), ldy = a.i32(14);
  const int dt = a.dtype(0);
  uniql_chanmap im, om;
  const uniql_chanmap *ip = a.map(9, &im), *op = a.map(11, &om);
  size_t ws_bytes;
  void* ws = a.workspace(15, &ws_bytes);
  if (!a.ok) return nullptr;
  void* stream = a.stream(16);
  if (!a.ok) return nullptr;
  return DONE(uniql_qlinear_ex(x, ldx, dt, (const uint8_t*)w, s, z, b, M, K, N, ip, k_in, op, k_out, y, ldy, ws, ws_bytes, stream),
              "uniql_qlinear_ex");
}

// jobs: dicts with packed_w, scales, zeros, bias (optional), N, k_out (optional), out_map (optional), y, ldy
FAST(qlinear_multi) {
  SIGNATURE(R("x"), R("ldx"), R("M"), R("K"), R("in_map"), R("k_in"), R("jobs"), O("workspace"), O("stream"))
  PARSE("qlinear_multi")
  void* x = a.ptr(0);
  const int ldx = a.i32(1), M = a.i32(2), K = a.i32(3), k_in = a.i32(5), dt = a.dtype(0);
  uniql_chanmap im, om[UNIQL_MAX_JOBS];
  const uniql_chanmap* ip = a.map(4, &im);
  size_t ws_bytes;
  void* ws = a.workspace(7, &ws_bytes);
  if (!a.ok) return nullptr;
  PyObject* seq = PySequence_Fast(a.v[6], "jobs: a sequence of dicts is expected");
  if (!seq) return nullptr;
  const int n = (int)PySequence_Fast_GET_SIZE(seq);
  uniql_job jobs[UNIQL_MAX_JOBS];
  memset(jobs, 0, sizeof(jobs));
  for (int j = 0; j < n && j < UNIQL_MAX_JOBS && a.ok; ++j) {       // (more jobs: the library says UNIQL_ERR_SHAPE)
    PyObject* d = PySequence_Fast_GET_ITEM(seq, j);
    auto item = [&](const char* key, bool required) -> PyObject* {
      PyObject* o = PyDict_Check(d) ? PyDict_GetItemString(d, key) : nullptr;
      if (!o && required && a.ok) { PyErr_Format(PyExc_KeyError, "%s", key); a.ok = false; }
      return o;
    };
    auto address = [&](const char* key, bool required) -> void* {
      PyObject* o = item(key, required);
      if (!o || (o == Py_None && !required)) return nullptr;
      if (!THPVariable_Check(o)) { if (a.ok) PyErr_Format(PyExc_TypeError, "job %d: %s: a torch tensor is expected", j, key); a.ok = false; return nullptr; }
      const at::Tensor& v = THPVariable_Unpack(o);
      return strcmp(key, "y") == 0 ? v.mutable_data_ptr() : const_cast<void*>(v.const_data_ptr());
    };
    auto number = [&](const char* key, bool required) -> int32_t {
      PyObject* o = item(key, required);
      if (!o) return 0;
      const long r = PyLong_AsLong(o);
      if (PyErr_Occurred()) a.ok = false;
      return (int32_t)r;
    };
    uniql_job& t = jobs[j];
    t.packed_w = (const uint8_t*)address("packed_w", true);
    t.scales = address("scales", true);
    t.zeros = address("zeros", true);
    t.bias = address("bias", false);
    t.N = number("N", true);
    t.k_out = number("k_out", false);
    PyObject* m = item("out_map", false);
    t.out_map = m && m != Py_None ? a.map_of(m, &om[j], 6) : nullptr;
    t.y = address("y", true);
    t.ldy = number("ldy", true);
  }
  Py_DECREF(seq);
  if (!a.ok) return nullptr;
  void* stream = a.stream(8);
  if (!a.ok) return nullptr;
  return DONE(uniql_qlinear_multi(x, ldx, dt, M, K, ip, k_in, n, jobs, ws, ws_bytes, stream), "uniql_qlinear_multi");
}

FAST(qk_rope_proj) {
  SIGNATURE(R("x"), R("ldx"), R("wq"), R("sq"), R("zq"), R("wk"), R("sk"), R("zk"), R("bq"), R("bk"), R("M"), R("K"),
            R("n_q_heads"), R("n_kv_heads"), R("head_dim"), R("head_keep"), R("retained_idx"), R("pos"), R("theta"),
            R("inv_freq"), R("q_out"), R("ldq"), R("k_out"), R("ldk"), O("workspace"), O("stream"))
  PARSE("qk_rope_proj")
  void* p[10];
  for (int i = 0; i < 10; ++i) p[i] = i == 1 ? nullptr : a.ptr(i);
  const int ldx = a.i32(1), M = a.i32(10), K = a.i32(11), hq = a.i32(12), hkv = a.i32(13), hd = a.i32(14), keep = a.i32(15);
  void *idx = a.ptr(16), *pos = a.ptr(17), *q = a.out(20), *k = a.out(22);
  const double theta = a.real(18);
  double buf[512] = {0};
  const double* f = a.table(19, buf, 512);
  const int ldq = a.i32(21), ldk = a.i32(23), dt = a.dtype(0);
  size_t ws_bytes;
  void* ws = a.workspace(24, &ws_bytes);
  if (!a.ok) return nullptr;
  void* stream = a.stream(25);
  if (!a.ok) return nullptr;
  return DONE(uniql_qk_rope_proj(p[0], ldx, dt, (const uint8_t*)p[2], p[3], p[4], (const uint8_t*)p[5], p[6], p[7], p[8], p[9],
                                 M, K, hq, hkv, hd, keep, (const int32_t*)idx, (const int32_t*)pos, theta, f, q, ldq, k, ldk,
                                 ws, ws_bytes, stream), "uniql_qk_rope_proj");
}

FAST(qkv_rope_proj) {
  SIGNATURE(R("x"), R("ldx"), R("wq"), R("sq"), R("zq"), R("wk"), R("sk"), R("zk"), R("wv"), R("sv"), R("zv"), R("bq"),
            R("bk"), R("bv"), R("M"), R("K"), R("n_q_heads"), R("n_kv_heads"), R("head_dim"), R("head_keep"), R("v_keep"),
            R("retained_idx"), R("pos"), R("theta"), R("inv_freq"), R("q_out"), R("ldq"), R("k_out"), R("ldk"), R("v_out"),
            R("ldv"), O("workspace"), O("stream"))
  PARSE("qkv_rope_proj")
  void* p[14];
  for (int i = 0; i < 14; ++i) p[i] = i == 1 ? nullptr : a.ptr(i);
  const int ldx = a.i32(1), M = a.i32(14), K = a.i32(15), hq = a.i32(16), hkv = a.i32(17), hd = a.i32(18), keep = a.i32(19),
            vkeep = a.i32(20);
  void *idx = a.ptr(21), *pos = a.ptr(22), *q = a.out(25), *k = a.out(27), *v = a.out(29);
  const double theta = a.real(23);
  double buf[512] = {0};
  const double* f = a.table(24, buf, 512);
  const int ldq = a.i32(26), ldk = a.i32(28), ldv = a.i32(30), dt = a.dtype(0);
  size_t ws_bytes;
  void* ws = a.workspace(31, &ws_bytes);
  if (!a.ok) return nullptr;
  void* stream = a.stream(32);
  if (!a.ok) return nullptr;
  return DONE(uniql_qkv_rope_proj(p[0], ldx, dt, (const uint8_t*)p[2], p[3], p[4], (const uint8_t*)p[5], p[6], p[7],
                                  (const uint8_t*)p[8], p[9], p[10], p[11], p[12], p[13], M, K, hq, hkv, hd, keep, vkeep,
                                  (const int32_t*)idx, (const int32_t*)pos, theta, f, q, ldq, k, ldk, v, ldv, ws, ws_bytes,
                                  stream), "uniql_qkv_rope_proj");
}

FAST(mlp_swiglu_decode) {
  SIGNATURE(R("x"), R("ldx"), R("wg"), R("sg"), R("zg"), R("wu"), R("su"), R("zu"), R("wd"), R("sd"), R("zd"), R("M"),
            R("hidden"), R("inter"), R("k_int"), R("h"), R("ldh"), R("y"), R("ldy"), O("fuse"), O("workspace"), O("stream"))
  PARSE("mlp_swiglu_decode")
  void* p[11];
  for (int i = 0; i < 11; ++i) p[i] = i == 1 ? nullptr : a.ptr(i);
  const int ldx = a.i32(1), M = a.i32(11), hidden = a.i32(12), inter = a.i32(13), k_int = a.i32(14), ldh = a.i32(16), ldy = a.i32(18);
  void *h = a.out(15), *y = a.out(17);
  const int fuse = a.i32(19, -1);
  for (int i : {0, 15, 17})
    if (a.ok && a.tensor(i) && a.tensor(i)->scalar_type() != at::kHalf) {
      PyErr_SetString(PyExc_TypeError, "uniql_mlp_swiglu_decode computes in fp16");
      a.ok = false;
    }
  size_t ws_bytes;
  void* ws = a.workspace(20, &ws_bytes);
  if (!a.ok) return nullptr;
  void* stream = a.stream(21);
  if (!a.ok) return nullptr;
  return DONE(uniql_mlp_swiglu_decode(p[0], ldx, (const uint8_t*)p[2], p[3], p[4], (const uint8_t*)p[5], p[6], p[7],
                                      (const uint8_t*)p[8], p[9], p[10], M, hidden, inter, k_int, h, ldh, y, ldy, fuse, ws,
                                      ws_bytes, stream), "uniql_mlp_swiglu_decode");
}

// the SwiGLU MLP block for fp16 or bf16 activations and any M (x, h, y of one type)
FAST(mlp_swiglu) {
  SIGNATURE(R("x"), R("ldx"), R("wg"), R("sg"), R("zg"), R("wu"), R("su"), R("zu"), R("wd"), R("sd"), R("zd"), R("M"),
            R("hidden"), R("inter"), R("k_int"), R("h"), R("ldh"), R("y"), R("ldy"), O("workspace"), O("stream"))
  PARSE("mlp_swiglu")
  void* p[11];
  for (int i = 0; i < 11; ++i) p[i] = i == 1 ? nullptr : a.ptr(i);
  const int ldx = a.i32(1), M = a.i32(11), hidden = a.i32(12), inter = a.i32(13), k_int = a.i32(14), ldh = a.i32(16), ldy = a.i32(18);
  void *h = a.out(15), *y = a.out(17);
  const int dt = a.dtype(0);
  for (int i : {15, 17})
    if (a.ok && a.tensor(i) && a.tensor(i)->scalar_type() != a.tensor(0)->scalar_type()) {
      PyErr_SetString(PyExc_TypeError, "x, h and y must have the same type");
      a.ok = false;
    }
  size_t ws_bytes;
  void* ws = a.workspace(19, &ws_bytes);
  if (!a.ok) return nullptr;
  void* stream = a.stream(20);
  if (!a.ok) return nullptr;
  return DONE(uniql_mlp_swiglu(p[0], ldx, dt, (const uint8_t*)p[2], p[3], p[4], (const uint8_t*)p[5], p[6], p[7],
                               (const uint8_t*)p[8], p[9], p[10], M, hidden, inter, k_int, h, ldh, y, ldy, ws, ws_bytes, stream),
              "uniql_mlp_swiglu");
}

FAST(embed_rows) {
  SIGNATURE(R("packed"), R("scales"), R("zeros"), R("ids"), R("out"), O("bad_id"), O("stream"))
  PARSE("embed_rows")
  for (int i : {0, 3, 4})
    if (!a.tensor(i)) { a.fail(PyExc_TypeError, "a torch tensor is expected", i); return nullptr; }
  const at::Tensor &packed = *a.tensor(0), &ids = *a.tensor(3), &out = *a.tensor(4);
  void *s = a.ptr(1), *z = a.ptr(2), *bad = a.out(5);
  const int dt = a.dtype(4);
  if (!a.ok) return nullptr;
  if (packed.dim() != 2 || out.dim() < 1) { PyErr_SetString(PyExc_ValueError, "embed_rows: packed is [V][K/2], out [M][K]"); return nullptr; }
  void* stream = a.stream(6);
  if (!a.ok) return nullptr;
  return DONE(uniql_embed_rows((const uint8_t*)packed.const_data_ptr(), s, z, packed.size(0), packed.size(1) * 2,
                               (const int32_t*)ids.const_data_ptr(), ids.numel(), dt, out.mutable_data_ptr(),
                               out.stride(0), (int*)bad, stream), "uniql_embed_rows");
}

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

// (exceptions of torch's C++ API, such as no CUDA device, become Python errors)
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t, PyObject*)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  try {
    return F(self, args, nargs, kwnames);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
#define ENTRY(fn) {#fn, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<fn>)), METH_FASTCALL | METH_KEYWORDS, nullptr}
PyMethodDef kMethods[] = {
    ENTRY(qlinear), ENTRY(qlinear_noalloc), ENTRY(qlinear_ex), ENTRY(qlinear_multi), ENTRY(qk_rope_proj), ENTRY(qkv_rope_proj),
    ENTRY(mlp_swiglu_decode), ENTRY(mlp_swiglu), ENTRY(embed_rows),
    {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_calls", "Hot entry points of libuniql.so", -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&kModule); }
