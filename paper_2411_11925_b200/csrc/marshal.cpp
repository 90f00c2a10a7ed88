// Argument marshalling of the library's short calls (ratio / accept, resampling, mixtures) for Python.  Each of them is one
// kernel of a few microseconds, and through ctypes the binding itself - one Python call per tensor for the contiguity check
// and one for the address, then a conversion per argument - took longer than the launch (measured at 64 sequences:
// csd_accept_scan 5.3 us of host time, 2.4 us of it in the library).  Here a tensor costs a type check and two field reads.
// No arithmetic and no policy: pointers and sizes go to the C ABI as they are, the status code comes back.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <exception>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/csd.h"

namespace {

PyObject* g_ptr_of = nullptr;   // the binding's address function for anything that is not a tensor (NumPy arrays)

struct Args {
  PyObject* const* a;
  bool ok = true;
  template <typename T> T* ptr(PyObject* o) {
    if (!ok || o == Py_None) return nullptr;
    if (THPVariable_Check(o)) {
      // a tensor without strides or storage (nested, sparse, vmapped) throws: that stays a Python error
      try {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_contiguous()) return static_cast<T*>(t.data_ptr());
        PyErr_SetString(PyExc_AssertionError, "tensor must be contiguous");
      } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
      }
      ok = false;
      return nullptr;
    }
    PyObject* r = PyObject_CallOneArg(g_ptr_of, o);
    void* v = r ? PyLong_AsVoidPtr(r) : nullptr;
    Py_XDECREF(r);
    if (PyErr_Occurred()) ok = false;
    return static_cast<T*>(v);
  }
  template <typename T> T* p(int i) { return ptr<T>(a[i]); }
  int n(int i) {
    const long v = ok ? PyLong_AsLong(a[i]) : 0;
    if (v == -1 && PyErr_Occurred()) ok = false;
    if (v != static_cast<int>(v)) { if (ok) PyErr_SetString(PyExc_OverflowError, "size exceeds a C int"); ok = false; }
    return static_cast<int>(v);
  }
  double d(int i) {
    const double v = ok ? PyFloat_AsDouble(a[i]) : 0.0;
    if (v == -1.0 && PyErr_Occurred()) ok = false;
    return v;
  }
  csd_ctx* ctx() {
    csd_ctx* c = ok ? static_cast<csd_ctx*>(PyLong_AsVoidPtr(a[0])) : nullptr;
    if (PyErr_Occurred()) ok = false;
    return c;
  }
  // (logw [rows, K], mu [rows, K, C], log_sigma [rows, K, C])
  csd_gmm gmm(int i) {
    csd_gmm m{};
    PyObject* s = ok ? PySequence_Fast(a[i], "a mixture is (logw, mu, log_sigma)") : nullptr;
    if (!s) { ok = false; return m; }
    if (PySequence_Fast_GET_SIZE(s) != 3) {
      PyErr_SetString(PyExc_ValueError, "a mixture is (logw, mu, log_sigma)");
      ok = false;
    } else {
      PyObject** it = PySequence_Fast_ITEMS(s);
      m.logw = ptr<const float>(it[0]); m.mu = ptr<const float>(it[1]); m.log_sigma = ptr<const float>(it[2]);
      if (ok) {
        PyObject* sh = PyObject_GetAttrString(it[0], "shape");
        PyObject* k = sh ? PySequence_GetItem(sh, 1) : nullptr;
        m.K = k ? static_cast<int>(PyLong_AsLong(k)) : 0;
        Py_XDECREF(k); Py_XDECREF(sh);
        if (PyErr_Occurred()) ok = false;
      }
    }
    Py_DECREF(s);
    return m;
  }
};

bool count_is(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return false;
}

#define CSD_MARSHAL(NAME, COUNT, ...)                                                 \
  PyObject* NAME(PyObject*, PyObject* const* args, Py_ssize_t nargs) {                 \
    if (!count_is(nargs, COUNT)) return nullptr;                                       \
    Args x{args};                                                                      \
    csd_ctx* ctx = x.ctx();                                                            \
    int rc = CSD_OK;                                                                   \
    __VA_ARGS__                                                                               \
    return x.ok ? PyLong_FromLong(rc) : nullptr;                                       \
  }
#define CSD_RUN(EXPR) if (x.ok) { Py_BEGIN_ALLOW_THREADS rc = (EXPR); Py_END_ALLOW_THREADS }

CSD_MARSHAL(accept_scan, 14, {
  const int B = x.n(1), gamma = x.n(2), C = x.n(3);
  const double ls = x.d(4), sp = x.d(5), sq = x.d(6);
  const float *x0 = x.p<const float>(7), *mq = x.p<const float>(8), *mp = x.p<const float>(9), *u = x.p<const float>(10);
  float* lr = x.p<float>(11);
  int32_t* na = x.p<int32_t>(12);
  uint32_t* mask = x.p<uint32_t>(13);
  CSD_RUN(csd_accept_scan(ctx, B, gamma, C, ls, static_cast<float>(sp), static_cast<float>(sq), x0, mq, mp, u, lr, na, mask))
})

CSD_MARSHAL(resample, 17, {
  const int B = x.n(1), gamma = x.n(2), C = x.n(3), cap = x.n(4);
  const double ls = x.d(5), sp = x.d(6), sq = x.d(7);
  const int32_t* na = x.p<const int32_t>(8);
  const float *mp = x.p<const float>(9), *mq = x.p<const float>(10), *xi = x.p<const float>(11), *v = x.p<const float>(12);
  float* xn = x.p<float>(13);
  int32_t* np = x.p<int32_t>(14);
  uint32_t* fl = x.p<uint32_t>(15);
  int32_t* ch = x.p<int32_t>(16);
  CSD_RUN(csd_resample(ctx, B, gamma, C, cap, ls, static_cast<float>(sp), static_cast<float>(sq), na, mp, mq, xi, v, xn, np, fl, ch))
})

CSD_MARSHAL(resample_lv, 17, {
  const int B = x.n(1), gamma = x.n(2), C = x.n(3), cap = x.n(4);
  const float* ls = x.p<const float>(5);
  const int32_t* na = x.p<const int32_t>(6);
  const float *mp = x.p<const float>(7), *lp = x.p<const float>(8), *mq = x.p<const float>(9), *lq = x.p<const float>(10),
              *xi = x.p<const float>(11), *v = x.p<const float>(12);
  float* xn = x.p<float>(13);
  int32_t* np = x.p<int32_t>(14);
  uint32_t* fl = x.p<uint32_t>(15);
  int32_t* ch = x.p<int32_t>(16);
  CSD_RUN(csd_resample_lv(ctx, B, gamma, C, cap, ls, na, mp, lp, mq, lq, xi, v, xn, np, fl, ch))
})

CSD_MARSHAL(gmm_draft_sample, 8, {
  const int R = x.n(1), C = x.n(2);
  const csd_gmm q = x.gmm(3);
  const float *u = x.p<const float>(4), *nz = x.p<const float>(5);
  float* xo = x.p<float>(6);
  int32_t* comp = x.p<int32_t>(7);
  CSD_RUN(csd_gmm_draft_sample(ctx, R, C, &q, u, nz, xo, comp))
})

CSD_MARSHAL(gmm_verify, 11, {
  const int B = x.n(1), gamma = x.n(2), C = x.n(3);
  const csd_gmm q = x.gmm(4), p = x.gmm(5);
  const float *xi = x.p<const float>(6), *u = x.p<const float>(7);
  float* lr = x.p<float>(8);
  int32_t* na = x.p<int32_t>(9);
  uint32_t* mask = x.p<uint32_t>(10);
  CSD_RUN(csd_gmm_verify(ctx, B, gamma, C, &q, &p, xi, u, lr, na, mask))
})

CSD_MARSHAL(gmm_resample, 15, {
  const int B = x.n(1), gamma = x.n(2), C = x.n(3), cap = x.n(4);
  const csd_gmm q = x.gmm(5), p = x.gmm(6);
  const int32_t* na = x.p<const int32_t>(7);
  const float *w = x.p<const float>(8), *xi = x.p<const float>(9), *v = x.p<const float>(10);
  float* xn = x.p<float>(11);
  int32_t* np = x.p<int32_t>(12);
  uint32_t* fl = x.p<uint32_t>(13);
  int32_t* ch = x.p<int32_t>(14);
  CSD_RUN(csd_gmm_resample(ctx, B, gamma, C, cap, &q, &p, na, w, xi, v, xn, np, fl, ch))
})

PyObject* set_ptr_of(PyObject*, PyObject* f) {
  Py_INCREF(f);
  Py_XSETREF(g_ptr_of, f);
  Py_RETURN_NONE;
}

#define CSD_METHOD(NAME) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(NAME)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {CSD_METHOD(accept_scan), CSD_METHOD(resample), CSD_METHOD(resample_lv), CSD_METHOD(gmm_draft_sample),
                          CSD_METHOD(gmm_verify), CSD_METHOD(gmm_resample), {"set_ptr_of", set_ptr_of, METH_O, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&kModule); }
