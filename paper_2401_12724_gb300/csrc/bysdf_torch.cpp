// The call path of api.py in native code: takes a record dict, checks its
// tensors, allocates the outputs and calls libbysdf's C entry points.
//
// A call through ctypes costs ~30 us on a Grace core (seven allocations, a
// stream lookup, eighteen pointer checks and conversions) against 10 us of
// kernel for a small batch.  Each function here returns NotImplemented
// whenever an argument is not the plain case it knows (another type than a
// torch.Tensor, no storage, not on the GPU, not contiguous, a missing key);
// api.py then takes the general path, which converts it or raises as it
// always has.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <optional>

#include "bysdf.h"

namespace {

struct Lib {
  decltype(&bysdf_workspace_size) workspace_size;
  decltype(&bysdf_eval) eval;
  decltype(&bysdf_sample) sample;
  decltype(&bysdf_pdf) pdf;
  decltype(&bysdf_eval_sample_pdf) fused;
  decltype(&bysdf_eval_backward) backward;
  decltype(&bysdf_eval_backward_ext) backward_ext;
  decltype(&bysdf_eval_l2_backward) l2;
  decltype(&bysdf_set_params) set_params;
  decltype(&bysdf_set_params_ext) set_params_ext;
} L;

// interned names
PyObject *k_h, *k_u, *k_v, *k_wi, *k_wo, *k_ratio, *k_mat_id, *k_seg, *k_u0, *k_u1, *k_f, *k_pdf,
    *k_status, *k_weight, *k_pdf_s, *k_lobe, *k_handle, *k_value, *k_ws, *k_n_mat, *k_keep, *k_workspace;

// Not the plain case: api.py's general path takes the call.
struct Other {};

const at::Tensor& plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) throw Other();
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.is_contiguous() ||
      !t.has_storage() || t.unsafeGetTensorImpl()->is_python_dispatch())
    throw Other();
  return t;
}
PyObject* item(PyObject* rec, PyObject* key) {
  PyObject* o = PyDict_GetItemWithError(rec, key);  // borrowed
  if (!o && PyErr_Occurred()) {
    PyErr_Clear();
    throw Other();
  }
  return o;
}
template <class T>
T* need(PyObject* rec, PyObject* key) {
  PyObject* o = item(rec, key);
  if (!o) throw Other();
  return static_cast<T*>(plain(o).data_ptr());
}
template <class T>
T* maybe(PyObject* rec, PyObject* key) {
  PyObject* o = item(rec, key);
  return !o || o == Py_None ? nullptr : static_cast<T*>(plain(o).data_ptr());
}

struct Call {
  bysdf_materials* mats;
  bysdf_hits hits;
  int64_t n, n_mat;
  at::Device device{at::kCUDA};
  at::Tensor ws_t;  // held while the call runs
  void* ws;
  size_t ws_bytes;
  void* stream;

  Call(PyObject* m, PyObject* rec, PyObject* st, bool with_wo) {
    if (!PyDict_CheckExact(rec)) throw Other();
    PyObject* po = item(rec, k_h);
    if (!po) throw Other();
    const at::Tensor& h = plain(po);
    if (h.dim() < 1) throw Other();
    n = h.size(0);
    device = h.device();
    mats = static_cast<bysdf_materials*>(handle(m));
    n_mat = number(m, k_n_mat);
    hits = bysdf_hits{};
    hits.h = static_cast<const float*>(h.data_ptr());
    hits.u = need<const float>(rec, k_u);
    hits.v = need<const float>(rec, k_v);
    hits.wi = need<const float>(rec, k_wi);
    hits.wo = with_wo ? maybe<const float>(rec, k_wo) : nullptr;
    hits.ratio = maybe<const float>(rec, k_ratio);
    hits.mat_id = maybe<const int32_t>(rec, k_mat_id);
    hits.seg_offsets = maybe<const int64_t>(rec, k_seg);
    PyObject* w = PyObject_GetAttr(m, k_ws);
    if (w && (w == Py_None || !holds(w))) {
      // none yet, or for fewer records: the object makes it
      Py_DECREF(w);
      PyObject* count = PyLong_FromLongLong(n);
      w = count ? PyObject_CallMethodOneArg(m, k_workspace, count) : nullptr;
      Py_XDECREF(count);
    }
    const bool ok = w && holds(w);
    Py_XDECREF(w);
    if (PyErr_Occurred()) PyErr_Clear();
    if (!ok) throw Other();
    ws = ws_t.data_ptr();
    ws_bytes = (size_t)ws_t.numel();
    if (st == Py_None) {
      stream = c10::cuda::getCurrentCUDAStream().stream();
    } else {
      stream = PyLong_AsVoidPtr(st);
      if (PyErr_Occurred()) {
        PyErr_Clear();
        throw Other();
      }
    }
  }
  // Takes a workspace tensor if it is large enough for the call.
  bool holds(PyObject* w) {
    try {
      ws_t = plain(w);
    } catch (const Other&) {
      return false;
    }
    return (size_t)ws_t.numel() >= L.workspace_size(mats, n);
  }
  static int64_t number(PyObject* o, PyObject* name) {
    PyObject* v = PyObject_GetAttr(o, name);
    const int64_t x = v ? PyLong_AsLongLong(v) : -1;
    Py_XDECREF(v);
    if (PyErr_Occurred()) {
      PyErr_Clear();
      throw Other();
    }
    return x;
  }
  static void* handle(PyObject* m) {
    PyObject* h = PyObject_GetAttr(m, k_handle);
    PyObject* v = h ? PyObject_GetAttr(h, k_value) : nullptr;  // None has no value
    Py_XDECREF(h);
    void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
    Py_XDECREF(v);
    if (PyErr_Occurred()) PyErr_Clear();
    if (!p) throw Other();
    return p;
  }
};

struct Out {
  at::Tensor t;
  Out(const Call& c, std::initializer_list<int64_t> shape, at::ScalarType type)
      : t(at::empty(at::IntArrayRef(shape), at::TensorOptions().dtype(type).device(c.device))) {
    // under a fake or functional mode the result holds no memory
    if (!t.has_storage() || t.unsafeGetTensorImpl()->is_python_dispatch()) throw Other();
  }
  float* f() const { return static_cast<float*>(t.data_ptr()); }
  uint8_t* b() const { return static_cast<uint8_t*>(t.data_ptr()); }
  PyObject* py() const { return THPVariable_Wrap(t); }
};

PyObject* none() {
  Py_RETURN_NONE;
}
PyObject* tuple(std::initializer_list<PyObject*> xs) {
  PyObject* r = PyTuple_New((Py_ssize_t)xs.size());
  Py_ssize_t i = 0;
  for (PyObject* x : xs) PyTuple_SET_ITEM(r, i++, x);
  return r;
}
void put(PyObject* d, PyObject* key, PyObject* v) {
  PyDict_SetItem(d, key, v);
  Py_DECREF(v);
}

template <class F>
int unlocked(F&& f) {
  PyThreadState* s = PyEval_SaveThread();
  const int rc = f();
  PyEval_RestoreThread(s);
  return rc;
}

// A C++ exception of a tensor operation leaves the call to the general path,
// which meets it again where Python reports it.
template <class F>
PyObject* guarded(F&& f) {
  try {
    return f();
  } catch (const Other&) {
  } catch (const std::exception&) {
  }
  PyErr_Clear();
  Py_RETURN_NOTIMPLEMENTED;
}

// forward(op, mats, rec, u0, u1, with_pdf, stream): the outputs, an error
// code, or NotImplemented.  op: BYSDF_OP_*.
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t na) {
  if (na != 7) Py_RETURN_NOTIMPLEMENTED;
  return guarded([&]() -> PyObject* {
    const long op = PyLong_AsLong(a[0]);
    const bool samples = op == BYSDF_OP_SAMPLE || op == BYSDF_OP_FUSED;
    Call c(a[1], a[2], a[6], op != BYSDF_OP_SAMPLE);
    const float *u0 = nullptr, *u1 = nullptr;
    if (samples) {
      u0 = a[3] == Py_None ? need<const float>(a[2], k_u0)
                           : static_cast<const float*>(plain(a[3]).data_ptr());
      u1 = a[4] == Py_None ? need<const float>(a[2], k_u1)
                           : static_cast<const float*>(plain(a[4]).data_ptr());
    }
    const int64_t n = c.n;
    if (op == BYSDF_OP_EVAL) {
      const bool with_pdf = a[5] == Py_True;
      Out f(c, {3, n}, at::kFloat);
      std::optional<Out> p;
      if (with_pdf) p.emplace(c, std::initializer_list<int64_t>{n}, at::kFloat);
      Out st(c, {n}, at::kByte);
      const int rc = unlocked([&] {
        return L.eval(c.mats, &c.hits, n, f.f(), p ? p->f() : nullptr, st.b(), c.ws, c.ws_bytes,
                      c.stream);
      });
      if (rc) return PyLong_FromLong(rc);
      return tuple({f.py(), p ? p->py() : none(), st.py()});
    }
    if (op == BYSDF_OP_PDF) {
      Out p(c, {n}, at::kFloat), st(c, {n}, at::kByte);
      const int rc = unlocked([&] {
        return L.pdf(c.mats, &c.hits, n, p.f(), st.b(), c.ws, c.ws_bytes, c.stream);
      });
      if (rc) return PyLong_FromLong(rc);
      return tuple({p.py(), st.py()});
    }
    if (op == BYSDF_OP_SAMPLE) {
      Out wo(c, {3, n}, at::kFloat), w(c, {3, n}, at::kFloat), p(c, {n}, at::kFloat),
          ls(c, {n}, at::kByte);
      const int rc = unlocked([&] {
        return L.sample(c.mats, &c.hits, u0, u1, n, wo.f(), w.f(), p.f(), ls.b(), c.ws,
                        c.ws_bytes, c.stream);
      });
      if (rc) return PyLong_FromLong(rc);
      return tuple({wo.py(), w.py(), p.py(), ls.py()});
    }
    if (op != BYSDF_OP_FUSED) throw Other();
    Out f(c, {3, n}, at::kFloat), p(c, {n}, at::kFloat), st(c, {n}, at::kByte),
        wo(c, {3, n}, at::kFloat), w(c, {3, n}, at::kFloat), ps(c, {n}, at::kFloat),
        ls(c, {n}, at::kByte);
    const int rc = unlocked([&] {
      return L.fused(c.mats, &c.hits, u0, u1, n, f.f(), p.f(), st.b(), wo.f(), w.f(), ps.f(),
                     ls.b(), c.ws, c.ws_bytes, c.stream);
    });
    if (rc) return PyLong_FromLong(rc);
    PyObject* d = PyDict_New();
    put(d, k_f, f.py());
    put(d, k_pdf, p.py());
    put(d, k_status, st.py());
    put(d, k_wo, wo.py());
    put(d, k_weight, w.py());
    put(d, k_pdf_s, ps.py());
    put(d, k_lobe, ls.py());
    return d;
  });
}

// backward(kind, mats, rec, x, weight, flag, deterministic, stream).  kind 0:
// x = grad_f, returns grad; 1: extended set, flag = directions, returns
// (grad, gwi, gwo); 2: L2, x = target, flag = with_f, returns (grad, loss, f).
PyObject* backward(PyObject*, PyObject* const* a, Py_ssize_t na) {
  if (na != 8) Py_RETURN_NOTIMPLEMENTED;
  return guarded([&]() -> PyObject* {
    const long kind = PyLong_AsLong(a[0]);
    Call c(a[1], a[2], a[7], true);
    const float* x = static_cast<const float*>(plain(a[3]).data_ptr());
    const float* weight =
        a[4] == Py_None ? nullptr : static_cast<const float*>(plain(a[4]).data_ptr());
    const bool flag = a[5] == Py_True;
    const int det = a[6] == Py_True ? 1 : 0;
    const int64_t n = c.n;
    Out g(c, {c.n_mat, kind == 1 ? BYSDF_NPARAM_EXT : BYSDF_NPARAM}, at::kFloat);
    if (kind == 0) {
      const int rc = unlocked([&] {
        return L.backward(c.mats, &c.hits, n, x, g.f(), det, c.ws, c.ws_bytes, c.stream);
      });
      return rc ? PyLong_FromLong(rc) : g.py();
    }
    std::optional<Out> p, q;
    if (kind == 1) {
      if (flag) {
        p.emplace(c, std::initializer_list<int64_t>{3, n}, at::kFloat);
        q.emplace(c, std::initializer_list<int64_t>{3, n}, at::kFloat);
      }
      const int rc = unlocked([&] {
        return L.backward_ext(c.mats, &c.hits, n, x, g.f(), p ? p->f() : nullptr,
                              q ? q->f() : nullptr, det, c.ws, c.ws_bytes, c.stream);
      });
      if (rc) return PyLong_FromLong(rc);
      return tuple({g.py(), p ? p->py() : none(), q ? q->py() : none()});
    }
    if (kind != 2) throw Other();
    p.emplace(c, std::initializer_list<int64_t>{c.n_mat}, at::kFloat);
    if (flag) q.emplace(c, std::initializer_list<int64_t>{3, n}, at::kFloat);
    const int rc = unlocked([&] {
      return L.l2(c.mats, &c.hits, n, x, weight, q ? q->f() : nullptr, p->f(), g.f(), det, c.ws,
                  c.ws_bytes, c.stream);
    });
    if (rc) return PyLong_FromLong(rc);
    return tuple({g.py(), p->py(), q ? q->py() : none()});
  });
}

// set_params(columns, mats, params, stream): None, an error code, or
// NotImplemented.  The tensor is kept by the materials object until the next
// update, as the library reads it on the stream.
PyObject* set_params(PyObject*, PyObject* const* a, Py_ssize_t na) {
  if (na != 4) Py_RETURN_NOTIMPLEMENTED;
  return guarded([&]() -> PyObject* {
    const long cols = PyLong_AsLong(a[0]);
    auto* m = static_cast<bysdf_materials*>(Call::handle(a[1]));
    const at::Tensor& p = plain(a[2]);
    if (p.scalar_type() != at::kFloat || p.dim() != 2 ||
        p.size(0) != Call::number(a[1], k_n_mat) || p.size(1) != cols ||
        p.get_device() != c10::cuda::current_device())
      throw Other();
    void* stream = a[3] == Py_None ? (void*)c10::cuda::getCurrentCUDAStream().stream()
                                   : PyLong_AsVoidPtr(a[3]);
    if (PyErr_Occurred()) throw Other();
    const float* x = static_cast<const float*>(p.data_ptr());
    const int rc = unlocked([&] {
      return cols == BYSDF_NPARAM ? L.set_params(m, x, stream) : L.set_params_ext(m, x, stream);
    });
    if (rc) return PyLong_FromLong(rc);
    PyObject* keep = THPVariable_Wrap(p.detach());
    PyObject_SetAttr(a[1], k_keep, keep);
    Py_DECREF(keep);
    if (PyErr_Occurred()) PyErr_Clear();
    Py_RETURN_NONE;
  });
}

// bind(addresses): the C entry points of the library in use, by name.
PyObject* bind(PyObject*, PyObject* d) {
  auto get = [&](const char* name) -> void* {
    PyObject* v = PyDict_GetItemString(d, name);
    return v ? PyLong_AsVoidPtr(v) : nullptr;
  };
#define BIND(field, name)                                           \
  L.field = reinterpret_cast<decltype(L.field)>(get(#name));        \
  if (!L.field) return PyErr_Format(PyExc_ValueError, "no %s", #name)
  BIND(workspace_size, bysdf_workspace_size);
  BIND(eval, bysdf_eval);
  BIND(sample, bysdf_sample);
  BIND(pdf, bysdf_pdf);
  BIND(fused, bysdf_eval_sample_pdf);
  BIND(backward, bysdf_eval_backward);
  BIND(backward_ext, bysdf_eval_backward_ext);
  BIND(l2, bysdf_eval_l2_backward);
  BIND(set_params, bysdf_set_params);
  BIND(set_params_ext, bysdf_set_params_ext);
#undef BIND
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(forward)), METH_FASTCALL,
     nullptr},
    {"backward", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(backward)), METH_FASTCALL,
     nullptr},
    {"set_params", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(set_params)),
     METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_bysdf_torch", nullptr, -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__bysdf_torch(void) {
  k_h = PyUnicode_InternFromString("h");
  k_u = PyUnicode_InternFromString("u");
  k_v = PyUnicode_InternFromString("v");
  k_wi = PyUnicode_InternFromString("wi");
  k_wo = PyUnicode_InternFromString("wo");
  k_ratio = PyUnicode_InternFromString("ratio");
  k_mat_id = PyUnicode_InternFromString("mat_id");
  k_seg = PyUnicode_InternFromString("seg_offsets");
  k_u0 = PyUnicode_InternFromString("u0");
  k_u1 = PyUnicode_InternFromString("u1");
  k_f = PyUnicode_InternFromString("f");
  k_pdf = PyUnicode_InternFromString("pdf");
  k_status = PyUnicode_InternFromString("status");
  k_weight = PyUnicode_InternFromString("weight");
  k_pdf_s = PyUnicode_InternFromString("pdf_s");
  k_lobe = PyUnicode_InternFromString("lobe_status");
  k_handle = PyUnicode_InternFromString("handle");
  k_value = PyUnicode_InternFromString("value");
  k_ws = PyUnicode_InternFromString("_ws");
  k_n_mat = PyUnicode_InternFromString("n_mat");
  k_keep = PyUnicode_InternFromString("_params_keepalive");
  k_workspace = PyUnicode_InternFromString("workspace");
  return PyModule_Create(&module_def);
}
