// Python side of the hot calls: turns tensors into pointers and calls the C ABI.
//
// binding.py declares every call; the ones a training or serving loop makes each step come here.
// What bounds a small batch is the host: through ctypes a call with three tensors cost 2.6 us before
// it reached the library (two Python method calls per tensor, argument conversion), a grouped call
// over 64 tables 85 us.  Here a tensor is unpacked in a few nanoseconds.  No work of the table is
// done in this file.
#include <Python.h>

#include <cstdint>
#include <exception>
#include <new>
#include <vector>

#include <ATen/PythonTorchFunctionTLS.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using u32 = uint32_t;
using i64 = int64_t;
using ptr = void*;

// Addresses of the library's functions, set once by bind().
enum Fn {
  F_LOOKUP, F_LOOKUP_NOALLOC, F_LOOKUP_HOST, F_APPLY, F_APPLY_HOST, F_PREPARE, F_AHEAD, F_EXPIRE, F_EXPIRE_SLICE, F_FENCE,
  F_GROUP_PREPARE, F_GROUP_LOOKUP, F_GROUP_APPLY, F_COUNT
};
const char* const kNames[F_COUNT] = {
  "mono_lookup_pool", "mono_lookup_pool_noalloc", "mono_lookup_pool_host", "mono_apply_grads", "mono_apply_grads_host",
  "mono_prepare_push", "mono_group_ahead", "mono_expire", "mono_expire_slice", "mono_fence", "mono_group_prepare_push",
  "mono_group_lookup_pool", "mono_group_apply_grads"
};
ptr g_fn[F_COUNT] = {};
PyObject* g_address_of = nullptr;      // binding._ptr, for what is neither a tensor, an int nor None

template <typename F>
F fn(Fn which) { return reinterpret_cast<F>(g_fn[which]); }

PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 2 || !PyDict_Check(args[0])) { PyErr_SetString(PyExc_TypeError, "bind(addresses, address_of)"); return nullptr; }
  for (int k = 0; k < F_COUNT; ++k) {
    PyObject* v = PyDict_GetItemString(args[0], kNames[k]);
    if (!v) { PyErr_SetString(PyExc_KeyError, kNames[k]); return nullptr; }
    g_fn[k] = PyLong_AsVoidPtr(v);
    if (PyErr_Occurred()) return nullptr;
  }
  Py_INCREF(args[1]);
  Py_XSETREF(g_address_of, args[1]);
  Py_RETURN_NONE;
}

bool expects(Py_ssize_t got, Py_ssize_t want) {
  if (got == want) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, got);
  return false;
}

// A reference that is given back whichever way its scope is left.
struct Owned {
  PyObject* o;
  explicit Owned(PyObject* p) : o(p) {}
  Owned(const Owned&) = delete;
  Owned& operator=(const Owned&) = delete;
  ~Owned() { Py_XDECREF(o); }
};

// Whether x is a torch.Tensor (or Parameter) itself, with nobody listening to its methods: only then may its
// fields be read here.  A subclass may answer for itself, and so may a torch function mode.
bool plain_tensor(PyObject* x) { return THPVariable_CheckExact(x) && !at::impl::torch_function_mode_enabled(); }

// Raw address of a tensor / int / None / anything binding._ptr knows.  What a plain tensor refuses
// (one without storage: inside vmap, grad or jvp, sparse, opaque) is asked for again through Python, which says why.
bool address(PyObject* x, ptr* out) {
  if (plain_tensor(x)) {
    try {
      const at::Tensor& t = THPVariable_Unpack(x);
      if (t.is_contiguous()) { *out = t.data_ptr(); return true; }
    } catch (const std::exception&) {
    }
  }
  if (x == Py_None) { *out = nullptr; return true; }
  if (!PyLong_Check(x)) {
    const Owned r(PyObject_CallOneArg(g_address_of, x));
    if (!r.o) return false;
    *out = PyLong_AsVoidPtr(r.o);
    return !PyErr_Occurred();
  }
  *out = PyLong_AsVoidPtr(x);
  return !PyErr_Occurred();
}

bool integer(PyObject* x, i64* out) {
  *out = PyLong_AsLongLong(x);
  return !(*out == -1 && PyErr_Occurred());
}

template <typename C>
PyObject* without_gil(C&& call) {
  struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }
  };
  int rc;
  { const Released released; rc = call(); }
  return PyLong_FromLong(rc);
}

// Every method is entered through this: a C++ exception that left one would end the process.
using Method = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);
template <Method F>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t n) noexcept {
  try {
    return F(self, args, n);
  } catch (const std::bad_alloc&) {
    return PyErr_NoMemory();
  } catch (const std::exception& e) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
  } catch (...) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
  }
  return nullptr;
}

// (t, ids, n_ids, offsets, n_bags)
struct Batch { ptr t, ids, off; i64 n_ids, n_bags; };
bool batch(PyObject* const* a, Batch* b) {
  return address(a[0], &b->t) && address(a[1], &b->ids) && integer(a[2], &b->n_ids) && address(a[3], &b->off) &&
         integer(a[4], &b->n_bags);
}

template <Fn W>
PyObject* announce(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Batch b;
  if (!expects(n, 5) || !batch(a, &b)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr, ptr, i64, ptr, i64)>(W)(b.t, b.ids, b.n_ids, b.off, b.n_bags); });
}

template <Fn W>
PyObject* pull(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Batch b;
  ptr out;
  if (!expects(n, 6) || !batch(a, &b) || !address(a[5], &out)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr, ptr, i64, ptr, i64, ptr)>(W)(b.t, b.ids, b.n_ids, b.off, b.n_bags, out); });
}

template <Fn W>
PyObject* push(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Batch b;
  ptr grad;
  i64 now;
  if (!expects(n, 7) || !batch(a, &b) || !address(a[5], &grad) || !integer(a[6], &now)) return nullptr;
  return without_gil([&] {
    return fn<int (*)(ptr, ptr, i64, ptr, i64, ptr, i64)>(W)(b.t, b.ids, b.n_ids, b.off, b.n_bags, grad, now);
  });
}

PyObject* expire(PyObject*, PyObject* const* a, Py_ssize_t n) {
  ptr t;
  i64 now;
  if (!expects(n, 2) || !address(a[0], &t) || !integer(a[1], &now)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr, i64)>(F_EXPIRE)(t, now); });
}

PyObject* expire_slice(PyObject*, PyObject* const* a, Py_ssize_t n) {
  ptr t;
  i64 now, slice, slices;
  if (!expects(n, 4) || !address(a[0], &t) || !integer(a[1], &now) || !integer(a[2], &slice) || !integer(a[3], &slices)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr, i64, u32, u32)>(F_EXPIRE_SLICE)(t, now, (u32)slice, (u32)slices); });
}

PyObject* fence(PyObject*, PyObject* const* a, Py_ssize_t n) {
  ptr t;
  if (!expects(n, 1) || !address(a[0], &t)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr)>(F_FENCE)(t); });
}

// Pulls with the arguments of MonoTable.lookup_pool as they are: returns None, having done nothing,
// unless ids and offsets are contiguous 64-bit tensors on the table's device, and out a tensor, all of them plain.
// (handle, device, ids, offsets, out)
PyObject* table_pull(PyObject*, PyObject* const* a, Py_ssize_t n) {
  ptr t, out;
  i64 device;
  if (!expects(n, 5) || !address(a[0], &t) || !integer(a[1], &device)) return nullptr;
  if (!plain_tensor(a[2]) || !plain_tensor(a[3]) || !plain_tensor(a[4])) Py_RETURN_NONE;
  ptr pi, po;
  i64 n_ids, n_bags;
  try {
    const at::Tensor &ids = THPVariable_Unpack(a[2]), &off = THPVariable_Unpack(a[3]);
    for (const at::Tensor* x : {&ids, &off}) {
      const bool words = x->scalar_type() == at::kLong || x->scalar_type() == at::kUInt64;
      if (!words || !x->is_cuda() || x->get_device() != device || !x->is_contiguous()) Py_RETURN_NONE;
    }
    pi = ids.data_ptr(), po = off.data_ptr();
    n_ids = ids.numel(), n_bags = off.numel() - 1;
  } catch (const std::exception&) {
    Py_RETURN_NONE;                                          // (no storage: the Python way says why)
  }
  if (!address(a[4], &out)) return nullptr;
  return without_gil([&] { return fn<int (*)(ptr, ptr, i64, ptr, i64, ptr)>(F_LOOKUP)(t, pi, n_ids, po, n_bags, out); });
}

// Host arrays of the grouped calls: one entry per table.
struct Group {
  std::vector<ptr> t, ids, off, vec;
  std::vector<i64> n_ids, n_bags;
};

bool entries(PyObject* list, size_t n, std::vector<ptr>* p, std::vector<i64>* numel, i64 less) {
  const Owned own(PySequence_Fast(list, "grouped calls take lists, one entry per table"));
  PyObject* const seq = own.o;
  if (!seq) return false;
  bool ok = (size_t)PySequence_Fast_GET_SIZE(seq) == n;
  if (!ok) PyErr_SetString(PyExc_ValueError, "grouped calls take one batch per table");
  p->resize(n);
  if (numel) numel->resize(n);
  for (size_t i = 0; ok && i < n; ++i) {
    PyObject* x = PySequence_Fast_GET_ITEM(seq, i);
    ok = address(x, &(*p)[i]);
    if (!ok || !numel) continue;
    if (plain_tensor(x)) { (*numel)[i] = THPVariable_Unpack(x).numel() - less; continue; }
    const Owned r(PyObject_CallMethod(x, "numel", nullptr));
    ok = r.o && integer(r.o, &(*numel)[i]);
    (*numel)[i] -= less;
  }
  return ok;
}

bool group(PyObject* handles, PyObject* ids, PyObject* off, PyObject* vec, Group* g) {
  const Py_ssize_t n = PySequence_Size(handles);
  return n >= 0 && entries(handles, (size_t)n, &g->t, nullptr, 0) && entries(ids, (size_t)n, &g->ids, &g->n_ids, 0) &&
         entries(off, (size_t)n, &g->off, &g->n_bags, 1) && (!vec || entries(vec, (size_t)n, &g->vec, nullptr, 0));
}

// (handles, ids, offsets, stream)
PyObject* group_prepare(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Group g;
  ptr s;
  if (!expects(n, 4) || !group(a[0], a[1], a[2], nullptr, &g) || !address(a[3], &s)) return nullptr;
  return without_gil([&] {
    return fn<int (*)(int32_t, ptr*, ptr*, i64*, ptr*, i64*, ptr)>(F_GROUP_PREPARE)(
        (int32_t)g.t.size(), g.t.data(), g.ids.data(), g.n_ids.data(), g.off.data(), g.n_bags.data(), s);
  });
}

// (handles, ids, offsets, outs, stream)
PyObject* group_pull(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Group g;
  ptr s;
  if (!expects(n, 5) || !group(a[0], a[1], a[2], a[3], &g) || !address(a[4], &s)) return nullptr;
  return without_gil([&] {
    return fn<int (*)(int32_t, ptr*, ptr*, i64*, ptr*, i64*, ptr*, ptr)>(F_GROUP_LOOKUP)(
        (int32_t)g.t.size(), g.t.data(), g.ids.data(), g.n_ids.data(), g.off.data(), g.n_bags.data(), g.vec.data(), s);
  });
}

// (handles, ids, offsets, grads, now, stream)
PyObject* group_push(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Group g;
  ptr s;
  i64 now;
  if (!expects(n, 6) || !group(a[0], a[1], a[2], a[3], &g) || !integer(a[4], &now) || !address(a[5], &s)) return nullptr;
  return without_gil([&] {
    return fn<int (*)(int32_t, ptr*, ptr*, i64*, ptr*, i64*, ptr*, i64, ptr)>(F_GROUP_APPLY)(
        (int32_t)g.t.size(), g.t.data(), g.ids.data(), g.n_ids.data(), g.off.data(), g.n_bags.data(), g.vec.data(), now, s);
  });
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(static_cast<Method>(guarded<f>))), METH_FASTCALL, nullptr
PyMethodDef kMethods[] = {
  {"bind", FAST(bind)},
  {"lookup_pool", FAST(pull<F_LOOKUP>)},
  {"lookup_pool_noalloc", FAST(pull<F_LOOKUP_NOALLOC>)},
  {"lookup_pool_host", FAST(pull<F_LOOKUP_HOST>)},
  {"apply_grads", FAST(push<F_APPLY>)},
  {"apply_grads_host", FAST(push<F_APPLY_HOST>)},
  {"prepare_push", FAST(announce<F_PREPARE>)},
  {"group_ahead", FAST(announce<F_AHEAD>)},
  {"expire", FAST(expire)},
  {"expire_slice", FAST(expire_slice)},
  {"fence", FAST(fence)},
  {"table_pull", FAST(table_pull)},
  {"group_prepare_push", FAST(group_prepare)},
  {"group_lookup_pool", FAST(group_pull)},
  {"group_apply_grads", FAST(group_push)},
  {nullptr, nullptr, 0, nullptr}
};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding_native", "pointers of tensors handed to the C ABI of mono.h", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding_native() { return PyModule_Create(&kModule); }
