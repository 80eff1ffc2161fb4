// Python entry points of the hot-path calls: argument checks, output allocation, workspace lookup and
// the C-ABI call in one native function each.  The same work in Python (ctypes marshalling of twenty
// arguments, torch.empty, the stream lookup) and the C call took 24 us a call on the host, longer than
// the kernels of a small call; both take 8 us now (a decode step of one sequence: 24.7 -> 10.7 us a
// step, a turn of one request, two calls: 54 -> 39 us).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "recache.h"

namespace {

// The library's functions, by the addresses that the binding resolved when it loaded it.
struct Lib {
  decltype(&recache_encode_workspace_bytes) encode_ws;
  decltype(&recache_compact_workspace_bytes) compact_ws;
  decltype(&recache_prefill_workspace_bytes) prefill_ws;
  decltype(&recache_prefill_history_workspace_bytes) prefill_history_ws;
  decltype(&recache_decode_workspace_bytes) decode_ws;
  decltype(&recache_encode_resources) encode;
  decltype(&recache_compact_routes) compact;
  decltype(&recache_attend_prefill) prefill;
  decltype(&recache_attend_prefill_gather) prefill_gather;
  decltype(&recache_attend_prefill_history) prefill_history;
  decltype(&recache_attend_decode) decode;
  decltype(&recache_attend_decode_gather) decode_gather;
} lib;

PyObject *s_ws, *s_workspace, *s_check;   // interned attribute names of the Python context object

struct Error {};   // a Python exception has been set

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor"); throw Error(); }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || !t.is_contiguous()) { PyErr_SetString(PyExc_AssertionError, "device, contiguous tensors only"); throw Error(); }
  return t;
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
template <typename T> T* ptr_as(PyObject* o) { return static_cast<T*>(ptr(o)); }
long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) {   // numpy integers and the like
    PyErr_Clear();
    PyObject* i = PyNumber_Long(o);
    if (!i) throw Error();
    const long long w = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (w == -1 && PyErr_Occurred()) throw Error();
    return w;
  }
  return v;
}

// What every call carries: the context object, its handle and its storage dtype.
struct Ctx {
  PyObject* self; recache_ctx* h; int dtype;
  explicit Ctx(PyObject* const* a) : self(a[0]), h(nullptr), dtype((int)integer(a[2])) {
    if (a[1] != Py_None) h = static_cast<recache_ctx*>(PyLong_AsVoidPtr(a[1]));
    if (PyErr_Occurred()) throw Error();
  }
  // the caller's workspace, or the context's own, grown by its Python method
  at::Tensor workspace(PyObject* given, int64_t need) const {
    if (given != Py_None) return tensor(given);
    PyObject* ws = PyObject_GetAttr(self, s_ws);
    if (!ws) throw Error();
    if (ws == Py_None || !THPVariable_Check(ws) || THPVariable_Unpack(ws).numel() < (need > 256 ? need : 256)) {
      Py_DECREF(ws);
      PyObject* n = PyLong_FromLongLong(need);
      ws = PyObject_CallMethodObjArgs(self, s_workspace, n, nullptr);
      Py_XDECREF(n);
      if (!ws) throw Error();
    }
    at::Tensor t = THPVariable_Unpack(ws);
    Py_DECREF(ws);
    return t;
  }
  at::ScalarType out_type(PyObject* out_dtype) const {
    if (out_dtype == Py_None) return dtype == RECACHE_F32 ? at::kFloat : at::kBFloat16;
    if (!THPDtype_Check(out_dtype)) { PyErr_SetString(PyExc_TypeError, "out_dtype must be a torch.dtype"); throw Error(); }
    return reinterpret_cast<THPDtype*>(out_dtype)->scalar_type;
  }
  void check(recache_status st, const char* what) const {
    if (st == RECACHE_OK) return;
    PyObject* n = PyLong_FromLong(st);
    PyObject* w = PyUnicode_FromString(what);
    PyObject* r = PyObject_CallMethodObjArgs(self, s_check, n, w, nullptr);   // raises
    Py_XDECREF(n); Py_XDECREF(w); Py_XDECREF(r);
    throw Error();
  }
};
int out_code(at::ScalarType t) { return t == at::kFloat ? RECACHE_F32 : RECACHE_BF16; }
at::Tensor given_or_empty(PyObject* o, at::IntArrayRef sizes, at::ScalarType t, const at::Tensor& like) {
  if (o != Py_None) return tensor(o);
  return at::empty(sizes, at::TensorOptions().dtype(t).device(like.device()));
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Other Python threads run while the launches are made.  (The lock is taken again also where f throws: a tensor
// without memory does when it is asked for its address.)
struct Unlock {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlock() { PyEval_RestoreThread(state); }
};
template <typename F> recache_status unlocked(F f) {
  const Unlock u;
  return f();
}

// Runs a call's body; exceptions become Python ones.
template <typename F> PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n); return nullptr; }
  try {
    return f();
  } catch (const Error&) {
    return nullptr;
  } catch (const std::exception&) {
    torch::translate_exception_to_python(std::current_exception());   // OutOfMemoryError, IndexError ... as torch raises them
    return nullptr;
  }
}

PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx x3, q k v cu max_len slot k_cache v_cache out out_dtype workspace
  return guarded(n, 14, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &q = tensor(a[3]), &cu = tensor(a[6]), &kc = tensor(a[9]);
    const at::ScalarType ot = c.out_type(a[12]);
    const at::Tensor out = given_or_empty(a[11], q.sizes(), ot, q);
    const int n_res = (int)cu.numel() - 1, total = (int)q.size(0), max_len = (int)integer(a[7]);
    const at::Tensor ws = c.workspace(a[13], lib.encode_ws(c.h, n_res, total, max_len));
    void *k = ptr(a[4]), *v = ptr(a[5]), *vc = ptr(a[10]);
    const int32_t* slot = ptr_as<int32_t>(a[8]);
    c.check(unlocked([&] {
      return lib.encode(c.h, q.data_ptr(), k, v, (const int32_t*)cu.data_ptr(), n_res, total, max_len, slot, kc.data_ptr(), vc, kc.size(1),
                        out.data_ptr(), out_code(ot), ws.data_ptr(), ws.numel(), stream());
    }), "recache_encode_resources");
    return THPVariable_Wrap(out);
  });
}

// ctx x3, k_cache v_cache keep res_off res_slot res_len vis mode route_cu route_idx k_out v_out route_len page_table free_pages workspace
PyObject* compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 19, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &kc = tensor(a[3]), &res_off = tensor(a[6]), &res_slot = tensor(a[7]), &route_idx = tensor(a[12]);
    const int n_req = (int)res_off.numel() - 1, listed = (int)res_slot.numel(), mode = (int)integer(a[10]);
    const bool paged = mode == RECACHE_PAGED;
    const at::Tensor ws = c.workspace(a[18], lib.compact_ws(c.h, n_req, listed));
    int64_t capacity = route_idx.numel(), n_free = 0, n_pool = 0;
    int max_pages = 0;
    if (paged) {
      max_pages = (int)tensor(a[16]).size(1); n_free = tensor(a[17]).numel(); n_pool = tensor(a[13]).size(0);
    } else if (a[13] != Py_None) {
      capacity = std::min(capacity, tensor(a[13]).size(0));
    }
    void *vc = ptr(a[4]), *k_out = ptr(a[13]), *v_out = ptr(a[14]);
    const uint8_t *keep = ptr_as<uint8_t>(a[5]), *vis = ptr_as<uint8_t>(a[9]);
    int32_t *res_len = ptr_as<int32_t>(a[8]), *route_cu = ptr_as<int32_t>(a[11]), *route_len = ptr_as<int32_t>(a[15]),
            *table = ptr_as<int32_t>(a[16]), *free_pages = ptr_as<int32_t>(a[17]);
    c.check(unlocked([&] {
      return lib.compact(c.h, kc.data_ptr(), vc, kc.size(1), keep, (const int32_t*)res_off.data_ptr(), (const int32_t*)res_slot.data_ptr(),
                         res_len, n_req, listed, vis, mode, route_cu, route_len, (int32_t*)route_idx.data_ptr(), capacity, k_out, v_out, table,
                         max_pages, free_pages, n_free, n_pool, ws.data_ptr(), ws.numel(), stream());
    }), "recache_compact_routes");
    Py_RETURN_NONE;
  });
}

// ctx x3, q k v cu_q q_pos0 max_q k_route v_route route_cu k_conv_out v_conv_out out out_dtype workspace [route_idx: gather, k/v_route = caches]
PyObject* prefill(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 18, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &q = tensor(a[3]), &k = tensor(a[4]), &cu = tensor(a[6]), &kr = tensor(a[9]);
    const int n_req = (int)cu.numel() - 1, total = (int)q.size(0), max_q = (int)integer(a[8]);
    const at::ScalarType ot = c.out_type(a[15]);
    const at::Tensor out = given_or_empty(a[14], q.sizes(), ot, q);
    const std::array<int64_t, 3> conv = {k.size(1), total, k.size(2)};
    const at::Tensor ko = given_or_empty(a[12], conv, k.scalar_type(), q), vo = given_or_empty(a[13], conv, k.scalar_type(), q);
    const at::Tensor ws = c.workspace(a[16], lib.prefill_ws(c.h, n_req, total, max_q));
    void *v = ptr(a[5]), *vr = ptr(a[10]);
    const int32_t *pos0 = ptr_as<int32_t>(a[7]), *route_cu = ptr_as<int32_t>(a[11]);
    if (a[17] == Py_None) {
      c.check(unlocked([&] {
        return lib.prefill(c.h, q.data_ptr(), k.data_ptr(), v, (const int32_t*)cu.data_ptr(), pos0, n_req, total, max_q, kr.data_ptr(), vr, route_cu,
                           kr.size(0), ko.data_ptr(), vo.data_ptr(), out.data_ptr(), out_code(ot), ws.data_ptr(), ws.numel(), stream());
      }), "recache_attend_prefill");
    } else {
      const at::Tensor& idx = tensor(a[17]);
      c.check(unlocked([&] {
        return lib.prefill_gather(c.h, q.data_ptr(), k.data_ptr(), v, (const int32_t*)cu.data_ptr(), pos0, n_req, total, max_q, kr.data_ptr(), vr,
                                  kr.size(1), (const int32_t*)idx.data_ptr(), route_cu, idx.numel(), ko.data_ptr(), vo.data_ptr(), out.data_ptr(),
                                  out_code(ot), ws.data_ptr(), ws.numel(), stream());
      }), "recache_attend_prefill_gather");
    }
    PyObject* r = PyTuple_New(3);
    if (!r) throw Error();
    PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(out));
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(ko));
    PyTuple_SET_ITEM(r, 2, THPVariable_Wrap(vo));
    return r;
  });
}

// ctx x3, q k v cu_q q_pos0 max_q k_route v_route route_cu k_cache v_cache conv_slot hist_len out out_dtype workspace
PyObject* prefill_history(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 19, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &q = tensor(a[3]), &cu = tensor(a[6]), &kr = tensor(a[9]), &kc = tensor(a[12]);
    const int n_req = (int)cu.numel() - 1, total = (int)q.size(0), max_q = (int)integer(a[8]);
    const at::ScalarType ot = c.out_type(a[17]);
    const at::Tensor out = given_or_empty(a[16], q.sizes(), ot, q);
    const at::Tensor ws = c.workspace(a[18], lib.prefill_history_ws(c.h, n_req, total, max_q));
    void *k = ptr(a[4]), *v = ptr(a[5]), *vr = ptr(a[10]), *vc = ptr(a[13]);
    const int32_t *pos0 = ptr_as<int32_t>(a[7]), *route_cu = ptr_as<int32_t>(a[11]), *slot = ptr_as<int32_t>(a[14]), *hist = ptr_as<int32_t>(a[15]);
    c.check(unlocked([&] {
      return lib.prefill_history(c.h, q.data_ptr(), k, v, (const int32_t*)cu.data_ptr(), pos0, n_req, total, max_q, kr.data_ptr(), vr, route_cu,
                                 kr.size(0), kc.data_ptr(), vc, kc.size(1), slot, hist, out.data_ptr(), out_code(ot), ws.data_ptr(), ws.numel(),
                                 stream());
    }), "recache_attend_prefill_history");
    return THPVariable_Wrap(out);
  });
}

// ctx x3, q q_pos k_pages v_pages res_table res_len hist_table hist_len k_new v_new out out_dtype workspace
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 16, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &q = tensor(a[3]), &kp = tensor(a[5]), &rt = tensor(a[7]), &ht = tensor(a[9]);
    const int batch = (int)q.size(0), mr = (int)rt.size(1), mh = (int)ht.size(1);
    const at::ScalarType ot = c.out_type(a[14]);
    const at::Tensor out = given_or_empty(a[13], q.sizes(), ot, q);
    const at::Tensor ws = c.workspace(a[15], lib.decode_ws(c.h, batch, mr, mh));
    void *vp = ptr(a[6]), *kn = ptr(a[11]), *vn = ptr(a[12]);
    const int32_t *pos = ptr_as<int32_t>(a[4]), *rl = ptr_as<int32_t>(a[8]), *hl = ptr_as<int32_t>(a[10]);
    c.check(unlocked([&] {
      return lib.decode(c.h, q.data_ptr(), pos, batch, kn, vn, kp.data_ptr(), vp, kp.size(0), (const int32_t*)rt.data_ptr(), mr, rl,
                        (const int32_t*)ht.data_ptr(), mh, hl, out.data_ptr(), out_code(ot), ws.data_ptr(), ws.numel(), stream());
    }), "recache_attend_decode");
    return THPVariable_Wrap(out);
  });
}

// ctx x3, q q_pos k_cache v_cache route_idx route_cu max_res_pages k_pages v_pages hist_table hist_len k_new v_new out out_dtype workspace
PyObject* decode_gather(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 19, [&]() -> PyObject* {
    const Ctx c(a);
    const at::Tensor &q = tensor(a[3]), &kc = tensor(a[5]), &idx = tensor(a[7]), &kp = tensor(a[10]), &ht = tensor(a[12]);
    const int batch = (int)q.size(0), mr = (int)integer(a[9]), mh = (int)ht.size(1);
    const at::ScalarType ot = c.out_type(a[17]);
    const at::Tensor out = given_or_empty(a[16], q.sizes(), ot, q);
    const at::Tensor ws = c.workspace(a[18], lib.decode_ws(c.h, batch, mr, mh));
    void *vc = ptr(a[6]), *vp = ptr(a[11]), *kn = ptr(a[14]), *vn = ptr(a[15]);
    const int32_t *pos = ptr_as<int32_t>(a[4]), *cu = ptr_as<int32_t>(a[8]), *hl = ptr_as<int32_t>(a[13]);
    c.check(unlocked([&] {
      return lib.decode_gather(c.h, q.data_ptr(), pos, batch, kn, vn, kc.data_ptr(), vc, kc.size(1), (const int32_t*)idx.data_ptr(), cu, idx.numel(),
                               mr, kp.data_ptr(), vp, kp.size(0), (const int32_t*)ht.data_ptr(), mh, hl, out.data_ptr(), out_code(ot),
                               ws.data_ptr(), ws.numel(), stream());
    }), "recache_attend_decode_gather");
    return THPVariable_Wrap(out);
  });
}

// the library's addresses, in the order of struct Lib
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, (Py_ssize_t)(sizeof(Lib) / sizeof(void*)), [&]() -> PyObject* {
    void** to = reinterpret_cast<void**>(&lib);
    for (Py_ssize_t i = 0; i < n; ++i) {
      to[i] = PyLong_AsVoidPtr(a[i]);
      if (PyErr_Occurred()) throw Error();
    }
    Py_RETURN_NONE;
  });
}

#define RC_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {RC_METHOD(bind), RC_METHOD(encode), RC_METHOD(compact), RC_METHOD(prefill), RC_METHOD(prefill_history),
                         RC_METHOD(decode), RC_METHOD(decode_gather), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  s_ws = PyUnicode_InternFromString("_ws");
  s_workspace = PyUnicode_InternFromString("workspace");
  s_check = PyUnicode_InternFromString("_check");
  return PyModule_Create(&module);
}
