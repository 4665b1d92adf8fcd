// The calls of a training step, and the row builder's, as CPython functions on torch tensors: argument checks, output
// allocation, current device and stream, and the C ABI call, without interpreter code or ctypes
// in between.  On small steps the host is what a call costs (a 144-token step has 28 us of
// kernels): plan, forward and backward took 12.6, 11.1 and 18.7 us through ctypes, of which 4.8,
// 3.7 and 10.1 were the library's own; now 4.4, 5.2 and 12.5.  The call that builds
// the rows of 4096 groups took 94 us through ctypes with a copy of the row count, now 56 (13 of the difference
// are its packing kernel's), the one that deals them out 19.5, now 13.
// Only marshalling lives here; everything is computed by libpp_attn.so, whose entry points are
// looked up once (bind).  Anything unusual -- a tensor that fails a check, descriptors that are not
// contiguous int32 arrays, an error code -- goes back to the Python side, which raises.
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/types.h>

#include "../../include/pp_attn.h"

namespace {

struct Api {
  decltype(&pp_build_plan) build_plan = nullptr;
  decltype(&pp_attn_fwd) fwd = nullptr;
  decltype(&pp_attn_bwd) bwd = nullptr, bwd_det = nullptr;
  decltype(&pp_build_rows_workspace_bytes) rows_bytes = nullptr;
  decltype(&pp_build_rows) build_rows = nullptr;
  decltype(&pp_assign_rows) assign_rows = nullptr;
} api;
PyObject* g_error = nullptr;  // PPError(code, where)
PyObject* g_chk = nullptr;    // _chk(tensor, shape, dtype, name): raises what is wrong with it

pp_stream_t stream_of(c10::DeviceIndex index) {
  return reinterpret_cast<pp_stream_t>(c10::cuda::getCurrentCUDAStream(index).stream());
}

PyObject* raise_code(int rc, const char* where) {
  PyObject* e = PyObject_CallFunction(g_error, "is", rc, where);
  if (e) {
    PyErr_SetObject(reinterpret_cast<PyObject*>(Py_TYPE(e)), e);
    Py_DECREF(e);
  }
  return nullptr;
}

struct Dims {
  int64_t T, Hq, Hkv, D;
};

// The tensor of `o` if it is a contiguous CUDA tensor of that type and shape, on the device of `on`
// (if given); otherwise the Python check is called to raise, and null comes back.
const at::Tensor* take(PyObject* o, at::ScalarType type, const char* type_name, at::IntArrayRef shape,
                       const char* name, const at::Tensor* on = nullptr) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.scalar_type() == type && t.sizes() == shape && t.is_contiguous()) {
      if (!on || t.device() == on->device()) return &t;
      PyErr_Format(PyExc_ValueError, "%s: on another device than q", name);
      return nullptr;
    }
  }
  PyObject* torch = PyImport_ImportModule("torch");
  PyObject* dtype = torch ? PyObject_GetAttrString(torch, type_name) : nullptr;
  PyObject* tup = PyTuple_New(Py_ssize_t(shape.size()));
  for (size_t i = 0; i < shape.size(); ++i) PyTuple_SET_ITEM(tup, Py_ssize_t(i), PyLong_FromLongLong(shape[i]));
  PyObject* r = dtype ? PyObject_CallFunction(g_chk, "OOOs", o, tup, dtype, name) : nullptr;
  if (r && !PyErr_Occurred()) PyErr_Format(PyExc_ValueError, "%s: unsuitable tensor", name);
  Py_XDECREF(r);
  Py_XDECREF(tup);
  Py_XDECREF(dtype);
  Py_XDECREF(torch);
  return nullptr;
}

// A buffer the caller provides, sized by its elements: a contiguous CUDA tensor.
const at::Tensor* take_buffer(PyObject* o, const char* name, const at::Tensor* on = nullptr) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.is_contiguous() && (!on || t.device() == on->device())) return &t;
  }
  PyErr_Format(PyExc_ValueError, "%s: expected a contiguous CUDA tensor%s", name, on ? " on q's device" : "");
  return nullptr;
}

bool nargs(Py_ssize_t n, Py_ssize_t want, const char* what) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "%s: %zd arguments, expected %zd", what, n, want);
  return false;
}

#define PP_GUARD_BEGIN try {
#define PP_GUARD_END                                   \
  }                                                    \
  catch (const std::exception& e) {                    \
    PyErr_SetString(PyExc_RuntimeError, e.what());     \
    return nullptr;                                    \
  }

// bind(library path, PPError, _chk)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 3, "bind")) return nullptr;
  const char* path = PyUnicode_AsUTF8(a[0]);
  if (!path) return nullptr;
  void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (!lib) {
    PyErr_SetString(PyExc_RuntimeError, dlerror());
    return nullptr;
  }
  Api x;
  x.build_plan = reinterpret_cast<decltype(x.build_plan)>(dlsym(lib, "pp_build_plan"));
  x.fwd = reinterpret_cast<decltype(x.fwd)>(dlsym(lib, "pp_attn_fwd"));
  x.bwd = reinterpret_cast<decltype(x.bwd)>(dlsym(lib, "pp_attn_bwd"));
  x.bwd_det = reinterpret_cast<decltype(x.bwd_det)>(dlsym(lib, "pp_attn_bwd_deterministic"));
  x.rows_bytes = reinterpret_cast<decltype(x.rows_bytes)>(dlsym(lib, "pp_build_rows_workspace_bytes"));
  x.build_rows = reinterpret_cast<decltype(x.build_rows)>(dlsym(lib, "pp_build_rows"));
  x.assign_rows = reinterpret_cast<decltype(x.assign_rows)>(dlsym(lib, "pp_assign_rows"));
  if (!x.build_plan || !x.fwd || !x.bwd || !x.bwd_det || !x.rows_bytes || !x.build_rows || !x.assign_rows) {
    PyErr_SetString(PyExc_RuntimeError, "libpp_attn.so lacks an entry point");
    return nullptr;
  }
  api = x;
  Py_INCREF(a[1]);
  Py_XSETREF(g_error, a[1]);
  Py_INCREF(a[2]);
  Py_XSETREF(g_chk, a[2]);
  Py_RETURN_NONE;
}

// build_plan((4 int32 arrays), Hq, Hkv, D, T, workspace): the plan handle, or None when an array is
// not a contiguous one of native int32 (the caller converts it and comes again)
PyObject* build_plan(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 6, "build_plan")) return nullptr;
  PP_GUARD_BEGIN
  if (!PyTuple_Check(a[0]) || PyTuple_GET_SIZE(a[0]) != 4 || !THPVariable_Check(a[5])) Py_RETURN_NONE;
  Py_buffer buf[4];
  int have = 0;
  bool ok = true;
  for (; have < 4 && ok; ++have) {
    if (PyObject_GetBuffer(PyTuple_GET_ITEM(a[0], have), &buf[have], PyBUF_ND | PyBUF_FORMAT) != 0) {
      PyErr_Clear();
      ok = false;
      break;
    }
    const Py_buffer& b = buf[have];
    ok = b.ndim == 1 && b.itemsize == 4 && b.format && b.format[0] == 'i' && b.format[1] == 0;
  }
  auto release = [&] { for (int i = 0; i < have; ++i) PyBuffer_Release(&buf[i]); };
  if (!ok) {
    release();
    Py_RETURN_NONE;
  }
  pp_problem p{};
  p.num_rows = int32_t(buf[0].shape[0]) - 1;
  p.row_group_off = static_cast<const int32_t*>(buf[0].buf);
  p.grp_prompt_len = static_cast<const int32_t*>(buf[1].buf);
  p.grp_resp_off = static_cast<const int32_t*>(buf[2].buf);
  p.resp_len = static_cast<const int32_t*>(buf[3].buf);
  p.num_groups = int32_t(buf[1].shape[0]);
  p.num_responses = int32_t(buf[3].shape[0]);
  p.num_q_heads = int32_t(PyLong_AsLong(a[1]));
  p.num_kv_heads = int32_t(PyLong_AsLong(a[2]));
  p.head_dim = int32_t(PyLong_AsLong(a[3]));
  p.total_tokens = int32_t(PyLong_AsLong(a[4]));
  if (PyErr_Occurred()) {
    release();
    return nullptr;
  }
  const at::Tensor* w = take_buffer(a[5], "workspace");
  if (!w) {
    release();
    return nullptr;
  }
  const at::Tensor& ws = *w;
  const c10::cuda::CUDAGuard guard(ws.device());
  const pp_stream_t s = stream_of(ws.get_device());
  pp_plan* plan = nullptr;
  int rc;
  void* wp = ws.data_ptr();
  const size_t wn = size_t(ws.numel());
  Py_BEGIN_ALLOW_THREADS
  rc = api.build_plan(&p, wp, wn, s, &plan);
  Py_END_ALLOW_THREADS
  release();
  if (rc == PP_ERR_WORKSPACE_TOO_SMALL) {
    PyErr_SetString(PyExc_ValueError, "workspace too small");
    return nullptr;
  }
  if (rc) return raise_code(rc, "pp_build_plan");
  return PyLong_FromVoidPtr(plan);
  PP_GUARD_END
}

bool take_dims(PyObject* const* a, void*& handle, Dims& d) {
  handle = PyLong_AsVoidPtr(a[0]);
  d = {PyLong_AsLongLong(a[1]), PyLong_AsLongLong(a[2]), PyLong_AsLongLong(a[3]), PyLong_AsLongLong(a[4])};
  return !PyErr_Occurred();
}

constexpr at::ScalarType kBf16 = at::kBFloat16, kF32 = at::kFloat;

// fwd(handle, T, Hq, Hkv, D, q, k, v, scale, o | None, lse | None, scratch | None) -> (o, lse)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 12, "fwd")) return nullptr;
  PP_GUARD_BEGIN
  void* handle;
  Dims d;
  if (!take_dims(a, handle, d)) return nullptr;
  const int64_t qs[3] = {d.T, d.Hq, d.D}, ks[3] = {d.T, d.Hkv, d.D}, ls[2] = {d.Hq, d.T};
  const at::Tensor *q, *k, *v;
  if (!(q = take(a[5], kBf16, "bfloat16", qs, "q")) || !(k = take(a[6], kBf16, "bfloat16", ks, "k", q)) ||
      !(v = take(a[7], kBf16, "bfloat16", ks, "v", q)))
    return nullptr;
  const double scale = PyFloat_AsDouble(a[8]);
  if (scale == -1.0 && PyErr_Occurred()) return nullptr;
  if (a[9] != Py_None && !take(a[9], kBf16, "bfloat16", qs, "o", q)) return nullptr;
  if (a[10] != Py_None && !take(a[10], kF32, "float32", ls, "lse", q)) return nullptr;
  const c10::cuda::CUDAGuard guard(q->device());
  const at::Tensor o = a[9] == Py_None ? at::empty(qs, q->options()) : THPVariable_Unpack(a[9]);
  const at::Tensor lse = a[10] == Py_None ? at::empty(ls, q->options().dtype(kF32)) : THPVariable_Unpack(a[10]);
  void* sp = nullptr;
  size_t sn = 0;
  if (a[11] != Py_None) {
    const at::Tensor* t = take_buffer(a[11], "scratch", q);
    if (!t) return nullptr;
    sp = t->data_ptr();
    sn = size_t(t->numel());
  }
  const pp_stream_t s = stream_of(q->get_device());
  const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr();
  void* op = o.data_ptr();
  float* lp = static_cast<float*>(lse.data_ptr());
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = api.fwd(static_cast<const pp_plan*>(handle), qp, kp, vp, float(scale), op, lp, sp, sn, s);
  Py_END_ALLOW_THREADS
  if (rc) return raise_code(rc, "pp_attn_fwd");
  PyObject* r = PyTuple_New(2);
  if (!r) return nullptr;
  PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(o));
  PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(lse));
  return r;
  PP_GUARD_END
}

// bwd(handle, T, Hq, Hkv, D, q, k, v, o, lse, d_o, scale, d_q | None, d_k | None, d_v | None, scratch,
//     deterministic) -> (d_q, d_k, d_v)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 17, "bwd")) return nullptr;
  PP_GUARD_BEGIN
  void* handle;
  Dims d;
  if (!take_dims(a, handle, d)) return nullptr;
  const int64_t qs[3] = {d.T, d.Hq, d.D}, ks[3] = {d.T, d.Hkv, d.D}, ls[2] = {d.Hq, d.T};
  const at::Tensor *q, *k, *v, *o, *lse, *d_o;
  if (!(q = take(a[5], kBf16, "bfloat16", qs, "q")) || !(k = take(a[6], kBf16, "bfloat16", ks, "k", q)) ||
      !(v = take(a[7], kBf16, "bfloat16", ks, "v", q)) || !(o = take(a[8], kBf16, "bfloat16", qs, "o", q)) ||
      !(lse = take(a[9], kF32, "float32", ls, "lse", q)) || !(d_o = take(a[10], kBf16, "bfloat16", qs, "d_o", q)))
    return nullptr;
  const double scale = PyFloat_AsDouble(a[11]);
  if (scale == -1.0 && PyErr_Occurred()) return nullptr;
  const int det = PyObject_IsTrue(a[16]);
  if (det < 0) return nullptr;
  if ((a[12] != Py_None && !take(a[12], kBf16, "bfloat16", qs, "d_q", q)) ||
      (a[13] != Py_None && !take(a[13], kBf16, "bfloat16", ks, "d_k", q)) ||
      (a[14] != Py_None && !take(a[14], kBf16, "bfloat16", ks, "d_v", q)))
    return nullptr;
  const at::Tensor* scratch = take_buffer(a[15], "scratch", q);
  if (!scratch) return nullptr;
  const c10::cuda::CUDAGuard guard(q->device());
  auto out = [&](PyObject* x, const at::Tensor& like, at::IntArrayRef shape) {
    return x == Py_None ? at::empty(shape, like.options()) : THPVariable_Unpack(x);
  };
  const at::Tensor dq = out(a[12], *q, qs), dk = out(a[13], *k, ks), dv = out(a[14], *v, ks);
  const pp_stream_t s = stream_of(q->get_device());
  const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr(),
             *gp = d_o->data_ptr();
  const float* lp = static_cast<const float*>(lse->data_ptr());
  void *dqp = dq.data_ptr(), *dkp = dk.data_ptr(), *dvp = dv.data_ptr(), *sp = scratch->data_ptr();
  const size_t sn = size_t(scratch->numel());
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = (det ? api.bwd_det : api.bwd)(static_cast<const pp_plan*>(handle), qp, kp, vp, op, lp, gp, float(scale),
                                     dqp, dkp, dvp, sp, sn, s);
  Py_END_ALLOW_THREADS
  if (rc) return raise_code(rc, "pp_attn_bwd");
  PyObject* r = PyTuple_New(3);
  if (!r) return nullptr;
  PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(dq));
  PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(dk));
  PyTuple_SET_ITEM(r, 2, THPVariable_Wrap(dv));
  return r;
  PP_GUARD_END
}

// build_rows(prompt_len, resp_off, resp_len, groups, responses, capacity) -> dict
PyObject* build_rows(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 6, "build_rows")) return nullptr;
  PP_GUARD_BEGIN
  const int64_t G = PyLong_AsLongLong(a[3]), N = PyLong_AsLongLong(a[4]), capacity = PyLong_AsLongLong(a[5]);
  if (PyErr_Occurred()) return nullptr;
  const int64_t gs[1] = {G}, os[1] = {G + 1}, ns[1] = {N};
  const at::Tensor *P, *off, *R;
  if (!(P = take(a[0], at::kInt, "int32", gs, "grp_prompt_len")) ||
      !(off = take(a[1], at::kInt, "int32", os, "grp_resp_off")) || !(R = take(a[2], at::kInt, "int32", ns, "resp_len")))
    return nullptr;
  size_t bytes = 0;
  if (const int rc = api.rows_bytes(int32_t(G), &bytes)) return raise_code(rc, "pp_build_rows_workspace_bytes");
  const c10::cuda::CUDAGuard guard(P->device());
  const auto i32 = P->options(), i64 = P->options().dtype(at::kLong);
  const at::Tensor ws = at::empty({int64_t(bytes)}, P->options().dtype(at::kByte));
  const at::Tensor order = at::empty({G}, i32), rgo = at::empty({G + 1}, i32), rtok = at::empty({G}, i64),
                   rcost = at::empty({G}, i64), op = at::empty({G}, i32), ooff = at::empty({G + 1}, i32),
                   orl = at::empty({N}, i32);
  // status code, detail and number of rows: written by the kernel to page-locked memory, which is read
  // behind the synchronisation that the number of rows needs anyway, without a copy
  const at::Tensor meta = at::empty({3}, at::TensorOptions().dtype(at::kInt).pinned_memory(true));
  const volatile int32_t* m = meta.data_ptr<int32_t>();
  void* dm = nullptr;
  if (cudaHostGetDevicePointer(&dm, meta.data_ptr(), 0) != cudaSuccess) {
    PyErr_SetString(PyExc_RuntimeError, "page-locked memory is not mapped into the device");
    return nullptr;
  }
  const c10::cuda::CUDAStream stream = c10::cuda::getCurrentCUDAStream(P->get_device());
  int32_t* meta_dev = static_cast<int32_t*>(dm);
  int rc;
  cudaError_t e = cudaSuccess;
  const int32_t *pp = P->data_ptr<int32_t>(), *po = off->data_ptr<int32_t>(), *pr = R->data_ptr<int32_t>();
  Py_BEGIN_ALLOW_THREADS
  rc = api.build_rows(int32_t(G), int32_t(N), pp, po, pr, int32_t(capacity), ws.data_ptr(), bytes,
                      order.data_ptr<int32_t>(), rgo.data_ptr<int32_t>(), meta_dev + 2, rtok.data_ptr<int64_t>(),
                      rcost.data_ptr<int64_t>(), op.data_ptr<int32_t>(), ooff.data_ptr<int32_t>(),
                      orl.data_ptr<int32_t>(), meta_dev, reinterpret_cast<pp_stream_t>(stream.stream()));
  if (rc == PP_OK) e = cudaStreamSynchronize(stream.stream());
  Py_END_ALLOW_THREADS
  if (rc) return raise_code(rc, "pp_build_rows");
  if (e != cudaSuccess) {
    PyErr_SetString(PyExc_RuntimeError, cudaGetErrorString(e));
    return nullptr;
  }
  const int64_t rows = m[2];
  const int code = m[0], detail = m[1];
  return Py_BuildValue("{sNsNsNsNsNsNsNs(ii)}", "order", THPVariable_Wrap(order), "row_group_off",
                       THPVariable_Wrap(rgo.narrow(0, 0, rows + 1)), "row_tokens",
                       THPVariable_Wrap(rtok.narrow(0, 0, rows)), "row_cost",
                       THPVariable_Wrap(rcost.narrow(0, 0, rows)), "grp_prompt_len", THPVariable_Wrap(op),
                       "grp_resp_off", THPVariable_Wrap(ooff), "resp_len", THPVariable_Wrap(orl), "status", code, detail);
  PP_GUARD_END
}

// assign_rows(row_cost, rows, ranks) -> (order, rank_of_row, rank_cost)
PyObject* assign_rows(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs(n, 3, "assign_rows")) return nullptr;
  PP_GUARD_BEGIN
  const int64_t R = PyLong_AsLongLong(a[1]), ranks = PyLong_AsLongLong(a[2]);
  if (PyErr_Occurred()) return nullptr;
  const int64_t rs[1] = {R};
  const at::Tensor* cost = take(a[0], at::kLong, "int64", rs, "row_cost");
  if (!cost) return nullptr;
  const c10::cuda::CUDAGuard guard(cost->device());
  const auto i32 = cost->options().dtype(at::kInt);
  const at::Tensor order = at::empty({R}, i32), rank_of_row = at::empty({R}, i32),
                   rank_cost = at::empty({ranks}, cost->options());
  const pp_stream_t s = stream_of(cost->get_device());
  const int64_t* cp = cost->data_ptr<int64_t>();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = api.assign_rows(int32_t(R), cp, int32_t(ranks), order.data_ptr<int32_t>(), rank_of_row.data_ptr<int32_t>(),
                       rank_cost.data_ptr<int64_t>(), s);
  Py_END_ALLOW_THREADS
  if (rc) return raise_code(rc, "pp_assign_rows");
  return Py_BuildValue("(NNN)", THPVariable_Wrap(order), THPVariable_Wrap(rank_of_row), THPVariable_Wrap(rank_cost));
  PP_GUARD_END
}

#define PP_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PP_METHOD(bind), PP_METHOD(build_plan), PP_METHOD(fwd), PP_METHOD(bwd),
                         PP_METHOD(build_rows), PP_METHOD(assign_rows),
                         {nullptr, nullptr, 0, nullptr}};
#define PP_STR2(x) #x
#define PP_STR(x) PP_STR2(x)
#define PP_INIT2(x) PyInit_##x
#define PP_INIT(x) PP_INIT2(x)
PyModuleDef module = {PyModuleDef_HEAD_INIT, PP_STR(PP_MODULE), nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PP_INIT(PP_MODULE)() { return PyModule_Create(&module); }   // (PP_MODULE: see build.py)
