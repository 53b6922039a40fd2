// The per-layer calls of the Python binding as one native call each: unpacks the tensors (pointers, sizes, strides), makes
// what the caller left out (output, statistics, workspace), reads the current stream and calls the C ABI.
// The same steps through ctypes and tensor methods took 17 to 29 us of host time per call, more than the kernels of a
// decode step or a short prompt; here it is 1 to 2 us plus the launches.  No arithmetic and no CUDA call of its own.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "cascade.h"

namespace {

struct Api {
  decltype(&cascade_last_error) last_error;
  decltype(&cascade_workspace_bytes) workspace_bytes;
  decltype(&cascade_attn_sharded) attn_sharded;
  decltype(&cascade_attn_sharded_rope) attn_sharded_rope;
  decltype(&cascade_attn_partials) attn_partials;
  decltype(&cascade_merge) merge;
  decltype(&cascade_decode_step_rope) decode_step_rope;
  decltype(&cascade_attn_decode_static) decode_static;
  decltype(&cascade_plan_advance) plan_advance;
};
Api api;
PyObject* cascade_error = nullptr;  // CascadeError(status, message)

struct PyFailure {};  // a Python exception is set

void raise_status(int status, const char* message) {
  PyObject* e = PyObject_CallFunction(cascade_error, "is", status, message);
  if (e) {
    PyErr_SetObject(cascade_error, e);
    Py_DECREF(e);
  }
  throw PyFailure();
}
void check(cascade_status_t status) {
  if (status != CASCADE_OK) raise_status(status, api.last_error());
}
[[noreturn]] void raise(PyObject* type, const char* message) {
  PyErr_SetString(type, message);
  throw PyFailure();
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, "a tensor is expected");
  return THPVariable_Unpack(o);
}
cascade_strides_t strides(const at::Tensor& t) {
  if (t.dim() != 4 || t.stride(3) != 1)
    raise(PyExc_AssertionError, "expected [batch, tokens, heads, head_dim] with contiguous head_dim");
  return {t.stride(0), t.stride(1), t.stride(2)};
}
cascade_dtype_t dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return CASCADE_F32;
  if (t.scalar_type() != at::kBFloat16)
    raise_status(CASCADE_ERR_UNSUPPORTED, ("dtype " + std::string(c10::toString(t.scalar_type())) + " unsupported").c_str());
  return CASCADE_BF16;
}
int32_t size(const at::Tensor& t, int dim) { return (int32_t)t.size(dim); }
void need_dims(const at::Tensor& t, int n) {
  if (t.dim() != n) raise(PyExc_ValueError, "wrong number of tensor dimensions");
}
void* stream() {  // of the current device, as torch.cuda.current_stream()
  static const bool any = c10::cuda::device_count() > 0;
  return any ? c10::cuda::getCurrentCUDAStream().stream() : nullptr;
}
long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyFailure();
  return v;
}
template <typename T>
T* address(PyObject* o) {
  if (o == Py_None) return nullptr;
  void* p = PyLong_AsVoidPtr(o);
  if (!p && PyErr_Occurred()) throw PyFailure();
  return static_cast<T*>(p);
}
float number(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyFailure();
  return (float)v;
}
bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw PyFailure();
  return v != 0;
}

at::Tensor output_or(PyObject* out, const at::Tensor& like, at::IntArrayRef shape) {
  return out == Py_None ? at::empty(shape, like.options()) : tensor(out);
}
at::Tensor lse_for(bool want, const at::Tensor& q) {
  if (!want) return at::Tensor();
  return at::empty({q.size(0), q.size(1), q.size(2)}, q.options().dtype(at::kFloat));
}
float* data_or_null(const at::Tensor& t) { return t.defined() ? static_cast<float*>(t.data_ptr()) : nullptr; }

struct Scratch {
  at::Tensor own;
  void* ptr = nullptr;
  size_t bytes = 0;
};
Scratch scratch(const cascade_plan_t* plan, int call, cascade_dtype_t code, const at::Tensor& q, int n_kv_heads,
                PyObject* given) {
  Scratch s;
  size_t need = 0;
  check(api.workspace_bytes(plan, call, code, size(q, 0), size(q, 2), n_kv_heads, size(q, 3), &need));
  if (need == 0) return s;
  s.own = given == Py_None ? at::empty({(int64_t)need}, q.options().dtype(at::kByte)) : tensor(given);
  s.ptr = s.own.data_ptr();
  s.bytes = (size_t)s.own.numel() * s.own.element_size();
  return s;
}

PyObject* wrap(const at::Tensor& t) {
  if (!t.defined()) Py_RETURN_NONE;
  return THPVariable_Wrap(t);
}
PyObject* pair(PyObject* given_out, const at::Tensor& o, const at::Tensor& lse) {
  PyObject* r = PyTuple_New(2);
  if (!r) throw PyFailure();
  if (given_out != Py_None) {
    Py_INCREF(given_out);
    PyTuple_SET_ITEM(r, 0, given_out);
  } else {
    PyTuple_SET_ITEM(r, 0, wrap(o));
  }
  PyTuple_SET_ITEM(r, 1, wrap(lse));
  return r;
}

// The C calls run without the interpreter lock.  `f` must not throw, which would leave the lock behind: sizes and data pointers
// are taken before (a tensor without storage, as torch.func.vmap hands out, throws when asked for its pointer).
template <typename F>
cascade_status_t unlocked(F&& f) {
  cascade_status_t status;
  Py_BEGIN_ALLOW_THREADS
  status = f();
  Py_END_ALLOW_THREADS
  return status;
}

template <int N, PyObject* (*F)(PyObject* const*)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments are expected, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (const PyFailure&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

// (plan, q, k, v, scale, rope_table or None, out or None, want_lse, workspace or None) -> (o, lse or None)
PyObject* attn_sharded(PyObject* const* a) {
  const auto* plan = address<const cascade_plan_t>(a[0]);
  const at::Tensor &q = tensor(a[1]), &k = tensor(a[2]), &v = tensor(a[3]);
  need_dims(q, 4);
  const cascade_strides_t qs = strides(q), ks = strides(k), vs = strides(v);
  const cascade_dtype_t code = dtype_code(q);
  const float scale = number(a[4]);
  const int32_t B = size(q, 0), H = size(q, 2), Hkv = size(k, 2), d = size(q, 3);
  const at::Tensor o = output_or(a[6], q, q.sizes());
  const cascade_strides_t os = strides(o);
  const at::Tensor lse = lse_for(truth(a[7]), q);
  const Scratch ws = scratch(plan, CASCADE_CALL_SHARDED, code, q, Hkv, a[8]);
  void *st = stream(), *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr(), *op = o.data_ptr();
  float* lp = data_or_null(lse);
  if (a[5] == Py_None) {
    check(unlocked([&] {
      return api.attn_sharded(plan, code, B, H, Hkv, d, scale, qp, qs, kp, ks, vp, vs, op, os, lp, ws.ptr, ws.bytes, st);
    }));
  } else {
    const at::Tensor& table = tensor(a[5]);
    if (table.scalar_type() != at::kFloat || !table.is_contiguous() || table.dim() != 3 || table.size(1) != d / 2 ||
        table.size(2) != 2)
      raise(PyExc_AssertionError, "the positional table is fp32 [positions, head_dim / 2, 2], contiguous");
    const auto* tp = static_cast<const float*>(table.data_ptr());
    const int32_t n_positions = size(table, 0);
    check(unlocked([&] {
      return api.attn_sharded_rope(plan, code, B, H, Hkv, d, scale, qp, qs, kp, ks, vp, vs, tp, n_positions, op, os, lp,
                                   ws.ptr, ws.bytes, st);
    }));
  }
  return pair(a[6], o, lse);
}

// (plan, n_kv_shards, q, k, v, scale, out or None, workspace or None) -> (o_part, m_part, l_part)
PyObject* attn_partials(PyObject* const* a) {
  const auto* plan = address<const cascade_plan_t>(a[0]);
  const int64_t P = integer(a[1]);
  const at::Tensor &q = tensor(a[2]), &k = tensor(a[3]), &v = tensor(a[4]);
  need_dims(q, 4);
  const cascade_strides_t qs = strides(q), ks = strides(k), vs = strides(v);
  const cascade_dtype_t code = dtype_code(q);
  const float scale = number(a[5]);
  at::Tensor o, m, l;
  if (a[6] == Py_None) {
    const int64_t B = q.size(0), n = q.size(1), H = q.size(2);
    o = at::empty({B, P, n, H, q.size(3)}, q.options());
    m = at::empty({B, P, n, H}, q.options().dtype(at::kFloat));
    l = at::empty_like(m);
  } else {
    PyObject* seq = PySequence_Fast(a[6], "out: (o_part, m_part, l_part) is expected");
    if (!seq) throw PyFailure();
    if (PySequence_Fast_GET_SIZE(seq) != 3) {
      Py_DECREF(seq);
      raise(PyExc_ValueError, "out: (o_part, m_part, l_part) is expected");
    }
    PyObject** item = PySequence_Fast_ITEMS(seq);
    const bool fine = THPVariable_Check(item[0]) && THPVariable_Check(item[1]) && THPVariable_Check(item[2]);
    if (fine) {
      o = THPVariable_Unpack(item[0]);
      m = THPVariable_Unpack(item[1]);
      l = THPVariable_Unpack(item[2]);
    }
    Py_DECREF(seq);
    if (!fine) raise(PyExc_TypeError, "out: three tensors are expected");
  }
  const int32_t B = size(q, 0), H = size(q, 2), Hkv = size(k, 2), d = size(q, 3);
  const Scratch ws = scratch(plan, CASCADE_CALL_PARTIALS, code, q, Hkv, a[7]);
  void *st = stream(), *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr(), *op = o.data_ptr();
  float *mp = static_cast<float*>(m.data_ptr()), *lp = static_cast<float*>(l.data_ptr());
  check(unlocked([&] {
    return api.attn_partials(plan, code, B, H, Hkv, d, scale, qp, qs, kp, ks, vp, vs, op, mp, lp, ws.ptr, ws.bytes, st);
  }));
  PyObject* r = PyTuple_New(3);
  if (!r) throw PyFailure();
  PyTuple_SET_ITEM(r, 0, wrap(o));
  PyTuple_SET_ITEM(r, 1, wrap(m));
  PyTuple_SET_ITEM(r, 2, wrap(l));
  return r;
}

// (o_part, m_part, l_part, row_scatter address, batch stride, out or None, want_lse) -> (o, lse or None)
PyObject* merge(PyObject* const* a) {
  const at::Tensor &parts = tensor(a[0]), &m = tensor(a[1]), &l = tensor(a[2]);
  need_dims(parts, 5);
  const cascade_dtype_t code = dtype_code(parts);
  const int64_t B = parts.size(0), n = parts.size(2), H = parts.size(3), d = parts.size(4);
  const int32_t n_parts = size(parts, 1);
  const auto* rows = address<const int32_t>(a[3]);
  const int64_t row_stride = integer(a[4]);
  const at::Tensor o = output_or(a[5], parts, {B, n, H, d});
  const cascade_strides_t os = strides(o);
  at::Tensor lse;
  if (truth(a[6])) lse = at::empty({B, n, H}, parts.options().dtype(at::kFloat));
  void *st = stream(), *pp = parts.data_ptr(), *op = o.data_ptr();
  const auto *mp = static_cast<const float*>(m.data_ptr()), *lp = static_cast<const float*>(l.data_ptr());
  float* lse_p = data_or_null(lse);
  check(unlocked([&] {
    return api.merge(code, (int32_t)B, n_parts, (int32_t)n, (int32_t)H, (int32_t)d, pp, mp, lp, rows, row_stride, op, os,
                     lse_p, st);
  }));
  return pair(a[5], o, lse);
}

// (plan, q_new, k_new, v_new, k_cache, v_cache, position, scale, rope_table, out or None, want_lse, workspace or None)
PyObject* decode_step_rope(PyObject* const* a) {
  auto* plan = address<cascade_plan_t>(a[0]);
  const at::Tensor &q = tensor(a[1]), &kn = tensor(a[2]), &vn = tensor(a[3]), &kc = tensor(a[4]), &vc = tensor(a[5]);
  const at::Tensor& table = tensor(a[8]);
  need_dims(q, 4);
  const cascade_strides_t qs = strides(q), kns = strides(kn), vns = strides(vn), kcs = strides(kc), vcs = strides(vc);
  const int32_t position = (int32_t)integer(a[6]);
  const float scale = number(a[7]);
  const at::Tensor o = a[9] == Py_None ? at::empty_like(q) : tensor(a[9]);
  const cascade_strides_t os = strides(o);
  const at::Tensor lse = lse_for(truth(a[10]), q);
  const int32_t B = size(q, 0), H = size(q, 2), Hkv = size(kn, 2), n_positions = size(table, 0);
  const Scratch ws = scratch(plan, CASCADE_CALL_DECODE_STEP_ROPE, CASCADE_BF16, q, Hkv, a[11]);
  void *st = stream(), *qp = q.data_ptr(), *knp = kn.data_ptr(), *vnp = vn.data_ptr(), *kcp = kc.data_ptr(),
       *vcp = vc.data_ptr(), *op = o.data_ptr();
  const auto* tp = static_cast<const float*>(table.data_ptr());
  float* lp = data_or_null(lse);
  check(unlocked([&] {
    return api.decode_step_rope(plan, B, H, Hkv, scale, qp, qs, knp, kns, vnp, vns, kcp, kcs, vcp, vcs, position, tp,
                                n_positions, op, os, lp, ws.ptr, ws.bytes, st);
  }));
  return pair(a[9], o, lse);
}

// (plan, q, k, v, scale, out or None, want_lse) -> (o, lse or None)
PyObject* attn_decode_static(PyObject* const* a) {
  const auto* plan = address<const cascade_plan_t>(a[0]);
  const at::Tensor &q = tensor(a[1]), &k = tensor(a[2]), &v = tensor(a[3]);
  need_dims(q, 4);
  if (q.size(1) != 1 || q.size(3) != 128 || q.scalar_type() != at::kBFloat16)
    raise(PyExc_AssertionError, "one bf16 query row of head_dim 128 per sequence is expected");
  const cascade_strides_t qs = strides(q), ks = strides(k), vs = strides(v);
  const float scale = number(a[4]);
  const at::Tensor o = output_or(a[5], q, q.sizes());
  const cascade_strides_t os = strides(o);
  const at::Tensor lse = lse_for(truth(a[6]), q);
  const int32_t B = size(q, 0), H = size(q, 2), Hkv = size(k, 2);
  void *st = stream(), *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr(), *op = o.data_ptr();
  float* lp = data_or_null(lse);
  check(unlocked([&] {
    return api.decode_static(plan, B, H, Hkv, scale, qp, qs, kp, ks, vp, vs, op, os, lp, st);
  }));
  return pair(a[5], o, lse);
}

// (plan, q_pos_offset)
PyObject* plan_advance(PyObject* const* a) {
  auto* plan = address<cascade_plan_t>(a[0]);
  const int32_t offset = (int32_t)integer(a[1]);
  void* st = stream();
  check(unlocked([&] { return api.plan_advance(plan, offset, st); }));
  Py_RETURN_NONE;
}

// load(path of the CUDA library, CascadeError)
PyObject* load(PyObject*, PyObject* args) {
  const char* path = nullptr;
  PyObject* error = nullptr;
  if (!PyArg_ParseTuple(args, "sO", &path, &error)) return nullptr;
  void* h = dlopen(path, RTLD_NOW);
  if (!h) {
    PyErr_SetString(PyExc_ImportError, dlerror());
    return nullptr;
  }
  auto find = [&](auto& fn, const char* name) {
    fn = reinterpret_cast<std::remove_reference_t<decltype(fn)>>(dlsym(h, name));
    if (!fn && !PyErr_Occurred()) PyErr_Format(PyExc_ImportError, "%s has no %s", path, name);
  };
  find(api.last_error, "cascade_last_error");
  find(api.workspace_bytes, "cascade_workspace_bytes");
  find(api.attn_sharded, "cascade_attn_sharded");
  find(api.attn_sharded_rope, "cascade_attn_sharded_rope");
  find(api.attn_partials, "cascade_attn_partials");
  find(api.merge, "cascade_merge");
  find(api.decode_step_rope, "cascade_decode_step_rope");
  find(api.decode_static, "cascade_attn_decode_static");
  find(api.plan_advance, "cascade_plan_advance");
  if (PyErr_Occurred()) return nullptr;
  Py_INCREF(error);
  Py_XDECREF(cascade_error);
  cascade_error = error;
  Py_RETURN_NONE;
}

template <int N, PyObject* (*F)(PyObject* const*)>
constexpr PyCFunction fast() {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<N, F>));
}

PyMethodDef methods[] = {
    {"load", load, METH_VARARGS, nullptr},
    {"attn_sharded", fast<9, attn_sharded>(), METH_FASTCALL, nullptr},
    {"attn_partials", fast<8, attn_partials>(), METH_FASTCALL, nullptr},
    {"merge", fast<7, merge>(), METH_FASTCALL, nullptr},
    {"decode_step_rope", fast<12, decode_step_rope>(), METH_FASTCALL, nullptr},
    {"attn_decode_static", fast<7, attn_decode_static>(), METH_FASTCALL, nullptr},
    {"plan_advance", fast<2, plan_advance>(), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__fastcall(void) { return PyModule_Create(&module); }
