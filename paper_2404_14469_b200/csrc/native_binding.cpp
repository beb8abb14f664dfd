// CPython extension behind the hot calls of binding.py: argument checks, output and workspace
// tensors, and the call into libsnapkv.so, in one native function per entry point.
//
// A call on a short prompt, and every decode step, is over on the GPU in 10-30 us, and the same
// work done in Python (tensor checks, four torch.empty, ctypes marshalling of 17 arguments) took
// 17-20 us of host time per call before the first launch: the GPU waited for the host.  From here
// a whole-step call with its four launches takes 13 us of host time in all, a decode step with its
// one 5, a ragged batch of eight 15.  The library itself is reached through addresses that binding.py looks up in the
// one copy of libsnapkv.so that the process has loaded, so nothing is linked twice.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>
#include <vector>

#include "snapkv_binding.h"

namespace {

struct Fail {  // becomes a SnapKVError
  std::string what;
};

PyObject* g_error = nullptr;

struct Library {
  decltype(&snapkv_status_string) status_string;
  decltype(&snapkv_workspace_size) workspace_size;
  decltype(&snapkv_compress) compress;
  decltype(&snapkv_compress_lse) compress_lse;
  decltype(&snapkv_compress_strided) compress_strided;
  decltype(&snapkv_compress_grouped) compress_grouped;
  decltype(&snapkv_varlen_workspace_size) varlen_workspace_size;
  decltype(&snapkv_binding_varlen) binding_varlen;
  decltype(&snapkv_binding_paged) binding_paged;
  decltype(&snapkv_decode_workspace_size) decode_workspace_size;
  decltype(&snapkv_decode_attention) decode_attention;
} g_lib;

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) throw Fail{std::string(name) + " must be a tensor"};
  return THPVariable_Unpack(o);
}

int to_int(PyObject* o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw nullptr;
  return static_cast<int>(v);
}

const at::Tensor& dev_bf16(PyObject* o, const char* name, int dims) {
  const at::Tensor& t = tensor(o, name);
  if (!(t.is_cuda() && t.scalar_type() == at::kBFloat16 && t.is_contiguous()))
    throw Fail{std::string(name) + " must be a contiguous CUDA bf16 tensor"};
  if (t.dim() != dims) throw Fail{std::string(name) + " has the wrong number of dimensions"};
  return t;
}

// a 4-D view whose rows of d elements are contiguous; the other strides are free
const at::Tensor& dev_bf16_rows(PyObject* o, const char* name) {
  const at::Tensor& t = tensor(o, name);
  if (!(t.is_cuda() && t.scalar_type() == at::kBFloat16 && t.dim() == 4 && t.stride(3) == 1))
    throw Fail{std::string(name) + " must be a CUDA bf16 [B, Hkv, L, d] view with contiguous rows"};
  return t;
}

const float* lse_arg(PyObject* o, int64_t B, int64_t Hq, int64_t W) {
  if (o == Py_None) return nullptr;
  const at::Tensor& t = tensor(o, "lse_obs");
  if (!(t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous() && t.dim() == 3 &&
        t.size(0) == B && t.size(1) == Hq && t.size(2) == W))
    throw Fail{"lse_obs must be a contiguous CUDA fp32 [B, Hq, W] tensor"};
  return static_cast<const float*>(t.data_ptr());
}

at::Tensor empty(std::initializer_list<int64_t> sizes, at::ScalarType type, const at::Device& dev) {
  return at::Tensor(at::detail::empty_cuda(at::IntArrayRef(sizes.begin(), sizes.size()), type, dev, std::nullopt));
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

void check(int code, const char* what) {
  if (code != SNAPKV_OK) throw Fail{std::string(what) + " failed: " + g_lib.status_string(code)};
}

// Attribute of the workspaces that were allocated here, as opposed to the caller's own.
constexpr const char* ALLOCATED = "snapkv_allocated";

// A tensor the caller may have passed in: its own object is handed back, else a new one.
struct Out {
  PyObject* given = nullptr;
  bool workspace = false;
  at::Tensor t;
  void* data() const { return t.data_ptr(); }
  PyObject* release() {
    if (given) {
      Py_INCREF(given);
      return given;
    }
    PyObject* o = THPVariable_Wrap(t);
    if (o && workspace && PyObject_SetAttrString(o, ALLOCATED, Py_True) != 0) {
      Py_DECREF(o);
      return nullptr;
    }
    return o;
  }
};

Out given_or(PyObject* o, const char* name) {
  Out r;
  if (o != Py_None) {
    r.given = o;
    r.t = tensor(o, name);
  }
  return r;
}

// The caller's workspace if it is large enough, else a new one.
Out workspace_for(PyObject* o, size_t need, const at::Device& dev) {
  Out w = given_or(o, "workspace");
  if (!w.given || static_cast<size_t>(w.t.numel()) < need) {
    w.given = nullptr;
    w.workspace = true;
    w.t = empty({static_cast<int64_t>(need > 256 ? need : 256)}, at::kByte, dev);
  }
  return w;
}

PyObject* tuple4(Out& a, Out& b, Out& c, Out& d) {
  PyObject* t = PyTuple_New(4);
  if (!t) throw nullptr;
  Out* all[4] = {&a, &b, &c, &d};
  for (int i = 0; i < 4; ++i) {
    PyObject* o = all[i]->release();
    if (!o) {
      Py_DECREF(t);
      throw nullptr;
    }
    PyTuple_SET_ITEM(t, i, o);
  }
  return t;
}

// Runs `f` (which may throw Fail, or nullptr with a Python error set) for a METH_FASTCALL function.
template <typename F>
PyObject* guarded(Py_ssize_t nargs, Py_ssize_t want, F&& f) {
  if (nargs != want) {
    PyErr_Format(PyExc_TypeError, "%zd arguments are needed, got %zd", want, nargs);
    return nullptr;
  }
  try {
    return f();
  } catch (const Fail& e) {
    PyErr_SetString(g_error ? g_error : PyExc_RuntimeError, e.what.c_str());
  } catch (std::nullptr_t) {
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

struct NoGil {
  PyThreadState* s = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(s); }
};

// A sequence of whole numbers (anything int() takes).
template <typename I>
std::vector<I> whole_numbers(PyObject* o, const char* name) {
  PyObject* seq = PySequence_Fast(o, name);
  if (!seq) throw nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  std::vector<I> v(static_cast<size_t>(n));
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* item = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, i));
    const long long x = item ? PyLong_AsLongLong(item) : -1;
    Py_XDECREF(item);
    if (x == -1 && PyErr_Occurred()) {
      Py_DECREF(seq);
      throw nullptr;
    }
    v[static_cast<size_t>(i)] = static_cast<I>(x);
  }
  Py_DECREF(seq);
  return v;
}

// q_obs, k, v, pool_kernel, pool_type, budget, out_k, out_v, out_idx, workspace, lse_obs, grouped
PyObject* py_compress(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 12, [&]() -> PyObject* {
    const at::Tensor& q = dev_bf16(a[0], "q_obs", 4);
    const at::Tensor& k = dev_bf16_rows(a[1], "k");
    const at::Tensor& v = dev_bf16_rows(a[2], "v");
    if (v.sizes() != k.sizes()) throw Fail{"k and v must have the same shape"};
    const int64_t B = q.size(0), Hq = q.size(1), W = q.size(2), d = q.size(3), Hkv = k.size(1), L = k.size(2);
    if (k.size(0) != B || k.size(3) != d) throw Fail{"q_obs and k disagree on batch or head dimension"};
    const int pk = to_int(a[3]), pt = to_int(a[4]), want = to_int(a[5]);
    const bool grouped = PyObject_IsTrue(a[11]) == 1;
    const bool strided = !(k.is_contiguous() && v.is_contiguous());
    // the library addresses outputs with `budget` rows per head; on the identity path it is
    // called with budget = L so that the tensors stay dense
    const int rows = want < L ? want : static_cast<int>(L);
    const at::Device dev = k.device();
    const int64_t Ho = grouped ? Hkv : Hq;
    Out ok = given_or(a[6], "out_k"), ov = given_or(a[7], "out_v"), oi = given_or(a[8], "out_idx");
    if (!ok.given) ok.t = empty({B, Ho, rows, d}, at::kBFloat16, dev);
    if (!ov.given) ov.t = empty({B, Ho, rows, d}, at::kBFloat16, dev);
    if (!oi.given) oi.t = empty({B, Ho, rows - W}, at::kInt, dev);
    const int iB = static_cast<int>(B), iHq = static_cast<int>(Hq), iHkv = static_cast<int>(Hkv),
              iL = static_cast<int>(L), id = static_cast<int>(d), iW = static_cast<int>(W);
    Out ws = workspace_for(a[9], g_lib.workspace_size(iB, iHq, iHkv, iL, id, iW, pk, pt, rows), dev);
    const float* lse = lse_arg(a[10], B, Hq, W);
    int code;
    {
      void* s = stream();
      const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
      void *okp = ok.data(), *ovp = ov.data(), *wsp = ws.data();
      int32_t* oip = static_cast<int32_t*>(oi.data());
      const size_t wsn = static_cast<size_t>(ws.t.numel());
      const int64_t ks[3] = {k.stride(0), k.stride(1), k.stride(2)}, vs[3] = {v.stride(0), v.stride(1), v.stride(2)};
      NoGil unlocked;
      if (strided || grouped)
        code = (grouped ? g_lib.compress_grouped : g_lib.compress_strided)(
            qp, kp, vp, strided ? ks : nullptr, strided ? vs : nullptr, lse, iB, iHq, iHkv, iL, id, iW, pk, pt,
            rows, okp, ovp, oip, wsp, wsn, s);
      else if (lse)
        code = g_lib.compress_lse(qp, kp, vp, lse, iB, iHq, iHkv, iL, id, iW, pk, pt, rows, okp, ovp, oip, wsp,
                                  wsn, s);
      else
        code = g_lib.compress(qp, kp, vp, iB, iHq, iHkv, iL, id, iW, pk, pt, rows, okp, ovp, oip, wsp, wsn, s);
    }
    check(code, "snapkv_compress");
    return tuple4(ok, ov, oi, ws);
  });
}

// The workspace of a ragged batch.  The call requires room for its largest single sequence, and with
// no more it takes the sequences one after the other; with `want` all go through in one set of launches.
// A caller's own workspace is used as it is when it meets the requirement.  One that an earlier call
// allocated, for a smaller batch perhaps, gives way to a larger one where it would cost launches.
Out ragged_workspace(PyObject* given, const std::vector<int32_t>& lens, int Hq, int Hkv, int d, int W, int pk, int pt,
                     int budget, const at::Device& dev) {
  const size_t want =
      g_lib.varlen_workspace_size(lens.data(), static_cast<int>(lens.size()), Hq, Hkv, d, W, pk, pt, budget);
  if (given != Py_None) {
    const size_t have = static_cast<size_t>(tensor(given, "workspace").numel());
    if (have >= want) return workspace_for(given, 0, dev);
    if (!PyObject_HasAttrString(given, ALLOCATED)) {
      size_t least = 256;
      for (int32_t x : lens)
        if (x > budget) {
          const size_t one = g_lib.workspace_size(1, Hq, Hkv, x, d, W, pk, pt, budget);
          if (one > least) least = one;
        }
      if (have >= least) return workspace_for(given, least, dev);
    }
  }
  return workspace_for(Py_None, want, dev);
}

struct RaggedOut {
  Out ok, ov, oi;
};
// the library writes all of it: rows behind a sequence's own become zero, positions -1
RaggedOut ragged_outputs(int64_t B, int64_t Hq, int64_t budget, int64_t W, int64_t d, const at::Device& dev) {
  RaggedOut r;
  r.ok.t = empty({B, Hq, budget, d}, at::kBFloat16, dev);
  r.ov.t = empty({B, Hq, budget, d}, at::kBFloat16, dev);
  r.oi.t = empty({B, Hq, budget - W}, at::kInt, dev);
  return r;
}

// q_obs, k, v, seq_lens, pool_kernel, pool_type, budget, cu_seqlens, lse_obs, workspace
PyObject* py_varlen(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 10, [&]() -> PyObject* {
    const at::Tensor& q = dev_bf16(a[0], "q_obs", 4);
    const int64_t B = q.size(0), Hq = q.size(1), W = q.size(2), d = q.size(3);
    const std::vector<int32_t> lens = whole_numbers<int32_t>(a[3], "seq_lens");
    if (static_cast<int64_t>(lens.size()) != B) throw Fail{"one length per sequence is needed"};
    const int pk = to_int(a[4]), pt = to_int(a[5]), budget = to_int(a[6]);
    const at::Tensor &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
    int64_t ks[3], vs[3], Hkv, Lmax;
    std::vector<int64_t> off;
    if (a[7] == Py_None) {
      dev_bf16_rows(a[1], "k");
      dev_bf16_rows(a[2], "v");
      Hkv = k.size(1);
      Lmax = k.size(2);
      for (int i = 0; i < 3; ++i) {
        ks[i] = k.stride(i);
        vs[i] = v.stride(i);
      }
    } else {
      if (!(k.is_cuda() && k.scalar_type() == at::kBFloat16 && k.dim() == 3 && k.is_contiguous() &&
            v.sizes() == k.sizes() && v.is_contiguous() && v.scalar_type() == at::kBFloat16))
        throw Fail{"packed k and v must be contiguous CUDA bf16 [total_tokens, Hkv, d]"};
      Hkv = k.size(1);
      Lmax = 0;
      for (int32_t x : lens) Lmax = x > Lmax ? x : Lmax;
      const int64_t row = Hkv * d;
      ks[0] = vs[0] = row * 8;  // the batch stride is not used: offsets are given
      ks[1] = vs[1] = d;
      ks[2] = vs[2] = row;
      off = whole_numbers<int64_t>(a[7], "cu_seqlens");
      for (int64_t& c : off) c *= row;
      if (static_cast<int64_t>(off.size()) != B) throw Fail{"one starting token per sequence is needed"};
    }
    const at::Device dev = k.device();
    const int iHq = static_cast<int>(Hq), iHkv = static_cast<int>(Hkv), id = static_cast<int>(d),
              iW = static_cast<int>(W);
    RaggedOut out = ragged_outputs(B, Hq, budget, W, d, dev);
    Out ws = ragged_workspace(a[9], lens, iHq, iHkv, id, iW, pk, pt, budget, dev);
    const float* lse = lse_arg(a[8], B, Hq, W);
    const int64_t* offp = off.empty() ? nullptr : off.data();
    int code;
    {
      void* s = stream();
      NoGil unlocked;
      code = g_lib.binding_varlen(q.data_ptr(), k.data_ptr(), v.data_ptr(), ks, vs, offp, offp, lens.data(), lse,
                                  static_cast<int>(B), iHq, iHkv, static_cast<int>(Lmax), id, iW, pk, pt, budget,
                                  out.ok.data(), out.ov.data(), static_cast<int32_t*>(out.oi.data()), ws.data(),
                                  static_cast<size_t>(ws.t.numel()), s, 1);
    }
    check(code, "snapkv_compress_varlen");
    return tuple4(out.ok, out.ov, out.oi, ws);
  });
}

// q_obs, k_pool, v_pool, page_table, L, pool_kernel, pool_type, budget, seq_lens, lse_obs, workspace
PyObject* py_paged(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 11, [&]() -> PyObject* {
    const at::Tensor& q = dev_bf16(a[0], "q_obs", 4);
    const at::Tensor& k = dev_bf16_rows(a[1], "k_pool");
    const at::Tensor& v = dev_bf16_rows(a[2], "v_pool");
    const at::Tensor& table = tensor(a[3], "page_table");
    const int64_t B = q.size(0), Hq = q.size(1), W = q.size(2), d = q.size(3);
    if (!(table.is_cuda() && table.scalar_type() == at::kInt && table.is_contiguous() && table.dim() == 2 &&
          table.size(0) == B))
      throw Fail{"page_table must be a contiguous CUDA int32 [B, pages_per_seq] tensor"};
    if (v.sizes() != k.sizes()) throw Fail{"k_pool and v_pool must have the same shape"};
    if (k.size(3) != d) throw Fail{"q_obs and k_pool disagree on the head dimension"};
    const int64_t Hkv = k.size(1);
    const int L = to_int(a[4]), pk = to_int(a[5]), pt = to_int(a[6]), want = to_int(a[7]);
    const at::Device dev = k.device();
    const int iB = static_cast<int>(B), iHq = static_cast<int>(Hq), iHkv = static_cast<int>(Hkv),
              id = static_cast<int>(d), iW = static_cast<int>(W);
    const bool ragged = a[8] != Py_None;
    const int budget = ragged || want < L ? want : L;
    std::vector<int32_t> lens;
    RaggedOut out = ragged_outputs(B, Hq, budget, W, d, dev);
    Out ws;
    if (ragged) {
      lens = whole_numbers<int32_t>(a[8], "seq_lens");
      if (static_cast<int64_t>(lens.size()) != B) throw Fail{"one length per sequence is needed"};
      ws = ragged_workspace(a[10], lens, iHq, iHkv, id, iW, pk, pt, budget, dev);
    } else {
      ws = workspace_for(a[10], g_lib.workspace_size(iB, iHq, iHkv, L, id, iW, pk, pt, budget), dev);
    }
    const float* lse = lse_arg(a[9], B, Hq, W);
    int code;
    {
      void* s = stream();
      const int64_t ks[3] = {k.stride(0), k.stride(1), k.stride(2)}, vs[3] = {v.stride(0), v.stride(1), v.stride(2)};
      NoGil unlocked;
      code = g_lib.binding_paged(q.data_ptr(), k.data_ptr(), v.data_ptr(), ks, vs,
                                 static_cast<const int32_t*>(table.data_ptr()), static_cast<int>(table.size(1)),
                                 static_cast<int>(k.size(2)), static_cast<int>(k.size(0)),
                                 ragged ? lens.data() : nullptr, lse, iB, iHq, iHkv, L, id, iW, pk, pt, budget,
                                 out.ok.data(), out.ov.data(), static_cast<int32_t*>(out.oi.data()), ws.data(),
                                 static_cast<size_t>(ws.t.numel()), s, 1);
    }
    check(code, "snapkv_compress_paged");
    return tuple4(out.ok, out.ov, out.oi, ws);
  });
}

// q_cur, cache_k, cache_v, workspace, want_lse
PyObject* py_decode(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 5, [&]() -> PyObject* {
    const at::Tensor& q = dev_bf16(a[0], "q_cur", 3);
    const at::Tensor& k = dev_bf16(a[1], "cache_k", 4);
    const at::Tensor& v = dev_bf16(a[2], "cache_v", 4);
    const int64_t B = q.size(0), Hq = q.size(1), d = q.size(2);
    if (k.size(0) != B || k.size(3) != d || v.sizes() != k.sizes())
      throw Fail{"q_cur, cache_k and cache_v disagree on their shapes"};
    const at::Device dev = q.device();
    const int iB = static_cast<int>(B), iHq = static_cast<int>(Hq), rows = static_cast<int>(k.size(2)),
              id = static_cast<int>(d);
    Out ws = workspace_for(a[3], g_lib.decode_workspace_size(iB, iHq, rows, id), dev);
    Out out, lse;
    out.t = empty({B, Hq, d}, at::kFloat, dev);
    const bool want = PyObject_IsTrue(a[4]) == 1;
    if (want) lse.t = empty({B, Hq}, at::kFloat, dev);
    int code;
    {
      void* s = stream();
      float* lp = want ? static_cast<float*>(lse.data()) : nullptr;
      NoGil unlocked;
      code = g_lib.decode_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), iB, iHq, static_cast<int>(k.size(1)),
                                    rows, id, static_cast<float*>(out.data()), lp, ws.data(),
                                    static_cast<size_t>(ws.t.numel()), s);
    }
    check(code, "snapkv_decode_attention");
    PyObject* l = Py_None;
    if (want) {
      l = lse.release();
      if (!l) throw nullptr;
    } else {
      Py_INCREF(l);
    }
    PyObject *o = out.release(), *w = ws.release();
    PyObject* t = o && w ? PyTuple_Pack(3, o, l, w) : nullptr;
    Py_XDECREF(o);
    Py_XDECREF(l);
    Py_XDECREF(w);
    return t;
  });
}

// {name: address} of the library's functions, and the exception class for failures
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 2, [&]() -> PyObject* {
    auto at = [&](const char* name) -> void* {
      PyObject* o = PyDict_GetItemString(a[0], name);
      void* p = o ? PyLong_AsVoidPtr(o) : nullptr;
      if (!p) throw Fail{std::string("no address for ") + name};
      return p;
    };
#define SNAPKV_BIND(field) g_lib.field = reinterpret_cast<decltype(g_lib.field)>(at("snapkv_" #field))
    SNAPKV_BIND(status_string);
    SNAPKV_BIND(workspace_size);
    SNAPKV_BIND(compress);
    SNAPKV_BIND(compress_lse);
    SNAPKV_BIND(compress_strided);
    SNAPKV_BIND(compress_grouped);
    SNAPKV_BIND(varlen_workspace_size);
    SNAPKV_BIND(binding_varlen);
    SNAPKV_BIND(binding_paged);
    SNAPKV_BIND(decode_workspace_size);
    SNAPKV_BIND(decode_attention);
#undef SNAPKV_BIND
    Py_INCREF(a[1]);
    g_error = a[1];
    Py_RETURN_NONE;
  });
}

#define SNAPKV_FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {
    {"bind", SNAPKV_FAST(py_bind)},     {"compress", SNAPKV_FAST(py_compress)},
    {"varlen", SNAPKV_FAST(py_varlen)}, {"paged", SNAPKV_FAST(py_paged)},
    {"decode", SNAPKV_FAST(py_decode)}, {nullptr, nullptr, 0, nullptr}};
#undef SNAPKV_FAST

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" PyObject* PyInit__native(void) { return PyModule_Create(&module); }
