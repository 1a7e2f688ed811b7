// The Python methods' way into libfact for the ordinary call: plain CUDA tensors on the handle's device, the library's
// own configuration, torch's current stream.
//
// A call costs more time on the host than most kernels of this library take on the device; marshalling it in Python
// (a dozen attribute reads, torch.empty, the stream object, a foreign call of twenty arguments) was most of that.
// Here the tensors are read, the output allocated and the C entry point called without going back to the interpreter: a
// call takes the host 4 us instead of 15-20 (512^3 with bias and ReLU, one after another: 16.6 -> 5.1 us, the kernel 4.7).
//
// Every function returns the output tensor, or None if anything about the call is not ordinary or the library refused
// it: the Python method then goes its own way, whose checks name the mistake.  Nothing has been launched when the answer is
// None; where the library failed after a launch (a late stage of a block, the reduction behind a sliced product), it is the
// library's status, which the Python method raises.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <vector>

#include "fact.h"

namespace {

using at::ScalarType;
using at::Tensor;

// The tensor in `o` if it is an ordinary strided CUDA tensor on `dev` of that type with contiguous rows.
const Tensor* plain(PyObject* o, ScalarType dtype, int64_t ndim, int dev) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || t.layout() != at::kStrided || !t.is_cuda() || t.device().index() != dev) return nullptr;
  if (t.scalar_type() != dtype || t.dim() != ndim) return nullptr;
  if (ndim > 0 && t.size(-1) > 1 && t.stride(-1) != 1) return nullptr;
  return &t;
}

// Leading dimension of the last two dimensions; a one-row matrix may carry any stride.
int64_t ld(const Tensor& t) { return t.size(-2) > 1 ? t.stride(-2) : std::max<int64_t>(t.size(-1), t.stride(-2)); }

// One call: the handle and its device as the Python object holds them, the current stream.
struct Call {
  fact_handle_t h = nullptr;
  int dev = 0;
  cudaStream_t stream = nullptr;
  bool ok = false;
  int64_t launches = 0;  // of the handle, before this call
  Call(PyObject* handle, PyObject* device) {
    h = reinterpret_cast<fact_handle_t>(PyLong_AsVoidPtr(handle));
    dev = (int)PyLong_AsLong(device);
    ok = h != nullptr && !PyErr_Occurred();
    if (!ok) return;
    stream = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream();
    launches = fact_launch_count(h);
  }
  template <typename O>
  PyObject* answer(fact_status_t st, O& out) const {
    if (st == FACT_OK) return out.result();
    return fact_launch_count(h) != launches ? PyLong_FromLong((long)st) : nullptr;
  }
};

// The output: the caller's (of exactly this shape, BF16 or FP32) or a new one.
struct Out {
  Tensor made;
  const Tensor* t = nullptr;
  PyObject* given = nullptr;
  bool ok = false;
  // `code`: the type of a new one (fact_out_t; anything else is not ordinary)
  Out(PyObject* out, at::IntArrayRef shape, long code, bool bf16_only, int dev) {
    if (out != Py_None) {
      const ScalarType dt = THPVariable_CheckExact(out) ? THPVariable_Unpack(out).scalar_type() : ScalarType::Undefined;
      if (dt != at::kBFloat16 && (dt != at::kFloat || bf16_only)) return;
      t = plain(out, dt, (int64_t)shape.size(), dev);
      if (t == nullptr || t->sizes() != shape) return;
      given = out;
    } else {
      if (code != FACT_OUT_BF16 && code != FACT_OUT_F32) return;
      made = Tensor(at::detail::empty_cuda(shape, code == FACT_OUT_F32 ? at::kFloat : at::kBFloat16,
                                           c10::Device(at::kCUDA, (c10::DeviceIndex)dev), std::nullopt));
      t = &made;
    }
    ok = true;
  }
  fact_out_t type() const { return t->scalar_type() == at::kFloat ? FACT_OUT_F32 : FACT_OUT_BF16; }
  PyObject* result() {
    if (given) return Py_NewRef(given);
    return THPVariable_Wrap(std::move(made));
  }
};

// The handle's workspace (a torch tensor that the Python object grows) if it is large enough and the object already
// knows that this stream uses it; `need` == 0 asks for nothing.
bool workspace_for(PyObject* ws, PyObject* streams, size_t need, const Call& c, void** ptr) {
  *ptr = nullptr;
  if (need == 0) return true;
  if (!THPVariable_CheckExact(ws)) return false;
  const Tensor& t = THPVariable_Unpack(ws);
  if ((size_t)t.numel() < need) return false;
  PyObject* key = PyLong_FromVoidPtr(c.stream);
  const int known = key ? PyDict_Contains(streams, key) : -1;
  Py_XDECREF(key);
  if (known != 1) return false;
  *ptr = t.data_ptr();
  return true;
}

template <typename F>
fact_status_t without_gil(F&& f) {
  fact_status_t st;
  Py_BEGIN_ALLOW_THREADS st = f();
  Py_END_ALLOW_THREADS return st;
}

// An exception of torch's (out of memory, ...) must not cross into the interpreter: the Python path raises it again.
template <typename F>
PyObject* guarded(F&& f) {
  try {
    PyObject* r = f();
    if (r != nullptr) return r;
  } catch (const std::exception&) {
  }
  PyErr_Clear();
  Py_RETURN_NONE;
}

// (handle, device, ws, streams, op, A, B, layout, out, type of a new one): C = A . B for the ops GEMM, GEMM_BATCHED and
// GEMM_SPLITK
PyObject* matmul(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 10) return nullptr;
    Call c(a[0], a[1]);
    const auto op = (fact_op_t)PyLong_AsLong(a[4]);
    const auto layout = (fact_blayout_t)PyLong_AsLong(a[7]);
    const int nd = op == FACT_OP_GEMM_BATCHED ? 3 : 2;
    const Tensor *A = plain(a[5], at::kBFloat16, nd, c.dev), *B = plain(a[6], at::kBFloat16, nd, c.dev);
    if (!c.ok || !A || !B || PyErr_Occurred()) return nullptr;
    const int64_t M = A->size(-2), K = A->size(-1), batch = nd == 3 ? A->size(0) : 1;
    const int64_t N = layout == FACT_B_KN ? B->size(-1) : B->size(-2), Kb = layout == FACT_B_KN ? B->size(-2) : B->size(-1);
    if (Kb != K || (nd == 3 && B->size(0) != batch)) return nullptr;
    const int64_t shape[3] = {batch, M, N};
    Out out(a[8], nd == 3 ? at::IntArrayRef(shape, 3) : at::IntArrayRef(shape + 1, 2), PyLong_AsLong(a[9]), false, c.dev);
    if (!out.ok) return nullptr;
    size_t need = 0;
    void* ws = nullptr;
    if (fact_workspace_bytes(c.h, op, batch, M, N, K, FACT_EPI_NONE, layout, out.type(), nullptr, &need) != FACT_OK ||
        !workspace_for(a[2], a[3], need, c, &ws))
      return nullptr;
    const int64_t lda = ld(*A), ldb = ld(*B), ldc = ld(*out.t);
    const void *pa = A->const_data_ptr(), *pb = B->const_data_ptr();
    void* pc = out.t->data_ptr();
    const fact_out_t ot = out.type();
    fact_status_t st;
    if (op == FACT_OP_GEMM_BATCHED) {
      const int64_t sa = A->stride(0), sb = B->stride(0), sc = out.t->stride(0);
      st = without_gil([&] {
        return fact_gemm_batched(c.h, batch, M, N, K, pa, lda, sa, pb, ldb, sb, layout, pc, ldc, sc, ot, nullptr, ws, need,
                                 c.stream);
      });
    } else if (op == FACT_OP_GEMM_SPLITK) {
      st = without_gil(
          [&] { return fact_gemm_splitk(c.h, M, N, K, pa, lda, pb, ldb, layout, pc, ldc, ot, 0, nullptr, ws, need, c.stream); });
    } else {
      st = without_gil([&] { return fact_gemm(c.h, M, N, K, pa, lda, pb, ldb, layout, pc, ldc, ot, nullptr, ws, need, c.stream); });
    }
    return c.answer(st, out);
  });
}

// 8-bit operands: E4M3 tensors, or their codes as bytes
const Tensor* codes(PyObject* o, int64_t ndim, int dev) {
  const Tensor* t = plain(o, at::kFloat8_e4m3fn, ndim, dev);
  return t != nullptr ? t : plain(o, at::kByte, ndim, dev);
}

// (handle, device, ws, streams, X, W, scale, bias, residual, epilogue, layout, out, type of a new one, group rows, which):
// the linear layers; bit 0 of `which`: FP8 operands with their scale, bit 1: one weight matrix per group of rows
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 15) return nullptr;
    Call c(a[0], a[1]);
    if (!c.ok) return nullptr;
    const long which = PyLong_AsLong(a[14]);
    const bool fp8 = which & 1, grouped = which & 2;
    const auto epi = (fact_epilogue_t)PyLong_AsLong(a[9]);
    const auto layout = (fact_blayout_t)PyLong_AsLong(a[10]);
    const double scale = fp8 ? PyFloat_AsDouble(a[6]) : 1.0;
    if (PyErr_Occurred()) return nullptr;
    const int64_t wd = grouped ? 3 : 2;
    const Tensor* X = fp8 ? codes(a[4], 2, c.dev) : plain(a[4], at::kBFloat16, 2, c.dev);
    const Tensor* W = fp8 ? codes(a[5], wd, c.dev) : plain(a[5], at::kBFloat16, wd, c.dev);
    if (!X || !W) return nullptr;
    const int64_t M = X->size(0), K = X->size(1);
    const int64_t Nw = layout == FACT_B_KN ? W->size(-1) : W->size(-2);
    if ((layout == FACT_B_KN ? W->size(-2) : W->size(-1)) != K) return nullptr;
    if (epi == FACT_EPI_SILU_GATE && Nw % 2) return nullptr;
    const int64_t N = epi == FACT_EPI_SILU_GATE ? Nw / 2 : Nw;
    const void *bias = nullptr, *res = nullptr;
    int64_t ldr = 0;
    if (a[7] != Py_None) {
      const Tensor* t = plain(a[7], at::kBFloat16, 1, c.dev);
      if (!t || t->size(0) != N) return nullptr;
      bias = t->const_data_ptr();
    }
    if (a[8] != Py_None) {
      const Tensor* t = plain(a[8], at::kBFloat16, 2, c.dev);
      if (!t || t->size(0) != M || t->size(1) != N) return nullptr;
      res = t->const_data_ptr();
      ldr = ld(*t);
    }
    std::vector<int64_t> rows;
    if (grouped) {
      if (!PyList_CheckExact(a[13]) || PyList_GET_SIZE(a[13]) != W->size(0)) return nullptr;
      int64_t sum = 0;
      rows.reserve((size_t)W->size(0));
      for (Py_ssize_t i = 0; i < PyList_GET_SIZE(a[13]); ++i) {
        rows.push_back(PyLong_AsLongLong(PyList_GET_ITEM(a[13], i)));
        sum += rows.back();
      }
      if (PyErr_Occurred() || sum != M) return nullptr;
    }
    const int64_t shape[2] = {M, N};
    Out out(a[11], at::IntArrayRef(shape, 2), PyLong_AsLong(a[12]), false, c.dev);
    if (!out.ok) return nullptr;
    const int64_t ldx = ld(*X), ldw = ld(*W), ldy = ld(*out.t);
    const void *px = X->const_data_ptr(), *pw = W->const_data_ptr();
    void* py = out.t->data_ptr();
    const fact_out_t ot = out.type();
    fact_status_t st;
    if (grouped) {
      const int G = (int)rows.size();
      const int64_t sw = G > 1 ? W->stride(0) : W->size(1) * W->stride(1);
      st = without_gil([&] {
        return fp8 ? fact_linear_grouped_fp8(c.h, G, rows.data(), N, K, px, ldx, pw, ldw, sw, (float)scale, bias, res, ldr, py,
                                             ldy, ot, epi, nullptr, c.stream)
                   : fact_linear_grouped(c.h, G, rows.data(), N, K, px, ldx, pw, ldw, sw, layout, bias, res, ldr, py, ldy, ot,
                                         epi, nullptr, c.stream);
      });
    } else {
      size_t need = 0;
      void* ws = nullptr;
      if (fact_workspace_bytes(c.h, fp8 ? FACT_OP_LINEAR_FP8 : FACT_OP_LINEAR, 1, M, N, K, epi, layout, ot, nullptr, &need) !=
              FACT_OK ||
          !workspace_for(a[2], a[3], need, c, &ws))
        return nullptr;
      st = without_gil([&] {
        return fp8 ? fact_linear_fp8(c.h, M, N, K, px, ldx, pw, ldw, (float)scale, bias, res, ldr, py, ldy, ot, epi, nullptr, ws,
                                     need, c.stream)
                   : fact_linear(c.h, M, N, K, px, ldx, pw, ldw, layout, bias, res, ldr, py, ldy, ot, epi, nullptr, ws, need,
                                 c.stream);
      });
    }
    return c.answer(st, out);
  });
}

// (handle, device, q, k, v, causal, scale, out)
PyObject* attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 8) return nullptr;
    Call c(a[0], a[1]);
    const Tensor *q = plain(a[2], at::kBFloat16, 4, c.dev), *k = plain(a[3], at::kBFloat16, 4, c.dev),
                 *v = plain(a[4], at::kBFloat16, 4, c.dev);
    const int causal = PyObject_IsTrue(a[5]);
    const double scale = PyFloat_AsDouble(a[6]);
    if (!c.ok || !q || !k || !v || causal < 0 || PyErr_Occurred()) return nullptr;
    const int64_t B = q->size(0), D = q->size(3), Tk = k->size(1), Hkv = k->size(2);
    if (k->sizes() != v->sizes() || k->size(0) != B || k->size(3) != D) return nullptr;
    Out out(a[7], q->sizes(), FACT_OUT_BF16, true, c.dev);
    if (!out.ok) return nullptr;
    const fact_status_t st = without_gil([&] {
      return fact_attention(c.h, B, q->size(1), Tk, q->size(2), Hkv, D, q->const_data_ptr(), q->stride(0), q->stride(1),
                            q->stride(2), k->const_data_ptr(), k->stride(0), k->stride(1), k->stride(2), v->const_data_ptr(),
                            v->stride(0), v->stride(1), v->stride(2), out.t->data_ptr(), out.t->stride(0), out.t->stride(1),
                            out.t->stride(2), causal, (float)scale, c.stream);
    });
    return c.answer(st, out);
  });
}

// (handle, device, x, gamma, beta, kind, eps, out)
PyObject* norm(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 8) return nullptr;
    Call c(a[0], a[1]);
    const Tensor *x = plain(a[2], at::kBFloat16, 2, c.dev), *g = plain(a[3], at::kBFloat16, 1, c.dev);
    const Tensor* b = a[4] != Py_None ? plain(a[4], at::kBFloat16, 1, c.dev) : nullptr;
    const auto kind = (fact_norm_t)PyLong_AsLong(a[5]);
    const double eps = PyFloat_AsDouble(a[6]);
    if (!c.ok || !x || !g || (a[4] != Py_None && !b) || PyErr_Occurred()) return nullptr;
    if (g->size(0) != x->size(1) || (b && b->size(0) != x->size(1))) return nullptr;
    Out out(a[7], x->sizes(), FACT_OUT_BF16, true, c.dev);
    if (!out.ok) return nullptr;
    const fact_status_t st = without_gil([&] {
      return fact_norm(c.h, kind, x->size(0), x->size(1), x->const_data_ptr(), ld(*x), g->const_data_ptr(),
                       b ? b->const_data_ptr() : nullptr, (float)eps, out.t->data_ptr(), ld(*out.t), c.stream);
    });
    return c.answer(st, out);
  });
}

// (handle, device, ws, streams, address of the descriptor, x, out)
PyObject* block_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 7) return nullptr;
    Call c(a[0], a[1]);
    const auto* desc = reinterpret_cast<const fact_block_t*>(PyLong_AsVoidPtr(a[4]));
    const Tensor* x = plain(a[5], at::kBFloat16, 2, c.dev);
    if (!c.ok || !desc || !x || !x->is_contiguous() || PyErr_Occurred()) return nullptr;
    if (x->size(0) != desc->batch * desc->seq || x->size(1) != desc->hidden) return nullptr;
    Out out(a[6], x->sizes(), FACT_OUT_BF16, true, c.dev);
    if (!out.ok || !out.t->is_contiguous()) return nullptr;
    void* ws = nullptr;
    const size_t need = fact_block_workspace_bytes(desc);
    if (need == 0 || !workspace_for(a[2], a[3], need, c, &ws)) return nullptr;
    const fact_status_t st = without_gil(
        [&] { return fact_block_forward(c.h, desc, x->const_data_ptr(), out.t->data_ptr(), ws, need, c.stream); });
    return c.answer(st, out);
  });
}

PyMethodDef kMethods[] = {
    {"matmul", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(matmul)), METH_FASTCALL, nullptr},
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr},
    {"attention", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(attention)), METH_FASTCALL, nullptr},
    {"norm", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(norm)), METH_FASTCALL, nullptr},
    {"block_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(block_forward)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_fact_bind", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fact_bind() { return PyModule_Create(&kModule); }
