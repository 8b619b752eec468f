// Native half of autograd.py: one Python call per forward, one autograd node per backward.
//
// A call on a short batch is host time: as a Python autograd.Function around ctypes the forward
// cost 75-90 us of interpreter, marshalling and allocator time and a training step 210-240 us, on
// kernels that need a fraction of that.  Here the arguments are read with the C API of Python, the
// buffers come from PyTorch's caching allocator without the dispatcher, what only the library and the
// backward read (saved branch outputs, log-sum-exps, workspace) is one allocation, and the backward is a C++
// node of the autograd graph.  Without a gradient to compute nothing is saved at all.
//
// Plumbing only, as in autograd.py: every step of the method runs behind the C ABI (blossom.h).
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/function.h>
#include <torch/csrc/autograd/functions/utils.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/autograd/saved_variable.h>
#include <torch/csrc/autograd/variable.h>

#include <stdexcept>
#include <string>

#include "../../include/blossom.h"

namespace {

using at::Tensor;
using torch::autograd::Node;
using torch::autograd::SavedVariable;
using torch::autograd::variable_list;

// the tensor's elements tile its storage span without gaps or overlap, so that a buffer of numel elements laid
// out with the same strides holds every one
bool dense(const Tensor &t) {
  int64_t span = 1;
  for (int64_t i = 0; i < t.dim(); ++i) {
    if (t.stride(i) <= 0) return false;
    span += (t.size(i) - 1) * t.stride(i);
  }
  return t.numel() > 0 && span == t.numel();
}

// an uninitialised tensor with exactly t's shape and strides (empty_like does not keep those of a view that is
// not dense, and the library writes every q-shaped buffer with the strides it is given)
Tensor like(const Tensor &t) {
  if (!t.is_cuda()) return at::empty_strided(t.sizes(), t.strides(), t.options());
  return at::detail::empty_strided_cuda(t.sizes(), t.strides(), t.scalar_type(), t.device());
}
Tensor fresh(at::IntArrayRef sizes, at::ScalarType type, const at::Device &dev) {
  return at::detail::empty_cuda(sizes, type, dev, std::nullopt);
}

// src's values in `dst` (same sizes, another layout) by the library's copy of rows in 16-byte pieces.  False, and
// nothing done, for every other form: types, strides of the last dimension, views that have to be resolved, tensors
// without memory of their own, empty ones.
bool copy_rows(const Tensor &src, const Tensor &dst) {
  if (!src.is_cuda() || !src.has_storage() || src.unsafeGetTensorImpl()->is_python_dispatch() || src.dim() != 4 ||
      src.scalar_type() != dst.scalar_type() || src.device() != dst.device() || src.sizes() != dst.sizes() ||
      src.numel() == 0 || src.stride(3) != 1 || dst.stride(3) != 1 || src.is_neg() || src._is_zerotensor() ||
      src.size(0) > INT32_MAX || src.size(1) > INT32_MAX || src.size(2) > INT32_MAX || src.size(3) > 1024)
    return false;
  const int64_t e = src.element_size();
  const int64_t ss[3] = {src.stride(0) * e, src.stride(1) * e, src.stride(2) * e},
                ds[3] = {dst.stride(0) * e, dst.stride(1) * e, dst.stride(2) * e};
  return blossom_copy_rows((int32_t)src.size(0), (int32_t)src.size(1), (int32_t)src.size(2), (int32_t)(src.size(3) * e),
                           src.data_ptr(), ss, dst.data_ptr(), ds,
                           (blossom_stream_t)c10::cuda::getCurrentCUDAStream(dst.device().index()).stream()) == BLOSSOM_OK;
}
Tensor copied(const Tensor &src, const Tensor &dst) { return copy_rows(src, dst) ? dst : dst.copy_(src); }
Tensor packed(const Tensor &t) {
  if (t.is_contiguous() || !t.is_cuda() || !t.has_storage() || t.unsafeGetTensorImpl()->is_python_dispatch())
    return t.contiguous();
  const Tensor dst = at::empty(t.sizes(), t.options());
  return copy_rows(t, dst) ? dst : t.contiguous();
}

// Makes `t`, whose layout is already the one wanted, plain memory: the library reads addresses, which know nothing of a view
// that negates (wrong signs) and of a zero tensor (no memory).
void make_plain(Tensor &t) {
  if (t.defined() && (t.is_neg() || t._is_zerotensor())) t = like(t).copy_(t);
}

std::string failure(const char *where, int rc) {
  return std::string(where) + ": " + blossom_status_string(rc) + " (status " + std::to_string(rc) + ")";
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// What the backward needs beside q, k, v, the gate and the indices: one allocation
// [out_lt | out_st | lse | workspace].
struct Scratch {
  size_t span, lse_bytes, ws_bytes;
  size_t bytes() const { return 2 * span + lse_bytes + ws_bytes; }
  void *out_lt(char *base) const { return base; }
  void *out_st(char *base) const { return base + span; }
  float *lse(char *base) const { return reinterpret_cast<float *>(base + 2 * span); }
  void *workspace(char *base) const { return base + 2 * span + lse_bytes; }
};

struct BlossomAttentionBackward : public Node {
  // (the scratch buffer, the largest of them, goes through the saved-tensor hooks like the rest: offloading and
  // checkpointing free it between the passes)
  SavedVariable q_, k_, v_, gate_, idx_, buf_;
  Tensor lens_, phi_;  // (the params hold phi's address)
  Scratch scratch_;
  blossom_params params_;
  at::ScalarType gate_type_;

  std::string name() const override { return "BlossomAttentionBackward"; }
  void release_variables() override {
    q_.reset_data();
    k_.reset_data();
    v_.reset_data();
    gate_.reset_data();
    idx_.reset_data();
    buf_.reset_data();
  }
  variable_list apply(variable_list &&grads) override {
    at::NoGradGuard no_grad;
    variable_list res(4);
    if (!grads[0].defined()) return res;
    const Tensor q = q_.unpack(), k = k_.unpack(), v = v_.unpack(), gate = gate_.unpack(), idx = idx_.unpack(),
                 buf = buf_.unpack();
    if (buf.device() != q.device() || (size_t)buf.nbytes() != scratch_.bytes() || !buf.is_contiguous())
      throw std::runtime_error("blossom_attention: a saved-tensor hook returned another tensor than it was given");
    char *const base = static_cast<char *>(buf.data_ptr());
    c10::cuda::CUDAGuard guard(q.device());
    Tensor dout = grads[0];
    if (dout.strides() != q.strides() || dout.scalar_type() != q.scalar_type())  // the library wants q's layout
      dout = copied(dout, like(q));
    make_plain(dout);
    Tensor dq = like(q), dk = like(k), dv = like(k);
    Tensor dgate = fresh(gate.sizes(), at::kFloat, q.device());
    // The workspace is this call's own and its last user was the training forward (or an earlier
    // backward, which leaves the lists alone): the tile lists of that call are still in it.
    blossom_params p = params_;
    p.reuse_tile_lists = 1;
    const int rc = blossom_attn_bwd(
        &p, q.data_ptr(), k.data_ptr(), v.data_ptr(), gate.data_ptr<float>(),
        lens_.defined() ? lens_.data_ptr<int32_t>() : nullptr, idx.data_ptr<int32_t>(), scratch_.out_lt(base),
        scratch_.out_st(base), scratch_.lse(base), dout.data_ptr(), dq.data_ptr(), dk.data_ptr(), dv.data_ptr(),
        dgate.data_ptr<float>(), scratch_.workspace(base), scratch_.ws_bytes,
        (blossom_stream_t)c10::cuda::getCurrentCUDAStream(q.device().index()).stream());
    if (rc) throw std::runtime_error(failure("blossom_attn_bwd", rc));
    res[0] = dq;
    res[1] = dk;
    res[2] = dv;
    res[3] = gate_type_ == at::kFloat ? dgate : dgate.to(gate_type_);
    return res;
  }
};

bool read_int(PyObject *o, int32_t *out) {
  long x;
  if (PyLong_Check(o)) {
    x = PyLong_AsLong(o);
  } else {  // bool, numpy integers, floats: what int() takes
    PyObject *n = PyNumber_Long(o);
    if (!n) return false;
    x = PyLong_AsLong(n);
    Py_DECREF(n);
  }
  if (x == -1 && PyErr_Occurred()) return false;
  *out = static_cast<int32_t>(x);
  return true;
}
bool read_float(PyObject *o, float *out) {
  const double x = PyFloat_AsDouble(o);
  if (x == -1.0 && PyErr_Occurred()) return false;
  *out = static_cast<float>(x);
  return true;
}

// Raises binding.BlossomError(status, where).
PyObject *raise_blossom(int rc, const char *where) {
  PyObject *mod = PyImport_ImportModule("paper_2512_13368_b200.binding");
  PyObject *cls = mod ? PyObject_GetAttrString(mod, "BlossomError") : nullptr;
  PyObject *exc = cls ? PyObject_CallFunction(cls, "is", rc, where) : nullptr;
  if (exc) PyErr_SetObject(cls, exc);
  Py_XDECREF(exc);
  Py_XDECREF(cls);
  Py_XDECREF(mod);
  return nullptr;
}

// attention(q, k, v, gate, seq_lens, phi, block, topk, window, sm_scale, stis_mode, stis_block,
//           cmp_block, cmp_stride, per_query, gate_mode, causal, rope_theta) -> (out, idx)
// None: the arguments are not what the library can be handed (autograd.check_arguments says why).
PyObject *attention(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (n != 18) {
    PyErr_SetString(PyExc_TypeError, "attention() takes 18 arguments");
    return nullptr;
  }
  for (int i = 0; i < 4; ++i)
    if (!THPVariable_Check(a[i])) Py_RETURN_NONE;
  blossom_params p = {};
  if (!read_int(a[6], &p.block_size) || !read_int(a[7], &p.top_k) || !read_int(a[8], &p.window) ||
      !read_float(a[9], &p.sm_scale) || !read_int(a[10], &p.stis_mode) || !read_int(a[11], &p.stis_block) ||
      !read_int(a[12], &p.cmp_block) || !read_int(a[13], &p.cmp_stride) || !read_int(a[14], &p.select_mode) ||
      !read_int(a[15], &p.gate_mode) || !read_int(a[16], &p.causal) || !read_float(a[17], &p.rope_theta))
    return nullptr;
  try {
    const Tensor &q0 = THPVariable_Unpack(a[0]), &k0 = THPVariable_Unpack(a[1]), &v0 = THPVariable_Unpack(a[2]),
                 &gate0 = THPVariable_Unpack(a[3]);
    const at::ScalarType dt = q0.scalar_type();
    if (dt != at::kFloat && dt != at::kBFloat16) Py_RETURN_NONE;
    if (!q0.is_cuda() || q0.dim() != 4 || k0.dim() != 4 || k0.sizes() != v0.sizes() || k0.scalar_type() != dt ||
        v0.scalar_type() != dt || k0.device() != q0.device() || v0.device() != q0.device())
      Py_RETURN_NONE;
    const int64_t B = q0.size(0), H = q0.size(1), L = q0.size(2), D = q0.size(3), Hkv = k0.size(1);
    if (k0.size(0) != B || k0.size(2) != L || k0.size(3) != D || Hkv < 1 || H % Hkv) Py_RETURN_NONE;
    if (gate0.dim() != 2 || gate0.size(0) != H || gate0.size(1) != (p.gate_mode ? 2 * D + 1 : 2) ||
        gate0.device() != q0.device() || !at::isFloatingType(gate0.scalar_type()))
      Py_RETURN_NONE;
    Tensor lens;
    if (a[4] != Py_None) {
      if (!THPVariable_Check(a[4])) Py_RETURN_NONE;
      lens = THPVariable_Unpack(a[4]);
      if (lens.dim() != 1 || lens.size(0) != B || lens.device() != q0.device() ||
          (lens.scalar_type() != at::kInt && lens.scalar_type() != at::kLong))
        Py_RETURN_NONE;
      if (lens.scalar_type() != at::kInt || !lens.is_contiguous()) lens = lens.to(at::kInt).contiguous();
    }
    Tensor phi;
    if (a[5] != Py_None) phi = THPVariable_Unpack(a[5]);  // (checked by the caller)

    // (the tangents would be dropped without a word)
    for (const Tensor *t : {&q0, &k0, &v0, &gate0})
      if (t->_fw_grad(/*level=*/0).defined()) {
        PyErr_SetString(PyExc_NotImplementedError, "blossom_attention has no forward-mode derivative");
        return nullptr;
      }

    c10::cuda::CUDAGuard guard(q0.device());
    Tensor q = q0, k = k0, v = v0, gate = gate0;
    {
      at::NoGradGuard no_grad;
      // The library addresses every q-shaped buffer with q's strides and every k-shaped one with k's:
      // views that are not dense (a slice of a packed projection) are copied first.
      if (!(dense(q) && q.stride(3) == 1)) q = packed(q);
      if (!(dense(k) && k.stride(3) == 1 && k.strides() == v.strides())) {
        k = packed(k);
        v = packed(v);
      }
      if (Hkv == H && k.strides() != q.strides()) {
        k = copied(k, like(q));
        v = copied(v, like(q));
      }
      if (gate.scalar_type() != at::kFloat || !gate.is_contiguous()) gate = gate.to(at::kFloat).contiguous();
      for (Tensor *t : {&q, &k, &v, &gate, &lens, &phi}) make_plain(*t);
    }
    p.batch = (int32_t)B;
    p.heads = (int32_t)H;
    p.kv_heads = (int32_t)Hkv;
    p.seq_len = (int32_t)L;
    p.head_dim = (int32_t)D;
    p.dtype = dt == at::kFloat ? BLOSSOM_DTYPE_FP32 : BLOSSOM_DTYPE_BF16;
    p.stride_b = q.stride(0);
    p.stride_h = q.stride(1);
    p.stride_l = q.stride(2);
    p.kv_stride_b = k.stride(0);
    p.kv_stride_h = k.stride(1);
    p.kv_stride_l = k.stride(2);
    p.phi_logits = phi.defined() ? phi.data_ptr<float>() : nullptr;
    const size_t ws_bytes = blossom_workspace_bytes(&p);
    if (ws_bytes == 0) return raise_blossom(BLOSSOM_ERR_UNSUPPORTED, "blossom_workspace_bytes");

    const bool grad = torch::autograd::compute_requires_grad(q0, k0, v0, gate0);
    const at::Device dev = q.device();
    Scratch s;
    s.span = grad ? align256((size_t)q.numel() * q.element_size()) : 0;
    s.lse_bytes = grad ? align256((size_t)2 * B * H * L * sizeof(float)) : 0;
    s.ws_bytes = ws_bytes;
    const Tensor buf = fresh({(int64_t)s.bytes()}, at::kByte, dev);
    char *const base = static_cast<char *>(buf.data_ptr());
    const int64_t rows = p.select_mode ? L : (L + p.block_size - 1) / p.block_size;
    Tensor out = like(q), idx = fresh({B, Hkv, rows, p.top_k}, at::kInt, dev);
    const blossom_stream_t st = (blossom_stream_t)c10::cuda::getCurrentCUDAStream(dev.index()).stream();
    // Every address is taken before the interpreter is let go: a tensor without memory of its own (a batched
    // one inside vmap) throws here, and an exception must not leave the block below.
    const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
    const float *gp = gate.data_ptr<float>();
    const int32_t *np = lens.defined() ? lens.data_ptr<int32_t>() : nullptr;
    int32_t *ip = idx.data_ptr<int32_t>();
    void *op = out.data_ptr(), *lp = grad ? s.out_lt(base) : nullptr, *sp = grad ? s.out_st(base) : nullptr,
         *wp = s.workspace(base);
    float *ep = grad ? s.lse(base) : nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS;
    rc = blossom_attn_fwd(&p, qp, kp, vp, gp, np, ip, 0, op, lp, sp, ep, wp, ws_bytes, st);
    Py_END_ALLOW_THREADS;
    if (rc) return raise_blossom(rc, "blossom_attn_fwd");
    if (grad) {
      auto node = std::shared_ptr<BlossomAttentionBackward>(new BlossomAttentionBackward(), torch::autograd::deleteNode);
      node->set_next_edges(torch::autograd::collect_next_edges(q0, k0, v0, gate0));
      node->q_ = SavedVariable(q, false);
      node->k_ = SavedVariable(k, false);
      node->v_ = SavedVariable(v, false);
      node->gate_ = SavedVariable(gate.is_same(gate0) ? gate : gate.detach(), false);
      node->idx_ = SavedVariable(idx, false);
      node->buf_ = SavedVariable(buf, false);
      node->lens_ = lens;
      node->phi_ = phi;
      node->scratch_ = s;
      node->params_ = p;
      node->gate_type_ = gate0.scalar_type();
      torch::autograd::set_history(out, node);
    }
    PyObject *res = PyTuple_New(2);
    if (!res) return nullptr;
    PyTuple_SET_ITEM(res, 0, THPVariable_Wrap(std::move(out)));
    PyTuple_SET_ITEM(res, 1, THPVariable_Wrap(std::move(idx)));
    return res;
  } catch (const std::exception &e) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// dense(tensor) -> bool, like(tensor) -> tensor: the two rules above, for the host-side tests
PyObject *py_dense(PyObject *, PyObject *t) {
  if (!THPVariable_Check(t)) return PyErr_Format(PyExc_TypeError, "dense() takes a tensor");
  return PyBool_FromLong(dense(THPVariable_Unpack(t)));
}
PyObject *py_like(PyObject *, PyObject *t) {
  if (!THPVariable_Check(t)) return PyErr_Format(PyExc_TypeError, "like() takes a tensor");
  try {
    return THPVariable_Wrap(like(THPVariable_Unpack(t)));
  } catch (const std::exception &e) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {
    {"dense", py_dense, METH_O, nullptr},
    {"like", py_like, METH_O, nullptr},
    {"attention", (PyCFunction)(void (*)(void))attention, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_front", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__front(void) { return PyModule_Create(&module); }
