// _marshal: what binding.py does per call, in native code - tensor and shape arguments to pointers, outputs from
// torch's allocator, the current stream - for the entry points that a decode or prefill loop calls per token.  No
// arithmetic and no CUDA call of its own: it calls the library's entry points, whose addresses binding.py hands over
// (so there is one library, whichever file it was loaded from).
//
// Why: a decode step is 16 us of GPU time and two calls, and in Python a call cost more than that.  Measured on the
// B200 machine's host (us per call, the launch itself 2.4): slicemoe_route_topk 17.9 in Python (three torch.empty at 2.4,
// torch.cuda.current_stream 3.2, ctypes conversions), slicemoe_layer with a given y 9.5.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstring>

#include "slicemoe.h"

namespace {

struct Entry {
  decltype(&slicemoe_pack) pack;
  decltype(&slicemoe_plane_bytes) plane_bytes;
  decltype(&slicemoe_meta_count) meta_count;
  decltype(&slicemoe_route_topk) route_topk;
  decltype(&slicemoe_expert_ffn) expert_ffn;
  decltype(&slicemoe_layer_flags) layer_flags;
  decltype(&slicemoe_layer_routed) layer_routed;
  decltype(&slicemoe_layer_static) layer_static;
  decltype(&slicemoe_decode_step_host) decode_step_host;
  decltype(&slicemoe_prefill_layer) prefill_layer;
  decltype(&slicemoe_dbsc_assign) dbsc_assign;
} lib;
PyObject* error_type = nullptr;  // binding.SliceMoEError(code, where)
PyObject* s_data_ptr = nullptr;
PyObject* s_cuda_stream = nullptr;

struct Failed {};  // a Python error is set

// A tensor's (or any data_ptr()-bearing object's) address; None is a null pointer.
void* address(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
  PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) throw Failed();
  void* p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (!p && PyErr_Occurred()) throw Failed();
  return p;
}
const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s: a tensor is wanted, got %s", name, Py_TYPE(o)->tp_name);
    throw Failed();
  }
  return THPVariable_Unpack(o);
}
void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* v = PyObject_GetAttr(o, s_cuda_stream);
  if (!v) throw Failed();
  void* p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (!p && PyErr_Occurred()) throw Failed();
  return p;
}
int64_t integer(PyObject* o) {
  PyObject* idx = PyNumber_Index(o);
  if (!idx) throw Failed();
  const int64_t v = PyLong_AsLongLong(idx);
  Py_DECREF(idx);
  if (v == -1 && PyErr_Occurred()) throw Failed();
  return v;
}
// ctypes takes the low 32 bits of an int argument
int integer32(PyObject* o) { return (int)(uint32_t)(uint64_t)integer(o); }
float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Failed();
  return (float)v;
}
int truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Failed();
  return v;
}
// The ctypes Structure binding.Shape: its bytes are the struct.
struct ShapeArg {
  Py_buffer b;
  explicit ShapeArg(PyObject* o) {
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw Failed();
    if (b.len != (Py_ssize_t)sizeof(slicemoe_shape)) {
      PyBuffer_Release(&b);
      PyErr_SetString(PyExc_TypeError, "shape: a binding.Shape is wanted");
      throw Failed();
    }
  }
  ~ShapeArg() { PyBuffer_Release(&b); }
  ShapeArg(const ShapeArg&) = delete;
  const slicemoe_shape* get() const { return static_cast<const slicemoe_shape*>(b.buf); }
};
at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type, at::Device dev) {
  if (dev.is_cuda()) return at::Tensor(at::detail::empty_cuda(sizes, type, dev, std::nullopt));
  return at::empty(sizes, at::TensorOptions().dtype(type).device(dev));
}
// Several outputs of one call on one device.  Each has a storage of its own: torch.save refuses tensors of different types in
// one, and one that is kept would keep them all.  They are what empty_cuda makes, with the device looked at once for all.
// (A routing call takes the host 4.2 us with one allocation for its three lists, 5.1 with three calls of empty_cuda, 4.85 so.)
class Outputs {
 public:
  explicit Outputs(at::Device dev) : dev_(dev) {
    if (dev.is_cuda()) guard_.set_device(dev);
  }
  at::Tensor operator()(at::IntArrayRef sizes, at::ScalarType type) const {
    size_t n = 1;
    for (const int64_t s : sizes) {
      if (s < 0) return empty(sizes, type, dev_);  // which says what is wrong
      n *= (size_t)s;
    }
    if (!dev_.is_cuda()) return empty(sizes, type, dev_);
    c10::Allocator* from = c10::cuda::CUDACachingAllocator::get();
    const size_t bytes = n * c10::elementSize(type);
    at::Tensor t = at::detail::make_tensor<c10::TensorImpl>(
        c10::make_intrusive<c10::StorageImpl>(c10::StorageImpl::use_byte_size_t(), bytes, from->allocate(bytes), from, /*resizable=*/true),
        c10::DispatchKeySet(c10::DispatchKey::CUDA), c10::scalarTypeToTypeMeta(type));
    t.unsafeGetTensorImpl()->set_sizes_contiguous(sizes);
    return t;
  }

 private:
  at::Device dev_;
  c10::cuda::OptionalCUDAGuard guard_;
};
PyObject* wrap(const at::Tensor& t) {
  PyObject* o = THPVariable_Wrap(t);
  if (!o) throw Failed();
  return o;
}
PyObject* wrap_or_none(const at::Tensor& t) {
  if (t.defined()) return wrap(t);
  return Py_NewRef(Py_None);
}
PyObject* tuple_of(std::initializer_list<const at::Tensor*> ts) {
  PyObject* r = PyTuple_New((Py_ssize_t)ts.size());
  if (!r) throw Failed();
  Py_ssize_t i = 0;
  for (const at::Tensor* t : ts) {
    PyObject* o = nullptr;
    try {
      o = wrap_or_none(*t);
    } catch (...) {
      Py_DECREF(r);
      throw;
    }
    PyTuple_SET_ITEM(r, i++, o);
  }
  return r;
}
void check(int rc, const char* where) {
  if (rc == SLICEMOE_OK) return;
  PyObject* e = PyObject_CallFunction(error_type, "is", rc, where);
  if (e) {
    PyErr_SetObject(error_type, e);
    Py_DECREF(e);
  }
  throw Failed();
}
// Calls the library without the interpreter lock, as ctypes does: a launch may wait for room in the stream's queue.
template <class F>
int unlocked(F&& f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS rc = f();
  Py_END_ALLOW_THREADS return rc;
}
void want(Py_ssize_t n, Py_ssize_t k) {
  if (n == k) return;
  PyErr_Format(PyExc_TypeError, "%zd arguments are wanted, got %zd", k, n);
  throw Failed();
}
template <class F>
PyObject* guarded(F&& f) {
  try {
    return f();
  } catch (const Failed&) {
  } catch (const std::exception&) {  // torch's own kinds stay what they are: out of memory, an index out of range
    torch::translate_exception_to_python(std::current_exception());
  }
  return nullptr;
}
// y, or a new float32 [T, hidden] on x's device
at::Tensor output(PyObject* y, const at::Tensor& x, const slicemoe_shape* s, PyObject** given) {
  if (y != Py_None) {
    *given = y;
    return at::Tensor();
  }
  *given = nullptr;
  return Outputs(x.device())({x.size(0), s->hidden}, at::kFloat);
}

#define SM_ARGS PyObject *, PyObject *const *a, Py_ssize_t n

PyObject* py_setup(SM_ARGS) {  // (error type, dict name -> address)
  return guarded([&]() -> PyObject* {
    want(n, 2);
    auto load = [&](const char* name, auto& fn) {
      PyObject* v = PyDict_GetItemString(a[1], name);
      if (!v) {
        PyErr_Format(PyExc_KeyError, "%s", name);
        throw Failed();
      }
      fn = reinterpret_cast<std::decay_t<decltype(fn)>>(PyLong_AsVoidPtr(v));
    };
    load("slicemoe_pack", lib.pack);
    load("slicemoe_plane_bytes", lib.plane_bytes);
    load("slicemoe_meta_count", lib.meta_count);
    load("slicemoe_route_topk", lib.route_topk);
    load("slicemoe_expert_ffn", lib.expert_ffn);
    load("slicemoe_layer_flags", lib.layer_flags);
    load("slicemoe_layer_routed", lib.layer_routed);
    load("slicemoe_layer_static", lib.layer_static);
    load("slicemoe_decode_step_host", lib.decode_step_host);
    load("slicemoe_prefill_layer", lib.prefill_layer);
    load("slicemoe_dbsc_assign", lib.dbsc_assign);
    Py_XSETREF(error_type, Py_NewRef(a[0]));
    Py_RETURN_NONE;
  });
}

PyObject* py_pack(SM_ARGS) {  // PackedMat, W, group, b_high, b_low, stream, out -> out, or a new PackedMat
  return guarded([&]() -> PyObject* {
    want(n, 7);
    if (!THPVariable_Check(a[1])) {
      PyErr_Format(PyExc_AttributeError, "W: a tensor is wanted, got %s", Py_TYPE(a[1])->tp_name);
      throw Failed();
    }
    const at::Tensor& W = THPVariable_Unpack(a[1]);
    if (!(W.is_cuda() && W.scalar_type() == at::kFloat && W.is_contiguous() && W.dim() == 2)) {
      PyErr_SetString(PyExc_AssertionError, "W: a contiguous CUDA float32 matrix is wanted");
      throw Failed();
    }
    const int N = (int)W.size(0), K = (int)W.size(1), group = integer32(a[2]), bh = integer32(a[3]), bl = integer32(a[4]);
    void* st = stream_of(a[5]);
    auto call = [&](void* msb, void* lsb, void* scale, void* zp) {
      check(unlocked([&] {
              return lib.pack(static_cast<const float*>(W.data_ptr()), N, K, group, bh, bl, msb, lsb, static_cast<uint16_t*>(scale),
                              static_cast<uint8_t*>(zp), st);
            }),
            "slicemoe_pack");
    };
    if (a[6] != Py_None) {
      void* p[4];
      const char* names[4] = {"msb", "lsb", "scale", "zp"};
      for (int i = 0; i < 4; ++i) {
        PyObject* o = PyObject_GetAttrString(a[6], names[i]);
        if (!o) throw Failed();
        const at::Tensor* t = THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr;
        p[i] = t ? t->data_ptr() : o == Py_None ? nullptr : address(o);
        Py_DECREF(o);
      }
      call(p[0], p[1], p[2], p[3]);
      return Py_NewRef(a[6]);
    }
    const int64_t nb = std::max<int64_t>((int64_t)lib.plane_bytes(N, K), 1);
    const int64_t nm = std::max<int64_t>(group > 0 ? (int64_t)lib.meta_count(N, K, group) : 1, 1);
    const at::Device dev = W.device();
    at::Tensor msb, lsb, scale, zp;
    {
      const Outputs out(dev);
      msb = out({nb}, at::kByte), lsb = out({nb}, at::kByte), scale = out({nm}, at::kShort), zp = out({nm}, at::kByte);
    }
    call(msb.data_ptr(), lsb.data_ptr(), scale.data_ptr(), zp.data_ptr());
    PyObject* args[7] = {};
    PyObject* r = nullptr;
    args[0] = PyLong_FromLong(N);
    args[1] = PyLong_FromLong(K);
    args[2] = Py_NewRef(a[2]);
    const at::Tensor* t[4] = {&msb, &lsb, &scale, &zp};
    bool ok = args[0] && args[1];
    for (int i = 0; i < 4 && ok; ++i) ok = (args[3 + i] = THPVariable_Wrap(*t[i])) != nullptr;
    if (ok) r = PyObject_Vectorcall(a[0], args, 7, nullptr);
    for (PyObject* o : args) Py_XDECREF(o);
    if (!r) throw Failed();
    return r;
  });
}

PyObject* py_route_topk(SM_ARGS) {  // logits, k, bias, renorm, tau, rank_high, want_prec, stream -> (ids, weights, prec)
  return guarded([&]() -> PyObject* {
    want(n, 8);
    const at::Tensor& logits = tensor(a[0], "logits");
    if (!(logits.is_cuda() && logits.scalar_type() == at::kFloat && logits.is_contiguous() && logits.dim() == 2)) {
      PyErr_SetString(PyExc_AssertionError, "logits: a contiguous CUDA float32 matrix is wanted");
      throw Failed();
    }
    const int64_t T = logits.size(0), E = logits.size(1);
    const int k = integer32(a[1]), kk = std::max(k, 1);
    const at::Device dev = logits.device();
    at::Tensor ids, w, prec;
    const bool want_prec = truth(a[6]);
    {
      const Outputs out(dev);
      ids = out({T, kk}, at::kInt), w = out({T, kk}, at::kFloat);
      if (want_prec) prec = out({T, kk}, at::kByte);
    }
    const float* bias = static_cast<const float*>(address(a[2]));
    const int renorm = truth(a[3]), rank_high = integer32(a[5]);
    const float tau = real(a[4]);
    void* st = stream_of(a[7]);
    check(unlocked([&] {
            return lib.route_topk(static_cast<const float*>(logits.data_ptr()), (int)T, (int)E, k, bias, renorm, tau, rank_high,
                                  static_cast<int32_t*>(ids.data_ptr()), static_cast<float*>(w.data_ptr()),
                                  prec.defined() ? static_cast<uint8_t*>(prec.data_ptr()) : nullptr, st);
          }),
          "slicemoe_route_topk");
    return tuple_of({&ids, &w, &prec});
  });
}

// A contiguous buffer of `size`-byte items with one of the format characters in `kinds`; nothing is raised if it is not.
bool plain_buffer(PyObject* o, Py_buffer* b, Py_ssize_t size, const char* kinds) {
  if (PyObject_GetBuffer(o, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
    PyErr_Clear();
    return false;
  }
  const char* f = b->format ? b->format : "B";
  if (*f == '<' || *f == '=' || *f == '@') ++f;
  if (b->itemsize == size && *f && strchr(kinds, *f) && !f[1]) return true;
  PyBuffer_Release(b);
  return false;
}
// handle, step, layer, ids (int32), prec_req (uint8), prec_out (uint8, written); returns False if the buffers are of other types
PyObject* py_dbsc_assign(SM_ARGS) {
  return guarded([&]() -> PyObject* {
    want(n, 6);
    auto* c = a[0] == Py_None ? nullptr : static_cast<slicemoe_dbsc*>(PyLong_AsVoidPtr(a[0]));
    if (PyErr_Occurred()) throw Failed();
    const int step = integer32(a[1]), layer = integer32(a[2]);
    Py_buffer ids, req, out;
    if (!plain_buffer(a[3], &ids, 4, "il")) Py_RETURN_FALSE;
    int rc = 1;
    if (plain_buffer(a[4], &req, 1, "B")) {
      if (plain_buffer(a[5], &out, 1, "B")) {
        if (!out.readonly && req.len >= ids.len / 4 && out.len >= ids.len / 4)
          rc = unlocked([&] {
            return lib.dbsc_assign(c, step, layer, static_cast<const int32_t*>(ids.buf), static_cast<const uint8_t*>(req.buf),
                                   (int)(ids.len / 4), static_cast<uint8_t*>(out.buf));
          });
        PyBuffer_Release(&out);
      }
      PyBuffer_Release(&req);
    }
    PyBuffer_Release(&ids);
    if (rc == 1) Py_RETURN_FALSE;
    check(rc, "slicemoe_dbsc_assign");
    Py_RETURN_TRUE;
  });
}

PyObject* py_expert_ffn(SM_ARGS) {  // shape, experts, x, ids, prec, weights, ws, y, stream -> y
  return guarded([&]() -> PyObject* {
    want(n, 9);
    const ShapeArg s(a[0]);
    const at::Tensor &x = tensor(a[2], "x"), &ws = tensor(a[6], "ws");
    PyObject* given;
    const at::Tensor y = output(a[7], x, s.get(), &given);
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* ids = static_cast<const int32_t*>(address(a[3]));
    const auto* prec = static_cast<const uint8_t*>(address(a[4]));
    const auto* w = static_cast<const float*>(address(a[5]));
    float* yp = static_cast<float*>(given ? address(given) : y.data_ptr());
    void* st = stream_of(a[8]);
    check(unlocked([&] {
            return lib.expert_ffn(s.get(), ex, x.data_ptr(), (int)x.size(0), ids, prec, w, yp, ws.data_ptr(),
                                  (size_t)ws.numel(), st);
          }),
          "slicemoe_expert_ffn");
    return given ? Py_NewRef(given) : wrap(y);
  });
}

PyObject* py_layer(SM_ARGS) {  // shape, experts, shared, gate_vec, x, ids, prec, weights, ws, y, stream, flags -> y
  return guarded([&]() -> PyObject* {
    want(n, 12);
    const ShapeArg s(a[0]);
    const at::Tensor &x = tensor(a[4], "x"), &ws = tensor(a[8], "ws");
    PyObject* given;
    const at::Tensor y = output(a[9], x, s.get(), &given);
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* sh = static_cast<const slicemoe_expert*>(address(a[2]));
    const auto* gv = static_cast<const float*>(address(a[3]));
    const auto* ids = static_cast<const int32_t*>(address(a[5]));
    const auto* prec = static_cast<const uint8_t*>(address(a[6]));
    const auto* w = static_cast<const float*>(address(a[7]));
    float* yp = static_cast<float*>(given ? address(given) : y.data_ptr());
    void* st = stream_of(a[10]);
    const unsigned flags = (unsigned)integer32(a[11]);
    check(unlocked([&] {
            return lib.layer_flags(s.get(), ex, sh, gv, x.data_ptr(), (int)x.size(0), ids, prec, w, yp, ws.data_ptr(),
                                   (size_t)ws.numel(), flags, st);
          }),
          flags ? "slicemoe_layer_flags" : "slicemoe_layer");
    return given ? Py_NewRef(given) : wrap(y);
  });
}

PyObject* py_layer_static(SM_ARGS) {  // shape, experts, shared, gate_vec, x, ids, prec, weights, y, stream -> y
  return guarded([&]() -> PyObject* {
    want(n, 10);
    const ShapeArg s(a[0]);
    const at::Tensor& x = tensor(a[4], "x");
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* sh = static_cast<const slicemoe_expert*>(address(a[2]));
    const auto* gv = static_cast<const float*>(address(a[3]));
    const auto* ids = static_cast<const int32_t*>(address(a[5]));
    const auto* prec = static_cast<const uint8_t*>(address(a[6]));
    const auto* w = static_cast<const float*>(address(a[7]));
    float* yp = static_cast<float*>(address(a[8]));
    void* st = stream_of(a[9]);
    check(unlocked([&] { return lib.layer_static(s.get(), ex, sh, gv, x.data_ptr(), (int)x.size(0), ids, prec, w, yp, st); }),
          "slicemoe_layer_static");
    return Py_NewRef(a[8]);
  });
}

// shape, experts, shared, gate_vec, x, logits, ws, bias, renorm, tau, rank_high, y, want_lists, stream -> (y, ids, prec, weights)
PyObject* py_layer_routed(SM_ARGS) {
  return guarded([&]() -> PyObject* {
    want(n, 14);
    const ShapeArg s(a[0]);
    const at::Tensor &x = tensor(a[4], "x"), &ws = tensor(a[6], "ws");
    PyObject* given;
    const at::Tensor y = output(a[11], x, s.get(), &given);
    const int64_t T = x.size(0), k = s.get()->top_k;
    at::Tensor ids, prec, w;
    if (truth(a[12])) {
      const Outputs out(x.device());
      ids = out({T, k}, at::kInt), w = out({T, k}, at::kFloat), prec = out({T, k}, at::kByte);
    }
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* sh = static_cast<const slicemoe_expert*>(address(a[2]));
    const auto* gv = static_cast<const float*>(address(a[3]));
    const auto* logits = static_cast<const float*>(address(a[5]));
    const auto* bias = static_cast<const float*>(address(a[7]));
    const int renorm = truth(a[8]), rank_high = integer32(a[10]);
    const float tau = real(a[9]);
    float* yp = static_cast<float*>(given ? address(given) : y.data_ptr());
    void* st = stream_of(a[13]);
    auto ptr = [](const at::Tensor& t) -> void* { return t.defined() ? t.data_ptr() : nullptr; };
    check(unlocked([&] {
            return lib.layer_routed(s.get(), ex, sh, gv, x.data_ptr(), (int)T, logits, bias, renorm, tau, rank_high,
                                    static_cast<int32_t*>(ptr(ids)), static_cast<uint8_t*>(ptr(prec)),
                                    static_cast<float*>(ptr(w)), yp, ws.data_ptr(), (size_t)ws.numel(), st);
          }),
          "slicemoe_layer_routed");
    if (!given) return tuple_of({&y, &ids, &prec, &w});
    PyObject* r = tuple_of({&y, &ids, &prec, &w});  // y undefined: a place holder
    PyTuple_SetItem(r, 0, Py_NewRef(given));
    return r;
  });
}

// shape, experts, shared, gate_vec, x_host, logits_host, y_host, ws, bias, renorm, tau, rank_high, stream -> y_host
PyObject* py_decode_step_host(SM_ARGS) {
  return guarded([&]() -> PyObject* {
    want(n, 13);
    const ShapeArg s(a[0]);
    const at::Tensor& ws = tensor(a[7], "ws");
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* sh = static_cast<const slicemoe_expert*>(address(a[2]));
    const auto* gv = static_cast<const float*>(address(a[3]));
    const void* x = address(a[4]);
    const auto* logits = static_cast<const float*>(address(a[5]));
    float* y = static_cast<float*>(address(a[6]));
    const auto* bias = static_cast<const float*>(address(a[8]));
    const int renorm = truth(a[9]), rank_high = integer32(a[11]);
    const float tau = real(a[10]);
    void* st = stream_of(a[12]);
    check(unlocked([&] {
            return lib.decode_step_host(s.get(), ex, sh, gv, x, logits, bias, renorm, tau, rank_high, y, ws.data_ptr(),
                                        (size_t)ws.numel(), st);
          }),
          "slicemoe_decode_step_host");
    return Py_NewRef(a[6]);
  });
}

// shape, experts, shared, gate_vec, x, ids, weights, expert_prec, ws, y, status, stream -> (y, status)
PyObject* py_prefill_layer(SM_ARGS) {
  return guarded([&]() -> PyObject* {
    want(n, 12);
    const ShapeArg s(a[0]);
    const at::Tensor &x = tensor(a[4], "x"), &ws = tensor(a[8], "ws");
    PyObject* given;
    const at::Tensor y = output(a[9], x, s.get(), &given);
    at::Tensor status;
    if (a[10] == Py_None) status = Outputs(x.device())({1}, at::kInt);
    const auto* ex = static_cast<const slicemoe_expert*>(address(a[1]));
    const auto* sh = static_cast<const slicemoe_expert*>(address(a[2]));
    const auto* gv = static_cast<const float*>(address(a[3]));
    const auto* ids = static_cast<const int32_t*>(address(a[5]));
    const auto* w = static_cast<const float*>(address(a[6]));
    const auto* prec = static_cast<const uint8_t*>(address(a[7]));
    float* yp = static_cast<float*>(given ? address(given) : y.data_ptr());
    int* sp = static_cast<int*>(status.defined() ? status.data_ptr() : address(a[10]));
    void* st = stream_of(a[11]);
    check(unlocked([&] {
            return lib.prefill_layer(s.get(), ex, sh, gv, x.data_ptr(), (int)x.size(0), ids, w, prec, yp, ws.data_ptr(),
                                     (size_t)ws.numel(), sp, st);
          }),
          "slicemoe_prefill_layer");
    PyObject* r = tuple_of({&y, &status});
    if (given) PyTuple_SetItem(r, 0, Py_NewRef(given));
    if (!status.defined()) PyTuple_SetItem(r, 1, Py_NewRef(a[10]));
    return r;
  });
}

#define SM_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SM_METHOD(setup),        SM_METHOD(pack),         SM_METHOD(route_topk),
                         SM_METHOD(expert_ffn),   SM_METHOD(layer),            SM_METHOD(layer_static),
                         SM_METHOD(layer_routed), SM_METHOD(decode_step_host), SM_METHOD(prefill_layer),
                         SM_METHOD(dbsc_assign),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_cuda_stream) return nullptr;
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_for", SLICEMOE_BUILT_FOR) < 0) Py_CLEAR(m);
  return m;
}
