// Argument marshalling of the Python binding in native code: each function takes the torch tensors of one library call,
// checks them, takes the current CUDA stream and calls the C entry point of include/tweo.h with the GIL released.
// The same checks in Python through ctypes cost 7 to 12 microseconds a call (attribute look-ups, conversions of up to
// seventeen arguments, the stream object), more than the kernels of a few-token call take.  Nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <string>
#include <vector>

#include "tweo.h"

namespace {

PyObject* g_tweo_error = nullptr;   // binding.TweoError, given by set_error()

struct PyFailure {};   // a Python exception is set

[[noreturn]] void fail(PyObject* type, const std::string& text) {
  PyErr_SetString(type, text.c_str());
  throw PyFailure{};
}

enum Kind : unsigned { kBf16 = 1, kF32 = 2, kU8 = 4, kI8 = 8, kCodes = 16, kAny = 32 };   // kCodes: uint8 or an FP8 type

const char* kind_text(unsigned k) {
  switch (k) {
    case kBf16: return "torch.bfloat16";
    case kF32: return "torch.float32";
    case kU8: return "torch.uint8";
    case kI8: return "torch.int8";
    default: return "(torch.uint8, torch.float8_e4m3fn, torch.float8_e5m2)";
  }
}

unsigned kind_of(at::ScalarType t) {
  switch (t) {
    case at::kBFloat16: return kBf16;
    case at::kFloat: return kF32;
    case at::kByte: return kU8 | kCodes;
    case at::kChar: return kI8;
    case at::kFloat8_e4m3fn:
    case at::kFloat8_e5m2: return kCodes;
    default: return 0;
  }
}

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o) || !THPVariable_Unpack(o).is_cuda())
    fail(PyExc_TypeError, std::string(name) + " must be a CUDA tensor (no CPU fallback exists)");
  return THPVariable_Unpack(o);
}

void check_kind(const at::Tensor& t, unsigned want, const char* name) {
  if (want != kAny && !(kind_of(t.scalar_type()) & want))
    fail(PyExc_TypeError, std::string(name) + " has dtype " + c10::toString(t.scalar_type()) + ", expected " + kind_text(want));
}

void* dev(PyObject* o, unsigned want, const char* name) {
  const at::Tensor& t = tensor(o, name);
  check_kind(t, want, name);
  return t.data_ptr();
}
template <typename T>
T* dev(PyObject* o, unsigned want, const char* name) { return static_cast<T*>(dev(o, want, name)); }
float* f32(PyObject* o, const char* name = "tensor") { return dev<float>(o, kF32, name); }
float* f32_or_null(PyObject* o, const char* name = "tensor") { return o == Py_None ? nullptr : f32(o, name); }

// A 2-D tensor whose rows are contiguous: pointer, shape and row pitch in elements.
struct Mat {
  void* p;
  int64_t rows, cols, ld;
};
Mat mat(PyObject* o, unsigned want, const char* name) {
  const at::Tensor& t = tensor(o, name);
  check_kind(t, want, name);
  if (t.dim() != 2 || t.stride(1) != 1) fail(PyExc_ValueError, std::string(name) + " must be 2-D with contiguous rows");
  return Mat{t.data_ptr(), t.size(0), t.size(1), t.stride(0)};
}

struct Ws {
  void* p;
  size_t n;
};
// any: storage of any type, of which a byte per element is used (the calls whose workspace is no option).
Ws workspace(PyObject* o, bool any = false) {
  if (o == Py_None) return Ws{nullptr, 0};
  const at::Tensor& t = tensor(o, "ws");
  if (!any) check_kind(t, kU8, "ws");
  return Ws{t.data_ptr(), (size_t)t.numel()};
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

int32_t i32(PyObject* o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyFailure{};
  if (v < INT32_MIN || v > INT32_MAX) fail(PyExc_OverflowError, "integer out of range");
  return (int32_t)v;
}
float flt(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyFailure{};
  return (float)v;
}
bool flag(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw PyFailure{};
  return v != 0;
}

// Owns a reference.
struct Ref {
  PyObject* o;
  explicit Ref(PyObject* p) : o(p) {
    if (!p) throw PyFailure{};
  }
  Ref(const Ref&) = delete;
  Ref& operator=(const Ref&) = delete;
  ~Ref() { Py_XDECREF(o); }
};

PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

template <typename F>
auto without_gil(F&& f) {
  struct Save {
    PyThreadState* s = PyEval_SaveThread();
    ~Save() { PyEval_RestoreThread(s); }
  } save;
  return f();
}

at::Tensor empty(at::IntArrayRef shape, at::ScalarType type, const at::Device& device) {
  return without_gil([&] { return at::empty(shape, at::TensorOptions().dtype(type).device(device)); });
}

// Calls the entry point with the GIL released; a status other than TWEO_OK becomes TweoError(status, where).
template <typename F>
void call(const char* where, F&& f) {
  const tweo_status_t s = without_gil(f);
  if (s == TWEO_OK) return;
  Ref err(PyObject_CallFunction(g_tweo_error, "is", (int)s, where));
  PyErr_SetObject(g_tweo_error, err.o);
  throw PyFailure{};
}

// The body of one Python-callable function: argument count, and C++ exceptions to Python ones.
template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& f) {
  try {
    if (n != want) fail(PyExc_TypeError, "wrong number of arguments");
    return f();
  } catch (const PyFailure&) {
    return nullptr;
  } catch (...) {   // as torch's own functions report it: torch.OutOfMemoryError where an output does not fit, and so on
    torch::translate_exception_to_python(std::current_exception());
    return nullptr;
  }
}
#define FN(name, count, ...)                                                   \
  PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n) {                \
    return guarded(n, count, [&]() -> PyObject* { __VA_ARGS__ });              \
  }

// Names of attributes and dictionary keys, interned once at import.
struct Names {
  PyObject *q, *scale, *scale_inv, *amax, *sat_count, *fmt;
  PyObject *product, *fmt_x, *fmt_w, *fmt_dy, *xq, *wq, *dyq, *sx_inv, *sw_inv, *sdy_inv, *out, *out_amax, *out_q, *q_fmt, *q_scale, *get;
} N;

struct Epi {
  tweo_epilogue_t e{};
  const tweo_epilogue_t* p = nullptr;
  void fill(PyObject* amax, PyObject* q, PyObject* q_fmt, PyObject* q_scale) {
    if (amax == Py_None && q == Py_None) return;
    if (amax != Py_None) e.out_amax = f32(amax, "out_amax");
    if (q != Py_None) {
      const Mat m = mat(q, kCodes, "out_q");
      e.out_q = (uint8_t*)m.p;
      e.ldq = m.ld;
      e.q_fmt = i32(q_fmt);
      e.q_scale = f32(q_scale, "q_scale");
    }
    p = &e;
  }
};

const at::Tensor& contiguous_bf16(PyObject* o, const char* name) {
  const at::Tensor& t = tensor(o, name);
  check_kind(t, kBf16, name);
  if (!t.is_contiguous()) fail(PyExc_ValueError, std::string(name) + " must be contiguous");
  return t;
}

// What a Quantized record holds, for the cast of x.  typed: the outputs must have the types the cast writes (a batch); a single
// cast writes into the memory of any CUDA tensors, bytes of int8 storage for instance.
void fill_desc(tweo_quant_desc_t& d, PyObject* x, PyObject* out, int32_t fmt, int32_t mode, bool typed) {
  const at::Tensor& t = contiguous_bf16(x, "x");
  Ref scale(PyObject_GetAttr(out, N.scale)), inv(PyObject_GetAttr(out, N.scale_inv)), amax(PyObject_GetAttr(out, N.amax)),
      q(PyObject_GetAttr(out, N.q)), sat(PyObject_GetAttr(out, N.sat_count));
  d.x = (const uint16_t*)t.data_ptr();
  d.n = t.numel();
  d.fmt = fmt;
  d.mode = mode;
  d.scale = f32(scale.o, "scale");
  d.scale_inv = dev<float>(inv.o, typed ? kF32 : kAny, "scale_inv");
  d.amax = dev<float>(amax.o, typed ? kF32 : kAny, "amax");
  d.q = dev<uint8_t>(q.o, typed ? kCodes : kAny, "q");
  d.sat_count = sat.o == Py_None ? nullptr : (uint32_t*)tensor(sat.o, "sat_count").data_ptr();
}

// quantize(x, out, fmt, mode, ws)
FN(quantize, 5, {
  tweo_quant_desc_t d;
  fill_desc(d, a[0], a[1], i32(a[2]), i32(a[3]), false);
  const Ws w = workspace(a[4]);
  void* st = stream();
  call("tweo_quantize_per_tensor", [&] {
    return tweo_quantize_per_tensor(d.x, d.n, d.fmt, d.mode, d.scale, d.scale_inv, d.amax, d.q, d.sat_count, w.p, w.n, st);
  });
  Py_RETURN_NONE;
})

// The casts of a batch, at least `least` of them.
struct Casts {
  Ref xs, outs, modes;
  Py_ssize_t count;
  Casts(PyObject* xs_, PyObject* outs_, PyObject* modes_, tweo_quant_desc_t* d, Py_ssize_t least)
      : xs(PySequence_Fast(xs_, "xs must be a sequence")), outs(PySequence_Fast(outs_, "outs must be a sequence")),
        modes(modes_ == Py_None ? Py_NewRef(Py_None) : PySequence_Fast(modes_, "modes must be a sequence")),
        count(PySequence_Fast_GET_SIZE(xs.o)) {
    if (count < least || count > TWEO_MAX_QUANT_BATCH || PySequence_Fast_GET_SIZE(outs.o) != count)
      fail(PyExc_ValueError, "need 1..MAX_QUANT_BATCH tensors with one output record each");
    if (modes.o != Py_None && PySequence_Fast_GET_SIZE(modes.o) < count) fail(PyExc_IndexError, "list index out of range");
    for (Py_ssize_t i = 0; i < count; ++i) {
      PyObject* o = PySequence_Fast_GET_ITEM(outs.o, i);
      Ref fmt(PyObject_GetAttr(o, N.fmt));
      fill_desc(d[i], PySequence_Fast_GET_ITEM(xs.o, i), o, i32(fmt.o),
                modes.o == Py_None ? TWEO_SCALE_CURRENT : i32(PySequence_Fast_GET_ITEM(modes.o, i)), true);
    }
  }
};

// quantize_batch(xs, outs, modes or None, ws)
FN(quantize_batch, 4, {
  tweo_quant_desc_t d[TWEO_MAX_QUANT_BATCH];
  const Casts casts(a[0], a[1], a[2], d, 1);
  const Ws w = workspace(a[3], true);
  void* st = stream();
  call("tweo_quantize_per_tensor_batch", [&] { return tweo_quantize_per_tensor_batch(d, (int32_t)casts.count, w.p, w.n, st); });
  Py_RETURN_NONE;
})

void same(int64_t x, int64_t y, const char* text) {
  if (x != y) fail(PyExc_ValueError, text);
}

// The output tensor of a product: the given one, or a new [rows, cols].
struct Out {
  PyObject* o;
  Mat m;
  Out(PyObject* given, int64_t rows, int64_t cols, const at::Device& device, const char* name, at::ScalarType type = at::kBFloat16) {
    o = given == Py_None ? wrap(empty({rows, cols}, type, device)) : Py_NewRef(given);
    if (!o) throw PyFailure{};
    try {
      m = mat(o, kind_of(type), name);
    } catch (...) {
      Py_DECREF(o);
      throw;
    }
  }
  Out(const Out&) = delete;
  Out& operator=(const Out&) = delete;
  ~Out() { Py_XDECREF(o); }
  PyObject* release() {
    PyObject* p = o;
    o = nullptr;
    return p;
  }
};

// linear_fwd(xq, wq, sx_inv, sw_inv, fmt_x, fmt_w, y, out_amax, out_q, q_fmt, q_scale, ws) -> y
FN(linear_fwd, 12, {
  const Mat x = mat(a[0], kCodes, "xq"), w = mat(a[1], kCodes, "wq");
  same(x.cols, w.cols, "inner dimensions differ");
  Out y(a[6], x.rows, w.rows, tensor(a[0], "xq").device(), "y");
  const float *sx = f32(a[2]), *sw = f32(a[3]);
  Epi e;
  e.fill(a[7], a[8], a[9], a[10]);
  const Ws ws = workspace(a[11]);
  const int32_t fx = i32(a[4]), fw = i32(a[5]);
  void* st = stream();
  call("tweo_fp8_linear_fwd", [&] {
    return tweo_fp8_linear_fwd((const uint8_t*)x.p, x.ld, (const uint8_t*)w.p, w.ld, sx, sw, (uint16_t*)y.m.p, y.m.ld, x.rows, w.rows,
                               x.cols, fx, fw, e.p, ws.p, ws.n, st);
  });
  return y.release();
})

// linear_fwd_act(xq, wq, sx_inv, sw_inv, act, fmt_x, fmt_w, y or None, want_y, out_amax, out_q, q_fmt, q_scale) -> y or None
FN(linear_fwd_act, 13, {
  const Mat x = mat(a[0], kCodes, "xq"), w = mat(a[1], kCodes, "wq");
  same(x.cols, w.cols, "inner dimensions differ");
  const int32_t act = i32(a[4]);
  int64_t cols = w.rows;
  if (act == TWEO_ACT_SWIGLU) {
    if (cols % 2) fail(PyExc_ValueError, "SwiGLU needs an even number of weight rows (gate rows, then up rows)");
    cols /= 2;
  }
  const float *sx = f32(a[2]), *sw = f32(a[3]);
  const int32_t fx = i32(a[5]), fw = i32(a[6]);
  Epi e;
  e.fill(a[9], a[10], a[11], a[12]);
  void* st = stream();
  auto run = [&](uint16_t* y, int64_t ldy) {
    call("tweo_fp8_linear_fwd_act", [&] {
      return tweo_fp8_linear_fwd_act((const uint8_t*)x.p, x.ld, (const uint8_t*)w.p, w.ld, sx, sw, act, y, ldy, x.rows, cols, x.cols,
                                     fx, fw, e.p, st);
    });
  };
  if (!flag(a[8])) {
    run(nullptr, 0);
    Py_RETURN_NONE;
  }
  Out y(a[7], x.rows, cols, tensor(a[0], "xq").device(), "y");
  run((uint16_t*)y.m.p, y.m.ld);
  return y.release();
})

// linear_dgrad(dyq, wq, sdy_inv, sw_inv, fmt_dy, fmt_w, dx, out_amax, out_q, q_fmt, q_scale, ws) -> dx
FN(linear_dgrad, 12, {
  const Mat dy = mat(a[0], kCodes, "dyq"), w = mat(a[1], kCodes, "wq");
  same(dy.cols, w.rows, "inner dimensions differ");
  Out dx(a[6], dy.rows, w.cols, tensor(a[0], "dyq").device(), "dx");
  const float *sd = f32(a[2]), *sw = f32(a[3]);
  Epi e;
  e.fill(a[7], a[8], a[9], a[10]);
  const Ws ws = workspace(a[11]);
  const int32_t fd = i32(a[4]), fw = i32(a[5]);
  void* st = stream();
  call("tweo_fp8_linear_bwd_dgrad", [&] {
    return tweo_fp8_linear_bwd_dgrad((const uint8_t*)dy.p, dy.ld, fd, (const uint8_t*)w.p, w.ld, fw, sd, sw, (uint16_t*)dx.m.p, dx.m.ld,
                                     dy.rows, dy.cols, w.cols, e.p, ws.p, ws.n, st);
  });
  return dx.release();
})

// linear_wgrad(xq, dyq, sx_inv, sdy_inv, fmt_x, fmt_dy, dw, dw_dtype, accumulate, ws) -> dw
FN(linear_wgrad, 10, {
  const Mat x = mat(a[0], kCodes, "xq"), dy = mat(a[1], kCodes, "dyq");
  same(x.rows, dy.rows, "token dimensions differ");
  const int32_t dt = i32(a[7]);
  const bool acc = flag(a[8]);
  if (a[6] == Py_None && acc) fail(PyExc_ValueError, "accumulate needs an existing dw");
  Out dw(a[6], dy.cols, x.cols, tensor(a[0], "xq").device(), "dw", dt == TWEO_BF16 ? at::kBFloat16 : at::kFloat);
  const float *sx = f32(a[2]), *sd = f32(a[3]);
  const Ws ws = workspace(a[9]);
  const int32_t fx = i32(a[4]), fd = i32(a[5]);
  void* st = stream();
  call("tweo_fp8_linear_bwd_wgrad", [&] {
    return tweo_fp8_linear_bwd_wgrad((const uint8_t*)x.p, x.ld, fx, (const uint8_t*)dy.p, dy.ld, fd, sx, sd, dw.m.p, dw.m.ld, dt,
                                     acc ? 1 : 0, x.rows, dy.cols, x.cols, ws.p, ws.n, st);
  });
  return dw.release();
})

// linear_bwd(dyq, xq, wq, sdy_inv, sx_inv, sw_inv, fmt_dy, fmt_x, fmt_w, dx, dw, ws) -> (dx, dw)
FN(linear_bwd, 12, {
  const Mat dy = mat(a[0], kCodes, "dyq"), x = mat(a[1], kCodes, "xq"), w = mat(a[2], kCodes, "wq");
  if (dy.rows != x.rows || dy.cols != w.rows || x.cols != w.cols)
    fail(PyExc_ValueError, "shapes of dyq [M,N], xq [M,K] and wq [N,K] do not agree");
  const at::Device device = tensor(a[0], "dyq").device();
  Out dx(a[9], dy.rows, x.cols, device, "dx");
  Out dw(a[10], dy.cols, x.cols, device, "dw");
  const float *sd = f32(a[3]), *sx = f32(a[4]), *sw = f32(a[5]);
  const Ws ws = workspace(a[11]);
  const int32_t fd = i32(a[6]), fx = i32(a[7]), fw = i32(a[8]);
  void* st = stream();
  call("tweo_fp8_linear_bwd", [&] {
    return tweo_fp8_linear_bwd((const uint8_t*)dy.p, dy.ld, fd, (const uint8_t*)x.p, x.ld, fx, (const uint8_t*)w.p, w.ld, fw, sd, sx, sw,
                               (uint16_t*)dx.m.p, dx.m.ld, (uint16_t*)dw.m.p, dw.m.ld, dy.rows, dy.cols, x.cols, ws.p, ws.n, st);
  });
  return PyTuple_Pack(2, dx.o, dw.o);
})

// What the mappings of a group handed out; kept until the call returns.
struct Held {
  std::vector<PyObject*> v;
  ~Held() {
    for (PyObject* o : v) Py_DECREF(o);
  }
  PyObject* keep(PyObject* o) {
    if (!o) throw PyFailure{};
    v.push_back(o);
    return o;
  }
};

// A problem's value for a key; None where there is none (borrowed).  A dict is read directly, another mapping through get().
PyObject* item(PyObject* map, PyObject* key, Held& held) {
  if (!PyDict_CheckExact(map)) return held.keep(PyObject_CallMethodOneArg(map, N.get, key));
  PyObject* v = PyDict_GetItemWithError(map, key);
  if (!v && PyErr_Occurred()) throw PyFailure{};
  return v ? v : Py_None;
}
PyObject* required(PyObject* map, PyObject* key, Held& held) { return held.keep(PyObject_GetItem(map, key)); }
int32_t item_i32(PyObject* map, PyObject* key, int32_t otherwise, Held& held) {
  PyObject* v = item(map, key, held);
  return v == Py_None ? otherwise : i32(v);
}

// The problems of a grouped launch.
struct Group {
  tweo_linear_problem_t pr[TWEO_MAX_GROUP] = {};
  Epi epi[TWEO_MAX_GROUP];
  Held held;
  Ref list;
  Py_ssize_t count;
  explicit Group(PyObject* problems) : list(PySequence_Fast(problems, "problems must be a sequence")), count(PySequence_Fast_GET_SIZE(list.o)) {
    if (count < 1 || count > TWEO_MAX_GROUP) fail(PyExc_ValueError, "need 1..MAX_GROUP problems");
    for (Py_ssize_t i = 0; i < count; ++i) fill(i);
  }
  void fill(Py_ssize_t i) {
    PyObject* d = PySequence_Fast_GET_ITEM(list.o, i);
    tweo_linear_problem_t& p = pr[i];
    PyObject* fmt = item(d, N.q_fmt, held);
    Ref q_fmt(fmt == Py_None ? PyLong_FromLong(TWEO_E4M3) : Py_NewRef(fmt));
    epi[i].fill(item(d, N.out_amax, held), item(d, N.out_q, held), q_fmt.o, item(d, N.q_scale, held));
    p.epi = epi[i].p;
    p.product = i32(required(d, N.product, held));
    p.fmt_x = item_i32(d, N.fmt_x, TWEO_E4M3, held);
    p.fmt_w = item_i32(d, N.fmt_w, TWEO_E4M3, held);
    p.fmt_dy = item_i32(d, N.fmt_dy, TWEO_E5M2, held);
    PyObject *xq = item(d, N.xq, held), *wq = item(d, N.wq, held), *dyq = item(d, N.dyq, held);
    Mat x{}, w{}, dy{};
    if (xq != Py_None || p.product == TWEO_PRODUCT_FWD || p.product == TWEO_PRODUCT_WGRAD) x = mat(xq, kCodes, "xq");
    if (wq != Py_None || p.product == TWEO_PRODUCT_FWD || p.product == TWEO_PRODUCT_DGRAD) w = mat(wq, kCodes, "wq");
    if (dyq != Py_None || p.product == TWEO_PRODUCT_DGRAD || p.product == TWEO_PRODUCT_WGRAD) dy = mat(dyq, kCodes, "dyq");
    if (p.product == TWEO_PRODUCT_FWD) {
      p.M = x.rows, p.K = x.cols, p.N = w.rows;
    } else if (p.product == TWEO_PRODUCT_DGRAD) {
      p.M = dy.rows, p.N = dy.cols, p.K = w.cols;
    } else if (p.product == TWEO_PRODUCT_WGRAD) {
      p.M = x.rows, p.K = x.cols, p.N = dy.cols;
    } else {
      fail(PyExc_ValueError, "product must be PRODUCT_FWD, PRODUCT_DGRAD or PRODUCT_WGRAD");
    }
    p.xq = (const uint8_t*)x.p, p.ldx = x.ld;
    p.wq = (const uint8_t*)w.p, p.ldw = w.ld;
    p.dyq = (const uint8_t*)dy.p, p.lddy = dy.ld;
    p.sx_inv = f32_or_null(item(d, N.sx_inv, held), "sx_inv");
    p.sw_inv = f32_or_null(item(d, N.sw_inv, held), "sw_inv");
    p.sdy_inv = f32_or_null(item(d, N.sdy_inv, held), "sdy_inv");
    const Mat o = mat(required(d, N.out, held), kBf16, "out");
    p.out = (uint16_t*)o.p;
    p.ldo = o.ld;
  }
};

// linear_group(problems)
FN(linear_group, 1, {
  const Group g(a[0]);
  void* st = stream();
  call("tweo_fp8_linear_group", [&] { return tweo_fp8_linear_group(g.pr, (int32_t)g.count, st); });
  Py_RETURN_NONE;
})

// The block outputs of a penalty and its gradients (None: no gradients).
struct Blocks {
  Ref blocks, grads;
  Py_ssize_t L;
  const uint16_t* pa[TWEO_MAX_BLOCKS];
  void* pg[TWEO_MAX_BLOCKS];
  int64_t numel = 0;
  Blocks(PyObject* blocks_, PyObject* grads_, int32_t gdt)
      : blocks(PySequence_Fast(blocks_, "blocks must be a sequence")),
        grads(grads_ == Py_None ? Py_NewRef(Py_None) : PySequence_Fast(grads_, "grads must be a sequence")),
        L(PySequence_Fast_GET_SIZE(blocks.o)) {
    if (L < 1) fail(PyExc_IndexError, "list index out of range");
    if (L > TWEO_MAX_BLOCKS) call("tweo_loss_fwd_bwd", [] { return TWEO_ERR_INVALID_ARG; });
    const Py_ssize_t ng = grads.o == Py_None ? 0 : PySequence_Fast_GET_SIZE(grads.o);
    if (ng > L) fail(PyExc_IndexError, "more gradients than block outputs");
    for (Py_ssize_t i = 0; i < L; ++i) {
      const at::Tensor& t = tensor(PySequence_Fast_GET_ITEM(blocks.o, i), "block output");
      if (i == 0) numel = t.numel();
      if (t.numel() != numel || !t.is_contiguous()) fail(PyExc_ValueError, "block outputs must be contiguous and of equal size");
      check_kind(t, kBf16, "block output");
      pa[i] = (const uint16_t*)t.data_ptr();
      pg[i] = nullptr;   // a missing gradient is refused by the library
      if (i < ng) pg[i] = dev(PySequence_Fast_GET_ITEM(grads.o, i), gdt == TWEO_BF16 ? kBf16 : kF32, "grad");
    }
  }
  at::Device device() const { return tensor(PySequence_Fast_GET_ITEM(blocks.o, 0), "block output").device(); }
};

// linear_group_beside(problems, xs, outs, modes or None, blocks or None, grads, tau, eps, grad_coeff, ws)
//   -> None, or with blocks (loss, per-block losses)
FN(linear_group_beside, 10, {
  const Group g(a[0]);
  tweo_quant_desc_t d[TWEO_MAX_QUANT_BATCH];
  tweo_beside_t w = {};
  Casts casts(a[1], a[2], a[3], d, 0);
  w.casts = d;
  w.n_casts = (int32_t)casts.count;
  const Ws ws = workspace(a[9], true);
  void* st = stream();
  auto run = [&] {
    call("tweo_fp8_linear_group_beside", [&] { return tweo_fp8_linear_group_beside(g.pr, (int32_t)g.count, &w, ws.p, ws.n, st); });
  };
  if (a[4] == Py_None) {
    run();
    Py_RETURN_NONE;
  }
  const Blocks b(a[4], a[5], TWEO_BF16);
  w.a = b.pa;
  w.grad = b.pg;
  w.L = (int32_t)b.L;
  w.n_per_tensor = b.numel;
  w.tau = flt(a[6]);
  w.eps = flt(a[7]);
  w.grad_coeff = flt(a[8]);
  const at::Tensor out = empty({1}, at::kFloat, b.device()), pb = empty({(int64_t)b.L}, at::kFloat, b.device());
  w.loss = (float*)out.data_ptr();
  w.loss_per_block = (float*)pb.data_ptr();
  run();
  Ref ro(wrap(out)), rp(wrap(pb));
  return PyTuple_Pack(2, ro.o, rp.o);
})

// loss(blocks, tau, eps, p, grad_coeff, grads or None, grad_dtype, ws, per_block) -> (loss, per-block losses or None)
FN(loss, 9, {
  const int32_t gdt = i32(a[6]);
  const Blocks b(a[0], a[5], gdt);
  const float tau = flt(a[1]), eps = flt(a[2]), p = flt(a[3]), c = flt(a[4]);
  const Ws w = workspace(a[7], true);
  const at::Tensor out = empty({1}, at::kFloat, b.device());
  at::Tensor pb;
  if (flag(a[8])) pb = empty({(int64_t)b.L}, at::kFloat, b.device());
  void* st = stream();
  call("tweo_loss_fwd_bwd", [&] {
    return tweo_loss_fwd_bwd(b.pa, (int32_t)b.L, b.numel, tau, eps, p, c, (float*)out.data_ptr(),
                             pb.defined() ? (float*)pb.data_ptr() : nullptr, b.grads.o != Py_None ? b.pg : nullptr, gdt, w.p, w.n, st);
  });
  Ref ro(wrap(out)), rp(pb.defined() ? wrap(pb) : Py_NewRef(Py_None));
  return PyTuple_Pack(2, ro.o, rp.o);
})

// w8a8(x, sx, wq, sw_inv, y, ws) -> y
FN(w8a8, 6, {
  const at::Tensor& t = tensor(a[0], "x");
  const unsigned k = kind_of(t.scalar_type());
  if (!(k & (kBf16 | kCodes))) fail(PyExc_TypeError, "x must be bf16 or uint8 E4M3 codes");
  const Mat x = mat(a[0], kBf16 | kCodes, "x"), w = mat(a[2], kCodes, "wq");
  same(x.cols, w.cols, "inner dimensions differ");
  Out y(a[4], x.rows, w.rows, t.device(), "y");
  const float *sx = f32(a[1], "sx"), *sw = f32(a[3]);
  const Ws ws = workspace(a[5], true);
  void* st = stream();
  call("tweo_w8a8_static_gemm", [&] {
    return tweo_w8a8_static_gemm(x.p, k & kBf16 ? TWEO_BF16 : TWEO_FP8_E4M3, x.ld, sx, (const uint8_t*)w.p, w.ld, sw, (uint16_t*)y.m.p,
                                 y.m.ld, x.rows, w.rows, x.cols, ws.p, ws.n, st);
  });
  return y.release();
})

// fp4_weight(xq, sx_inv, w4, sw_inv, fmt_x, y) -> y
FN(fp4_weight, 6, {
  const Mat x = mat(a[0], kCodes, "xq"), w = mat(a[2], kCodes, "w4");
  same(2 * w.cols, x.cols, "w4 must be [N, K // 2]");
  Out y(a[5], x.rows, w.rows, tensor(a[0], "xq").device(), "y");
  const float *sx = f32(a[1], "sx_inv"), *sw = f32(a[3], "sw_inv");
  const int32_t fx = i32(a[4]);
  void* st = stream();
  call("tweo_fp4_weight_linear", [&] {
    return tweo_fp4_weight_linear((const uint8_t*)x.p, x.ld, fx, sx, (const uint8_t*)w.p, w.ld, sw, (uint16_t*)y.m.p, y.m.ld, x.rows,
                                  w.rows, x.cols, st);
  });
  return y.release();
})

// block_output(x, f, tau, eps, p, grad_coeff, want_grad, q_fmt or None, q_scale, a, grad, aq, ws)
//   -> (a, loss, amax, grad or None, aq or None)
FN(block_output, 13, {
  const at::Tensor &x = tensor(a[0], "x"), &f = tensor(a[1], "f");
  if (x.sizes() != f.sizes() || !x.is_contiguous() || !f.is_contiguous())
    fail(PyExc_ValueError, "x and f must be contiguous and of equal shape");
  check_kind(x, kBf16, "x");
  check_kind(f, kBf16, "f");
  const at::Device device = x.device();
  auto given_or_new = [&](PyObject* o, at::ScalarType type) { return o == Py_None ? wrap(empty(x.sizes(), type, device)) : Py_NewRef(o); };
  Ref out(given_or_new(a[9], at::kBFloat16));
  Ref grad(flag(a[6]) ? given_or_new(a[10], at::kBFloat16) : Py_NewRef(Py_None));
  const bool cast = a[7] != Py_None;
  if (cast && a[8] == Py_None) fail(PyExc_ValueError, "the FP8 copy needs q_scale");
  Ref aq(cast ? given_or_new(a[11], at::kByte) : Py_NewRef(Py_None));
  uint16_t* po = dev<uint16_t>(out.o, kBf16, "a");
  uint16_t* pg = grad.o == Py_None ? nullptr : dev<uint16_t>(grad.o, kBf16, "grad");
  uint8_t* pq = cast ? dev<uint8_t>(aq.o, kCodes, "aq") : nullptr;
  const int32_t fmt = cast ? i32(a[7]) : 0;
  const float* qs = f32_or_null(a[8], "q_scale");
  const Ws w = workspace(a[12], true);
  const float tau = flt(a[2]), eps = flt(a[3]), p = flt(a[4]), c = flt(a[5]);
  const at::Tensor two = empty({2}, at::kFloat, device);
  float* scalars = (float*)two.data_ptr();
  void* st = stream();
  call("tweo_block_output_fused", [&] {
    return tweo_block_output_fused((const uint16_t*)x.data_ptr(), (const uint16_t*)f.data_ptr(), x.numel(), tau, eps, p, c, po, pg,
                                   scalars, scalars + 1, pq, fmt, qs, w.p, w.n, st);
  });
  Ref l(wrap(two.narrow(0, 0, 1))), m(wrap(two.narrow(0, 1, 1)));
  return PyTuple_Pack(5, out.o, l.o, m.o, grad.o, aq.o);
})

// layernorm(x, gamma, beta, eps, kind, want_y, q_fmt or None, q_scale, want_amax, want_stats, y, yq)
//   -> (y or None, yq or None, amax or None, mean or None, rstd or None)
FN(layernorm, 12, {
  const Mat x = mat(a[0], kBf16, "x");
  const at::Device device = tensor(a[0], "x").device();
  auto given_or_new = [&](PyObject* o, at::ScalarType type) {
    return o == Py_None ? wrap(empty({x.rows, x.cols}, type, device)) : Py_NewRef(o);
  };
  const bool cast = a[6] != Py_None;
  Ref y(flag(a[5]) ? given_or_new(a[10], at::kBFloat16) : Py_NewRef(Py_None));
  if (cast && a[7] == Py_None) fail(PyExc_ValueError, "the FP8 copy needs q_scale");
  Ref yq(cast ? given_or_new(a[11], at::kByte) : Py_NewRef(Py_None));
  Mat my{}, mq{};
  if (y.o != Py_None) my = mat(y.o, kBf16, "y");
  if (cast) mq = mat(yq.o, kCodes, "yq");
  at::Tensor amax, mean, rstd;
  if (flag(a[8])) amax = empty({1}, at::kFloat, device);
  if (flag(a[9])) {
    mean = empty({x.rows}, at::kFloat, device);
    rstd = empty({x.rows}, at::kFloat, device);
  }
  auto ptr = [](const at::Tensor& t) { return t.defined() ? (float*)t.data_ptr() : nullptr; };
  const float *gamma = f32(a[1], "gamma"), *beta = f32_or_null(a[2], "beta"), *qs = f32_or_null(a[7], "q_scale");
  const float eps = flt(a[3]);
  const int32_t kind = i32(a[4]), fmt = cast ? i32(a[6]) : 0;
  void* st = stream();
  call("tweo_layernorm_fp8", [&] {
    return tweo_layernorm_fp8((const uint16_t*)x.p, x.ld, x.rows, x.cols, kind, gamma, beta, eps, (uint16_t*)my.p, my.ld, (uint8_t*)mq.p,
                              mq.ld, fmt, qs, ptr(amax), ptr(mean), ptr(rstd), st);
  });
  auto obj = [](const at::Tensor& t) { return t.defined() ? wrap(t) : Py_NewRef(Py_None); };
  Ref oa(obj(amax)), om(obj(mean)), os(obj(rstd));
  return PyTuple_Pack(5, y.o, yq.o, oa.o, om.o, os.o);
})

// delayed_scaling(history, amax_new, scale, scale_inv, fmt)
FN(delayed_scaling, 5, {
  const at::Tensor& h = tensor(a[0], "amax_history");
  if (h.dim() != 2 || !h.is_contiguous()) fail(PyExc_ValueError, "amax_history must be contiguous [T, H]");
  const int64_t T = h.size(0);
  const char* names[3] = {"amax_new", "scale", "scale_inv"};
  for (int i = 0; i < 3; ++i) {
    const at::Tensor& t = tensor(a[1 + i], names[i]);
    if (t.numel() != T || !t.is_contiguous()) fail(PyExc_ValueError, std::string(names[i]) + " must hold one value per tensor");
  }
  float *ph = f32(a[0], "amax_history"), *pn = f32(a[1]), *ps = f32(a[2]), *pi = f32(a[3]);
  const int32_t fmt = i32(a[4]);
  void* st = stream();
  call("tweo_delayed_scaling_update", [&] { return tweo_delayed_scaling_update(ph, (int32_t)h.size(1), pn, ps, pi, (int32_t)T, fmt, st); });
  Py_RETURN_NONE;
})

// absmax(x, bits, granularity, eps, s or None, ws) -> (q, s)
FN(absmax, 6, {
  const Mat x = mat(a[0], kBf16, "x");
  const at::Device device = tensor(a[0], "x").device();
  const int32_t bits = i32(a[1]), gran = i32(a[2]);
  const bool given = a[4] != Py_None;
  Ref s(given ? Py_NewRef(a[4]) : wrap(empty({gran == TWEO_GRAN_ROW ? x.rows : (int64_t)1}, at::kFloat, device)));
  float* ps = f32(s.o, "s");
  const at::Tensor q = empty({x.rows, x.cols}, at::kChar, device);
  const Ws w = workspace(a[5]);
  const float eps = flt(a[3]);
  const int64_t ldq = q.stride(0);
  void* st = stream();
  call("tweo_absmax_quantize", [&] {
    return tweo_absmax_quantize((const uint16_t*)x.p, x.rows, x.cols, x.ld, bits, gran, given ? TWEO_SCALE_GIVEN : TWEO_SCALE_CURRENT, eps, ps,
                                (int8_t*)q.data_ptr(), ldq, w.p, w.n, st);
  });
  Ref rq(wrap(q));
  return PyTuple_Pack(2, rq.o, s.o);
})

int32_t per_row(PyObject* o, const char* name) { return tensor(o, name).numel() > 1 ? 1 : 0; }

// int8_linear(xq, sx, wq, sw, bits, y) -> y
FN(int8_linear, 6, {
  const Mat x = mat(a[0], kI8, "xq"), w = mat(a[2], kI8, "wq");
  same(x.cols, w.cols, "inner dimensions differ");
  Out y(a[5], x.rows, w.rows, tensor(a[0], "xq").device(), "y");
  const float *sx = f32(a[1], "sx"), *sw = f32(a[3], "sw");
  const int32_t px = per_row(a[1], "sx"), pw = per_row(a[3], "sw"), bits = i32(a[4]);
  void* st = stream();
  call("tweo_int8_linear", [&] {
    return tweo_int8_linear((const int8_t*)x.p, x.ld, sx, px, (const int8_t*)w.p, w.ld, sw, pw, bits, (uint16_t*)y.m.p, y.m.ld, x.rows,
                            w.rows, x.cols, st);
  });
  return y.release();
})

// residual_rows(xq, sx, fq, sf, bits, eps, yq) -> (yq, sy)
FN(residual_rows, 7, {
  const at::Tensor &x = tensor(a[0], "xq"), &f = tensor(a[2], "fq");
  if (x.dim() != 2 || x.sizes() != f.sizes() || !x.is_contiguous() || !f.is_contiguous())
    fail(PyExc_ValueError, "xq and fq must be contiguous 2-D tensors of equal shape");
  check_kind(x, kI8, "xq");
  check_kind(f, kI8, "fq");
  const int64_t rows = x.size(0), cols = x.size(1);
  if (tensor(a[1], "sx").numel() != rows || tensor(a[3], "sf").numel() != rows) fail(PyExc_ValueError, "one scale per row");
  const float *sx = f32(a[1], "sx"), *sf = f32(a[3], "sf");
  Ref y(a[6] == Py_None ? wrap(empty(x.sizes(), at::kChar, x.device())) : Py_NewRef(a[6]));
  int8_t* py = dev<int8_t>(y.o, kI8, "yq");
  const at::Tensor sy = empty({rows}, at::kFloat, x.device());
  const int32_t bits = i32(a[4]);
  const float eps = flt(a[5]);
  void* st = stream();
  call("tweo_residual_add_q8_rows", [&] {
    return tweo_residual_add_q8_rows((const int8_t*)x.data_ptr(), sx, (const int8_t*)f.data_ptr(), sf, rows, cols, bits, eps, py,
                                     rows ? (float*)sy.data_ptr() : nullptr, st);
  });
  Ref rs(wrap(sy));
  return PyTuple_Pack(2, y.o, rs.o);
})

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_XSETREF(g_tweo_error, Py_NewRef(cls));
  Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"set_error", set_error, METH_O, nullptr},
    ENTRY(quantize), ENTRY(quantize_batch), ENTRY(linear_fwd), ENTRY(linear_fwd_act), ENTRY(linear_dgrad), ENTRY(linear_wgrad),
    ENTRY(linear_bwd), ENTRY(linear_group), ENTRY(linear_group_beside), ENTRY(loss), ENTRY(w8a8), ENTRY(fp4_weight), ENTRY(block_output), ENTRY(layernorm),
    ENTRY(delayed_scaling), ENTRY(absmax), ENTRY(int8_linear), ENTRY(residual_rows),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of binding.py", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
  const char* const text[] = {"q", "scale", "scale_inv", "amax", "sat_count", "fmt", "product", "fmt_x", "fmt_w", "fmt_dy", "xq", "wq",
                              "dyq", "sx_inv", "sw_inv", "sdy_inv", "out", "out_amax", "out_q", "q_fmt", "q_scale", "get"};
  PyObject** const slot = reinterpret_cast<PyObject**>(&N);
  static_assert(sizeof(text) / sizeof(text[0]) == sizeof(Names) / sizeof(PyObject*), "one name per slot");
  for (size_t i = 0; i < sizeof(text) / sizeof(text[0]); ++i)
    if (!(slot[i] = PyUnicode_InternFromString(text[i]))) return nullptr;
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "BUILT_FOR", TWEO_BUILT_FOR) < 0) Py_CLEAR(m);
  return m;
}
