// Native part of the Python binding: the calls of binding.py and autograd.py that a
// training step makes, with tensor checks, output allocation and argument marshalling
// in C++ (a call through ctypes cost 15-40 us of host time, several times what the
// kernels of a small layer take), and the autograd function behind LbpLinear, whose
// backward pass then runs without the interpreter.
//
// Conventions of the module functions: positional arguments as binding.py passes them.
// They return the call's result; an int, the lbp_status, where the library refused; None
// where an argument is not what they expect.  In that case nothing has been done, and
// binding.py goes through its own checks, which name the error.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/autocast_mode.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_cpp_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/pybind.h>

#include <optional>
#include <string>
#include <vector>

#include "lbp.h"

namespace {

using at::Tensor;

// ---- the C library, resolved from the file binding.py has loaded ----
struct Library {
  decltype(&lbp_status_string) status_string;
  decltype(&lbp_status_bytes) status_bytes;
  decltype(&lbp_workspace_bytes) workspace_bytes;
  decltype(&lbp_workspace_bytes_ex) workspace_bytes_ex;
  decltype(&lbp_workspace_bytes_projected) workspace_bytes_projected;
  decltype(&lbp_spectrum_workspace_bytes) spectrum_workspace_bytes;
  decltype(&lbp_project) project;
  decltype(&lbp_spectrum) spectrum;
  decltype(&lbp_backward) backward;
  decltype(&lbp_backward_ex) backward_ex;
  decltype(&lbp_backward_batch) backward_batch;
  decltype(&lbp_backward_fullrank) backward_fullrank;
} lib;
PyObject* error_type = nullptr;   // binding.LbpError

template <class F>
bool resolve(void* handle, const char* name, F* fn) {
  *fn = reinterpret_cast<F>(dlsym(handle, name));
  return *fn != nullptr;
}

// ---- arguments ----
struct Bases {
  lbp_basis v[256];
  int r = 0;
};
// int(o), where that is an int32; false otherwise (no error is left behind).
bool index_of(PyObject* o, int32_t* v) {
  int over = 0;
  long l = 0;
  if (PyLong_Check(o)) {
    l = PyLong_AsLongAndOverflow(o, &over);
  } else {   // a numpy or torch scalar, a float
    PyObject* n = PyNumber_Long(o);
    if (n == nullptr) {
      PyErr_Clear();
      return false;
    }
    l = PyLong_AsLongAndOverflow(n, &over);
    Py_DECREF(n);
  }
  *v = static_cast<int32_t>(l);
  return over == 0 && *v == l;
}
// A sequence of pairs; whether a pair is a basis is the library's to say.
bool parse_pair(PyObject* p, lbp_basis* out) {
  if (PyTuple_Check(p) && PyTuple_GET_SIZE(p) == 2)
    return index_of(PyTuple_GET_ITEM(p, 0), &out->i) && index_of(PyTuple_GET_ITEM(p, 1), &out->j);
  PyObject* t = PySequence_Check(p) ? PySequence_Tuple(p) : nullptr;   // a list, a row of an array
  const bool ok = t != nullptr && PyTuple_GET_SIZE(t) == 2 && index_of(PyTuple_GET_ITEM(t, 0), &out->i) &&
                  index_of(PyTuple_GET_ITEM(t, 1), &out->j);
  Py_XDECREF(t);
  PyErr_Clear();
  return ok;
}
bool parse_bases(PyObject* o, Bases* out) {
  if (!PySequence_Check(o)) return false;
  PyObject* s = PySequence_Fast(o, "");
  if (s == nullptr) {
    PyErr_Clear();
    return false;
  }
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(s);
  bool ok = n <= 256;
  for (Py_ssize_t q = 0; q < n && ok; ++q) ok = parse_pair(PySequence_Fast_GET_ITEM(s, q), &out->v[q]);
  Py_DECREF(s);
  out->r = static_cast<int>(n);
  return ok;
}

bool parse_int(PyObject* o, int* v) {
  int32_t a = 0;
  if (!PyIndex_Check(o) || !index_of(o, &a) || a < 0 || a > (1 << 30)) return false;   // no floats
  *v = a;
  return true;
}

// A tensor, or an undefined one for None; false: neither.
bool parse_tensor(PyObject* o, Tensor* t) {
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) return false;
  *t = THPVariable_Unpack(o);
  return true;
}

int dtype_code(at::ScalarType t) {
  if (t == at::kFloat) return LBP_F32;
  if (t == at::kBFloat16) return LBP_BF16;
  return -1;
}
int parse_dtype(PyObject* o) {
  return THPDtype_Check(o) ? dtype_code(reinterpret_cast<THPDtype*>(o)->scalar_type) : -1;
}

bool int_size(int64_t v) { return v >= 0 && v <= (1ll << 30); }

// On the current CUDA device, and contiguous.
bool dense_on(const Tensor& t, int dev) {
  return t.is_cuda() && t.get_device() == dev && t.is_contiguous();
}

bool has_shape(const Tensor& t, at::IntArrayRef want) { return t.sizes() == want; }

// Strides of a (B,H,W,C) tensor as the library takes them (all zero: dense).
bool view_of(const Tensor& t, int dev, lbp_view* v) {
  *v = lbp_view{0, 0, 0};
  if (!t.is_cuda() || t.get_device() != dev) return false;
  if (t.is_contiguous()) return true;
  const int64_t B = t.size(0), H = t.size(1), W = t.size(2), C = t.size(3);
  if (C > 1 && t.stride(3) != 1) return false;
  const int64_t tok = W > 1 ? t.stride(2) : C;
  const int64_t row = H > 1 ? t.stride(1) : W * tok;
  const int64_t img = B > 1 ? t.stride(0) : H * row;
  *v = lbp_view{img, row, tok};
  return true;
}
// Row pitch of an (n, C) matrix (0: dense).
bool rows_of(const Tensor& t, int dev, int64_t* pitch) {
  *pitch = 0;
  if (!t.is_cuda() || t.get_device() != dev) return false;
  if (t.is_contiguous()) return true;
  if (t.size(1) > 1 && t.stride(1) != 1) return false;
  *pitch = t.size(0) > 1 ? t.stride(0) : 0;
  return true;
}

Tensor bytes_on(const Tensor& like, size_t n) {
  return at::empty({static_cast<int64_t>(n)}, like.options().dtype(at::kByte));
}
void* current_stream(int dev) { return c10::cuda::getCurrentCUDAStream(dev).stream(); }

PyObject* pair(const Tensor& a, const Tensor& b) {
  PyObject* t = PyTuple_New(2);
  if (t == nullptr) return nullptr;
  PyTuple_SET_ITEM(t, 0, THPVariable_Wrap(a));
  PyTuple_SET_ITEM(t, 1, THPVariable_Wrap(b));
  return t;
}
PyObject* not_handled() { Py_RETURN_NONE; }

// A call into the library: other Python threads run meanwhile (it may search a tile plan, wait
// for the batch section of another thread, or for room in a full launch queue).
template <class F>
auto without_gil(F call) {
  pybind11::gil_scoped_release no_gil;
  return call();
}

// One problem's shapes, dtypes and devices, as binding._check_layer_tensors has them.
struct Problem {
  lbp_layer L;
  int dev;
};
bool layer_of(const Tensor& g_y, const Tensor& W, const Tensor& x, int k, Problem* p) {
  if (!g_y.defined() || !W.defined() || g_y.dim() != 4 || W.dim() != 2 || !g_y.is_cuda()) return false;
  const int dt = dtype_code(g_y.scalar_type());
  if (dt < 0 || W.scalar_type() != g_y.scalar_type()) return false;
  const int64_t B = g_y.size(0), H = g_y.size(1), Wd = g_y.size(2), Cout = g_y.size(3), Cin = W.size(1);
  if (W.size(0) != Cout || !int_size(B) || !int_size(H) || !int_size(Wd) || !int_size(Cout) || !int_size(Cin))
    return false;
  p->dev = g_y.get_device();
  if (p->dev != c10::cuda::current_device() || !dense_on(W, p->dev)) return false;
  if (x.defined() && (!has_shape(x, {B, H, Wd, Cin}) || x.scalar_type() != g_y.scalar_type())) return false;
  p->L = lbp_layer{static_cast<int32_t>(B), static_cast<int32_t>(H), static_cast<int32_t>(Wd),
                   static_cast<int32_t>(Cin), static_cast<int32_t>(Cout), k, dt, LBP_F32};
  return true;
}
// The given output, checked, or a new one.
bool grad_x(Tensor* g_x, const Tensor& g_y, const lbp_layer& L) {
  if (!g_x->defined()) {
    *g_x = at::empty({L.B, L.H, L.W, L.Cin}, g_y.options());
    return true;
  }
  return has_shape(*g_x, {L.B, L.H, L.W, L.Cin}) && g_x->scalar_type() == g_y.scalar_type();
}
bool grad_w(Tensor* g_W, const Tensor& g_y, lbp_layer* L, int gw_code, int dev) {
  if (!g_W->defined()) {
    if (gw_code < 0) return false;
    *g_W = at::empty({L->Cout, L->Cin}, g_y.options().dtype(gw_code == LBP_BF16 ? at::kBFloat16 : at::kFloat));
  } else if (!has_shape(*g_W, {L->Cout, L->Cin}) || !dense_on(*g_W, dev)) {
    return false;
  }
  L->gw_dtype = dtype_code(g_W->scalar_type());
  return L->gw_dtype >= 0;
}

// project(t, k, bases, out, ws)
PyObject* py_project(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Tensor t, out, ws;
  int k = 0;
  Bases b;
  if (n != 5 || !parse_tensor(a[0], &t) || !parse_int(a[1], &k) || !parse_bases(a[2], &b) ||
      !parse_tensor(a[3], &out) || !parse_tensor(a[4], &ws) || !t.defined() || t.dim() != 4 || k < 1 || !t.is_cuda())
    return not_handled();
  const int dt = dtype_code(t.scalar_type()), dev = t.get_device();
  if (dt < 0 || dev != c10::cuda::current_device() || !t.is_contiguous()) return not_handled();
  for (int i = 0; i < 4; ++i)
    if (!int_size(t.size(i))) return not_handled();
  const int64_t shape[5] = {t.size(0), (t.size(1) + k - 1) / k, (t.size(2) + k - 1) / k, b.r, t.size(3)};
  if (!out.defined())
    out = at::empty(shape, t.options());
  else if (!has_shape(out, shape) || out.scalar_type() != t.scalar_type() || !dense_on(out, dev))
    return not_handled();
  if (!ws.defined()) ws = bytes_on(t, lib.status_bytes());
  if (!dense_on(ws, dev)) return not_handled();
  const int e = without_gil([&] {
    return lib.project(t.data_ptr(), out.data_ptr(), t.size(0), t.size(1), t.size(2), t.size(3), k, b.v, b.r, dt,
                       ws.data_ptr(), ws.numel(), current_stream(dev));
  });
  return e != LBP_OK ? PyLong_FromLong(e) : THPVariable_Wrap(out);
  END_HANDLE_TH_ERRORS
}

// spectrum(t, k, out, ws)
PyObject* py_spectrum(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Tensor t, out, ws;
  int k = 0;
  if (n != 4 || !parse_tensor(a[0], &t) || !parse_int(a[1], &k) || !parse_tensor(a[2], &out) ||
      !parse_tensor(a[3], &ws) || !t.defined() || t.dim() != 4 || !t.is_cuda())
    return not_handled();
  const int dt = dtype_code(t.scalar_type()), dev = t.get_device();
  if (dt < 0 || dev != c10::cuda::current_device() || !t.is_contiguous()) return not_handled();
  for (int i = 0; i < 4; ++i)
    if (!int_size(t.size(i))) return not_handled();
  if (!out.defined())
    out = at::empty({k, k}, t.options().dtype(at::kDouble));
  else if (!has_shape(out, {k, k}) || out.scalar_type() != at::kDouble || !dense_on(out, dev))
    return not_handled();
  if (!ws.defined()) {
    const size_t bytes = lib.spectrum_workspace_bytes(t.size(0), t.size(1), t.size(2), t.size(3), k, dt);
    if (bytes == 0) return not_handled();
    ws = bytes_on(t, bytes);
  }
  if (!dense_on(ws, dev)) return not_handled();
  const int e = without_gil([&] {
    return lib.spectrum(t.data_ptr(), out.data_ptr<double>(), t.size(0), t.size(1), t.size(2), t.size(3), k, dt,
                        ws.data_ptr(), ws.numel(), current_stream(dev));
  });
  return e != LBP_OK ? PyLong_FromLong(e) : THPVariable_Wrap(out);
  END_HANDLE_TH_ERRORS
}

// backward(x, g_y, W, k, bases | None, gw_dtype, g_x, g_W, ws); bases None: exact backpropagation
PyObject* py_backward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Tensor x, g_y, W, g_x, g_W, ws;
  int k = 0;
  Bases b;
  Problem p;
  if (n != 9 || !parse_tensor(a[0], &x) || !parse_tensor(a[1], &g_y) || !parse_tensor(a[2], &W) ||
      !parse_int(a[3], &k) || (a[4] != Py_None && !parse_bases(a[4], &b)) || !parse_tensor(a[6], &g_x) ||
      !parse_tensor(a[7], &g_W) || !parse_tensor(a[8], &ws) || !x.defined() || !layer_of(g_y, W, x, k, &p))
    return not_handled();
  const int dev = p.dev, r = a[4] == Py_None ? k * k : b.r;
  if (!dense_on(x, dev) || !dense_on(g_y, dev) || !grad_x(&g_x, g_y, p.L) || !dense_on(g_x, dev) ||
      !grad_w(&g_W, g_y, &p.L, parse_dtype(a[5]), dev))
    return not_handled();
  if (!ws.defined()) {
    const size_t bytes = lib.workspace_bytes(&p.L, r);
    if (bytes == 0) return not_handled();
    ws = bytes_on(g_y, bytes);
  }
  if (!dense_on(ws, dev)) return not_handled();
  const bool exact = a[4] == Py_None;
  const int e = without_gil([&] {
    return exact ? lib.backward_fullrank(x.data_ptr(), g_y.data_ptr(), W.data_ptr(), g_x.data_ptr(), g_W.data_ptr(),
                                         &p.L, ws.data_ptr(), ws.numel(), current_stream(dev))
                 : lib.backward(x.data_ptr(), g_y.data_ptr(), W.data_ptr(), g_x.data_ptr(), g_W.data_ptr(), &p.L, b.v,
                                b.r, ws.data_ptr(), ws.numel(), current_stream(dev));
  });
  return e != LBP_OK ? PyLong_FromLong(e) : pair(g_x, g_W);
  END_HANDLE_TH_ERRORS
}

// What lbp_backward_ex takes, as tensors; the optional ones may be undefined.
struct ExCall {
  Tensor x, x_hat, g_y, W, g_bias, x_extra, gy_extra, gx_extra, g_x, g_W, ws;
  double beta = 0.0;
  int k = 0, gw_code = LBP_F32;
};
// Returns the library's status, or -1 where a check does not hold (nothing done).
int run_ex(ExCall* c, const lbp_basis* set, int r) {
  Problem p;
  if (c->x.defined() == c->x_hat.defined() || !layer_of(c->g_y, c->W, c->x, c->k, &p) || c->k < 1) return -1;
  lbp_layer& L = p.L;
  const int dev = p.dev;
  const at::ScalarType dt = c->g_y.scalar_type();
  if (c->x_hat.defined()) {
    const int64_t shape[5] = {L.B, (L.H + c->k - 1) / c->k, (L.W + c->k - 1) / c->k, r, L.Cin};
    if (!has_shape(c->x_hat, shape) || c->x_hat.scalar_type() != dt || !dense_on(c->x_hat, dev)) return -1;
  }
  if (!c->g_W.defined() && c->beta != 0.0) return -1;
  if (!grad_x(&c->g_x, c->g_y, L) || !grad_w(&c->g_W, c->g_y, &L, c->gw_code, dev)) return -1;
  lbp_extras ex{};
  ex.beta = static_cast<float>(c->beta);
  if (c->g_bias.defined()) {
    const at::ScalarType bt = c->g_bias.scalar_type();
    if ((bt != at::kFloat && bt != dt) || !has_shape(c->g_bias, {L.Cout}) || !dense_on(c->g_bias, dev)) return -1;
    ex.g_bias = c->g_bias.data_ptr();
    ex.g_bias_dtype = dtype_code(bt);
  }
  if (c->x_extra.defined() || c->gy_extra.defined()) {
    if (!c->x_extra.defined() || !c->gy_extra.defined() || !c->gx_extra.defined() || c->x_extra.dim() != 2) return -1;
    const int64_t n = c->x_extra.size(0);
    if (!int_size(n) || !has_shape(c->x_extra, {n, L.Cin}) || !has_shape(c->gy_extra, {n, L.Cout}) ||
        !has_shape(c->gx_extra, {n, L.Cin}) || c->x_extra.scalar_type() != dt || c->gy_extra.scalar_type() != dt ||
        c->gx_extra.scalar_type() != dt)
      return -1;
    if (n > 0) {
      if (!rows_of(c->x_extra, dev, &ex.x_extra_pitch) || !rows_of(c->gy_extra, dev, &ex.gy_extra_pitch) ||
          !rows_of(c->gx_extra, dev, &ex.gx_extra_pitch))
        return -1;
      ex.x_extra = c->x_extra.data_ptr();
      ex.gy_extra = c->gy_extra.data_ptr();
      ex.gx_extra = c->gx_extra.data_ptr();
      ex.n_extra = static_cast<int32_t>(n);
    }
  }
  if ((c->x.defined() && !view_of(c->x, dev, &ex.x_view)) || !view_of(c->g_y, dev, &ex.gy_view) ||
      !view_of(c->g_x, dev, &ex.gx_view))
    return -1;
  if (!c->ws.defined()) {
    const size_t bytes = (c->x_hat.defined() ? lib.workspace_bytes_projected : lib.workspace_bytes_ex)(&L, r, &ex);
    if (bytes == 0) return -1;
    c->ws = bytes_on(c->g_y, bytes);
  }
  if (!dense_on(c->ws, dev)) return -1;
  return lib.backward_ex(c->x.defined() ? c->x.data_ptr() : nullptr,
                         c->x_hat.defined() ? c->x_hat.data_ptr() : nullptr, c->g_y.data_ptr(), c->W.data_ptr(),
                         c->g_x.data_ptr(), c->g_W.data_ptr(), &L, set, r, &ex, c->ws.data_ptr(), c->ws.numel(),
                         current_stream(dev));
}

// backward_ex(x, x_hat, g_y, W, k, bases, beta, g_bias, x_extra, gy_extra, gx_extra, gw_dtype, g_x, g_W, ws)
PyObject* py_backward_ex(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  ExCall c;
  Bases b;
  if (n != 15 || !parse_tensor(a[0], &c.x) || !parse_tensor(a[1], &c.x_hat) || !parse_tensor(a[2], &c.g_y) ||
      !parse_tensor(a[3], &c.W) || !parse_int(a[4], &c.k) || !parse_bases(a[5], &b) || !PyFloat_Check(a[6]) ||
      !parse_tensor(a[7], &c.g_bias) || !parse_tensor(a[8], &c.x_extra) || !parse_tensor(a[9], &c.gy_extra) ||
      !parse_tensor(a[10], &c.gx_extra) || !parse_tensor(a[12], &c.g_x) || !parse_tensor(a[13], &c.g_W) ||
      !parse_tensor(a[14], &c.ws) || (c.g_bias.defined() && c.g_bias.scalar_type() != at::kFloat))
    return not_handled();
  c.beta = PyFloat_AS_DOUBLE(a[6]);
  c.gw_code = parse_dtype(a[11]);
  const int e = without_gil([&] { return run_ex(&c, b.v, b.r); });
  if (e < 0) return not_handled();
  return e != LBP_OK ? PyLong_FromLong(e) : pair(c.g_x, c.g_W);
  END_HANDLE_TH_ERRORS
}

// backward_batch(xs, g_ys, Ws, k, bases, g_xs, g_Ws, wss) -> 0 or a status
PyObject* py_backward_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  int k = 0;
  Bases b;
  if (n != 8 || !parse_int(a[3], &k) || !parse_bases(a[4], &b)) return not_handled();
  PyObject* lists[6] = {a[0], a[1], a[2], a[5], a[6], a[7]};
  Py_ssize_t count = -1;
  for (PyObject* l : lists) {
    if (!PyList_Check(l) && !PyTuple_Check(l)) return not_handled();
    const Py_ssize_t m = PySequence_Fast_GET_SIZE(l);
    if (count >= 0 && m != count) return not_handled();
    count = m;
  }
  if (count < 1 || count > 64) return not_handled();
  std::vector<Tensor> held;   // the lists are the caller's to change once the lock is released
  held.reserve(6 * count);
  void* ptr[6][64];
  lbp_layer layers[64];
  size_t sizes[64];
  int dev = 0;
  for (Py_ssize_t i = 0; i < count; ++i) {
    Tensor t[6];
    for (int l = 0; l < 6; ++l)
      if (!parse_tensor(PySequence_Fast_GET_ITEM(lists[l], i), &t[l]) || !t[l].defined()) return not_handled();
    Problem p;
    if (!layer_of(t[1], t[2], t[0], k, &p)) return not_handled();
    dev = p.dev;
    if (!grad_x(&t[3], t[1], p.L) || !grad_w(&t[4], t[1], &p.L, -1, dev)) return not_handled();
    for (int l = 0; l < 6; ++l) {
      if (!dense_on(t[l], dev)) return not_handled();
      ptr[l][i] = t[l].data_ptr();
      held.push_back(t[l]);
    }
    layers[i] = p.L;
    sizes[i] = static_cast<size_t>(t[5].numel());
  }
  const int e = without_gil([&] {
    return lib.backward_batch(static_cast<int>(count), ptr[0], ptr[1], ptr[2], ptr[3], ptr[4], layers, b.v, b.r, ptr[5],
                              sizes, nullptr, current_stream(dev));
  });
  return PyLong_FromLong(e);
  END_HANDLE_TH_ERRORS
}

// Raises binding.LbpError(status, where) from any thread.
[[noreturn]] void raise_status(int status, const char* where) {
  pybind11::gil_scoped_acquire gil;
  PyObject* e = PyObject_CallFunction(error_type, "is", status, where);
  if (e != nullptr) {
    PyErr_SetObject(error_type, e);
    Py_DECREF(e);
  }
  python_error err;
  err.persist();
  throw err;
}

// y = x W^T (+ b);  backward: Algorithm 1 on the selected bases.  H, W: the token grid of
// a (B, n + H*W, Cin) sequence, 0: x is (B, H, W, Cin).  With save_projected the
// forward pass keeps x_hat = p(x) (Eq. 3) instead of x.
struct LinearFunction : public torch::autograd::Function<LinearFunction> {
  static Tensor forward(torch::autograd::AutogradContext* ctx, const Tensor& x, const Tensor& weight,
                        const std::optional<Tensor>& bias, int64_t k, const std::vector<int64_t>& bases,
                        bool save_projected, int64_t H, int64_t W) {
    auto& saved = ctx->saved_data;
    saved["k"] = k;
    saved["bases"] = bases;
    saved["bias"] = bias.has_value();
    saved["H"] = H;
    saved["W"] = W;
    bool projected = false;
    if (H > 0) {
      TORCH_CHECK_VALUE(x.dim() == 3 && x.size(1) >= H * W, "with a grid, x must be (B, n + H*W, Cin)");
    } else {
      TORCH_CHECK_VALUE(x.dim() == 4, "x must be (B, H, W, Cin)");
      projected = save_projected && x.is_cuda();
    }
    saved["projected"] = projected;
    if (projected) {
      const Tensor xc = x.contiguous();
      const int dt = dtype_code(xc.scalar_type()), dev = xc.get_device();
      TORCH_CHECK_TYPE(dt >= 0, "unsupported dtype ", xc.scalar_type());
      const std::vector<lbp_basis> set = unpack(bases);
      Tensor x_hat = at::empty({xc.size(0), (xc.size(1) + k - 1) / k, (xc.size(2) + k - 1) / k,
                                static_cast<int64_t>(set.size()), xc.size(3)},
                               xc.options());
      Tensor ws = bytes_on(xc, lib.status_bytes());
      const int e = lib.project(xc.data_ptr(), x_hat.data_ptr(), xc.size(0), xc.size(1), xc.size(2), xc.size(3),
                                static_cast<int>(k), set.data(), static_cast<int>(set.size()), dt, ws.data_ptr(),
                                ws.numel(), current_stream(dev));
      if (e != LBP_OK) raise_status(e, "lbp_project");
      ctx->save_for_backward({x_hat, weight});
    } else {
      ctx->save_for_backward({x, weight});
    }
    // The bias rides in the product's epilogue where that is all one type.  Otherwise (a bias
    // of another type, autocast, which casts the product's operands but not the sum's) torch's
    // rules for the two operations decide the type of y.
    const at::ScalarType dt = x.scalar_type();
    if (!bias.has_value() || (weight.scalar_type() == dt && bias->scalar_type() == dt &&
                              !at::autocast::is_autocast_enabled(x.device().type())))
      return at::linear(x, weight, bias);
    return at::matmul(x, weight.t()) + *bias;
  }

  static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx,
                                                 torch::autograd::variable_list grads) {
    at::AutoGradMode no_grad(false);
    auto& saved = ctx->saved_data;
    const auto vars = ctx->get_saved_variables();
    const std::vector<int64_t> flat = saved["bases"].toIntVector();
    const std::vector<lbp_basis> set = unpack(flat);
    const int64_t H = saved["H"].toInt(), W = saved["W"].toInt();
    const Tensor g_y = grads[0].contiguous();
    ExCall c;
    c.k = static_cast<int>(saved["k"].toInt());
    c.W = vars[1].contiguous();
    c.gw_code = dtype_code(c.W.scalar_type());
    TORCH_CHECK_TYPE(c.gw_code >= 0, "unsupported dtype ", c.W.scalar_type());
    TORCH_CHECK_VALUE(g_y.is_cuda(), "g_y must be a CUDA tensor (the library has no CPU path)");
    if (saved["bias"].toBool()) c.g_bias = at::empty({c.W.size(0)}, c.W.options());
    Tensor g_x, cls;
    int64_t n = 0;
    if (H > 0) {
      const Tensor x = vars[0].contiguous();
      const int64_t B = x.size(0);
      n = x.size(1) - H * W;
      g_x = at::empty_like(x);
      auto tokens = [&](const Tensor& t) {
        return t.as_strided({B, H, W, t.size(2)}, {t.stride(0), W * t.size(2), t.size(2), 1},
                            t.storage_offset() + n * t.size(2));
      };
      c.x = tokens(x);
      c.g_y = tokens(g_y);
      c.g_x = tokens(g_x);
      if (n == 1) {   // one class token per image: rows with the sequence's pitch, in place
        c.x_extra = x.select(1, 0);
        c.gy_extra = g_y.select(1, 0);
        c.gx_extra = g_x.select(1, 0);
      } else if (n > 1) {   // several: gathered (a few rows)
        c.x_extra = x.narrow(1, 0, n).reshape({B * n, x.size(2)});
        c.gy_extra = g_y.narrow(1, 0, n).reshape({B * n, g_y.size(2)});
        c.gx_extra = cls = at::empty({B * n, x.size(2)}, x.options());
      }
    } else {
      c.g_y = g_y;
      (saved["projected"].toBool() ? c.x_hat : c.x) = vars[0].contiguous();
    }
    const int e = run_ex(&c, set.data(), static_cast<int>(set.size()));
    TORCH_CHECK_VALUE(e >= 0, "LbpLinear: gradient, activation and weight do not fit together (shapes ",
                      g_y.sizes(), ", ", vars[0].sizes(), ", ", c.W.sizes(), "; one dtype, the current device)");
    if (e != LBP_OK) raise_status(e, "lbp_backward_ex");
    if (n > 1) g_x.narrow(1, 0, n).copy_(cls.view({g_x.size(0), n, g_x.size(2)}));
    return {H > 0 ? g_x : c.g_x, c.g_W, c.g_bias, Tensor(), Tensor(), Tensor(), Tensor(), Tensor()};
  }

  static std::vector<lbp_basis> unpack(const std::vector<int64_t>& flat) {
    std::vector<lbp_basis> v(flat.size() / 2);
    for (size_t q = 0; q < v.size(); ++q)
      v[q] = lbp_basis{static_cast<int32_t>(flat[2 * q]), static_cast<int32_t>(flat[2 * q + 1])};
    return v;
  }
};

// Whether torch's functions on a tensor of this type give tensors of it (unless the class has
// switched that off).
bool makes_subclasses(PyTypeObject* type) {
  const pybind11::object off = pybind11::module_::import("torch._C").attr("_disabled_torch_function_impl");
  return !pybind11::getattr(reinterpret_cast<PyObject*>(type), "__torch_function__", off).is(off);
}

// linear(x, weight, bias | None, k, bases, save_projected, H, W) -> y
PyObject* py_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Tensor x, weight, bias;
  int k = 0, H = 0, W = 0;
  Bases b;
  if (n != 8 || !parse_tensor(a[0], &x) || !parse_tensor(a[1], &weight) || !parse_tensor(a[2], &bias) ||
      !parse_int(a[3], &k) || k < 1 || !parse_bases(a[4], &b) || !parse_int(a[6], &H) || !parse_int(a[7], &W) ||
      !x.defined() || !weight.defined() || (H > 0) != (W > 0)) {
    PyErr_SetString(PyExc_ValueError,
                    "linear: x and weight are tensors, bases a list of (i, j) pairs, k and the grid positive");
    return nullptr;
  }
  std::vector<int64_t> flat(2 * b.r);
  for (int q = 0; q < b.r; ++q) {
    flat[2 * q] = b.v[q].i;
    flat[2 * q + 1] = b.v[q].j;
  }
  const bool projected = PyObject_IsTrue(a[5]) == 1;
  Tensor y;
  {
    pybind11::gil_scoped_release no_gil;
    y = LinearFunction::apply(x, weight, bias.defined() ? std::optional<Tensor>(bias) : std::nullopt,
                              static_cast<int64_t>(k), flat, projected, static_cast<int64_t>(H),
                              static_cast<int64_t>(W));
  }
  PyObject* out = THPVariable_Wrap(y);
  // a subclass among the operands makes the result one, as under torch's own functions
  for (int i = 0; i < 3 && out != nullptr && THPVariable_CheckExact(out); ++i)
    if (THPVariable_Check(a[i]) && !THPVariable_CheckExact(a[i]) && makes_subclasses(Py_TYPE(a[i]))) {
      PyObject* as = PyObject_CallMethod(out, "as_subclass", "O", Py_TYPE(a[i]));
      Py_DECREF(out);
      out = as;
    }
  return out;
  END_HANDLE_TH_ERRORS
}

// What a Python autograd function shows of the node: y.grad_fn.saved_tensors.
PyObject* node_saved_tensors(PyObject* self, void*) {
  HANDLE_TH_ERRORS
  using Node = torch::autograd::CppNode<LinearFunction>;
  auto* node = dynamic_cast<Node*>(reinterpret_cast<torch::autograd::THPCppFunction*>(self)->cdata.get());
  if (node == nullptr) {
    PyErr_SetString(PyExc_RuntimeError, "saved_tensors: not a node of LbpLinear");
    return nullptr;
  }
  const auto vars = node->ctx_.get_saved_variables();
  PyObject* t = PyTuple_New(static_cast<Py_ssize_t>(vars.size()));
  if (t == nullptr) return nullptr;
  for (size_t i = 0; i < vars.size(); ++i) PyTuple_SET_ITEM(t, i, THPVariable_Wrap(vars[i]));
  return t;
  END_HANDLE_TH_ERRORS
}
void register_node_type() {
  using namespace torch::autograd;
  static PyTypeObject type;
  static PyGetSetDef properties[] = {
      {const_cast<char*>("saved_tensors"), node_saved_tensors, nullptr, nullptr, nullptr},
      THP_FUNCTION_DEFAULT_PROPERTIES,
      {nullptr, nullptr, nullptr, nullptr, nullptr}};
  torch::autograd::_initFunctionPyTypeObject(type, "LbpLinearBackward", properties, nullptr);
  torch::autograd::registerCppFunction(typeid(torch::autograd::CppNode<LinearFunction>), &type);
}

// load(path of liblbp.so, LbpError)
PyObject* py_load(PyObject*, PyObject* args) {
  const char* path = nullptr;
  PyObject* err = nullptr;
  if (!PyArg_ParseTuple(args, "sO", &path, &err)) return nullptr;
  void* h = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (h == nullptr) {
    PyErr_SetString(PyExc_RuntimeError, dlerror());
    return nullptr;
  }
  const bool ok = resolve(h, "lbp_status_string", &lib.status_string) &&
                  resolve(h, "lbp_status_bytes", &lib.status_bytes) &&
                  resolve(h, "lbp_workspace_bytes", &lib.workspace_bytes) &&
                  resolve(h, "lbp_workspace_bytes_ex", &lib.workspace_bytes_ex) &&
                  resolve(h, "lbp_workspace_bytes_projected", &lib.workspace_bytes_projected) &&
                  resolve(h, "lbp_spectrum_workspace_bytes", &lib.spectrum_workspace_bytes) &&
                  resolve(h, "lbp_project", &lib.project) && resolve(h, "lbp_spectrum", &lib.spectrum) &&
                  resolve(h, "lbp_backward", &lib.backward) && resolve(h, "lbp_backward_ex", &lib.backward_ex) &&
                  resolve(h, "lbp_backward_batch", &lib.backward_batch) &&
                  resolve(h, "lbp_backward_fullrank", &lib.backward_fullrank);
  if (!ok) {
    PyErr_Format(PyExc_RuntimeError, "%s does not export what this binding calls", path);
    return nullptr;
  }
  if (error_type == nullptr) register_node_type();
  Py_INCREF(err);
  Py_XSETREF(error_type, err);
  Py_RETURN_NONE;
}

#define LBP_FAST(name, fn) \
  {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"load", py_load, METH_VARARGS, nullptr},
                         LBP_FAST("project", py_project),
                         LBP_FAST("spectrum", py_spectrum),
                         LBP_FAST("backward", py_backward),
                         LBP_FAST("backward_ex", py_backward_ex),
                         LBP_FAST("backward_batch", py_backward_batch),
                         LBP_FAST("linear", py_linear),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lbp_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lbp_torch() { return PyModule_Create(&module); }
