// The per-step calls of the binding as a CPython extension: the same checks as binding.py makes, on the tensors themselves instead of through
// attribute lookups, which bounded small steps and the decode loop's critical path: 16 rows of 4,096 13.1 -> 11.9 us a step, 32 iterations of
// one window 2,058 -> 1,655 us, 16 of sixteen windows 1,130 -> 934 us.
// Whatever is not the ordinary case (another type, a check that fails) is handed back untouched
// and takes the way through binding.py, which also words the errors.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAFunctions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/sjd.h"

namespace {

using StepFn = decltype(&sjd_step);
using AdvanceFn = decltype(&sjd_window_advance);
StepFn g_step = nullptr;
AdvanceFn g_advance = nullptr;
PyObject *s_tok_prob, *s_ids, *s_vals, *s_cnt;

constexpr long kHandBack = 1;  // (no code of the library: those are 0 and below)

struct HandBack {};

const at::Tensor& tensor_of(PyObject* o) {
  if (!THPVariable_CheckExact(o)) throw HandBack{};
  return THPVariable_Unpack(o);
}
// the address of a contiguous CUDA tensor of the given type
void* array_of(PyObject* o, at::ScalarType type) {
  const at::Tensor& t = tensor_of(o);
  if (!t.is_cuda() || t.scalar_type() != type || !t.is_contiguous()) throw HandBack{};
  return t.data_ptr();
}
void* optional_array_of(PyObject* o, at::ScalarType type) { return o == Py_None ? nullptr : array_of(o, type); }

void* attribute_array(PyObject* o, PyObject* name, at::ScalarType type) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) {
    PyErr_Clear();
    throw HandBack{};
  }
  void* p = nullptr;
  try {
    p = array_of(v, type);  // (the object keeps the tensor alive as well)
  } catch (...) {
    Py_DECREF(v);
    throw;
  }
  Py_DECREF(v);
  return p;
}
sjd_probs probs_of(PyObject* o) {
  sjd_probs p;
  p.tok_prob = static_cast<float*>(attribute_array(o, s_tok_prob, at::kFloat));
  p.ids = static_cast<int32_t*>(attribute_array(o, s_ids, at::kInt));
  p.vals = static_cast<float*>(attribute_array(o, s_vals, at::kFloat));
  p.cnt = static_cast<int32_t*>(attribute_array(o, s_cnt, at::kInt));
  return p;
}
uint64_t word_of(PyObject* o) {
  if (!PyLong_CheckExact(o)) throw HandBack{};
  const uint64_t v = PyLong_AsUnsignedLongLongMask(o);
  if (v == (uint64_t)-1 && PyErr_Occurred()) {
    PyErr_Clear();
    throw HandBack{};
  }
  return v;
}
// A CUDA tensor's device is current as long as this lives: a process that drives several GPUs need not switch itself.
class OnDeviceOf {
 public:
  explicit OnDeviceOf(const at::Tensor& t) {
    if (!t.is_cuda()) throw HandBack{};
    const c10::DeviceIndex current = c10::cuda::current_device();
    if (t.get_device() == current) return;
    c10::cuda::set_device(t.get_device());
    before_ = current;
  }
  ~OnDeviceOf() {
    if (before_ < 0) return;
    try {
      c10::cuda::set_device(before_);
    } catch (...) {  // (it was current before: the next CUDA call says what has happened to it)
    }
  }
  OnDeviceOf(const OnDeviceOf&) = delete;
  OnDeviceOf& operator=(const OnDeviceOf&) = delete;

 private:
  c10::DeviceIndex before_ = -1;
};

// step(params address, cond, uncond, drafts, draft_probs, seed, accept_len, tokens, out_probs)
PyObject* py_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9) {
    PyErr_SetString(PyExc_TypeError, "step() takes 9 arguments");
    return nullptr;
  }
  long code = kHandBack;
  try {
    const sjd_params* const params = reinterpret_cast<const sjd_params*>(word_of(a[0]));
    const at::Tensor& cond = tensor_of(a[1]);
    const OnDeviceOf on(cond);
    const void* uncond = nullptr;
    if (a[2] != Py_None) {
      const at::Tensor& u = tensor_of(a[2]);
      if (u.scalar_type() != cond.scalar_type() || u.device() != cond.device() || u.sizes() != cond.sizes() || u.strides() != cond.strides())
        throw HandBack{};
      uncond = u.data_ptr();
    }
    const int32_t* const drafts = static_cast<const int32_t*>(optional_array_of(a[3], at::kInt));
    sjd_probs q{}, out;
    if (a[4] != Py_None) q = probs_of(a[4]);
    const uint64_t seed = word_of(a[5]);
    int32_t* const accept_len = static_cast<int32_t*>(optional_array_of(a[6], at::kInt));
    int32_t* const tokens = static_cast<int32_t*>(optional_array_of(a[7], at::kInt));
    out = probs_of(a[8]);
    const void* const c = cond.data_ptr();
    const bool has_q = a[4] != Py_None;
    Py_BEGIN_ALLOW_THREADS
    code = g_step(c, uncond, drafts, has_q ? &q : nullptr, params, seed, accept_len, tokens, &out);
    Py_END_ALLOW_THREADS
  } catch (const HandBack&) {
  } catch (const std::exception&) {  // (a tensor without storage: the ordinary way says so)
  }
  return PyLong_FromLong(code);
}

// advance(params address, n_total, seed, accept_len, step_tokens, step_probs, win_len, pos_base, iteration, next_drafts, next_probs,
//         committed, n_committed)
PyObject* py_advance(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 13) {
    PyErr_SetString(PyExc_TypeError, "advance() takes 13 arguments");
    return nullptr;
  }
  long code = kHandBack;
  try {
    const sjd_params* const params = reinterpret_cast<const sjd_params*>(word_of(a[0]));
    if (!PyLong_CheckExact(a[1])) throw HandBack{};
    int overflow = 0;
    const long total = PyLong_AsLongAndOverflow(a[1], &overflow);
    if (overflow != 0 || total != (int32_t)total) throw HandBack{};
    const uint64_t seed = word_of(a[2]);
    auto words = [&](int i) { return static_cast<int32_t*>(optional_array_of(a[i], at::kInt)); };
    const OnDeviceOf on(tensor_of(a[4]));
    sjd_probs step = probs_of(a[5]), next = probs_of(a[10]);
    int32_t *const acc = words(3), *const tok = words(4), *const win = words(6), *const pos = words(7), *const iter = words(8), *const drafts = words(9),
                   *const committed = words(11), *const count = words(12);
    Py_BEGIN_ALLOW_THREADS
    code = g_advance(params, (int32_t)total, seed, acc, tok, &step, win, pos, iter, drafts, &next, committed, count);
    Py_END_ALLOW_THREADS
  } catch (const HandBack&) {
  } catch (const std::exception&) {
  }
  return PyLong_FromLong(code);
}

// set_entries(step, advance): addresses of the loaded library's functions
PyObject* py_set_entries(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2) {
    PyErr_SetString(PyExc_TypeError, "set_entries() takes 2 arguments");
    return nullptr;
  }
  const uint64_t step = PyLong_AsUnsignedLongLong(a[0]), advance = PyLong_AsUnsignedLongLong(a[1]);
  if (PyErr_Occurred()) return nullptr;
  g_step = reinterpret_cast<StepFn>(step);
  g_advance = reinterpret_cast<AdvanceFn>(advance);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_step)), METH_FASTCALL, nullptr},
    {"advance", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_advance)), METH_FASTCALL, nullptr},
    {"set_entries", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_set_entries)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  s_tok_prob = PyUnicode_InternFromString("tok_prob");
  s_ids = PyUnicode_InternFromString("ids");
  s_vals = PyUnicode_InternFromString("vals");
  s_cnt = PyUnicode_InternFromString("cnt");
  return PyModule_Create(&module);
}
