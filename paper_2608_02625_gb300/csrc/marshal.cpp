// Native marshalling of the Python binding: torch tensors to dlm_tensor
// descriptors, torch's current stream to dlm_set_stream, and the call.
//
// Every function takes the arguments of its Python entry point and returns the
// library's status, or None when it has done nothing because an argument is
// not of the ordinary form (a plain CUDA tensor of a supported type with
// storage, on the current device; a Python int; a RefineParams): the caller
// then takes the general path in Python, which marshals what can be marshalled
// and raises what has to be raised. What it is for: through ctypes, building
// the descriptors in Python took longer on a GB300's Grace host than the work on
// the GPU of a small call (calls issued one after another: the update of 8 x 2048
// 17.6 us, of which 8.7 on the GPU, now 10.3; one sequence's attention 13.9, now
// 12.3; a first call on new tensors about 20 us shorter).
#include <Python.h>

#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#include "dlmrefine.h"

namespace {

constexpr int kMaxTensors = 12;

PyObject* g_params_type = nullptr;  // RefineParams
PyObject *s_threshold, *s_k, *s_frac, *s_mask_id, *s_prompt, *s_seq;

// The tensors of one call. Every method returns false where the general path
// has to decide.
class Call {
 public:
  // Descriptor of `o` as argument slot n (null for None when `optional`).
  bool add(PyObject* o, bool optional = false) {
    if (optional && o == Py_None) {
      ptr_[n_++] = nullptr;
      return true;
    }
    at::Tensor* t = nullptr;
    if (!plain(o, &t)) return false;
    dlm_tensor& d = desc_[n_];
    switch (t->scalar_type()) {
      case at::kBFloat16: d.dtype = DLM_BF16; break;
      case at::kFloat: d.dtype = DLM_F32; break;
      case at::kInt: d.dtype = DLM_I32; break;
      case at::kByte: d.dtype = DLM_U8; break;
      default: return false;
    }
    const int64_t nd = t->dim();
    if (nd < 1 || nd > 4) return false;
    d.data = t->numel() ? t->data_ptr() : nullptr;
    d.ndim = static_cast<int32_t>(nd);
    for (int i = 0; i < 4; ++i) {
      d.shape[i] = i < nd ? t->size(i) : 0;
      d.stride[i] = i < nd ? t->stride(i) : 0;
    }
    ptr_[n_++] = &d;
    return true;
  }

  // Device memory the call works in: any type, contiguous.
  bool workspace(PyObject* o, void** data, size_t* bytes) {
    at::Tensor* t = nullptr;
    if (!plain(o, &t) || !t->is_contiguous()) return false;
    *bytes = static_cast<size_t>(t->numel()) * t->itemsize();
    *data = *bytes ? t->data_ptr() : nullptr;
    return true;
  }

  bool params(PyObject* o, dlm_refine_params* p) {
    if (reinterpret_cast<PyObject*>(Py_TYPE(o)) != g_params_type) return false;
    double threshold, frac;
    long k, mask_id;
    if (!number(o, s_threshold, &threshold) || !number(o, s_frac, &frac) || !integer(o, s_k, &k) ||
        !integer(o, s_mask_id, &mask_id))
      return false;
    p->edit_threshold = static_cast<float>(threshold);
    p->remask_frac = static_cast<float>(frac);
    p->remask_k = static_cast<int32_t>(k);
    p->mask_id = static_cast<int32_t>(mask_id);
    return lengths(o, s_prompt, &p->prompt_lens) && lengths(o, s_seq, &p->seq_lens);
  }

  // The current stream of the tensors' device, for the library.
  bool stream() {
    if (device_ < 0 || c10::cuda::current_device() != device_) return false;
    return dlm_set_stream(c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device_)).stream()) == DLM_OK;
  }

  dlm_tensor* operator[](int i) { return ptr_[i]; }

 private:
  bool plain(PyObject* o, at::Tensor** out) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage()) return false;
    const int dev = t.get_device();
    if (device_ >= 0 && dev != device_) return false;
    device_ = dev;
    *out = const_cast<at::Tensor*>(&t);
    return true;
  }

  static bool number(PyObject* o, PyObject* name, double* v) {
    PyObject* x = PyObject_GetAttr(o, name);
    if (!x) return false;
    const bool ok = PyFloat_CheckExact(x) || PyLong_CheckExact(x);
    if (ok) *v = PyFloat_AsDouble(x);
    Py_DECREF(x);
    return ok && !PyErr_Occurred();
  }

  static bool integer(PyObject* o, PyObject* name, long* v) {
    PyObject* x = PyObject_GetAttr(o, name);
    if (!x) return false;
    const bool ok = PyLong_CheckExact(x);
    if (ok) *v = PyLong_AsLong(x);
    Py_DECREF(x);
    return ok && !PyErr_Occurred() && *v >= INT32_MIN && *v <= INT32_MAX;
  }

  bool lengths(PyObject* o, PyObject* name, const int32_t** v) {
    PyObject* x = PyObject_GetAttr(o, name);
    if (!x) return false;
    at::Tensor* t = nullptr;
    const bool ok = plain(x, &t) && t->scalar_type() == at::kInt && t->is_contiguous();
    if (ok) *v = static_cast<const int32_t*>(t->data_ptr());
    Py_DECREF(x);  // the RefineParams keeps it
    return ok;
  }

  dlm_tensor desc_[kMaxTensors];
  dlm_tensor* ptr_[kMaxTensors];
  int n_ = 0, device_ = -1;
};

bool as_int32(PyObject* o, int32_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  const long x = PyLong_AsLong(o);
  if (PyErr_Occurred() || x < INT32_MIN || x > INT32_MAX) return false;
  *v = static_cast<int32_t>(x);
  return true;
}

PyObject* general_path() {
  PyErr_Clear();
  Py_RETURN_NONE;
}

// body(call, status): false for the general path. No C++ exception leaves.
template <typename Body>
PyObject* run(Py_ssize_t n, Py_ssize_t want, Body body) {
  if (n != want) return general_path();
  int status = 0;
  try {
    Call c;
    if (!body(c, &status)) return general_path();
  } catch (...) {
    return general_path();
  }
  return PyLong_FromLong(status);
}

// The library call without the interpreter lock (a launch may wait for queue space).
template <typename F>
int unlocked(F f) {
  int status;
  Py_BEGIN_ALLOW_THREADS status = f();
  Py_END_ALLOW_THREADS return status;
}

bool add_all(Call& c, PyObject* const* a, int first, int last) {
  for (int i = first; i < last; ++i)
    if (!c.add(a[i])) return false;
  return true;
}

PyObject* bidir_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 5, [&](Call& c, int* st) {
    if (!add_all(c, a, 0, 3) || !c.add(a[3], true) || !c.add(a[4]) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_bidir_attn(c[0], c[1], c[2], c[3], c[4]); });
    return true;
  });
}

PyObject* attn_masked(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 8, [&](Call& c, int* st) {
    int32_t mode, block;
    if (!add_all(c, a, 0, 3) || !c.add(a[3], true) || !c.add(a[4], true) || !as_int32(a[5], &mode) ||
        !as_int32(a[6], &block) || !c.add(a[7]) || !c.stream())
      return false;
    *st = unlocked([&] { return dlm_attn_masked(c[0], c[1], c[2], c[3], c[4], mode, block, c[5]); });
    return true;
  });
}

PyObject* vocab_confidence(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 4, [&](Call& c, int* st) {
    if (!add_all(c, a, 0, 4) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_vocab_confidence(c[0], c[1], c[2], c[3]); });
    return true;
  });
}

PyObject* token_prob(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 4, [&](Call& c, int* st) {
    if (!add_all(c, a, 0, 4) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_token_prob(c[0], c[1], c[2], c[3]); });
    return true;
  });
}

// tokens, mask, argmax, conf, params, new_tokens, new_mask, n_edits
PyObject* refine_update(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 8, [&](Call& c, int* st) {
    dlm_refine_params p;
    if (!add_all(c, a, 0, 4) || !c.params(a[4], &p) || !add_all(c, a, 5, 8) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_refine_update(c[0], c[1], c[2], c[3], &p, c[4], c[5], c[6]); });
    return true;
  });
}

// tokens, mask, argmax, conf, tok_prob, params, new_tokens, new_mask, n_edits
PyObject* refine_update_ranked(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 9, [&](Call& c, int* st) {
    dlm_refine_params p;
    if (!add_all(c, a, 0, 5) || !c.params(a[5], &p) || !add_all(c, a, 6, 9) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_refine_update_ranked(c[0], c[1], c[2], c[3], c[4], &p, c[5], c[6], c[7]); });
    return true;
  });
}

// logits, tokens, mask, params, argmax, conf, lse, new_tokens, new_mask, n_edits, workspace
PyObject* refine_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 11, [&](Call& c, int* st) {
    dlm_refine_params p;
    void* ws;
    size_t bytes;
    if (!add_all(c, a, 0, 3) || !c.params(a[3], &p) || !add_all(c, a, 4, 10) || !c.workspace(a[10], &ws, &bytes) ||
        !c.stream())
      return false;
    *st = unlocked([&] {
      return dlm_refine_step(c[0], c[1], c[2], &p, c[3], c[4], c[5], c[6], c[7], c[8], ws, bytes);
    });
    return true;
  });
}

// logits, tokens, mask, params, argmax, conf, lse, new_tokens, new_mask, n_edits
PyObject* refine_step_static(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 10, [&](Call& c, int* st) {
    dlm_refine_params p;
    if (!add_all(c, a, 0, 3) || !c.params(a[3], &p) || !add_all(c, a, 4, 10) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_refine_step_static(c[0], c[1], c[2], &p, c[3], c[4], c[5], c[6], c[7], c[8]); });
    return true;
  });
}

// hidden, weight, argmax, conf, lse, workspace
PyObject* lmhead_confidence(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 6, [&](Call& c, int* st) {
    void* ws;
    size_t bytes;
    if (!add_all(c, a, 0, 5) || !c.workspace(a[5], &ws, &bytes) || !c.stream()) return false;
    *st = unlocked([&] { return dlm_lmhead_confidence(c[0], c[1], c[2], c[3], c[4], ws, bytes); });
    return true;
  });
}

// handle (a non-zero int), device index
PyObject* loop_launch(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(n, 2, [&](Call&, int* st) {
    int32_t dev;
    if (!PyLong_CheckExact(a[0]) || !as_int32(a[1], &dev)) return false;
    void* handle = PyLong_AsVoidPtr(a[0]);
    if (!handle || c10::cuda::current_device() != dev ||
        dlm_set_stream(c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(dev)).stream()) != DLM_OK)
      return false;
    *st = unlocked([&] { return dlm_loop_launch(static_cast<dlm_loop*>(handle)); });
    return true;
  });
}

PyObject* set_params_type(PyObject*, PyObject* type) {
  Py_XDECREF(g_params_type);
  g_params_type = Py_NewRef(type);
  Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(bidir_attn),
                         FAST(attn_masked),
                         FAST(vocab_confidence),
                         FAST(token_prob),
                         FAST(refine_update),
                         FAST(refine_update_ranked),
                         FAST(refine_step),
                         FAST(refine_step_static),
                         FAST(lmhead_confidence),
                         FAST(loop_launch),
                         {"set_params_type", set_params_type, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) {
  s_threshold = PyUnicode_InternFromString("edit_threshold");
  s_k = PyUnicode_InternFromString("remask_k");
  s_frac = PyUnicode_InternFromString("remask_frac");
  s_mask_id = PyUnicode_InternFromString("mask_id");
  s_prompt = PyUnicode_InternFromString("prompt_lens");
  s_seq = PyUnicode_InternFromString("seq_lens");
  return PyModule_Create(&module);
}
