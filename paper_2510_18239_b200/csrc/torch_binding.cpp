// The calls of a request through the C ABI (`include/lime.h`) for torch tensors: what `binding.Lime` does per call - check the tensors,
// allocate the output, read the current stream, make the one library call - without the interpreter in between.  A request is four such
// calls with a few microseconds of GPU work each, and marshalled through ctypes they took 7 to 10 us of host time apiece, more than the
// kernels of a small batch.  Nothing is computed or kept here.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <dlfcn.h>

#include "lime.h"

namespace {

decltype(&lime_lengths_to_offsets) f_offsets;
decltype(&lime_gather_history) f_gather, f_gather_ln;
decltype(&lime_encode_user) f_encode, f_encode_ln;
decltype(&lime_precompute_candidate_links) f_precompute;
decltype(&lime_score_candidates) f_score;
decltype(&lime_score_candidates_head) f_score_head;
decltype(&lime_last_cuda_error) f_last_error;
PyObject* lime_error;                                            // binding.LimeError

struct Refused {};                                               // a Python error is set

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a torch.Tensor, got %s", Py_TYPE(o)->tp_name);
    throw Refused();
  }
  return THPVariable_Unpack(o);
}
void* pointer(const at::Tensor& t) {
  if (!t.is_cuda() || !t.is_contiguous()) {
    PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
    throw Refused();
  }
  return t.data_ptr();
}
void* pointer_or_null(PyObject* o) { return o == Py_None ? nullptr : pointer(tensor(o)); }
int64_t integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Refused();
  return v;
}
int32_t integer32(int64_t v) { return static_cast<int32_t>(v); }
lime_ctx* context(PyObject* o) { return o == Py_None ? nullptr : reinterpret_cast<lime_ctx*>(integer(o)); }

// f(a..., current stream)
template <typename F, typename... A>
void call(const char* where, F f, A... a) {
  if (f == nullptr) {
    PyErr_SetString(PyExc_RuntimeError, "the library is not loaded");
    throw Refused();
  }
  lime_status s;
  void* const st = c10::cuda::getCurrentCUDAStream().stream();
  Py_BEGIN_ALLOW_THREADS
  s = f(a..., st);
  Py_END_ALLOW_THREADS
  if (s == LIME_OK) return;
  PyObject* e = PyObject_CallFunction(lime_error, "iss", static_cast<int>(s), where, s == LIME_CUDA_ERROR ? f_last_error() : "");
  if (e != nullptr) {
    PyErr_SetObject(lime_error, e);
    Py_DECREF(e);
  }
  throw Refused();
}

template <typename Body>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, Body body) {
  if (n != want) return PyErr_Format(PyExc_TypeError, "%zd arguments instead of %zd", n, want);
  HANDLE_TH_ERRORS
  try {
    return THPVariable_Wrap(body());
  } catch (const Refused&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

// (ctx, lengths)
PyObject* lengths_to_offsets(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 2, [&] {
    const at::Tensor& len = tensor(a[1]);
    at::Tensor off = at::empty({len.numel() + 1}, len.options());
    call("lime_lengths_to_offsets", f_offsets, context(a[0]), static_cast<const int32_t*>(pointer(len)), integer32(len.numel()),
         static_cast<int32_t*>(pointer(off)));
    return off;
  });
}

// (ctx, d, table, ids, flag)
template <bool LN>
PyObject* gather(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 5, [&] {
    const at::Tensor &table = tensor(a[2]), &ids = tensor(a[3]);
    at::Tensor out = at::empty({ids.numel(), integer(a[1])}, table.options());
    call(LN ? "lime_gather_history_normalized" : "lime_gather_history", LN ? f_gather_ln : f_gather, context(a[0]),
         static_cast<const void*>(pointer(table)), table.size(0), static_cast<const int32_t*>(pointer(ids)), ids.numel(), pointer(out),
         static_cast<int32_t*>(pointer_or_null(a[4])));
    return out;
  });
}

// (ctx, ell_c, d, hist, off, link_ctx, ws)
template <bool LN>
PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 7, [&] {
    const at::Tensor &hist = tensor(a[3]), &off = tensor(a[4]), &ws = tensor(a[6]);
    const int64_t B = off.numel() - 1;
    at::Tensor ls = at::empty({B, integer(a[1]), integer(a[2])}, hist.options());
    call(LN ? "lime_encode_user_normalized" : "lime_encode_user", LN ? f_encode_ln : f_encode, context(a[0]),
         static_cast<const void*>(pointer(hist)), static_cast<const int32_t*>(pointer(off)), integer32(B), hist.size(0),
         static_cast<const float*>(pointer_or_null(a[5])), pointer(ls), pointer(ws), ws.nbytes());
    return ls;
  });
}

// (ctx, ell_c, cand_emb)
PyObject* precompute(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 3, [&] {
    const at::Tensor& emb = tensor(a[2]);
    at::Tensor out = at::empty({emb.size(0), integer(a[1])}, emb.options());
    call("lime_precompute_candidate_links", f_precompute, context(a[0]), static_cast<const void*>(pointer(emb)), emb.size(0), pointer(out));
    return out;
  });
}

// (ctx, link_states, cand_w, cand_emb, C, cand_off, cand_ids, total_cands, corpus_rows, dev_flag[, ws])
template <bool HEAD>
PyObject* score(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, HEAD ? 11 : 10, [&] {
    const at::Tensor &ls = tensor(a[1]), &w = tensor(a[2]), &emb = tensor(a[3]);
    const bool by_id = a[6] != Py_None;
    const int64_t total = a[7] != Py_None ? integer(a[7]) : by_id ? tensor(a[6]).numel() : emb.size(0);
    const int64_t rows = a[8] != Py_None ? integer(a[8]) : by_id ? emb.size(0) : 0;
    at::Tensor logits = at::empty({total}, ls.options().dtype(at::kFloat));
    const void *lp = pointer(ls), *wp = pointer(w), *ep = pointer(emb);
    const int32_t *off = static_cast<const int32_t*>(pointer_or_null(a[5])), *ids = static_cast<const int32_t*>(pointer_or_null(a[6]));
    int32_t* flag = static_cast<int32_t*>(pointer_or_null(a[9]));
    float* out = static_cast<float*>(pointer(logits));
    const int32_t B = integer32(ls.size(0)), C = integer32(integer(a[4]));
    if constexpr (HEAD) {
      const at::Tensor& ws = tensor(a[10]);
      call("lime_score_candidates_head", f_score_head, context(a[0]), lp, B, wp, ep, off, C, total, ids, rows, flag, out, pointer(ws), ws.nbytes());
    } else {
      call("lime_score_candidates", f_score, context(a[0]), lp, B, wp, ep, off, C, total, ids, rows, flag, out);
    }
    return logits;
  });
}

// (path of the library, LimeError)
PyObject* load(PyObject*, PyObject* args) {
  const char* path;
  PyObject* error;
  if (!PyArg_ParseTuple(args, "sO", &path, &error)) return nullptr;
  void* h = dlopen(path, RTLD_NOW);
  if (h == nullptr) return PyErr_Format(PyExc_RuntimeError, "%s", dlerror());
  bool all = true;
  auto get = [&](auto& f, const char* name) {
    f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(dlsym(h, name));
    all = all && f != nullptr;
  };
  get(f_offsets, "lime_lengths_to_offsets");
  get(f_gather, "lime_gather_history");
  get(f_gather_ln, "lime_gather_history_normalized");
  get(f_encode, "lime_encode_user");
  get(f_encode_ln, "lime_encode_user_normalized");
  get(f_precompute, "lime_precompute_candidate_links");
  get(f_score, "lime_score_candidates");
  get(f_score_head, "lime_score_candidates_head");
  get(f_last_error, "lime_last_cuda_error");
  if (!all) return PyErr_Format(PyExc_RuntimeError, "%s lacks an entry point", path);
  Py_INCREF(error);
  Py_XSETREF(lime_error, error);
  Py_RETURN_NONE;
}

#define LIME_FAST(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"load", load, METH_VARARGS, nullptr},
    LIME_FAST("lengths_to_offsets", &lengths_to_offsets),
    LIME_FAST("gather_history", &gather<false>),
    LIME_FAST("gather_history_normalized", &gather<true>),
    LIME_FAST("encode_user", &encode<false>),
    LIME_FAST("encode_user_normalized", &encode<true>),
    LIME_FAST("precompute_candidate_links", &precompute),
    LIME_FAST("score_candidates", &score<false>),
    LIME_FAST("score_candidates_head", &score<true>),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_binding(void) {
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr && PyModule_AddStringConstant(m, "made_for", LIME_MADE_FOR) < 0) Py_CLEAR(m);
  return m;
}
