// One call of cos_verify_run on device tensors, from Python: checks, outputs and arguments without going through the interpreter.
//
// What bounds small runs called from Python is the call itself: with its steps in Python one row of 5 x 2 x 32000 took 14.8 us a call, of
// which the device needs 12.4; now it takes 12.8.  Whatever does not fit here (other outputs, tensors that are not plain, anything to
// complain about) returns None, and the caller goes the long way, which has the messages.
#include <ATen/ops/as_strided.h>
#include <ATen/ops/empty.h>
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <new>

#include "cos_verify.h"

namespace {

using RunFn = cos_status (*)(cos_verify_ctx*, const cos_verify_args*, void*);

struct Callee {  // a context and what its calls have to look like
  RunFn run;
  cos_verify_ctx* ctx;
  int64_t n, positions, vocab;
  at::ScalarType dtype;
};
constexpr const char* kCapsule = "cos_verify.callee";

void drop(PyObject* capsule) { delete static_cast<Callee*>(PyCapsule_GetPointer(capsule, kCapsule)); }

// callee(address of cos_verify_run, address of the context, n, gamma + 1, vocab, dtype)
PyObject* callee(PyObject*, PyObject* args) {
  unsigned long long run = 0, ctx = 0;
  long long n = 0, positions = 0, vocab = 0;
  int dtype = 0;
  if (!PyArg_ParseTuple(args, "KKLLLi", &run, &ctx, &n, &positions, &vocab, &dtype)) return nullptr;
  Callee* c = new (std::nothrow) Callee{reinterpret_cast<RunFn>(run), reinterpret_cast<cos_verify_ctx*>(ctx), n, positions, vocab,
                                        dtype == COS_DTYPE_F32 ? at::kFloat : (dtype == COS_DTYPE_BF16 ? at::kBFloat16 : at::kHalf)};
  if (!c) return PyErr_NoMemory();
  PyObject* capsule = PyCapsule_New(c, kCapsule, drop);
  if (!capsule) delete c;
  return capsule;
}

// A plain int32 device tensor that is contiguous, with anything in it.
bool plain_int32(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.scalar_type() == at::kInt && t.is_cuda() && t.is_contiguous();
}
bool as_word(PyObject* o, unsigned long long* v) {
  if (!PyLong_Check(o)) return false;
  *v = PyLong_AsUnsignedLongLongMask(o);
  return true;
}

// run(callee, logits, drafts, proposer, seed, offset, row_base, flags, bonus_model, offset_device): the outputs, or the status of a call
// that failed, or None.
PyObject* run(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  if (nargs != 10) {
    PyErr_SetString(PyExc_TypeError, "run takes 10 arguments");
    return nullptr;
  }
  const Callee* c = static_cast<Callee*>(PyCapsule_GetPointer(a[0], kCapsule));
  if (!c) return nullptr;
  HANDLE_TH_ERRORS  // (what the allocation of the outputs raises is what torch raises from Python)
  {
    if (!THPVariable_CheckExact(a[1]) || !plain_int32(a[3])) Py_RETURN_NONE;
    const at::Tensor &logits = THPVariable_Unpack(a[1]), &proposer = THPVariable_Unpack(a[3]);
    if (!logits.is_cuda() || logits.layout() != at::kStrided || logits.dim() != 4 || logits.scalar_type() != c->dtype) Py_RETURN_NONE;
    const int64_t B = logits.size(1), P = c->positions;
    if (logits.size(0) != c->n || logits.size(2) != P || logits.size(3) != c->vocab || logits.stride(3) != 1 || B < 1 || B > INT32_MAX) Py_RETURN_NONE;
    cos_verify_args v = {};
    unsigned long long row_base = 0, flags = 0, seed = 0, offset = 0;
    if (!as_word(a[4], &seed) || !as_word(a[5], &offset) || !as_word(a[6], &row_base) || !as_word(a[7], &flags)) Py_RETURN_NONE;
    if (proposer.dim() == 2) {
      if (proposer.size(0) != B || proposer.size(1) != P) Py_RETURN_NONE;
      flags |= COS_RUN_PROPOSER_PER_POSITION;
    } else if (proposer.numel() != B) {
      Py_RETURN_NONE;
    }
    if (a[8] != Py_None) {
      const long model = PyLong_Check(a[8]) ? PyLong_AsLong(a[8]) : -2;
      if (model < INT32_MIN || model > INT32_MAX || (model == -1 && PyErr_Occurred()) || !PyLong_Check(a[8])) {
        PyErr_Clear();
        Py_RETURN_NONE;
      }
      if (model >= 0) {
        flags |= COS_RUN_BONUS_FROM_MODEL;
        v.bonus_model = static_cast<int32_t>(model);
      }
    }
    if (a[2] != Py_None) {
      if (!THPVariable_CheckExact(a[2])) Py_RETURN_NONE;
      const at::Tensor& drafts = THPVariable_Unpack(a[2]);
      if (drafts.numel() > 0) {
        if (!plain_int32(a[2])) Py_RETURN_NONE;
        v.draft_tokens = static_cast<const int32_t*>(drafts.data_ptr());
      }
    }
    if (a[9] != Py_None) {
      if (!THPVariable_CheckExact(a[9])) Py_RETURN_NONE;
      const at::Tensor& t = THPVariable_Unpack(a[9]);
      if (t.scalar_type() != at::kLong || !t.is_cuda()) Py_RETURN_NONE;
      v.offset_device = static_cast<const uint64_t*>(t.data_ptr());
    }
    v.logits = logits.data_ptr();
    v.stride_model = logits.stride(0);
    v.stride_row = logits.stride(1);
    v.stride_pos = logits.stride(2);
    v.proposer = static_cast<const int32_t*>(proposer.data_ptr());
    v.batch = static_cast<int32_t>(B);
    v.flags = static_cast<int32_t>(flags);
    v.row_base = static_cast<int64_t>(row_base);
    v.seed = seed;
    v.offset = offset;
    // one allocation for the small outputs
    const at::Tensor buf = at::empty({B * (P + 3)}, logits.options().dtype(at::kInt).requires_grad(false));
    int32_t* at0 = static_cast<int32_t*>(buf.data_ptr());
    v.accept_count = at0;
    v.row_status = reinterpret_cast<uint32_t*>(at0 + B);
    v.bonus_prob = reinterpret_cast<float*>(at0 + 2 * B);
    v.out_tokens = at0 + 3 * B;
    void* stream = c10::cuda::getCurrentCUDAStream(logits.get_device()).stream();
    cos_status st;
    Py_BEGIN_ALLOW_THREADS
    st = c->run(c->ctx, &v, stream);
    Py_END_ALLOW_THREADS
    if (st != COS_OK) return PyLong_FromLong(st);
    const at::Tensor outs[4] = {at::as_strided(buf, {B}, {1}, 0), at::as_strided(buf, {B, P}, {P, 1}, 3 * B), at::as_strided(buf, {B}, {1}, B),
                                at::as_strided(buf, {B}, {1}, 2 * B).view(at::kFloat)};
    static PyObject* const names[4] = {PyUnicode_InternFromString("accept_count"), PyUnicode_InternFromString("out_tokens"),
                                       PyUnicode_InternFromString("row_status"), PyUnicode_InternFromString("bonus_prob")};
    PyObject* d = PyDict_New();
    for (int k = 0; d && k < 4; ++k) {
      PyObject* t = THPVariable_Wrap(outs[k]);
      if (!t || PyDict_SetItem(d, names[k], t) != 0) Py_CLEAR(d);
      Py_XDECREF(t);
    }
    return d;
  }
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"callee", callee, METH_VARARGS, "a context, for run"},
                         {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(run)), METH_FASTCALL, "one call of cos_verify_run"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() { return PyModule_Create(&module); }
