// Python side of the C ABI: argument marshalling in native code.
//
// A step of a few rows takes 4 - 5 us on the GPU, less than Python needs to read twelve tensors' addresses and fill
// fly_verify_args_t through ctypes (7.5 us a call in all).  These functions do the same from C++: they read the
// tensors in place, fill the struct on the stack and call the library (0.5 us on top of the launch).  They keep
// nothing: no pointer, shape or check outlives the call.
//
// Reading a tensor may throw (a nested or sparse one has no strides or storage, a functorch wrapper no data): every
// function runs inside guarded(), which turns that into the Python exception that the same access raises there.
//
// The library itself stays free of torch types; its entry points are handed in by address (init), so that there is
// one copy of it in the process.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/Context.h>
#include <ATen/EmptyTensor.h>
#include <ATen/detail/CUDAHooksInterface.h>
#include <ATen/ops/empty.h>
#include <ATen/record_function.h>
#include <c10/core/DeviceGuard.h>
#include <c10/core/impl/LocalDispatchKeySet.h>

#include "fly_verify.h"

namespace {

struct Api {
  decltype(&fly_verify_run) run;
  decltype(&fly_verify_run_host) run_host;
  decltype(&fly_verify_reduce_shard) reduce_shard;
  decltype(&fly_verify_run_partials) run_partials;
  decltype(&fly_verify_run_static) run_static;
  decltype(&fly_pld_draft) pld_draft;
} api;

// Address of a tensor's storage; None is a null pointer.  Anything else that has data_ptr() is asked for it.
bool address(PyObject* o, void** p) {
  *p = nullptr;
  if (o == Py_None) return true;
  if (THPVariable_Check(o)) {
    *p = THPVariable_Unpack(o).data_ptr();
    return true;
  }
  PyObject* r = PyObject_CallMethod(o, "data_ptr", nullptr);
  if (!r) return false;
  *p = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !(*p == nullptr && PyErr_Occurred());
}

bool attribute(PyObject* o, PyObject* name, void** p) {
  struct Owned {
    PyObject* v;
    ~Owned() { Py_XDECREF(v); }
  } owned{PyObject_GetAttr(o, name)};
  return owned.v && address(owned.v, p);
}

bool as_text(PyObject* o, const char* what) { return PyUnicode_Check(o) && PyUnicode_CompareWithASCIIString(o, what) == 0; }

bool number(PyObject* o, double* v) {
  if (PyFloat_CheckExact(o)) {
    *v = PyFloat_AS_DOUBLE(o);
    return true;
  }
  PyObject* f = PyNumber_Float(o);  // as float(o) does
  if (!f) return false;
  *v = PyFloat_AS_DOUBLE(f);
  Py_DECREF(f);
  return true;
}
bool integer(PyObject* o, long long* v) {
  if (PyLong_CheckExact(o)) {
    *v = PyLong_AsLongLong(o);
  } else {  // as int(o) does
    PyObject* i = PyNumber_Long(o);
    if (!i) return false;
    *v = PyLong_AsLongLong(i);
    Py_DECREF(i);
  }
  return !(*v == -1 && PyErr_Occurred());
}
template <typename T>
bool integer_as(PyObject* o, T* v) {
  long long x;
  if (!integer(o, &x)) return false;
  *v = (T)x;
  return true;
}

bool expect(bool ok, const char* what) {
  if (!ok) PyErr_SetString(PyExc_AssertionError, what);
  return ok;
}

PyObject *s_accept_len, *s_rollback, *s_out_tokens, *s_target_argmax, *s_entropy, *s_row_flags, *s_state;

bool output_buffers(PyObject* out, bool carry, fly_verify_args_t* a) {
  void* state;
  if (!attribute(out, s_accept_len, (void**)&a->accept_len) || !attribute(out, s_rollback, (void**)&a->rollback) ||
      !attribute(out, s_out_tokens, (void**)&a->out_tokens) || !attribute(out, s_target_argmax, (void**)&a->target_argmax) ||
      !attribute(out, s_entropy, (void**)&a->entropy) || !attribute(out, s_row_flags, (void**)&a->row_flags) ||
      !attribute(out, s_state, &state))
    return false;
  a->state_in = carry ? (const fly_state_t*)state : nullptr;
  a->state_out = (fly_state_t*)state;
  return true;
}

// theta, W, theta unit and boundary of a round
bool rule(PyObject* theta, PyObject* W, PyObject* unit, PyObject* boundary, fly_verify_args_t* a) {
  if (!number(theta, &a->theta) || !integer_as(W, &a->W)) return false;
  a->theta_unit = as_text(unit, "nats") ? FLY_THETA_NATS : FLY_THETA_NORMALIZED;
  a->boundary = as_text(boundary, "carry") ? FLY_BOUNDARY_CARRY : FLY_BOUNDARY_REJECT;
  return true;
}

bool enough(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return n == want;
}

// Other threads run while this lives (taken back on every way out, an exception among them).
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};

// Whether at::empty is nothing but an allocation here: no dispatch mode, tracing or transform in this thread, no profiler, no fill.
bool plain_empty() {
  return (c10::impl::tls_local_dispatch_key_set().included_ - c10::default_included_set).empty() && !at::hasCallbacks() &&
         !(at::globalContext().deterministicAlgorithms() && at::globalContext().deterministicFillUninitializedMemory());
}

PyObject* status(fly_status_t s) { return PyLong_FromLong((long)s); }

// init(run, run_host, reduce_shard, run_partials, run_static, pld_draft): addresses of the library's entry points
PyObject* py_init(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 6)) return nullptr;
  void* p[6];
  for (int i = 0; i < 6; ++i) {
    p[i] = PyLong_AsVoidPtr(v[i]);
    if (!p[i] && PyErr_Occurred()) return nullptr;
  }
  api.run = (decltype(api.run))p[0];
  api.run_host = (decltype(api.run_host))p[1];
  api.reduce_shard = (decltype(api.reduce_shard))p[2];
  api.run_partials = (decltype(api.run_partials))p[3];
  api.run_static = (decltype(api.run_static))p[4];
  api.pld_draft = (decltype(api.pld_draft))p[5];
  Py_RETURN_NONE;
}

// fill(args, B, K, draft, accept_len, out_tokens, logits, row_stride, hidden, weight, theta, theta_unit, W, boundary,
//      state_in, state_out, rollback, target_argmax, entropy, row_flags, target_tokens, temperature, inputs_ready)
PyObject* py_fill(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 23)) return nullptr;
  fly_verify_args_t* a = (fly_verify_args_t*)PyLong_AsVoidPtr(v[0]);
  if (!a) return nullptr;
  if (!integer_as(v[1], &a->B) || !integer_as(v[2], &a->K) || !address(v[3], (void**)&a->draft) ||
      !address(v[4], (void**)&a->accept_len) || !address(v[5], (void**)&a->out_tokens) || !address(v[6], (void**)&a->logits) ||
      !integer_as(v[7], &a->row_stride) || !address(v[8], (void**)&a->hidden) || !address(v[9], (void**)&a->weight) ||
      !rule(v[10], v[12], v[11], v[13], a) || !address(v[14], (void**)&a->state_in) ||
      !address(v[15], (void**)&a->state_out) || !address(v[16], (void**)&a->rollback) ||
      !address(v[17], (void**)&a->target_argmax) || !address(v[18], (void**)&a->entropy) ||
      !address(v[19], (void**)&a->row_flags) || !address(v[20], (void**)&a->target_tokens) || !number(v[21], &a->temperature))
    return nullptr;
  const int ready = PyObject_IsTrue(v[22]);
  if (ready < 0) return nullptr;
  a->inputs_ready = ready;
  Py_RETURN_NONE;
}

// verify(handle, vocab, logits, draft, out, theta, W, theta_unit, boundary, stream, host, temperature, inputs_ready)
PyObject* py_verify(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 13)) return nullptr;
  fly_verify_t* h = (fly_verify_t*)PyLong_AsVoidPtr(v[0]);
  if (!h && PyErr_Occurred()) return nullptr;
  long long vocab;
  fly_verify_args_t a = {};
  if (!integer(v[1], &vocab) || !expect(THPVariable_Check(v[2]), "logits is a tensor")) return nullptr;
  const at::Tensor& logits = THPVariable_Unpack(v[2]);
  if (logits.dim() != 3) {
    PyErr_SetString(PyExc_ValueError, "logits is [B, K+1, V]");
    return nullptr;
  }
  const int64_t B = logits.size(0), K1 = logits.size(1), V = logits.size(2);
  if (!expect(V == vocab && logits.stride(2) == 1 && logits.stride(0) == K1 * logits.stride(1),
              "logits is [B, K+1, vocab] with rows at one stride"))
    return nullptr;
  a.B = (int32_t)B;
  a.K = (int32_t)(K1 - 1);
  a.row_stride = logits.stride(1);
  void* stream;
  if (!address(v[2], (void**)&a.logits) || !address(v[3], (void**)&a.draft) || !rule(v[5], v[6], v[7], v[8], &a) ||
      !output_buffers(v[4], a.boundary == FLY_BOUNDARY_CARRY, &a) || !number(v[11], &a.temperature))
    return nullptr;
  stream = PyLong_AsVoidPtr(v[9]);
  const int host = PyObject_IsTrue(v[10]), ready = PyObject_IsTrue(v[12]);
  if (PyErr_Occurred()) return nullptr;
  a.inputs_ready = ready;
  fly_status_t s;
  {
    Unlocked unlocked;
    s = host ? api.run_host(h, &a, stream) : api.run(h, &a, stream);
  }
  return status(s);
}

// verify_fused(handle, vocab, vocab_major, hidden, weight, draft, out, theta, W, theta_unit, boundary, stream, host,
//              temperature)
PyObject* py_verify_fused(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 14)) return nullptr;
  fly_verify_t* h = (fly_verify_t*)PyLong_AsVoidPtr(v[0]);
  if (!h && PyErr_Occurred()) return nullptr;
  long long vocab;
  fly_verify_args_t a = {};
  if (!integer(v[1], &vocab) ||
      !expect(THPVariable_Check(v[3]) && THPVariable_Check(v[4]) && THPVariable_Check(v[5]), "hidden, weight and draft are tensors"))
    return nullptr;
  const at::Tensor &hidden = THPVariable_Unpack(v[3]), &weight = THPVariable_Unpack(v[4]), &draft = THPVariable_Unpack(v[5]);
  if (draft.dim() != 2 || hidden.dim() != 2 || weight.dim() != 2) {
    PyErr_SetString(PyExc_ValueError, "hidden is [B*(K+1), D], weight 2-D and draft [B, K]");
    return nullptr;
  }
  const int64_t B = draft.size(0), K = draft.size(1), rows = hidden.size(0), D = hidden.size(1);
  const int major = PyObject_IsTrue(v[2]);
  if (!expect(rows == B * (K + 1), "hidden is [B*(K+1), D]") ||
      !expect(weight.size(0) == (major ? vocab : D) && weight.size(1) == (major ? D : vocab), "weight does not fit hidden and vocab") ||
      !expect(hidden.is_contiguous() && weight.is_contiguous(), "hidden and weight are contiguous"))
    return nullptr;
  a.B = (int32_t)B;
  a.K = (int32_t)K;
  if (!address(v[3], (void**)&a.hidden) || !address(v[4], (void**)&a.weight) || !address(v[5], (void**)&a.draft) ||
      !rule(v[7], v[8], v[9], v[10], &a) || !output_buffers(v[6], a.boundary == FLY_BOUNDARY_CARRY, &a) ||
      !number(v[13], &a.temperature))
    return nullptr;
  void* stream = PyLong_AsVoidPtr(v[11]);
  const int host = PyObject_IsTrue(v[12]);
  if (PyErr_Occurred()) return nullptr;
  fly_status_t s;
  {
    Unlocked unlocked;
    s = host ? api.run_host(h, &a, stream) : api.run(h, &a, stream);
  }
  return status(s);
}

// reduce_shard(handle, vocab, logits, vocab_offset, partial_out, stream, temperature)
PyObject* py_reduce_shard(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 7)) return nullptr;
  fly_verify_t* h = (fly_verify_t*)PyLong_AsVoidPtr(v[0]);
  if (!h && PyErr_Occurred()) return nullptr;
  long long vocab, offset;
  if (!integer(v[1], &vocab) || !expect(THPVariable_Check(v[2]), "logits is a tensor")) return nullptr;
  const at::Tensor& logits = THPVariable_Unpack(v[2]);
  if (!expect(logits.dim() >= 2 && logits.size(1) == vocab && logits.stride(1) == 1, "logits is [rows, vocab]")) return nullptr;
  void *src, *dst;
  double temperature;
  if (!address(v[2], &src) || !integer(v[3], &offset) || !address(v[4], &dst) || !number(v[6], &temperature)) return nullptr;
  void* stream = PyLong_AsVoidPtr(v[5]);
  if (PyErr_Occurred()) return nullptr;
  const int64_t rows = logits.size(0), stride = logits.stride(0);
  fly_status_t s;
  {
    Unlocked unlocked;
    s = api.reduce_shard(h, (int32_t)rows, src, stride, (int32_t)offset, temperature, (fly_partial_t*)dst, stream);
  }
  return status(s);
}

// run(handle, args, stream, host)
PyObject* py_run(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 4)) return nullptr;
  fly_verify_t* h = (fly_verify_t*)PyLong_AsVoidPtr(v[0]);
  fly_verify_args_t* a = (fly_verify_args_t*)PyLong_AsVoidPtr(v[1]);
  void* stream = PyLong_AsVoidPtr(v[2]);
  const int host = PyObject_IsTrue(v[3]);
  if (PyErr_Occurred()) return nullptr;
  fly_status_t s;
  {
    Unlocked unlocked;
    s = host ? api.run_host(h, a, stream) : api.run(h, a, stream);
  }
  return status(s);
}

// run_partials(handle, args, partials, world, total_vocab, stream)
PyObject* py_run_partials(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 6)) return nullptr;
  fly_verify_t* h = (fly_verify_t*)PyLong_AsVoidPtr(v[0]);
  fly_verify_args_t* a = (fly_verify_args_t*)PyLong_AsVoidPtr(v[1]);
  void* partials;
  int32_t world, total;
  if (PyErr_Occurred() || !address(v[2], &partials) || !integer_as(v[3], &world) || !integer_as(v[4], &total)) return nullptr;
  void* stream = PyLong_AsVoidPtr(v[5]);
  if (PyErr_Occurred()) return nullptr;
  fly_status_t s;
  {
    Unlocked unlocked;
    s = api.run_partials(h, a, (const fly_partial_t*)partials, world, total, stream);
  }
  return status(s);
}

// run_static(args, vocab, dtype, device, stream)
PyObject* py_run_static(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 5)) return nullptr;
  fly_verify_args_t* a = (fly_verify_args_t*)PyLong_AsVoidPtr(v[0]);
  int32_t vocab, dtype, device;
  if (PyErr_Occurred() || !integer_as(v[1], &vocab) || !integer_as(v[2], &dtype) || !integer_as(v[3], &device)) return nullptr;
  void* stream = PyLong_AsVoidPtr(v[4]);
  if (PyErr_Occurred()) return nullptr;
  fly_status_t s;
  {
    Unlocked unlocked;
    s = api.run_static(device, vocab, (fly_dtype_t)dtype, a, stream);
  }
  return status(s);
}

// pld_draft(tokens, lengths, K, max_ngram, min_ngram, device, stream) -> (status, draft, count, match_pos, match_ngram)
PyObject* py_pld_draft(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!enough(n, 7)) return nullptr;
  if (!expect(THPVariable_Check(v[0]) && THPVariable_Check(v[1]), "tokens and lengths are tensors")) return nullptr;
  const at::Tensor &tokens = THPVariable_Unpack(v[0]), &lengths = THPVariable_Unpack(v[1]);
  if (!expect(tokens.dim() >= 2 && tokens.scalar_type() == at::kInt && lengths.scalar_type() == at::kInt && tokens.stride(1) == 1,
              "tokens is [B, L] int32 with contiguous rows, lengths [B] int32"))
    return nullptr;
  int32_t K, mx, mn, device;
  if (!integer_as(v[2], &K) || !integer_as(v[3], &mx) || !integer_as(v[4], &mn) || !integer_as(v[5], &device)) return nullptr;
  void* stream = PyLong_AsVoidPtr(v[6]);
  if (PyErr_Occurred()) return nullptr;
  fly_status_t s;
  at::Tensor draft, count, pos, ngram;
  {
    Unlocked unlocked;
    const int64_t B = tokens.size(0);
    if (tokens.is_cuda() && plain_empty()) {
      // Straight from torch's allocator: through the dispatcher each of the four takes 0.5 us longer, and the call as long as
      // the kernel (32 contexts of 32768 tokens: 6.9 us a call, 5.6 so).
      const c10::DeviceGuard guard(tokens.device());
      c10::Allocator* const allocator = at::detail::getCUDAHooks().getCUDADeviceAllocator();
      auto empty = [&](at::IntArrayRef shape) {
        return at::Tensor(at::detail::empty_generic(shape, allocator, c10::DispatchKeySet(c10::DispatchKey::CUDA), at::kInt, std::nullopt));
      };
      draft = empty({B, K});
      count = empty({B});
      pos = empty({B});
      ngram = empty({B});
    } else {
      const auto opt = tokens.options().requires_grad(false);
      draft = at::empty({B, K}, opt);
      count = at::empty({B}, opt);
      pos = at::empty({B}, opt);
      ngram = at::empty({B}, opt);
    }
    s = api.pld_draft(device, (int32_t)B, (const int32_t*)tokens.data_ptr(), tokens.stride(0), (const int32_t*)lengths.data_ptr(), mx,
                      mn, K, (int32_t*)draft.data_ptr(), (int32_t*)count.data_ptr(), (int32_t*)pos.data_ptr(),
                      (int32_t*)ngram.data_ptr(), stream);
  }
  return Py_BuildValue("(iNNNN)", (int)s, THPVariable_Wrap(draft), THPVariable_Wrap(count), THPVariable_Wrap(pos),
                       THPVariable_Wrap(ngram));
}

// A C++ exception must not leave a function that Python calls.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* v, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  return F(self, v, n);
  END_HANDLE_TH_ERRORS
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))guarded<py_##name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(init),         FAST(fill), FAST(verify),       FAST(verify_fused), FAST(reduce_shard),
                         FAST(run_partials), FAST(run),  FAST(run_static), FAST(pld_draft),    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Native argument marshalling of the C ABI.", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
  s_accept_len = PyUnicode_InternFromString("accept_len");
  s_rollback = PyUnicode_InternFromString("rollback");
  s_out_tokens = PyUnicode_InternFromString("out_tokens");
  s_target_argmax = PyUnicode_InternFromString("target_argmax");
  s_entropy = PyUnicode_InternFromString("entropy");
  s_row_flags = PyUnicode_InternFromString("row_flags");
  s_state = PyUnicode_InternFromString("state");
  return PyModule_Create(&module);
}
