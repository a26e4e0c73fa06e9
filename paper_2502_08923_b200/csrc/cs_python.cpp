// The search call for Python, in native code: marshalling of cs_find_match with its outputs made by the allocator directly.
//
// The search takes 2.3 to 5.1 us on the device, a call through ctypes 10.7: three tensors made from Python, eleven
// arguments converted, two tensors looked at, the launch.  Here 5.0 - 5.3 for one history of 4,097 tokens, and 5.3 - 5.5 for 64 of 32,768, where the
// device sets the pace.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "copyspec.h"

namespace {

// (what vmap and other transforms hand in looks like a tensor, but has no memory of its own)
bool plain(const at::Tensor& t, int64_t dim) {
  return t.has_storage() && t.is_cuda() && t.scalar_type() == at::kInt && t.layout() == at::kStrided && t.dim() == dim && t.is_contiguous();
}

// find_match(hist, hist_len, gamma, k, policy) -> (match_pos [B], draft [B][k], draft_len [B]), or the call's status where that
// is an error, or None where the arguments are not plain ones: the caller's general path takes those.
PyObject* find_match(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  HANDLE_TH_ERRORS
  if (n_args != 5 || !THPVariable_CheckExact(args[0]) || !THPVariable_CheckExact(args[1]) || !PyLong_CheckExact(args[2]) ||
      !PyLong_CheckExact(args[3]) || !PyLong_CheckExact(args[4]) || c10::impl::TorchDispatchModeTLS::any_modes_set())
    Py_RETURN_NONE;
  const at::Tensor& hist = THPVariable_Unpack(args[0]);
  const at::Tensor& len = THPVariable_Unpack(args[1]);
  int overflow[3];
  const long gamma = PyLong_AsLongAndOverflow(args[2], &overflow[0]), k = PyLong_AsLongAndOverflow(args[3], &overflow[1]),
             policy = PyLong_AsLongAndOverflow(args[4], &overflow[2]);
  constexpr int64_t kMost = 1 << 30;
  if (overflow[0] || overflow[1] || overflow[2] || gamma < 0 || gamma > kMost || k < 0 || k > kMost || policy < 0 || policy > kMost ||
      !plain(hist, 2) || !plain(len, 1))
    Py_RETURN_NONE;
  const int64_t B = hist.size(0), stride = hist.size(1);
  if (B < 1 || B > kMost || stride > kMost || len.size(0) != B || len.device() != hist.device()) Py_RETURN_NONE;
  const at::Tensor pos = at::detail::empty_cuda({B}, at::kInt, hist.device(), std::nullopt);
  const at::Tensor draft = at::detail::empty_cuda({B, k}, at::kInt, hist.device(), std::nullopt);
  const at::Tensor draft_len = at::detail::empty_cuda({B}, at::kInt, hist.device(), std::nullopt);
  // (everything that may throw comes before the interpreter's lock is given up: the handler below needs it)
  void* const stream = c10::cuda::getCurrentCUDAStream().stream();
  const int32_t* const h = static_cast<const int32_t*>(hist.const_data_ptr());
  const int32_t* const n = static_cast<const int32_t*>(len.const_data_ptr());
  int32_t* const out_pos = static_cast<int32_t*>(pos.mutable_data_ptr());
  int32_t* const out_draft = k > 0 ? static_cast<int32_t*>(draft.mutable_data_ptr()) : nullptr;
  int32_t* const out_len = static_cast<int32_t*>(draft_len.mutable_data_ptr());
  cs_status s;
  Py_BEGIN_ALLOW_THREADS
  s = cs_find_match(h, n, (int)B, (int)stride, (int)gamma, (int)k, (cs_match_policy)policy, out_pos, out_draft, out_len, stream);
  Py_END_ALLOW_THREADS
  if (s != CS_OK) return PyLong_FromLong(s);
  PyObject* out = PyTuple_New(3);
  if (out == nullptr) return nullptr;
  PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(pos));
  PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(draft));
  PyTuple_SET_ITEM(out, 2, THPVariable_Wrap(draft_len));
  return out;
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"find_match", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(find_match)), METH_FASTCALL, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
