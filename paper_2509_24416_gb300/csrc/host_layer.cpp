// One call of a prepared layer from Python: the checks, the two output
// allocations and the two launches of rotate-quant + product in one native
// call.  A pass over a small layer lasts 8 us on the GPU; the same steps in
// Python took the host 32 us (three allocations 5, two stream look-ups 6, the two
// C calls with their launches 7, the rest interpreter time), this call about 9.
//
// Only the plain case is taken: a 2-D fp16 / bf16 CUDA tensor with unit column
// stride and the layer's K columns, and weights in a layout its width names.
// Anything else returns None, and the Python path goes on with it (and raises
// what it always raised).
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/clq.h"

namespace {

// Layout of a weight code array of `width` bytes a row for K codes, or -1.
int codes_layout(int64_t width, int64_t K) {
  if (width == K) return CLQ_CODES_E4M3;
  if (2 * width == K) return CLQ_CODES_INT4_PACKED;
  if (width == 2 * K) return CLQ_CODES_E4M3_SPLIT;
  if (4 * width == 3 * K) return CLQ_CODES_E2M3;
  return -1;
}

int64_t codes_width(int64_t codes, int64_t K) {
  switch (codes) {
    case CLQ_CODES_INT4_PACKED: return K / 2;
    case CLQ_CODES_E4M3: return K;
    case CLQ_CODES_E4M3_SPLIT: return 2 * K;
    case CLQ_CODES_E2M3: return K / 4 * 3;
    default: return -1;
  }
}

// layer(X, perm, We, s_w, bias | None, b, K, a_codes) -> Y [M, N] on the current
// stream, whose pool the buffers come from; None: not the plain case; an int:
// status | 256 * (0 rotate-quant, 1 product).
PyObject* layer(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  HANDLE_TH_ERRORS
  if (nargs != 8) {
    PyErr_SetString(PyExc_TypeError, "layer() takes 8 arguments");
    return nullptr;
  }
  for (int i = 0; i < 4; ++i)
    if (!THPVariable_Check(args[i])) Py_RETURN_NONE;
  const bool has_bias = args[4] != Py_None;
  if (has_bias && !THPVariable_Check(args[4])) Py_RETURN_NONE;
  const at::Tensor& X = THPVariable_Unpack(args[0]);
  const at::Tensor& We = THPVariable_Unpack(args[2]);
  const long b = PyLong_AsLong(args[5]);
  const long K = PyLong_AsLong(args[6]);
  const long a_codes = PyLong_AsLong(args[7]);
  if (PyErr_Occurred()) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
  if (!X.is_cuda() || X.dim() != 2 || X.stride(1) != 1 || X.size(1) != K || We.dim() != 2)
    Py_RETURN_NONE;
  const at::ScalarType dt = X.scalar_type();
  if (dt != at::kHalf && dt != at::kBFloat16) Py_RETURN_NONE;
  if (has_bias && THPVariable_Unpack(args[4]).scalar_type() != dt) Py_RETURN_NONE;
  const int64_t M = X.size(0), N = We.size(0), ld = X.stride(0);
  const int w_codes = codes_layout(We.size(1), K);
  const int64_t width = codes_width(a_codes, K);
  // (8-bit weights go with 8-bit activations only)
  if (w_codes < 0 || width < 0 ||
      (w_codes == CLQ_CODES_E4M3_SPLIT && a_codes != CLQ_CODES_E4M3_SPLIT) ||
      M > INT32_MAX || N > INT32_MAX || ld > INT32_MAX || b < 0 || b > INT32_MAX)
    Py_RETURN_NONE;
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  // Activation codes and, behind them, their fp32 scales: one buffer.
  const int64_t codes_bytes = (M * width + 15) / 16 * 16;
  at::Tensor codes = at::empty({codes_bytes + 4 * M}, X.options().dtype(at::kByte));
  at::Tensor Y = at::empty({M, N}, X.options());
  uint8_t* Xq = codes.data_ptr<uint8_t>();
  float* s_x = reinterpret_cast<float*>(Xq + codes_bytes);
  const clq_dtype cdt = dt == at::kHalf ? CLQ_F16 : CLQ_BF16;
  const void* x = X.data_ptr();
  const int32_t* perm = static_cast<const int32_t*>(THPVariable_Unpack(args[1]).data_ptr());
  const uint8_t* w = static_cast<const uint8_t*>(We.data_ptr());
  const float* s_w = static_cast<const float*>(THPVariable_Unpack(args[3]).data_ptr());
  const void* bias = has_bias ? THPVariable_Unpack(args[4]).data_ptr() : nullptr;
  void* y = Y.data_ptr();
  long where = 0;
  clq_status st;
  Py_BEGIN_ALLOW_THREADS
  st = clq_rotate_quant_act(x, cdt, static_cast<int32_t>(M), static_cast<int32_t>(K),
                            static_cast<int32_t>(ld), perm, static_cast<int32_t>(b),
                            static_cast<clq_codes>(a_codes), Xq, s_x, nullptr, stream);
  if (st == CLQ_OK) {
    where = 1;
    st = clq_linear(Xq, static_cast<clq_codes>(a_codes), s_x, w, w_codes, s_w, bias,
                    static_cast<int32_t>(M), static_cast<int32_t>(N), static_cast<int32_t>(K),
                    static_cast<int32_t>(b), cdt, y, nullptr, stream);
  }
  Py_END_ALLOW_THREADS
  if (st != CLQ_OK) return PyLong_FromLong(st | (where << 8));
  return THPVariable_Wrap(Y);
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"layer", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(layer)), METH_FASTCALL,
     "Rotate-quant and product of one prepared layer."},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_clq_host", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__clq_host(void) { return PyModule_Create(&module); }
