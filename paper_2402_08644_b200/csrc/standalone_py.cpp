// Python entry to the stand-alone kernels (decode attention, FF_Tandem projection, block linear) without the
// interpreter's share: the kernels run for 4-8 us, and through ctypes a projection call cost the host 13.9 us (two tensor
// allocations 3, argument conversion 2, the wrapper itself 2) and an attention call 6.0.  Arguments are unpacked and
// outputs allocated here.  Each function returns its result, or the library's status as an int where a call failed;
// binding.py wraps them and turns a status into its exception.
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "../../include/tandem.h"

namespace {

const at::Tensor* tensor_arg(PyObject* o) {
    if (THPVariable_Check(o)) return &THPVariable_Unpack(o);
    PyErr_SetString(PyExc_TypeError, "a torch.Tensor is expected");
    return nullptr;
}
// The kernels take plain addresses: whatever they would read or write lies on the first argument's GPU (t: null where an optional
// argument is absent; an empty tensor is never touched).  Ranks of the first argument as documented.
void check_arguments(const at::Tensor* const* t, int n, int rank) {
    const at::Tensor& first = *t[0];
    TORCH_CHECK_VALUE(first.dim() == rank, "the first argument must have " + std::to_string(rank) + " dimensions, it has " + std::to_string(first.dim()));
    TORCH_CHECK_VALUE(first.is_cuda(), "expected a tensor on a CUDA device, got one on " + first.device().str());
    for (int i = 1; i < n; ++i)
        if (t[i] && t[i]->numel())
            TORCH_CHECK_VALUE(t[i]->device() == first.device(),
                              "argument " + std::to_string(i + 1) + " is on " + t[i]->device().str() + ", the first one on " + first.device().str());
}
const void* ptr_of(const at::Tensor& t) { return t.numel() ? t.const_data_ptr() : nullptr; }
void* stream_of(const at::Tensor& t) { return c10::cuda::getCurrentCUDAStream(t.get_device()).stream(); }
at::Tensor empty_like_device(at::IntArrayRef size, at::ScalarType type, const at::Tensor& t) {
    return at::detail::empty_cuda(size, type, t.device(), std::nullopt);
}
PyObject* result(tandem_status st, const at::Tensor& t) { return st == TANDEM_OK ? THPVariable_Wrap(t) : PyLong_FromLong(st); }

// (q, k_derived, v_derived, k_own, v_own, out or None, scratch or None)
PyObject* decode_attention(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 7) { PyErr_SetString(PyExc_TypeError, "seven arguments are expected"); return nullptr; }
    const at::Tensor* t[7] = {};
    for (int i = 0; i < 7; ++i)
        if (i < 5 || args[i] != Py_None)
            if (!(t[i] = tensor_arg(args[i]))) return nullptr;
    check_arguments(t, 7, 3);
    const at::Tensor& q = *t[0];
    const int B = (int)q.size(0), H = (int)q.size(1), dh = (int)q.size(2), Td = (int)t[1]->size(2), To = (int)t[3]->size(2);
    const at::Tensor out = t[5] ? *t[5] : empty_like_device(q.sizes(), q.scalar_type(), q);
    const at::Tensor scratch = t[6] ? *t[6] : empty_like_device({(int64_t)tandem_decode_attention_scratch_bytes(B, H, dh, Td, To)}, at::kByte, q);
    const tandem_status st = tandem_decode_attention(q.const_data_ptr(), ptr_of(*t[1]), ptr_of(*t[2]), ptr_of(*t[3]), ptr_of(*t[4]), out.mutable_data_ptr(),
                                                     scratch.mutable_data_ptr(), (size_t)scratch.numel(), B, H, dh, Td, To, stream_of(q));
    return result(st, out);
    END_HANDLE_TH_ERRORS
}

// (x, w_t, ln_g, ln_b, wk, wv, scratch or None)
PyObject* ff_tandem_project(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 7) { PyErr_SetString(PyExc_TypeError, "seven arguments are expected"); return nullptr; }
    const at::Tensor* t[7] = {};
    for (int i = 0; i < 7; ++i)
        if (i < 6 || args[i] != Py_None)
            if (!(t[i] = tensor_arg(args[i]))) return nullptr;
    check_arguments(t, 7, 2);
    const at::Tensor& x = *t[0];
    const int rows = (int)x.size(0), d_l = (int)x.size(1), d_s = (int)t[1]->size(0);
    const at::Tensor k = empty_like_device({rows, d_s}, at::kBFloat16, x), v = empty_like_device({rows, d_s}, at::kBFloat16, x);
    const at::Tensor scratch = t[6] ? *t[6] : empty_like_device({(int64_t)tandem_ff_tandem_project_scratch_bytes(rows, d_s)}, at::kByte, x);
    const tandem_status st = tandem_ff_tandem_project(x.const_data_ptr(), t[1]->const_data_ptr(), t[2]->const_data_ptr(), t[3]->const_data_ptr(),
                                                      t[4]->const_data_ptr(), t[5]->const_data_ptr(), k.mutable_data_ptr(), v.mutable_data_ptr(),
                                                      scratch.mutable_data_ptr(), (size_t)scratch.numel(), rows, d_l, d_s, stream_of(x));
    if (st != TANDEM_OK) return PyLong_FromLong(st);
    PyObject* pair = PyTuple_New(2);
    if (!pair) return nullptr;
    PyTuple_SET_ITEM(pair, 0, THPVariable_Wrap(k));
    PyTuple_SET_ITEM(pair, 1, THPVariable_Wrap(v));
    return pair;
    END_HANDLE_TH_ERRORS
}

// (x, w, y or None)
PyObject* block_linear(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 3) { PyErr_SetString(PyExc_TypeError, "three arguments are expected"); return nullptr; }
    const at::Tensor* t[3] = {};
    for (int i = 0; i < 3; ++i)
        if (i < 2 || args[i] != Py_None)
            if (!(t[i] = tensor_arg(args[i]))) return nullptr;
    check_arguments(t, 3, 2);
    const at::Tensor &x = *t[0], &w = *t[1];
    const int rows = (int)x.size(0), k = (int)x.size(1), nf = (int)w.size(0);
    const at::Tensor y = t[2] ? *t[2] : empty_like_device({rows, nf}, at::kBFloat16, x);
    return result(tandem_block_linear(x.const_data_ptr(), w.const_data_ptr(), y.mutable_data_ptr(), rows, k, nf, stream_of(x)), y);
    END_HANDLE_TH_ERRORS
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL
PyMethodDef methods[] = {{"decode_attention", FAST(decode_attention), nullptr},
                         {"ff_tandem_project", FAST(ff_tandem_project), nullptr},
                         {"block_linear", FAST(block_linear), nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_standalone", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__standalone(void) { return PyModule_Create(&module); }
