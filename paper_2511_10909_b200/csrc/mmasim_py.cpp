// The call path of mmasim.gemm and mmasim.dot_batch in native code: argument checks, output allocation, current
// stream, library call.  In Python these cost 13 us a call (probe batch of 2048 dots: 17.4 us with the launch), more than
// the kernels of small problems run.  Every function answers None when the call is not plain (anything but CUDA tensors of the expected
// types and strides, a status other than OK): the Python code then does it, and names what is wrong.
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include "../../include/mmasim.h"

namespace {

decltype(&mmasim_gemm_ex) p_gemm_ex;
decltype(&mmasim_dot_batch) p_dot_batch;
decltype(&mmasim_model_info) p_model_info;

// bind(gemm_ex, dot_batch, model_info): addresses of the library's entry points.
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 3) { PyErr_SetString(PyExc_TypeError, "bind takes three addresses"); return nullptr; }
    void* p[3];
    for (int i = 0; i < 3; ++i) p[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
    p_gemm_ex = reinterpret_cast<decltype(p_gemm_ex)>(p[0]);
    p_dot_batch = reinterpret_cast<decltype(p_dot_batch)>(p[1]);
    p_model_info = reinterpret_cast<decltype(p_model_info)>(p[2]);
    Py_RETURN_NONE;
}

const at::Tensor* tensor(PyObject* o) {                 // a plain CUDA tensor, or nothing
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.defined() && t.layout() == at::kStrided && t.is_cuda() ? &t : nullptr;
}
// Row stride of a matrix of at least rows x cols words of `bytes` bytes on `dev`, or -1.
int64_t matrix(const at::Tensor* t, int64_t rows, int64_t cols, int bytes, at::Device dev) {
    if (!t || t->device() != dev || t->itemsize() != bytes || t->dim() != 2 || t->size(0) < rows || t->size(1) < cols) return -1;
    if (t->size(1) > 1 && t->stride(1) != 1) return -1;
    const int64_t ld = t->size(0) > 1 ? t->stride(0) : std::max(t->stride(0), t->size(1));
    return ld < cols ? -1 : ld;
}
bool vector(const at::Tensor* t, int64_t n, int bytes, at::Device dev) {
    return t && t->device() == dev && t->is_contiguous() && t->itemsize() == bytes && t->numel() >= n;
}
at::ScalarType word(int bytes) { return bytes == 8 ? at::kLong : (bytes == 4 ? at::kInt : at::kShort); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// gemm(model, A, B, C, out, K, sfa, sfb, k_chunk, row_scale, col_scale, flags) -> D or None
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 12) Py_RETURN_NONE;
    const auto* model = static_cast<const mmasim_model*>(PyLong_AsVoidPtr(a[0]));
    mmasim_info info;
    if (PyErr_Occurred() || !model || p_model_info(model, &info)) { PyErr_Clear(); Py_RETURN_NONE; }
    const at::Tensor *A = tensor(a[1]), *B = tensor(a[2]);
    if (!A || !B || A->dim() != 2 || B->dim() != 2) Py_RETURN_NONE;
    const at::Device dev = A->device();
    const int64_t per_word = info.a_bits == 4 ? 2 : 1, M = A->size(0), N = B->size(0);
    const int64_t K = a[5] == Py_None ? A->size(1) * per_word : PyLong_AsLongLong(a[5]);
    const int64_t k_chunk = PyLong_AsLongLong(a[8]);
    const long flags = PyLong_AsLong(a[11]);
    if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
    const int64_t words = (K + per_word - 1) / per_word, ld_a = matrix(A, M, words, std::max(info.a_bits, 8) / 8, dev),
                  ld_b = matrix(B, N, words, std::max(info.b_bits, 8) / 8, dev);
    if (K < 1 || ld_a < 0 || ld_b < 0) Py_RETURN_NONE;
    mmasim_gemm_opts o = {};
    o.lda = ld_a * per_word;
    o.ldb = ld_b * per_word;
    o.k_chunk = k_chunk;
    o.flags = int32_t(flags);
    const at::Tensor* C = nullptr;
    if (a[3] != Py_None) {
        C = tensor(a[3]);
        if ((o.ldc = matrix(C, M, N, info.acc_bytes, dev)) < 0) Py_RETURN_NONE;
    }
    if (info.k_block) {
        const int64_t nsf = (K + info.k_block - 1) / info.k_block;
        const at::Tensor *sa = tensor(a[6]), *sb = tensor(a[7]);
        if (matrix(sa, M, nsf, 1, dev) != nsf || matrix(sb, N, nsf, 1, dev) != nsf) Py_RETURN_NONE;
        o.sfa = sa->data_ptr();
        o.sfb = sb->data_ptr();
    } else if (a[6] != Py_None || a[7] != Py_None) Py_RETURN_NONE;
    if (a[9] != Py_None || a[10] != Py_None) {
        const at::Tensor *rs = tensor(a[9]), *cs = tensor(a[10]);
        if (!vector(rs, M, 4, dev) || !vector(cs, N, 4, dev)) Py_RETURN_NONE;
        o.row_scale = static_cast<const float*>(rs->data_ptr());
        o.col_scale = static_cast<const float*>(cs->data_ptr());
    }
    try {
        at::Tensor fresh;
        const at::Tensor* out = &fresh;
        if (a[4] == Py_None) fresh = at::empty({M, N}, at::TensorOptions().dtype(word(info.acc_bytes)).device(dev));
        else out = tensor(a[4]);
        if ((o.ldd = matrix(out, M, N, info.acc_bytes, dev)) < 0) Py_RETURN_NONE;
        const void *a_ptr = A->data_ptr(), *b_ptr = B->data_ptr(), *c_ptr = C ? C->data_ptr() : nullptr;
        void *d_ptr = out->data_ptr(), *s = stream();
        int st;
        Py_BEGIN_ALLOW_THREADS                              // (a launch waits where the stream's queue is full, an allocation too)
        st = p_gemm_ex(model, M, N, K, a_ptr, b_ptr, c_ptr, d_ptr, &o, s);
        Py_END_ALLOW_THREADS
        if (st) Py_RETURN_NONE;
        if (a[4] == Py_None) return THPVariable_Wrap(fresh);
        Py_INCREF(a[4]);
        return a[4];
    } catch (const std::exception&) { Py_RETURN_NONE; }
}

// dot_batch(model, A, B, C, out) -> D or None
PyObject* dot_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 5) Py_RETURN_NONE;
    const auto* model = static_cast<const mmasim_model*>(PyLong_AsVoidPtr(a[0]));
    mmasim_info info;
    if (PyErr_Occurred() || !model || p_model_info(model, &info)) { PyErr_Clear(); Py_RETURN_NONE; }
    const at::Tensor *A = tensor(a[1]), *B = tensor(a[2]), *C = a[3] == Py_None ? nullptr : tensor(a[3]);
    if (!A || A->dim() != 2 || (a[3] != Py_None && !C)) Py_RETURN_NONE;
    const at::Device dev = A->device();
    const int64_t dots = A->size(0), K = A->size(1);
    const int64_t ld_a = matrix(A, dots, K, std::max(info.a_bits, 8) / 8, dev), ld_b = matrix(B, dots, K, std::max(info.b_bits, 8) / 8, dev);
    if (K < 1 || ld_a < 0 || ld_b < 0 || (dots > 1 && (ld_a != K || ld_b != K))) Py_RETURN_NONE;
    if (C && !vector(C, dots, info.acc_bytes, dev)) Py_RETURN_NONE;
    try {
        at::Tensor fresh;
        const at::Tensor* out = &fresh;
        if (a[4] == Py_None) fresh = at::empty({dots}, at::TensorOptions().dtype(word(info.acc_bytes)).device(dev));
        else out = tensor(a[4]);
        if (!vector(out, dots, info.acc_bytes, dev)) Py_RETURN_NONE;
        const void *a_ptr = A->data_ptr(), *b_ptr = B->data_ptr(), *c_ptr = C ? C->data_ptr() : nullptr;
        void *d_ptr = out->data_ptr(), *s = stream();
        int st;
        Py_BEGIN_ALLOW_THREADS
        st = p_dot_batch(model, dots, K, a_ptr, b_ptr, c_ptr, d_ptr, s);
        Py_END_ALLOW_THREADS
        if (st) Py_RETURN_NONE;
        if (a[4] == Py_None) return THPVariable_Wrap(fresh);
        Py_INCREF(a[4]);
        return a[4];
    } catch (const std::exception&) { Py_RETURN_NONE; }
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bind)), METH_FASTCALL, nullptr},
    {"gemm", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(gemm)), METH_FASTCALL, nullptr},
    {"dot_batch", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(dot_batch)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mmasim_py", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mmasim_py() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_against", MMASIM_BUILT_AGAINST)) { Py_DECREF(m); return nullptr; }
    return m;
}
