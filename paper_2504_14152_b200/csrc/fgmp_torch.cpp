// CPython entry points of the calls that a decode or prefill step makes: they take torch tensors, allocate the
// result, look up the current stream and call the C ABI.  The arithmetic stays in libfgmp; this file only removes
// the interpreter's share of a call (a ctypes call with fifteen arguments, two allocations and a stream look-up
// through torch's Python layer took 13-14 us of host time per step, longer than the kernel of a small layer; here a
// step costs about 4 us, most of it the launch).
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include "fgmp.h"

namespace {

// The calls that can return a status raise it through here: the Python side turns the pair into its exception type.
PyObject* fail(fgmp_status st, const char* what) { return Py_BuildValue("is", (int)st, what); }

inline bool is_none(PyObject* o) { return o == Py_None; }
inline const at::Tensor& tensor_of(PyObject* o)
{
    TORCH_CHECK_TYPE(THPVariable_Check(o), "expected a tensor");
    return THPVariable_Unpack(o);
}
inline at::Tensor empty_cuda(c10::IntArrayRef sizes, at::ScalarType t, c10::Device dev)
{
    return at::detail::empty_cuda(sizes, t, dev, c10::nullopt);
}
// uint8 buffer whose data pointer is 1024-byte aligned (the allocator aligns to 512)
inline at::Tensor empty_aligned(int64_t nbytes, c10::Device dev)
{
    at::Tensor t = empty_cuda({nbytes + 1024}, at::kByte, dev);
    const int64_t off = (int64_t)((1024 - ((uintptr_t)t.data_ptr() & 1023)) & 1023);
    t.unsafeGetTensorImpl()->set_storage_offset(off);
    t.unsafeGetTensorImpl()->set_sizes_contiguous({nbytes});
    return t;
}
inline void* current_stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }
inline double as_double(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw python_error();
    return v;
}
inline int64_t as_int(PyObject* o)
{
    const int64_t v = (int64_t)PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}
inline at::Tensor optional_tensor(PyObject* o) { return is_none(o) ? at::Tensor() : tensor_of(o); }
// The interpreter lock is given up for what may wait: allocations, and launches on a full queue.
struct WithoutLock {
    PyThreadState* state = PyEval_SaveThread();
    ~WithoutLock() { PyEval_RestoreThread(state); }
};
// workspace given by the caller, or a cleared one of this call's own
inline at::Tensor workspace_for(const at::Tensor& given, int op, int64_t M, int64_t N, int64_t K, c10::Device dev, void* stream, fgmp_status* st)
{
    if (given.defined()) return given;
    at::Tensor ws = empty_aligned((int64_t)fgmp_workspace_bytes(op, M, N, K), dev);
    *st = fgmp_workspace_init(ws.data_ptr(), (size_t)ws.numel(), stream);
    return ws;
}
inline at::Tensor output_for(const at::Tensor& given, bool bf16, int64_t M, int64_t N, c10::Device dev)
{
    if (given.defined()) return given;
    return empty_cuda({M, N}, bf16 ? at::kBFloat16 : at::kFloat, dev);
}

// quantize_activations(X, fisher, scale_fp4, ratio, scale_fp8, score_mode, tau, out | None) -> blob
PyObject* py_quantize_activations(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    TORCH_CHECK_TYPE(n == 8, "quantize_activations takes 8 arguments");
    const at::Tensor &X = tensor_of(a[0]), &f = tensor_of(a[1]);
    const int64_t M = X.size(0), K = X.size(1);
    const size_t nbytes = fgmp_acts_bytes(M, K);
    if (nbytes == 0) return fail(FGMP_ERR_SHAPE, "fgmp_acts_bytes");
    const fgmp_scales sc{(float)as_double(a[2]), (int)as_int(a[3]), (float)as_double(a[4])};
    const int mode = (int)as_int(a[5]);
    const float tau = (float)as_double(a[6]);
    at::Tensor out = optional_tensor(a[7]);
    fgmp_status st = FGMP_OK;
    {
        WithoutLock no_lock;
        if (!out.defined()) out = empty_aligned((int64_t)nbytes, X.device());
        st = fgmp_quantize_activations(X.data_ptr(), X.stride(0), (const float*)f.data_ptr(), M, K, sc, (fgmp_score_mode)mode, tau,
                                       out.data_ptr(), (size_t)out.numel(), nullptr, 0, current_stream());
    }
    if (st != FGMP_OK) return fail(st, "fgmp_quantize_activations");
    return THPVariable_Wrap(std::move(out));
    END_HANDLE_TH_ERRORS
}

// linear(acts, weights, M, N, K, out | None, bf16, workspace | None, nvfp4) -> (Y, workspace)
PyObject* py_linear(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    TORCH_CHECK_TYPE(n == 9, "linear takes 9 arguments");
    const at::Tensor &acts = tensor_of(a[0]), &w = tensor_of(a[1]);
    const int64_t M = as_int(a[2]), N = as_int(a[3]), K = as_int(a[4]);
    const bool bf16 = PyObject_IsTrue(a[6]) == 1;
    const int nvfp4 = (int)as_int(a[8]);
    at::Tensor out = optional_tensor(a[5]), ws = optional_tensor(a[7]);
    fgmp_status st = FGMP_OK;
    const char* call = "fgmp_workspace_init";
    {
        WithoutLock no_lock;
        void* s = current_stream();
        out = output_for(out, bf16, M, N, acts.device());
        ws = workspace_for(ws, FGMP_OP_LINEAR, M, N, K, acts.device(), s, &st);
        if (st == FGMP_OK) {
            call = "fgmp_linear";
            st = fgmp_linear_expect(acts.data_ptr(), w.data_ptr(), out.data_ptr(), out.scalar_type() == at::kBFloat16 ? 1 : 0, out.stride(0),
                                    M, N, K, ws.data_ptr(), (size_t)ws.numel(), nvfp4, s);
        }
    }
    if (st != FGMP_OK) return fail(st, call);
    PyObject* r = PyTuple_New(2);
    PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(out)));
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(ws)));
    return r;
    END_HANDLE_TH_ERRORS
}

// linear_fused(X, fisher, weights, N, scale_fp4, ratio, score_mode, tau, out | None, bf16, packed_out | None, want_packed,
//              workspace | None) -> (Y, packed | None, workspace)
PyObject* py_linear_fused(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    TORCH_CHECK_TYPE(n == 13, "linear_fused takes 13 arguments");
    const at::Tensor &X = tensor_of(a[0]), &f = tensor_of(a[1]), &w = tensor_of(a[2]);
    const int64_t M = X.size(0), K = X.size(1), N = as_int(a[3]);
    const fgmp_scales sc{(float)as_double(a[4]), (int)as_int(a[5]), 0.f};
    const int mode = (int)as_int(a[6]);
    const float tau = (float)as_double(a[7]);
    const bool bf16 = PyObject_IsTrue(a[9]) == 1, want_packed = PyObject_IsTrue(a[11]) == 1;
    at::Tensor out = optional_tensor(a[8]), packed = optional_tensor(a[10]), ws = optional_tensor(a[12]);
    fgmp_status st = FGMP_OK;
    const char* call = "fgmp_workspace_init";
    {
        WithoutLock no_lock;
        void* s = current_stream();
        out = output_for(out, bf16, M, N, X.device());
        if (!packed.defined() && want_packed) packed = empty_aligned((int64_t)fgmp_acts_bytes(M, K), X.device());
        ws = workspace_for(ws, FGMP_OP_LINEAR_FUSED, M, N, K, X.device(), s, &st);
        if (st == FGMP_OK) {
            call = "fgmp_linear_fused";
            st = fgmp_linear_fused(X.data_ptr(), X.stride(0), (const float*)f.data_ptr(), sc, (fgmp_score_mode)mode, tau, w.data_ptr(),
                                   out.data_ptr(), out.scalar_type() == at::kBFloat16 ? 1 : 0, out.stride(0), M, N, K,
                                   packed.defined() ? packed.data_ptr() : nullptr, packed.defined() ? (size_t)packed.numel() : 0,
                                   ws.data_ptr(), (size_t)ws.numel(), s);
        }
    }
    if (st != FGMP_OK) return fail(st, call);
    PyObject* r = PyTuple_New(3);
    PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(out)));
    if (packed.defined()) PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(packed)));
    else { Py_INCREF(Py_None); PyTuple_SET_ITEM(r, 1, Py_None); }
    PyTuple_SET_ITEM(r, 2, THPVariable_Wrap(std::move(ws)));
    return r;
    END_HANDLE_TH_ERRORS
}

// linear_quantize(acts, weights, M, N, K, fisher_next, scale_fp4, ratio, score_mode, tau, workspace | None) -> (blob, workspace)
PyObject* py_linear_quantize(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    TORCH_CHECK_TYPE(n == 11, "linear_quantize takes 11 arguments");
    const at::Tensor &acts = tensor_of(a[0]), &w = tensor_of(a[1]), &f = tensor_of(a[5]);
    const int64_t M = as_int(a[2]), N = as_int(a[3]), K = as_int(a[4]);
    const fgmp_scales sc{(float)as_double(a[6]), (int)as_int(a[7]), 0.f};
    const int mode = (int)as_int(a[8]);
    const float tau = (float)as_double(a[9]);
    at::Tensor out, ws = optional_tensor(a[10]);
    fgmp_status st = FGMP_OK;
    const char* call = "fgmp_workspace_init";
    {
        WithoutLock no_lock;
        void* s = current_stream();
        out = empty_aligned((int64_t)fgmp_acts_bytes(M, N), acts.device());
        ws = workspace_for(ws, FGMP_OP_LINEAR_QUANTIZE, M, N, K, acts.device(), s, &st);
        if (st == FGMP_OK) {
            call = "fgmp_linear_quantize";
            st = fgmp_linear_quantize(acts.data_ptr(), w.data_ptr(), M, N, K, (const float*)f.data_ptr(), sc, (fgmp_score_mode)mode, tau,
                                      out.data_ptr(), (size_t)out.numel(), ws.data_ptr(), (size_t)ws.numel(), s);
        }
    }
    if (st != FGMP_OK) return fail(st, call);
    PyObject* r = PyTuple_New(2);
    PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(out)));
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(ws)));
    return r;
    END_HANDLE_TH_ERRORS
}

#define FASTCALL(f) (PyCFunction)(void (*)(void))(f), METH_FASTCALL
PyMethodDef methods[] = {
    {"quantize_activations", FASTCALL(py_quantize_activations), nullptr},
    {"linear", FASTCALL(py_linear), nullptr},
    {"linear_fused", FASTCALL(py_linear_fused), nullptr},
    {"linear_quantize", FASTCALL(py_linear_quantize), nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fgmp_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fgmp_torch(void) { return PyModule_Create(&module); }
