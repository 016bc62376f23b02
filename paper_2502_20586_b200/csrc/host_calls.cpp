// The host side of a layer's backward call in native code: the checks, the tensors that the caller did not bring, the current stream and
// the call of the C ABI.  binding.py does the same in Python for tensors of a subclass; its other backward calls use the checks.
//
// What bounds a small layer is host time (256 x 512 x 512: 10.0 us of GPU work).  Of 17.8 us through Python and ctypes 7 went to the library
// (tensor maps, two launches), 6.5 to three allocations, 4 to marshalling; here a call takes 10.9, with the caller's buffers 7.3
// (10.6), and a forward and backward step through autograd, 8192 x 1024 x 3072 with bias, 113 (127).  Calls back to back: 256 x 512 x 512 17.7 -> 10.4 - 11.2 us,
// the autograd step 135 -> 123.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/core/impl/VirtualGuardImpl.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <initializer_list>

#include "mxfp4.h"

namespace {

// Entry points of the library, as binding.py has loaded it.
decltype(&mxfp4_linear_backward_ex_workspace) g_workspace = nullptr;
decltype(&mxfp4_linear_backward_ex) g_backward = nullptr;

PyObject* bind(PyObject*, PyObject* args) {
    unsigned long long workspace = 0, backward = 0;
    if (!PyArg_ParseTuple(args, "KK", &workspace, &backward)) return nullptr;
    g_workspace = reinterpret_cast<decltype(g_workspace)>(workspace);
    g_backward = reinterpret_cast<decltype(g_backward)>(backward);
    Py_RETURN_NONE;
}

// Whether an argument is an integer by itself, and if so its low bits, as ctypes takes them.
bool integer(PyObject* o, uint64_t* out) {
    if (!PyIndex_Check(o)) return false;
    PyObject* i = PyNumber_Index(o);
    if (i == nullptr) return false;
    *out = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return *out != ~uint64_t(0) || PyErr_Occurred() == nullptr;
}

// The current device's current stream, by torch's interface for any device: this module needs no CUDA library of torch's to load.
void* current_stream() {
    const c10::impl::VirtualGuardImpl cuda(c10::DeviceType::CUDA);
    return cuda.getStreamNativeHandle(cuda.getStream(cuda.getDevice()));
}

// Other Python threads run while one of these lives, an exception included.  It goes around the allocations as well as the library: one
// that the caching allocator has no block for frees others and waits for the GPU, where a host callback may need the interpreter.
struct NoGil {
    PyThreadState* thread = PyEval_SaveThread();
    NoGil() = default;
    NoGil(const NoGil&) = delete;
    NoGil& operator=(const NoGil&) = delete;
    ~NoGil() { PyEval_RestoreThread(thread); }
};

bool refuse(PyObject* error, const char* why) {
    PyErr_SetString(error, why);
    return false;
}

// A tensor, or nothing for None.
at::Tensor tensor_or_none(PyObject* o) { return o == Py_None ? at::Tensor() : THPVariable_Unpack(o); }

bool are_tensors(PyObject* const* args, std::initializer_list<int> required, std::initializer_list<int> given) {
    for (int i : required)
        if (!THPVariable_Check(args[i])) return refuse(PyExc_TypeError, "a tensor is expected");
    for (int i : given)
        if (args[i] != Py_None && !THPVariable_Check(args[i])) return refuse(PyExc_TypeError, "a tensor is expected");
    return true;
}

// The tensors of a layer's backward call and the buffers that the caller has for it.  The kernels get addresses and b, m and n: no tensor
// may be smaller than these say, of another type or laid out otherwise.  binding.py's _layer says the same of tensors of a subclass.
bool layer_fits(const at::Tensor& dY, const at::Tensor& X, const at::Tensor& W, const at::Tensor& dX, const at::Tensor& dW, const at::Tensor& db,
                const at::Tensor& workspace, bool fp32) {
    if (dY.dim() != 2 || X.dim() != 2) return refuse(PyExc_ValueError, "dY and X have two dimensions");
    for (const at::Tensor* t : {&dY, &X, &W})
        if (!t->is_cuda() || t->scalar_type() != at::kBFloat16 || !t->is_contiguous())
            return refuse(PyExc_AssertionError, "contiguous bf16 tensors on the GPU are expected");
    const int64_t b = dY.size(0), m = dY.size(1), n = X.size(1);
    if (X.size(0) != b || W.numel() != m * n || (W.dim() == 2 && W.size(1) != n) || X.device() != dY.device() || W.device() != dY.device())
        return refuse(PyExc_AssertionError, "dY [b, m], X [b, n] and W [m, n] on one GPU are expected");
    auto in_place = [&](const at::Tensor& t) { return !t.defined() || (t.device() == dY.device() && t.is_contiguous()); };
    auto holds = [&](const at::Tensor& t, int64_t elements, at::ScalarType type) {
        return !t.defined() || (in_place(t) && t.scalar_type() == type && t.numel() >= elements);
    };
    auto rows_of_n = [&](const at::Tensor& t) { return !t.defined() || t.dim() != 2 || t.size(1) == n; };
    const at::ScalarType result = fp32 ? at::kFloat : at::kBFloat16;
    if (!holds(dX, b * n, result) || !rows_of_n(dX) || !holds(dW, m * n, result) || !rows_of_n(dW) || !holds(db, m, at::kFloat) || !in_place(workspace))
        return refuse(PyExc_AssertionError, "a buffer has another type or device, is not contiguous or too small");
    return true;
}

// layer(dY, X, W, dX, dW, workspace, fp32) -> (b, m, n), or the exception that the caller gets.
PyObject* layer(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
    HANDLE_TH_ERRORS
    if (n_args != 7) {
        PyErr_SetString(PyExc_TypeError, "layer: 7 arguments");
        return nullptr;
    }
    if (!are_tensors(args, {0, 1, 2}, {3, 4, 5})) return nullptr;
    const at::Tensor &dY = THPVariable_Unpack(args[0]), &X = THPVariable_Unpack(args[1]), &W = THPVariable_Unpack(args[2]);
    if (!layer_fits(dY, X, W, tensor_or_none(args[3]), tensor_or_none(args[4]), at::Tensor(), tensor_or_none(args[5]), args[6] == Py_True)) return nullptr;
    return Py_BuildValue("LLL", (long long)dY.size(0), (long long)dY.size(1), (long long)X.size(1));
    END_HANDLE_TH_ERRORS
}

// backward(dY, X, W, g, seed, rounding, out_dtype, dX, dW, db, with_bias, accumulate, workspace) -> (status, dX, dW, db): Algorithm 3.
// None for dX, dW, db (with_bias) or workspace: made here.  The result is None where g, seed, rounding or out_dtype is no integer by itself.
PyObject* backward(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
    HANDLE_TH_ERRORS
    if (n_args != 13) {
        PyErr_SetString(PyExc_TypeError, "backward: 13 arguments");
        return nullptr;
    }
    if (!are_tensors(args, {0, 1, 2}, {7, 8, 9, 12})) return nullptr;
    uint64_t g, seed, rounding, out_dtype;
    if (!integer(args[3], &g) || !integer(args[4], &seed) || !integer(args[5], &rounding) || !integer(args[6], &out_dtype)) {
        if (PyErr_Occurred() != nullptr) return nullptr;
        Py_RETURN_NONE;                                               // ctypes may know what to do with it
    }
    const int with_bias = PyObject_IsTrue(args[10]), accumulate = PyObject_IsTrue(args[11]);
    if (with_bias < 0 || accumulate < 0) return nullptr;
    const at::Tensor &dY = THPVariable_Unpack(args[0]), &X = THPVariable_Unpack(args[1]), &W = THPVariable_Unpack(args[2]);
    at::Tensor dX = tensor_or_none(args[7]), dW = tensor_or_none(args[8]), db = tensor_or_none(args[9]), workspace = tensor_or_none(args[12]);
    const bool fp32 = (int)out_dtype == MXFP4_OUT_FP32;
    if (!layer_fits(dY, X, W, dX, dW, db, workspace, fp32)) return nullptr;
    if (accumulate != 0 && (!dW.defined() || (with_bias != 0 && !db.defined()))) {
        PyErr_SetString(PyExc_AssertionError, "accumulation needs an existing dW, and db");
        return nullptr;
    }
    const int64_t b = dY.size(0), m = dY.size(1), n = X.size(1);
    mxfp4_status status;
    {
        const NoGil others_run;
        const auto like = dY.options().requires_grad(false), result = like.dtype(fp32 ? at::kFloat : at::kBFloat16);
        if (!dX.defined()) dX = at::empty({b, n}, result);
        if (!dW.defined()) dW = at::empty({m, n}, result);
        if (with_bias != 0 && !db.defined()) db = at::empty({m}, like.dtype(at::kFloat));
        if (!workspace.defined()) workspace = at::empty({(int64_t)g_workspace(b, m, n, db.defined() ? 1 : 0)}, like.dtype(at::kByte));
        status = g_backward(dY.data_ptr(), X.data_ptr(), W.data_ptr(), b, m, n, (int)g, (int)rounding, seed, dX.data_ptr(), dW.data_ptr(),
                            db.defined() ? static_cast<float*>(db.data_ptr()) : nullptr, (int)out_dtype, accumulate, workspace.data_ptr(),
                            (size_t)workspace.numel(), current_stream());
    }
    PyObject* out[4] = {PyLong_FromLong(status), nullptr, nullptr, nullptr};
    const at::Tensor* made[3] = {&dX, &dW, &db};
    for (int i = 0; i < 3; ++i) {
        if (args[7 + i] != Py_None) { out[1 + i] = args[7 + i]; Py_INCREF(args[7 + i]); }
        else out[1 + i] = THPVariable_Wrap(*made[i]);                 // (None for a tensor that is not defined)
    }
    PyObject* tuple = PyTuple_New(4);
    if (tuple == nullptr || !out[0] || !out[1] || !out[2] || !out[3]) {
        for (PyObject* o : out) Py_XDECREF(o);
        Py_XDECREF(tuple);
        return nullptr;
    }
    for (int i = 0; i < 4; ++i) PyTuple_SET_ITEM(tuple, i, out[i]);
    return tuple;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, "addresses of mxfp4_linear_backward_ex_workspace and mxfp4_linear_backward_ex"},
    {"layer", (PyCFunction)(void (*)(void))layer, METH_FASTCALL, "(b, m, n)"},
    {"backward", (PyCFunction)(void (*)(void))backward, METH_FASTCALL, "(status, dX, dW, db)"},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_calls() {
    PyObject* m = PyModule_Create(&module);
    // the torch and Python whose headers are compiled in here (build.py): binding.py compares it with the running ones
    if (m != nullptr && PyModule_AddStringConstant(m, "built_for", MXFP4_HOST_STAMP) != 0) Py_CLEAR(m);
    return m;
}
