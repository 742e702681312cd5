// The tensor-level call of fff_forward_infer for Python, as a CPython extension module.
//
// Checks of type, shape and contiguity, two allocations, the current stream's handle and the call cost 9.4 us of host time per
// forward when Python and ctypes make them, more than the kernel of a small batch takes (5 to 8.5 us); here they cost about
// half of that, and a batch of one image (197 tokens, D = 768) went from 9.6 us to the 8.6 us that its kernel takes.  The
// module computes nothing: it calls fff_forward_infer, whose address it is given, with the tensors' addresses.  For arguments
// that it does not take as they are it returns None, and the caller's own checks then say what is wrong with them.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using ForwardInfer = int (*)(void*, const void*, void*, int32_t*, int64_t, void*);
ForwardInfer g_forward = nullptr;

bool matches(const at::Tensor& t, at::ScalarType type, int64_t rows, int64_t cols) {
    if (!t.is_cuda() || t.layout() != at::kStrided || t.scalar_type() != type || !t.is_contiguous()) return false;
    if (cols < 0) return t.dim() == 1 && t.size(0) == rows;
    return t.dim() == 2 && t.size(0) == rows && t.size(1) == cols;
}

PyObject* set_address(PyObject*, PyObject* arg) {
    g_forward = reinterpret_cast<ForwardInfer>(PyLong_AsVoidPtr(arg));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

// forward(handle, D, O, is_bf16, x, y or None, leaf_idx or None, want_leaf_idx, stream address or None)
//   -> (status, y, leaf_idx or None), or None when the arguments are not what the call takes
// (A tensor may answer any question about itself with an exception, a Python one from a subclass's dispatch among them: all of
// it stands between the macros that turn C++ exceptions into Python errors, each into the type that torch raises for it.)
PyObject* forward(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 9 || !g_forward || !THPVariable_Check(args[4])) Py_RETURN_NONE;
    void* handle = args[0] == Py_None ? nullptr : PyLong_AsVoidPtr(args[0]);
    const int64_t D = PyLong_AsLongLong(args[1]), O = PyLong_AsLongLong(args[2]);
    const bool bf16 = PyObject_IsTrue(args[3]) == 1, want_leaf = PyObject_IsTrue(args[7]) == 1;
    if (PyErr_Occurred()) return nullptr;
    const at::ScalarType type = bf16 ? at::kBFloat16 : at::kFloat;
    const at::Tensor& x = THPVariable_Unpack(args[4]);
    if (x.dim() != 2 || !matches(x, type, x.size(0), D)) Py_RETURN_NONE;
    const int64_t B = x.size(0);
    if (args[5] != Py_None && (!THPVariable_Check(args[5]) || !matches(THPVariable_Unpack(args[5]), type, B, O))) Py_RETURN_NONE;
    if (args[6] != Py_None && (!THPVariable_Check(args[6]) || !matches(THPVariable_Unpack(args[6]), at::kInt, B, -1))) Py_RETURN_NONE;
    at::Tensor y, leaf;
    void* stream = nullptr;
    if (args[8] == Py_None) stream = c10::cuda::getCurrentCUDAStream().stream();
    else stream = PyLong_AsVoidPtr(args[8]);
    if (PyErr_Occurred()) return nullptr;
    if (args[5] != Py_None) y = THPVariable_Unpack(args[5]);
    else y = at::empty({B, O}, x.options().requires_grad(false));
    if (args[6] != Py_None) leaf = THPVariable_Unpack(args[6]);
    else if (want_leaf) leaf = at::empty({B}, x.options().requires_grad(false).dtype(at::kInt));
    const void* xp = x.data_ptr();
    void* yp = y.data_ptr();
    int32_t* lp = leaf.defined() ? static_cast<int32_t*>(leaf.data_ptr()) : nullptr;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = g_forward(handle, xp, yp, lp, B, stream);
    Py_END_ALLOW_THREADS
    PyObject* py = args[5] != Py_None ? (Py_INCREF(args[5]), args[5]) : THPVariable_Wrap(std::move(y));
    PyObject* pl = args[6] != Py_None   ? (Py_INCREF(args[6]), args[6])
                   : leaf.defined()     ? THPVariable_Wrap(std::move(leaf))
                                        : (Py_INCREF(Py_None), Py_None);
    PyObject* ps = PyLong_FromLong(status);
    PyObject* out = py && pl && ps ? PyTuple_New(3) : nullptr;
    if (!out) {
        Py_XDECREF(py); Py_XDECREF(pl); Py_XDECREF(ps);
        return nullptr;
    }
    PyTuple_SET_ITEM(out, 0, ps);
    PyTuple_SET_ITEM(out, 1, py);
    PyTuple_SET_ITEM(out, 2, pl);
    return out;
    END_HANDLE_TH_ERRORS
}

PyMethodDef kMethods[] = {
    {"set_address", set_address, METH_O, "Address of fff_forward_infer."},
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, "Tensor-level fff_forward_infer."},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "torch_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_torch_call() { return PyModule_Create(&kModule); }
