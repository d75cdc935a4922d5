// The plain forms of the smallest calls without the interpreter's part: rows in, new buffers out, on the current stream.  A call of a
// few microseconds on the GPU is bound by what happens before it; the checks, the allocations and the argument marshalling of
// binding.py take 6 us, here about one.  Whatever is not plain (given buffers, other types, shapes, strides or devices, anything
// that throws) is answered with None, and binding.py does the call or raises as it always did: there is no second set of rules.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/bfq.h"

namespace {

using ForwardQuant = int (*)(bfq_plan*, const void*, bfq_dtype, int64_t, int64_t, int, uint8_t*, uint16_t*, void*);
using Rows = int (*)(bfq_plan*, const void*, bfq_dtype, int64_t, int64_t, void*, bfq_dtype, int64_t, void*);
ForwardQuant forward_quant_fn = nullptr;
Rows forward_fn = nullptr, inverse_fn = nullptr;

struct Call {
    bfq_plan* plan;
    int64_t n;
    int device;
    const at::Tensor* x;
    bfq_dtype type;
    int64_t rows, ld;
};

// arguments (plan handle, n, device index, x): false if x is not plain rows of n numbers on that device
bool plain_rows(PyObject* const* args, Call* call) {
    if (!THPVariable_CheckExact(args[3])) return false;
    call->plan = static_cast<bfq_plan*>(PyLong_AsVoidPtr(args[0]));
    call->n = PyLong_AsLongLong(args[1]);
    call->device = static_cast<int>(PyLong_AsLong(args[2]));
    if (PyErr_Occurred() || call->plan == nullptr) {
        PyErr_Clear();
        return false;
    }
    const at::Tensor& x = THPVariable_Unpack(args[3]);
    if (!x.is_cuda() || x.get_device() != call->device || x.dim() != 2) return false;
    const auto type = x.scalar_type();
    if (type != at::kBFloat16 && type != at::kFloat) return false;
    call->x = &x, call->type = type == at::kFloat ? BFQ_F32 : BFQ_BF16;
    call->rows = x.size(0), call->ld = x.stride(0);
    return call->rows > 0 && x.size(1) == call->n && x.stride(1) == 1 && call->ld >= call->n;
}

// f(stream) without the interpreter's lock
template <class F>
int launch(const Call& call, F&& f) {
    void* stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(call.device)).stream();
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = f(stream);
    Py_END_ALLOW_THREADS
    return status;
}

// forward_quant(plan, n, device, x, bits) -> (codes, scales), or a status, or None
PyObject* forward_quant(PyObject*, PyObject* const* args, Py_ssize_t count) {
    try {
        Call call;
        if (count != 5 || forward_quant_fn == nullptr || !PyLong_CheckExact(args[4]) || !plain_rows(args, &call)) Py_RETURN_NONE;
        const long bits = PyLong_AsLong(args[4]);
        if (bits != 2 && bits != 4 && bits != 8) {
            PyErr_Clear();
            Py_RETURN_NONE;
        }
        const c10::Device device(c10::kCUDA, static_cast<c10::DeviceIndex>(call.device));
        at::Tensor codes = at::empty({call.rows, call.n * bits / 8}, at::TensorOptions().dtype(at::kByte).device(device));
        at::Tensor scales = at::empty({call.rows}, at::TensorOptions().dtype(at::kHalf).device(device));
        const void* x = call.x->data_ptr();
        uint8_t* to = static_cast<uint8_t*>(codes.data_ptr());
        uint16_t* scale = static_cast<uint16_t*>(scales.data_ptr());
        const int status = launch(call, [&](void* stream) {
            return forward_quant_fn(call.plan, x, call.type, call.rows, call.ld, static_cast<int>(bits), to, scale, stream);
        });
        if (status != BFQ_OK) return PyLong_FromLong(status);
        PyObject* first = THPVariable_Wrap(std::move(codes));
        PyObject* second = first != nullptr ? THPVariable_Wrap(std::move(scales)) : nullptr;
        PyObject* both = second != nullptr ? PyTuple_Pack(2, first, second) : nullptr;
        Py_XDECREF(first), Py_XDECREF(second);
        return both;
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// forward / inverse(plan, n, device, x) -> rows in the type of x, or a status, or None
PyObject* rows_call(Rows fn, PyObject* const* args, Py_ssize_t count) {
    try {
        Call call;
        if (count != 4 || fn == nullptr || !plain_rows(args, &call)) Py_RETURN_NONE;
        at::Tensor y = at::empty({call.rows, call.n}, call.x->options());
        const void* x = call.x->data_ptr();
        void* to = y.data_ptr();
        const int status = launch(call, [&](void* stream) { return fn(call.plan, x, call.type, call.rows, call.ld, to, call.type, call.n, stream); });
        if (status != BFQ_OK) return PyLong_FromLong(status);
        return THPVariable_Wrap(std::move(y));
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}
PyObject* forward(PyObject*, PyObject* const* args, Py_ssize_t count) { return rows_call(forward_fn, args, count); }
PyObject* inverse(PyObject*, PyObject* const* args, Py_ssize_t count) { return rows_call(inverse_fn, args, count); }

// attach(path of libbfq.so): the library binding.py has loaded
PyObject* attach(PyObject*, PyObject* path) {
    const char* name = PyUnicode_AsUTF8(path);
    if (name == nullptr) return nullptr;
    void* lib = dlopen(name, RTLD_NOW | RTLD_LOCAL);
    void* found[3] = {};
    const char* names[3] = {"bfq_forward_quant", "bfq_forward", "bfq_inverse"};
    for (int i = 0; i < 3; ++i)
        if (lib == nullptr || (found[i] = dlsym(lib, names[i])) == nullptr) {
            const char* why = dlerror();
            PyErr_SetString(PyExc_OSError, why != nullptr ? why : names[i]);
            return nullptr;
        }
    forward_quant_fn = reinterpret_cast<ForwardQuant>(found[0]);
    forward_fn = reinterpret_cast<Rows>(found[1]), inverse_fn = reinterpret_cast<Rows>(found[2]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"attach", attach, METH_O, nullptr},
    {"forward_quant", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward_quant)), METH_FASTCALL, nullptr},
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, nullptr},
    {"inverse", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(inverse)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "fast_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_fast_calls() {
    PyObject* m = PyModule_Create(&module);
    // calls nothing of torch's: the binding asks for this before it uses the module with the torch that is there
    if (m != nullptr && PyModule_AddStringConstant(m, "torch_version", BFQ_TORCH) < 0) Py_CLEAR(m);
    return m;
}
