// The Python binding's short way into the two products (lowra_lora_forward, lowra_lora_backward_input): tensor checks, the output's and
// the scratch's memory and the call itself without an interpreted line between them; and the tensor checks of the other calls.  A call for few tokens is two launches of 2.5 us each
// and 10 us on the GPU; with every check, pointer and argument handled by the interpreter its host side took 12 to 14 us.
//
// forward / backward_input(layout address, its device, packed, absmax, maps, act, A, B, s, out or None, workspace or None) returns the output,
// a status that is not LOWRA_OK, or None for everything that is not the ordinary case - other types, memory of other devices than the
// current one, other layouts in memory, shapes that do not fit, arrays that are too short, subclasses, errors: the caller then takes the
// interpreted way, which says what is wrong.
#include <torch/extension.h>

#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>

#include "lowra.h"

namespace {

using Product = lowra_status (*)(const lowra_layout*, const uint8_t*, const float*, const float*, const uint16_t*, int32_t, const uint16_t*,
                                 const uint16_t*, int32_t, float, uint16_t*, void*, size_t, void*);
using WorkspaceBytes = size_t (*)(const lowra_layout*, int32_t, int32_t);
using WorkspaceInit = lowra_status (*)(void*, size_t, void*);
struct Library {
    Product forward, backward_input;
    WorkspaceBytes workspace_bytes;
    WorkspaceInit workspace_init;
} library;

bool plain(PyObject* o) { return THPVariable_CheckExact(o); }

// memory of device `dev` without gaps
bool on(const at::Tensor& t, int64_t dev) { return t.device() == at::Device(at::kCUDA, (c10::DeviceIndex)dev) && t.is_contiguous(); }
bool matrix(const at::Tensor& t, int64_t rows, int64_t cols, int64_t dev) {
    return on(t, dev) && t.scalar_type() == at::kBFloat16 && t.dim() == 2 && t.size(0) == rows && t.size(1) == cols;
}
bool array(const at::Tensor& t, at::ScalarType type, int64_t least, int64_t dev) { return on(t, dev) && t.scalar_type() == type && t.numel() >= least; }

// Other Python threads run while one of these lives.
struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }
};

PyObject* product(PyObject* const* args, Py_ssize_t n, bool backward) {
    if (n != 11 || library.forward == nullptr) Py_RETURN_NONE;
    for (int i = 2; i <= 7; ++i)
        if (!plain(args[i])) Py_RETURN_NONE;
    const bool out_given = args[9] != Py_None, workspace_given = args[10] != Py_None;
    if ((out_given && !plain(args[9])) || (workspace_given && !plain(args[10])) || !(PyFloat_CheckExact(args[8]) || PyLong_CheckExact(args[8]))) Py_RETURN_NONE;
    const lowra_layout* layout = static_cast<const lowra_layout*>(PyLong_AsVoidPtr(args[0]));
    const long dev = PyLong_AsLong(args[1]);
    const double s = PyFloat_AsDouble(args[8]);
    if (PyErr_Occurred() != nullptr || layout == nullptr) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    try {
        const at::Tensor &packed = THPVariable_Unpack(args[2]), &absmax = THPVariable_Unpack(args[3]), &maps = THPVariable_Unpack(args[4]);
        const at::Tensor &act = THPVariable_Unpack(args[5]), &A = THPVariable_Unpack(args[6]), &B = THPVariable_Unpack(args[7]);
        if (act.dim() != 2 || A.dim() != 2 || dev != c10::cuda::current_device()) Py_RETURN_NONE;
        const int64_t M = act.size(0), r = A.size(1), N = layout->N, K = layout->K, cols = backward ? K : N;
        if (!matrix(act, M, backward ? N : K, dev) || !matrix(A, K, r, dev) || !matrix(B, r, N, dev) || M > INT32_MAX || r > INT32_MAX) Py_RETURN_NONE;
        if (!on(packed, dev) || packed.nbytes() < layout->packed_bytes || !array(absmax, at::kFloat, N * (K / 64), dev) || !array(maps, at::kFloat, N * 16, dev)) Py_RETURN_NONE;
        if (out_given && !array(THPVariable_Unpack(args[9]), at::kBFloat16, M * cols, dev)) Py_RETURN_NONE;
        if (workspace_given && !on(THPVariable_Unpack(args[10]), dev)) Py_RETURN_NONE;
        const Product call = backward ? library.backward_input : library.forward;
        const auto* packed_p = static_cast<const uint8_t*>(packed.data_ptr());
        const auto *absmax_p = static_cast<const float*>(absmax.data_ptr()), *maps_p = static_cast<const float*>(maps.data_ptr());
        const auto *act_p = static_cast<const uint16_t*>(act.data_ptr()), *A_p = static_cast<const uint16_t*>(A.data_ptr()), *B_p = static_cast<const uint16_t*>(B.data_ptr());
        const at::TensorOptions options = act.options().requires_grad(false);
        at::Tensor out, workspace;
        if (out_given) out = THPVariable_Unpack(args[9]);
        if (workspace_given) workspace = THPVariable_Unpack(args[10]);
        lowra_status st = LOWRA_ERR_WORKSPACE;
        bool called = false;
        {
            Released released;      // (allocations included: one that has to ask the driver for memory takes its time)
            void* stream = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream();
            if (!out_given) out = at::empty({M, cols}, options);
            bool ready = true;
            if (!workspace_given) {
                const size_t bytes = library.workspace_bytes(layout, (int32_t)M, (int32_t)r);
                ready = bytes > 0;
                if (ready) workspace = at::empty({(int64_t)bytes}, options.dtype(at::kByte));
                if (ready && layout->deal_dev != nullptr) ready = library.workspace_init(workspace.data_ptr(), bytes, stream) == LOWRA_OK;   // no prologue launch will clear it
            }
            if (ready) {
                st = call(layout, packed_p, absmax_p, maps_p, act_p, (int32_t)M, A_p, B_p, (int32_t)r, (float)s, static_cast<uint16_t*>(out.data_ptr()),
                          workspace.data_ptr(), (size_t)workspace.numel(), stream);
                called = true;
            }
        }
        if (!called) Py_RETURN_NONE;
        if (st != LOWRA_OK) return PyLong_FromLong(st);
        if (out_given) {
            Py_INCREF(args[9]);
            return args[9];
        }
        return THPVariable_Wrap(std::move(out));
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyObject* forward(PyObject*, PyObject* const* args, Py_ssize_t n) { return product(args, n, false); }
PyObject* backward_input(PyObject*, PyObject* const* args, Py_ssize_t n) { return product(args, n, true); }

// fits(device, then for each array: tensor or None, element type, least number of elements) -> whether every one is a plain tensor on that
// device, which is the current one, without gaps, of that type and long enough; None fits.  Types: 'B' bytes of any type, 'u' uint8, 'h' bf16,
// 'f' fp32, 'd' fp64.  The other calls' checks, a tenth of a microsecond an array where the interpreter takes one; what does not fit is looked at
// by the interpreter, which says what is wrong.
PyObject* fits(PyObject*, PyObject* const* args, Py_ssize_t n) {
    const long dev = n % 3 == 1 ? PyLong_AsLong(args[0]) : -1;
    bool good = dev >= 0;
    try {
        good = good && dev == c10::cuda::current_device();
        for (Py_ssize_t i = 1; good && i < n; i += 3) {
            if (args[i] == Py_None) continue;
            const Py_UCS4 type = PyUnicode_Check(args[i + 1]) && PyUnicode_GET_LENGTH(args[i + 1]) == 1 ? PyUnicode_READ_CHAR(args[i + 1], 0) : 0;
            const int64_t least = PyLong_AsLongLong(args[i + 2]);
            if (!plain(args[i])) { good = false; break; }
            const at::Tensor& t = THPVariable_Unpack(args[i]);
            if (type == 'B') good = on(t, dev) && (int64_t)t.nbytes() >= least;
            else good = type != 0 && array(t, type == 'u' ? at::kByte : type == 'h' ? at::kBFloat16 : type == 'f' ? at::kFloat : at::kDouble, least, dev);
        }
    } catch (...) {
        good = false;
    }
    if (PyErr_Occurred() != nullptr) {
        PyErr_Clear();
        good = false;
    }
    return PyBool_FromLong(good);
}

// bind(addresses of lowra_lora_forward, lowra_lora_backward_input, lowra_workspace_bytes, lowra_workspace_init)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    void* p[4] = {};
    for (int i = 0; i < 4; ++i) {
        p[i] = i < n ? PyLong_AsVoidPtr(args[i]) : nullptr;
        if (p[i] == nullptr) {
            if (PyErr_Occurred() == nullptr) PyErr_SetString(PyExc_ValueError, "bind takes four addresses");
            return nullptr;
        }
    }
    library = Library{reinterpret_cast<Product>(p[0]), reinterpret_cast<Product>(p[1]), reinterpret_cast<WorkspaceBytes>(p[2]), reinterpret_cast<WorkspaceInit>(p[3])};
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"forward", (PyCFunction)(void (*)())forward, METH_FASTCALL, nullptr},
    {"backward_input", (PyCFunction)(void (*)())backward_input, METH_FASTCALL, nullptr},
    {"fits", (PyCFunction)(void (*)())fits, METH_FASTCALL, nullptr},
    {"bind", (PyCFunction)(void (*)())bind, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_py_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__py_calls() { return PyModule_Create(&module); }
