// The Python binding's short way into the two products (lowra_lora_forward, lowra_lora_backward_input), their batches, and the gradients of the factors:
// tensor checks, the outputs' and the scratch's memory and the call itself without an interpreted line between them; and the tensor checks of the other calls.
// A call for few tokens is one or two launches of 2.5 us each and 5 to 9 us on the GPU; with every check, pointer and argument handled by the interpreter
// its host side took 12 to 14 us.  Host time of the others (256 x 512, 128 tokens, rank 48), us: a batch of three 16.3 -> 5.2, gradients 17.3 -> 8.6, from kept
// projections 13.5 -> 6.4, such a projection's view 5.2 -> 1.6; a training step of three weights 135 -> 66.
//
// forward / backward_input(layout address, its device, packed, absmax, maps, act, A, B, s, out or None, workspace or None) returns the output,
// a status that is not LOWRA_OK, or None for everything that is not the ordinary case - other types, memory of other devices than the
// current one, other layouts in memory, shapes that do not fit, arrays that are too short, subclasses, errors: the caller then takes the
// interpreted way, which says what is wrong.  Likewise
//   batch(backward, members, s, workspace)                                          the list of outputs
//   gradients(X, dY, A, B, s, dA or None, dB or None, workspace or None)            the pair of gradients
//   gradients_reuse(X, dY, T, U, r, dA or None, dB or None, workspace or None)      likewise
//   projection(workspace, M, r, member)                                             its view of the workspace
#include <torch/extension.h>

#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>

#include "lowra.h"

namespace {

using Product = lowra_status (*)(const lowra_layout*, const uint8_t*, const float*, const float*, const uint16_t*, int32_t, const uint16_t*,
                                 const uint16_t*, int32_t, float, uint16_t*, void*, size_t, void*);
using WorkspaceBytes = size_t (*)(const lowra_layout*, int32_t, int32_t);
using WorkspaceInit = lowra_status (*)(void*, size_t, void*);
using Batch = lowra_status (*)(const lowra_member*, int32_t, int32_t, int32_t, float, void*, size_t, void*);
using Gradients = lowra_status (*)(const uint16_t*, const uint16_t*, int32_t, int32_t, int32_t, const uint16_t*, const uint16_t*, int32_t, float, uint16_t*, uint16_t*,
                                   void*, size_t, void*);
using GradientsReuse = lowra_status (*)(const uint16_t*, const uint16_t*, int32_t, int32_t, int32_t, const uint16_t*, const uint16_t*, int32_t, uint16_t*, uint16_t*, void*,
                                        size_t, void*);
using GradientsBytes = size_t (*)(int32_t, int32_t);
using Projection = const uint16_t* (*)(const void*, int32_t, int32_t, int32_t);
struct Library {
    Product forward, backward_input;
    WorkspaceBytes workspace_bytes;
    WorkspaceInit workspace_init;
    Batch forward_batch, backward_input_batch;
    Gradients gradients;
    GradientsReuse gradients_reuse;
    GradientsBytes gradients_bytes;
    Projection projection;
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

// A reference of ours.
struct Held {
    PyObject* o = nullptr;
    ~Held() { Py_XDECREF(o); }
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

// A number, or not: an exact int within an int32, an exact float or int.
bool number(PyObject* o, int32_t* v) {
    int overflow = 0;
    const long long x = PyLong_CheckExact(o) ? PyLong_AsLongLongAndOverflow(o, &overflow) : -1;
    *v = (int32_t)x;
    return PyLong_CheckExact(o) && overflow == 0 && x >= 0 && x <= INT32_MAX;
}
bool number(PyObject* o, double* v) {
    if (!PyFloat_CheckExact(o) && !PyLong_CheckExact(o)) return false;
    *v = PyFloat_AsDouble(o);
    if (PyErr_Occurred() == nullptr) return true;
    PyErr_Clear();
    return false;
}
uint16_t* bf16(const at::Tensor& t) { return static_cast<uint16_t*>(t.data_ptr()); }

// gradients(X, dY, A, B, s, dA, dB, workspace), and with `reuse` (X, dY, T, U, r, dA, dB, workspace)
PyObject* factor_gradients(PyObject* const* args, Py_ssize_t n, bool reuse) {
    double s = 0.0;
    int32_t rank = 0;
    if (n != 8 || library.forward == nullptr || !(reuse ? number(args[4], &rank) : number(args[4], &s))) Py_RETURN_NONE;
    for (int i = 0; i < 8; ++i)
        if (i != 4 && !(i > 4 && args[i] == Py_None) && !plain(args[i])) Py_RETURN_NONE;
    try {
        const int64_t dev = c10::cuda::current_device();
        const at::Tensor &X = THPVariable_Unpack(args[0]), &dY = THPVariable_Unpack(args[1]), &P = THPVariable_Unpack(args[2]), &Q = THPVariable_Unpack(args[3]);
        if (X.dim() != 2 || dY.dim() != 2 || P.dim() != 2) Py_RETURN_NONE;
        const int64_t M = X.size(0), K = X.size(1), N = dY.size(1), r = reuse ? rank : P.size(1), rp = (r + 63) / 64 * 64;
        if (M > INT32_MAX || K > INT32_MAX || N > INT32_MAX || r > INT32_MAX || !matrix(X, M, K, dev) || !matrix(dY, M, N, dev)) Py_RETURN_NONE;
        if (reuse ? !matrix(P, M, rp, dev) || !matrix(Q, M, rp, dev) : !matrix(P, K, r, dev) || !matrix(Q, r, N, dev)) Py_RETURN_NONE;
        at::Tensor out[2], workspace;
        for (int i = 0; i < 2; ++i) {
            if (args[5 + i] == Py_None) continue;
            out[i] = THPVariable_Unpack(args[5 + i]);
            if (!array(out[i], at::kBFloat16, i == 0 ? K * r : r * N, dev)) Py_RETURN_NONE;
        }
        if (args[7] != Py_None) {
            workspace = THPVariable_Unpack(args[7]);
            if (!on(workspace, dev)) Py_RETURN_NONE;
        }
        const size_t bytes = reuse ? 256 : library.gradients_bytes((int32_t)M, (int32_t)r);
        if (bytes == 0) Py_RETURN_NONE;
        const at::TensorOptions options = X.options().requires_grad(false);
        lowra_status st;
        {
            Released released;
            void* stream = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream();
            if (!out[0].defined()) out[0] = at::empty({K, r}, options);
            if (!out[1].defined()) out[1] = at::empty({r, N}, options);
            if (!workspace.defined()) workspace = at::empty({(int64_t)bytes}, options.dtype(at::kByte));
            const size_t size = (size_t)workspace.numel();
            st = reuse ? library.gradients_reuse(bf16(X), bf16(dY), (int32_t)M, (int32_t)K, (int32_t)N, bf16(P), bf16(Q), (int32_t)r, bf16(out[0]), bf16(out[1]),
                                                 workspace.data_ptr(), size, stream)
                       : library.gradients(bf16(X), bf16(dY), (int32_t)M, (int32_t)K, (int32_t)N, bf16(P), bf16(Q), (int32_t)r, (float)s, bf16(out[0]), bf16(out[1]),
                                           workspace.data_ptr(), size, stream);
        }
        if (st != LOWRA_OK) return PyLong_FromLong(st);
        PyObject* both = PyTuple_New(2);
        for (int i = 0; both != nullptr && i < 2; ++i) {
            PyObject* o = args[5 + i];
            if (o != Py_None) Py_INCREF(o);
            else o = THPVariable_Wrap(std::move(out[i]));
            PyTuple_SET_ITEM(both, i, o);
        }
        return both;
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyObject* gradients(PyObject*, PyObject* const* args, Py_ssize_t n) { return factor_gradients(args, n, false); }
PyObject* gradients_reuse(PyObject*, PyObject* const* args, Py_ssize_t n) { return factor_gradients(args, n, true); }

PyObject* projection(PyObject*, PyObject* const* args, Py_ssize_t n) {
    int32_t M = 0, r = 0, member = 0;
    if (n != 4 || library.forward == nullptr || !plain(args[0]) || !number(args[1], &M) || !number(args[2], &r) || !number(args[3], &member)) Py_RETURN_NONE;
    try {
        const at::Tensor& workspace = THPVariable_Unpack(args[0]);
        if (workspace.dim() != 1 || !array(workspace, at::kByte, 0, c10::cuda::current_device())) Py_RETURN_NONE;
        const auto* p = reinterpret_cast<const uint8_t*>(library.projection(workspace.data_ptr(), member, M, r));
        if (p == nullptr) Py_RETURN_NONE;
        const int64_t from = p - static_cast<const uint8_t*>(workspace.data_ptr()), rp = ((int64_t)r + 63) / 64 * 64, bytes = (int64_t)M * rp * 2;
        if (from + bytes > workspace.numel()) Py_RETURN_NONE;
        return THPVariable_Wrap(workspace.slice(0, from, from + bytes).view(at::kBFloat16).view({(int64_t)M, rp}));
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// batch(backward, members, s, workspace): a list of dicts with layout, packed, absmax, maps, act, A, B, out
PyObject* batch(PyObject*, PyObject* const* args, Py_ssize_t n) {
    double s = 0.0;
    if (n != 4 || library.forward == nullptr || !PyBool_Check(args[0]) || !PyList_CheckExact(args[1]) || !number(args[2], &s) || !plain(args[3])) Py_RETURN_NONE;
    const bool backward = args[0] == Py_True;
    const Py_ssize_t count = PyList_GET_SIZE(args[1]);
    if (count < 1 || count > LOWRA_MAX_BATCH) Py_RETURN_NONE;
    static PyObject* names[10] = {};      // (interned once)
    if (names[9] == nullptr) {
        constexpr const char* kNames[10] = {"packed", "absmax", "maps", "act", "A", "B", "out", "layout", "address", "device_index"};
        for (int i = 0; i < 10; ++i) names[i] = PyUnicode_InternFromString(kNames[i]);
    }
    // the members' arrays, layouts and outputs: their dicts are the caller's, and other threads run during the call
    at::Tensor arrays[LOWRA_MAX_BATCH][7];
    Held layouts[LOWRA_MAX_BATCH], outs[LOWRA_MAX_BATCH];
    lowra_member members[LOWRA_MAX_BATCH];
    try {
        const int64_t dev = c10::cuda::current_device();
        const at::Tensor& workspace = THPVariable_Unpack(args[3]);
        if (!on(workspace, dev)) Py_RETURN_NONE;
        int64_t M = 0, r = 0;
        for (Py_ssize_t i = 0; i < count; ++i) {
            PyObject* m = PyList_GET_ITEM(args[1], i);
            if (!PyDict_CheckExact(m)) Py_RETURN_NONE;
            PyObject* o = nullptr;
            for (int j = 0; j < 7; ++j) {
                o = PyDict_GetItemWithError(m, names[j]);
                if (o == nullptr || !plain(o)) {
                    PyErr_Clear();
                    Py_RETURN_NONE;
                }
                arrays[i][j] = THPVariable_Unpack(o);
            }
            outs[i].o = Py_NewRef(o);
            layouts[i].o = Py_XNewRef(PyDict_GetItemWithError(m, names[7]));
            Held address, where;
            if (layouts[i].o != nullptr) address.o = PyObject_GetAttr(layouts[i].o, names[8]);
            if (address.o != nullptr) where.o = PyObject_GetAttr(layouts[i].o, names[9]);
            const bool known = where.o != nullptr && PyLong_CheckExact(address.o) && PyLong_CheckExact(where.o);
            const auto* layout = known ? static_cast<const lowra_layout*>(PyLong_AsVoidPtr(address.o)) : nullptr;
            const bool here = known && PyLong_AsLong(where.o) == dev;
            PyErr_Clear();
            if (layout == nullptr || !here) Py_RETURN_NONE;
            const at::Tensor &packed = arrays[i][0], &absmax = arrays[i][1], &maps = arrays[i][2], &act = arrays[i][3], &A = arrays[i][4], &B = arrays[i][5], &out = arrays[i][6];
            const int64_t N = layout->N, K = layout->K;
            if (i == 0) {
                if (act.dim() != 2 || A.dim() != 2) Py_RETURN_NONE;
                M = act.size(0);
                r = A.size(1);
            }
            if (M > INT32_MAX || r > INT32_MAX || !matrix(act, M, backward ? N : K, dev) || !matrix(out, M, backward ? K : N, dev) || !matrix(A, K, r, dev) ||
                !matrix(B, r, N, dev) || !on(packed, dev) || packed.nbytes() < layout->packed_bytes || !array(absmax, at::kFloat, N * (K / 64), dev) ||
                !array(maps, at::kFloat, N * 16, dev))
                Py_RETURN_NONE;
            members[i] = lowra_member{layout, static_cast<const uint8_t*>(packed.data_ptr()), static_cast<const float*>(absmax.data_ptr()),
                                      static_cast<const float*>(maps.data_ptr()), bf16(act), bf16(A), bf16(B), bf16(out)};
        }
        lowra_status st;
        {
            Released released;
            st = (backward ? library.backward_input_batch : library.forward_batch)(members, (int32_t)count, (int32_t)M, (int32_t)r, (float)s, workspace.data_ptr(),
                                                                                  (size_t)workspace.numel(), c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream());
        }
        if (st != LOWRA_OK) return PyLong_FromLong(st);
        PyObject* list = PyList_New(count);
        for (Py_ssize_t i = 0; list != nullptr && i < count; ++i) PyList_SET_ITEM(list, i, Py_NewRef(outs[i].o));
        return list;
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

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

// bind(addresses of lowra_lora_forward, lowra_lora_backward_input, lowra_workspace_bytes, lowra_workspace_init, lowra_lora_forward_batch, lowra_lora_backward_input_batch,
// lowra_lora_backward_adapters, lowra_lora_backward_adapters_reuse, lowra_adapter_workspace_bytes, lowra_workspace_projection)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    void* p[10] = {};
    for (int i = 0; i < 10; ++i) {
        p[i] = i < n ? PyLong_AsVoidPtr(args[i]) : nullptr;
        if (p[i] == nullptr) {
            if (PyErr_Occurred() == nullptr) PyErr_SetString(PyExc_ValueError, "bind takes ten addresses");
            return nullptr;
        }
    }
    library = Library{reinterpret_cast<Product>(p[0]), reinterpret_cast<Product>(p[1]), reinterpret_cast<WorkspaceBytes>(p[2]), reinterpret_cast<WorkspaceInit>(p[3]),
                      reinterpret_cast<Batch>(p[4]), reinterpret_cast<Batch>(p[5]), reinterpret_cast<Gradients>(p[6]), reinterpret_cast<GradientsReuse>(p[7]),
                      reinterpret_cast<GradientsBytes>(p[8]), reinterpret_cast<Projection>(p[9])};
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"forward", (PyCFunction)(void (*)())forward, METH_FASTCALL, nullptr},
    {"backward_input", (PyCFunction)(void (*)())backward_input, METH_FASTCALL, nullptr},
    {"batch", (PyCFunction)(void (*)())batch, METH_FASTCALL, nullptr},
    {"gradients", (PyCFunction)(void (*)())gradients, METH_FASTCALL, nullptr},
    {"gradients_reuse", (PyCFunction)(void (*)())gradients_reuse, METH_FASTCALL, nullptr},
    {"projection", (PyCFunction)(void (*)())projection, METH_FASTCALL, nullptr},
    {"fits", (PyCFunction)(void (*)())fits, METH_FASTCALL, nullptr},
    {"bind", (PyCFunction)(void (*)())bind, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_py_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__py_calls() { return PyModule_Create(&module); }
