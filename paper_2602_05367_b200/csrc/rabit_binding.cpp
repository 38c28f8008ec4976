// The Python side of the hot calls, in native code: argument checks, output allocation, the current stream and the call
// into the C ABI, without the interpreter's and ctypes' cost per call.  At batch 1 a layer lasts two to seven
// microseconds on the device; the same steps in Python took 10.6 us per rabit_linear call (torch.empty 2.5,
// torch.cuda.current_stream 2.3, the ctypes call 3.3 of which the launch is most, the rest attribute look-ups), so an
// eager decoder was bound by its host.
//
// The module calls the library through addresses handed to init(), so that it serves whichever build of librabit.so the
// package has loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/Functions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <cstdint>
#include <vector>

namespace {

typedef int (*LinearFn)(const void*, const void*, void*, int, void*);
typedef int (*GroupFn)(const void* const*, const void* const*, void* const*, int, int, void*);
typedef int (*GroupHostFn)(const void* const*, const void* const*, void* const*, int, int, void*, size_t, void*);
typedef int (*DimFn)(const void*);
typedef const char* (*ErrorFn)();

LinearFn p_linear = nullptr;
GroupFn p_group = nullptr;
GroupHostFn p_group_host = nullptr;
DimFn p_M = nullptr, p_N = nullptr;
ErrorFn p_error = nullptr;
PyObject* g_error_type = nullptr;      // RabitError
PyObject* g_addr_name = nullptr;       // "_addr": the descriptor's address on a RabitLayer, None once freed

constexpr Py_ssize_t kInline = 16;     // layers of a group whose pointers need no allocation

PyObject* raise_code(int code, const char* msg) {
    PyObject* args = Py_BuildValue("(is)", code, msg);
    if (args) {
        PyErr_SetObject(g_error_type, args);          // the type is called with (code, message)
        Py_DECREF(args);
    }
    return nullptr;
}

void* layer_handle(PyObject* layer) {
    PyObject* a = PyObject_GetAttr(layer, g_addr_name);
    if (!a) return nullptr;
    void* p = nullptr;
    if (a == Py_None) raise_code(-1, "layer already freed");
    else p = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    return p;
}

// stream argument: an integer, or None for torch's current stream on that device
bool stream_of(PyObject* arg, c10::DeviceIndex device, void** out) {
    if (arg == Py_None) {
        *out = (void*)c10::cuda::getCurrentCUDAStream(device).stream();
        return true;
    }
    *out = PyLong_AsVoidPtr(arg);
    return !(*out == nullptr && PyErr_Occurred());
}

inline bool is_cuda_half(PyObject* o) {
    if (!THPVariable_Check(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.scalar_type() == at::kHalf && t.is_cuda() && t.is_contiguous();
}

// linear(layer, x, y | None, stream | None) -> y
PyObject* linear(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 4) return PyErr_Format(PyExc_TypeError, "linear takes 4 arguments");
    HANDLE_TH_ERRORS
    if (!is_cuda_half(args[1])) return PyErr_Format(PyExc_ValueError, "x must be a contiguous CUDA float16 tensor");
    const void* h = layer_handle(args[0]);
    if (!h) return nullptr;
    const at::Tensor& x = THPVariable_Unpack(args[1]);
    const int64_t M = p_M(h), N = p_N(h);
    const bool flat = x.dim() != 2;
    const int64_t batch = flat ? 1 : x.size(0), cols = flat ? x.numel() : x.size(1);
    if (cols != N) return PyErr_Format(PyExc_ValueError, "x has %lld columns, layer expects %lld", (long long)cols, (long long)N);
    at::Tensor made;
    void* yp;
    if (args[2] == Py_None) {
        made = at::empty({batch, M}, at::TensorOptions().dtype(at::kHalf).device(x.device()));
        yp = made.data_ptr();
    } else {
        if (!is_cuda_half(args[2]) || THPVariable_Unpack(args[2]).numel() != batch * M)
            return PyErr_Format(PyExc_ValueError, "y must be a contiguous CUDA float16 tensor of batch*M elements");
        yp = THPVariable_Unpack(args[2]).data_ptr();
    }
    void* stream;
    if (!stream_of(args[3], x.device().index(), &stream)) return nullptr;
    const void* xp = x.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = p_linear(h, xp, yp, (int)batch, stream);
    Py_END_ALLOW_THREADS
    if (rc != 0) return raise_code(rc, p_error());
    if (args[2] == Py_None) return THPVariable_Wrap(flat ? made.view({-1}) : made);
    if (flat) return THPVariable_Wrap(THPVariable_Unpack(args[2]).view({-1}));
    Py_INCREF(args[2]);
    return args[2];
    END_HANDLE_TH_ERRORS
}

// linear_group(layers, xs, ys, stream | None) -> ys
PyObject* linear_group(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 4) return PyErr_Format(PyExc_TypeError, "linear_group takes 4 arguments");
    HANDLE_TH_ERRORS
    THPObjectPtr ls(PySequence_Fast(args[0], "layers must be a sequence")), xs(PySequence_Fast(args[1], "xs must be a sequence")),
        ys(PySequence_Fast(args[2], "ys must be a sequence"));
    if (!ls || !xs || !ys) return nullptr;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(ls.get());
    if (n < 1 || PySequence_Fast_GET_SIZE(xs.get()) != n || PySequence_Fast_GET_SIZE(ys.get()) != n)
        return PyErr_Format(PyExc_ValueError, "layers, xs and ys must have the same, non-zero length");
    void* inl[3 * kInline];
    std::vector<void*> more;
    void** hp = inl;
    if (n > kInline) {
        more.resize(3 * (size_t)n);
        hp = more.data();
    }
    void **xp = hp + n, **yp = hp + 2 * n;
    int64_t batch = 0;
    c10::DeviceIndex device = 0;
    for (Py_ssize_t l = 0; l < n; ++l) {
        PyObject *xo = PySequence_Fast_GET_ITEM(xs.get(), l), *yo = PySequence_Fast_GET_ITEM(ys.get(), l);
        hp[l] = layer_handle(PySequence_Fast_GET_ITEM(ls.get(), l));
        if (!hp[l]) return nullptr;
        if (l == 0 && THPVariable_Check(xo)) {
            const at::Tensor& x0 = THPVariable_Unpack(xo);
            batch = x0.dim() == 1 ? 1 : x0.dim() > 0 ? x0.size(0) : 0;
            device = x0.device().index();
        }
        if (!is_cuda_half(xo) || THPVariable_Unpack(xo).numel() != batch * p_N(hp[l]))
            return PyErr_Format(PyExc_ValueError, "every x must be a contiguous CUDA float16 tensor of batch*N elements");
        if (!is_cuda_half(yo) || THPVariable_Unpack(yo).numel() != batch * p_M(hp[l]))
            return PyErr_Format(PyExc_ValueError, "every y must be a contiguous CUDA float16 tensor of batch*M elements");
        xp[l] = THPVariable_Unpack(xo).data_ptr();
        yp[l] = THPVariable_Unpack(yo).data_ptr();
    }
    void* stream;
    if (!stream_of(args[3], device, &stream)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = p_group(hp, xp, yp, (int)n, (int)batch, stream);
    Py_END_ALLOW_THREADS
    if (rc != 0) return raise_code(rc, p_error());
    Py_INCREF(args[2]);
    return args[2];
    END_HANDLE_TH_ERRORS
}

// group_host((layers*, xs*, ys*, n, batch, stage*, stage bytes, device), stream | None): a call whose arrays were laid out before
PyObject* group_host(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 2 || !PyTuple_Check(args[0]) || PyTuple_GET_SIZE(args[0]) != 8) return PyErr_Format(PyExc_TypeError, "group_host takes a prepared tuple and a stream");
    HANDLE_TH_ERRORS
    void* v[8];
    for (int i = 0; i < 8; ++i) v[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(args[0], i));
    if (PyErr_Occurred()) return nullptr;
    void* stream;
    if (!stream_of(args[1], (c10::DeviceIndex)(intptr_t)v[7], &stream)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = p_group_host((const void* const*)v[0], (const void* const*)v[1], (void* const*)v[2], (int)(intptr_t)v[3], (int)(intptr_t)v[4], v[5],
                      (size_t)v[6], stream);
    Py_END_ALLOW_THREADS
    if (rc != 0) return raise_code(rc, p_error());
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// current_stream(device index) -> the handle of torch's current stream
PyObject* current_stream(PyObject*, PyObject* arg) {
    HANDLE_TH_ERRORS
    const long d = PyLong_AsLong(arg);
    if (d == -1 && PyErr_Occurred()) return nullptr;
    return PyLong_FromVoidPtr((void*)c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)d).stream());
    END_HANDLE_TH_ERRORS
}

// init(error type, address of rabit_linear, _linear_group, _linear_group_host, _layer_M, _layer_N, _last_error)
PyObject* init(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 7) return PyErr_Format(PyExc_TypeError, "init takes 7 arguments");
    void* v[6];
    for (int i = 0; i < 6; ++i) v[i] = PyLong_AsVoidPtr(args[1 + i]);
    if (PyErr_Occurred()) return nullptr;
    p_linear = (LinearFn)v[0];
    p_group = (GroupFn)v[1];
    p_group_host = (GroupHostFn)v[2];
    p_M = (DimFn)v[3];
    p_N = (DimFn)v[4];
    p_error = (ErrorFn)v[5];
    Py_XSETREF(g_error_type, Py_NewRef(args[0]));
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, nullptr},
    {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, nullptr},
    {"linear_group", (PyCFunction)(void (*)(void))linear_group, METH_FASTCALL, nullptr},
    {"group_host", (PyCFunction)(void (*)(void))group_host, METH_FASTCALL, nullptr},
    {"current_stream", current_stream, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_rabit_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rabit_binding(void) {
    g_addr_name = PyUnicode_InternFromString("_addr");
    return g_addr_name ? PyModule_Create(&module) : nullptr;
}
