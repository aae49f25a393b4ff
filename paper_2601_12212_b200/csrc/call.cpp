// Python side of the C ABI: argument marshalling for the entry points of include/resps.h that
// enqueue work.  A decode loop makes one such call per layer, each worth 2-20 us of GPU time, so what
// the call costs on the host decides whether an eager loop is bound by the GPU: with ctypes the
// conversion of ~17 arguments and the tensor checks took 7-8 of the 10-13 us of a call.
//
// `bind(name, address)` returns a callable for one entry point of an already loaded library.  Every
// argument has a one-letter code (below); the C types come from the declarations in resps.h.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <type_traits>
#include <utility>

#include "resps.h"

namespace {

struct Slot {
    int64_t i = 0;
    double d = 0.0;
    template <typename T>
    T as() const {
        if constexpr (std::is_pointer_v<T>)
            return reinterpret_cast<T>(static_cast<intptr_t>(i));
        else if constexpr (std::is_floating_point_v<T>)
            return static_cast<T>(d);
        else
            return static_cast<T>(i);
    }
};
constexpr int kMaxArgs = 32;

template <typename R, typename... A, size_t... I>
int invoke_with(R (*fn)(A...), const Slot* s, std::index_sequence<I...>) {
    return fn(s[I].template as<A>()...);
}
template <typename F>
struct Invoke;
template <typename R, typename... A>
struct Invoke<R (*)(A...)> {
    static constexpr int kArgs = sizeof...(A);
    static_assert(kArgs <= kMaxArgs, "argument table");
    static int call(void* fn, const Slot* s) {
        return invoke_with(reinterpret_cast<R (*)(A...)>(fn), s, std::index_sequence_for<A...>{});
    }
};

// Codes: p address, i integer, f real; tensors (None = null): I int32, L int64, F fp32, D fp64, B bf16,
// T any dtype; s stream (None = the current one).
struct Spec {
    const char* name;
    const char* codes;
    int n_args;
    int (*call)(void*, const Slot*);
};
template <typename F, size_t N>
constexpr Spec make_spec(const char* name, const char (&codes)[N]) {
    static_assert(N - 1 == Invoke<F>::kArgs, "one code per argument");
    return {name, codes, Invoke<F>::kArgs, &Invoke<F>::call};
}
#define RESPS_SPEC(fn, codes) make_spec<decltype(&fn)>(#fn, codes)
const Spec kSpecs[] = {
    RESPS_SPEC(resps_tree_expand, "pIiFiiiiiIIIIITIIIs"),
    RESPS_SPEC(resps_tree_expand_begin, "pIii"),
    RESPS_SPEC(resps_tree_expand_level, "pIiiFiiIIIITDs"),
    RESPS_SPEC(resps_tree_expand_finish, "pIiIIIIITIIIs"),
    RESPS_SPEC(resps_tree_attention, "pIIiBBFBBiiiiTfs"),
    RESPS_SPEC(resps_verify_accept, "pIIiFiiIIIIIIIs"),
    RESPS_SPEC(resps_verify_accept_sampled, "pIIiFiiFiiifIIDDIIIIs"),
    RESPS_SPEC(resps_controller_step, "ppBBBiiifDIFIIFFIs"),
    RESPS_SPEC(resps_row_scan_shard, "pIiFiiiiiFIDs"),
    RESPS_SPEC(resps_tree_expand_merge, "pIiiiiFIDIIIIIITIIIs"),
    RESPS_SPEC(resps_target_argmax_shard, "pIiFiiLs"),
    RESPS_SPEC(resps_verify_accept_merge, "pIIiiLIIIIIIIIs"),
    RESPS_SPEC(resps_kv_compact, "pIiiIILLiiiiis"),
    RESPS_SPEC(resps_target_argmax_static, "IiiiFiiIs"),
};

struct Entry {
    const Spec* spec;
    void* fn;
};

const char* dtype_name(c10::ScalarType t) {
    switch (t) {
        case c10::kInt: return "torch.int32";
        case c10::kLong: return "torch.int64";
        case c10::kFloat: return "torch.float32";
        case c10::kDouble: return "torch.float64";
        case c10::kBFloat16: return "torch.bfloat16";
        default: return c10::toString(t);
    }
}

bool tensor_address(PyObject* o, char code, int64_t* out) {
    if (o == Py_None) {
        *out = 0;
        return true;
    }
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a CUDA tensor, got %s", Py_TYPE(o)->tp_name);
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
        return false;
    }
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "expected a contiguous tensor");
        return false;
    }
    if (code != 'T') {
        const c10::ScalarType want = code == 'I' ? c10::kInt : code == 'L' ? c10::kLong : code == 'F' ? c10::kFloat
                                   : code == 'D' ? c10::kDouble : c10::kBFloat16;
        if (t.scalar_type() != want) {
            PyErr_Format(PyExc_ValueError, "expected dtype %s, got %s", dtype_name(want), dtype_name(t.scalar_type()));
            return false;
        }
    }
    *out = static_cast<int64_t>(reinterpret_cast<intptr_t>(t.data_ptr()));
    return true;
}

// The interpreter lock is given up for the call and taken again on every way out of the scope, an exception's too
// (Python's own pair of macros leaves it with the lock given up).
struct WithoutLock {
    PyThreadState* const state = PyEval_SaveThread();
    ~WithoutLock() { PyEval_RestoreThread(state); }
};

PyObject* call_entry(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    const Entry* e = static_cast<const Entry*>(PyCapsule_GetPointer(self, nullptr));
    if (!e) return nullptr;
    if (n != e->spec->n_args)
        return PyErr_Format(PyExc_TypeError, "%s takes %d arguments, got %zd", e->spec->name, e->spec->n_args, n);
    Slot slots[kMaxArgs];
    int rc;
    try {
        for (Py_ssize_t k = 0; k < n; ++k) {
            PyObject* o = args[k];
            Slot& s = slots[k];
            switch (const char code = e->spec->codes[k]) {
                case 'p':
                    if (o != Py_None) s.i = static_cast<int64_t>(PyLong_AsUnsignedLongLong(o));
                    break;
                case 'i': s.i = PyLong_AsLongLong(o); break;
                case 'f': s.d = PyFloat_AsDouble(o); break;
                case 's':
                    if (o == Py_None) {
                        s.i = reinterpret_cast<intptr_t>(c10::cuda::getCurrentCUDAStream().stream());
                    } else {
                        PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
                        if (!h) return nullptr;
                        s.i = static_cast<int64_t>(PyLong_AsUnsignedLongLong(h));
                        Py_DECREF(h);
                    }
                    break;
                default:
                    if (!tensor_address(o, code, &s.i)) return nullptr;
            }
            if ((s.i == -1 || s.d == -1.0) && PyErr_Occurred()) return nullptr;
        }
        const WithoutLock unlocked;
        rc = e->spec->call(e->fn, slots);
    } catch (const std::exception& ex) {
        PyErr_SetString(PyExc_RuntimeError, ex.what());
        return nullptr;
    }
    return PyLong_FromLong(rc);
}

PyMethodDef kCallDef = {"resps_call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call_entry)),
                        METH_FASTCALL, nullptr};

PyObject* bind(PyObject*, PyObject* args) {
    const char* name;
    unsigned long long address;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return nullptr;
    for (const Spec& s : kSpecs) {
        if (std::strcmp(s.name, name)) continue;
        auto* e = new Entry{&s, reinterpret_cast<void*>(static_cast<uintptr_t>(address))};
        PyObject* cap = PyCapsule_New(e, nullptr, [](PyObject* c) { delete static_cast<Entry*>(PyCapsule_GetPointer(c, nullptr)); });
        if (!cap) {
            delete e;
            return nullptr;
        }
        PyObject* fn = PyCFunction_New(&kCallDef, cap);
        Py_DECREF(cap);
        return fn;
    }
    return PyErr_Format(PyExc_KeyError, "%s", name);
}

PyObject* names(PyObject*, PyObject*) {
    PyObject* list = PyList_New(0);
    for (const Spec& s : kSpecs) {
        PyObject* o = PyUnicode_FromString(s.name);
        if (!list || !o || PyList_Append(list, o) < 0) {
            Py_XDECREF(o);
            Py_XDECREF(list);
            return nullptr;
        }
        Py_DECREF(o);
    }
    return list;
}

PyMethodDef kMethods[] = {{"bind", bind, METH_VARARGS, "bind(name, address) -> callable for one entry point"},
                          {"names", names, METH_NOARGS, "names of the entry points that can be bound"},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() { return PyModule_Create(&kModule); }
