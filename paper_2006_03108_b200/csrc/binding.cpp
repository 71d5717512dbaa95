// Calls of the C ABI from Python: shards to arrays of pointers, the current stream, the call without the interpreter's lock.
//
// What bounds a small call is the host: H of 256 x 256 on 2 x 2 workers is 2 us on the device.  Through ctypes an array of pointers cost 0.24 us a
// shard and a call 0.6 us before the library was entered; here a shard is one method call (0.08 us) and the arguments of a call are converted by
// their types in the C prototype, so that the two cannot disagree.  Back to back (B200): H and H* of 256 x 256 9.1 -> 5.5 us, repartition of
// 280 x 333 and back 11.9 -> 5.7.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include "distdl.h"

namespace {

PyObject *g_data_ptr, *g_cuda_stream;                 // attribute names
PyObject *g_device, *g_raw_stream;                    // PyTorch's current device, and the handle of a device's current stream

bool pointer_of(PyObject *number, void **out) {       // takes the reference
    if (!number) return false;
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(number);
    Py_DECREF(number);
    return !PyErr_Occurred();
}

// Device (or host) address of a tensor, or of a raw int; None: NULL.
bool address(PyObject *o, void **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    return pointer_of(PyLong_Check(o) ? Py_NewRef(o) : PyObject_CallMethodNoArgs(o, g_data_ptr), out);
}

// Handle of a stream: an int, or an object with `cuda_stream`; None: PyTorch's current stream of the current device.
bool stream_handle(PyObject *o, void **out) {
    if (o != Py_None) return pointer_of(PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttr(o, g_cuda_stream), out);
    // the first lookup of the device puts others in the place of both
    PyObject *lookup = Py_NewRef(g_device), *device = PyObject_CallNoArgs(lookup);
    Py_DECREF(lookup);
    if (!device) return false;
    lookup = Py_NewRef(g_raw_stream);
    PyObject *stream = PyObject_CallOneArg(lookup, device);
    Py_DECREF(lookup);
    Py_DECREF(device);
    return pointer_of(stream, out);
}

template <typename T>
struct Arg {                                          // whole numbers
    T value;
    bool read(PyObject *o, bool) {
        value = (T)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    T get() { return value; }
};

template <typename T>
struct Arg<T *> {                                     // handles, buffers, the stream
    void *value;
    bool read(PyObject *o, bool is_stream) { return is_stream ? stream_handle(o, &value) : address(o, &value); }
    T *get() { return static_cast<T *>(value); }
};

template <>
struct Arg<const float *> {                           // what taps() returns
    const float *value;
    bool read(PyObject *o, bool) {
        value = reinterpret_cast<const float *>(PyBytes_AsString(o));
        return value != nullptr;
    }
    const float *get() { return value; }
};

struct Pointers {                                     // shards; None: no array
    void *few[64] = {};
    std::vector<void *> many;
    void **p = nullptr;
    Py_ssize_t size = 0;
    bool read(PyObject *o, bool) {
        if (o == Py_None) return true;
        PyObject *s = PySequence_Fast(o, "a sequence of shards is needed");
        if (!s) return false;
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(s);
        if (n > 64) many.resize((size_t)n);
        p = n > 64 ? many.data() : few;
        bool ok = true;
        for (; ok && size < n && size < PySequence_Fast_GET_SIZE(s); ++size) {      // another thread may change a list meanwhile
            PyObject *shard = Py_NewRef(PySequence_Fast_GET_ITEM(s, size));
            ok = address(shard, p + size);
            Py_DECREF(shard);
        }
        Py_DECREF(s);
        return ok;
    }
};
template <>
struct Arg<void *const *> : Pointers {
    void *const *get() { return p; }
};
template <>
struct Arg<const void *const *> : Pointers {
    const void *const *get() { return p; }
};

// What the library reads of a list: as many entries as the caller says the layer has.  A list that is too short is refused here, optional ones too (a
// missing bias or position would read as "none").  Beyond any layer's number the library refuses the layer before it reads the list.
constexpr long long kMostEntries = 4096;
static_assert(kMostEntries >= DISTDL_MAX_WORKERS, "");
template <typename T>
bool too_short(const Arg<T> &arg, PyObject *const *&need, int at, PyObject **why) {
    if constexpr (std::is_base_of_v<Pointers, Arg<T>>) {
        const long long entries = PyLong_AsLongLong(*need++);
        if (entries == -1 && PyErr_Occurred()) return true;
        if (arg.p && arg.size < entries && entries <= kMostEntries) {
            *why = PyUnicode_FromFormat("argument %d is a list of %zd entries, %lld are needed", at + 1, arg.size, entries);
            return true;
        }
    }
    return false;
}

// The stream is every function's last argument.  Behind it: how many entries each list has to have, in the lists' order.  Returns the status, or what is
// wrong with a list.
template <auto Function>
struct Call;
template <typename... A, distdl_status_t (*Function)(A...)>
struct Call<Function> {
    static constexpr size_t kLists = (std::is_base_of_v<Pointers, Arg<A>> + ... + 0);
    template <size_t... I>
    static PyObject *run(PyObject *const *args, std::index_sequence<I...>) {
        std::tuple<Arg<A>...> a;
        if (!(std::get<I>(a).read(args[I], I + 1 == sizeof...(A)) && ...)) return nullptr;
        PyObject *const *need = args + sizeof...(A);
        PyObject *why = nullptr;
        if ((too_short(std::get<I>(a), need, (int)I, &why) || ...)) return why;
        distdl_status_t status;
        Py_BEGIN_ALLOW_THREADS
        status = Function(std::get<I>(a).get()...);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong((long)status);
    }
    static PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
        constexpr Py_ssize_t needed = (Py_ssize_t)(sizeof...(A) + kLists);
        if (n != needed) return PyErr_Format(PyExc_TypeError, "%zd arguments, %zd needed", n, needed);
        return run(args, std::index_sequence_for<A...>{});
    }
};

// taps(w) -> (bytes of 3 x (2R+1) floats, R) of any nested sequence of numbers, or None if it has another shape
PyObject *taps(PyObject *, PyObject *w) {
    PyObject *rows = PySequence_Fast(w, "taps must have shape [3][2R+1]");
    if (!rows) return nullptr;
    std::vector<float> v;
    Py_ssize_t width = -1, count = 0;
    bool shaped = true, failed = false;
    // a number's own conversion may change the lists meanwhile: sizes are looked up at each step, and what is in hand is held
    for (; !failed && count < PySequence_Fast_GET_SIZE(rows); ++count) {
        PyObject *item = Py_NewRef(PySequence_Fast_GET_ITEM(rows, count)), *row = PySequence_Fast(item, "taps must have shape [3][2R+1]");
        Py_DECREF(item);
        failed = !row;
        Py_ssize_t n = 0;
        for (; !failed && n < PySequence_Fast_GET_SIZE(row); ++n) {
            PyObject *number = Py_NewRef(PySequence_Fast_GET_ITEM(row, n)), *f = PyNumber_Float(number);
            Py_DECREF(number);
            failed = !f;
            if (f) v.push_back((float)PyFloat_AS_DOUBLE(f));
            Py_XDECREF(f);
        }
        Py_XDECREF(row);
        shaped = shaped && n % 2 == 1 && (width < 0 || n == width);
        width = n;
    }
    shaped = shaped && count == 3;
    Py_DECREF(rows);
    if (failed) return nullptr;
    if (!shaped) Py_RETURN_NONE;
    return Py_BuildValue("y#n", (const char *)v.data(), (Py_ssize_t)(v.size() * sizeof(float)), width / 2);
}

PyObject *set_stream_lookup(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != 2) return PyErr_Format(PyExc_TypeError, "two functions are needed");
    Py_XSETREF(g_device, Py_NewRef(args[0]));
    Py_XSETREF(g_raw_stream, Py_NewRef(args[1]));
    Py_RETURN_NONE;
}

#define FUNCTION(name) {#name, (PyCFunction)(void (*)(void))Call<distdl_##name>::entry, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FUNCTION(broadcast_fwd), FUNCTION(broadcast_adj), FUNCTION(sumreduce_fwd), FUNCTION(sumreduce_adj), FUNCTION(allreduce),
    FUNCTION(halo_fwd), FUNCTION(halo_adj), FUNCTION(repartition_fwd), FUNCTION(repartition_adj),
    FUNCTION(conv_fwd), FUNCTION(conv_adj), FUNCTION(conv_adj_params), FUNCTION(convg_fwd), FUNCTION(convg_adj), FUNCTION(convg_adj_params),
    FUNCTION(stencil3d_fwd), FUNCTION(stencil3d_adj), FUNCTION(pool_fwd), FUNCTION(pool_adj),
    FUNCTION(affine_fwd), FUNCTION(affine_adj), FUNCTION(affine_adj_params),
    {"taps", taps, METH_O, nullptr},
    {"set_stream_lookup", (PyCFunction)(void (*)(void))set_stream_lookup, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    g_device = Py_NewRef(Py_None);
    g_raw_stream = Py_NewRef(Py_None);
    return PyModule_Create(&module);
}
