// CPython entry points of the data-path calls: argument conversion, the current stream, the call, the
// exception.  A ctypes call with a dozen tensor arguments costs 6 us of host time, more than many of the
// kernels behind it; this costs 0.3.
//
// The module knows no library path: binding.py hands it the addresses of the library's functions, the two
// torch functions that give the current stream, and the function that raises for a status code.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include <utility>

namespace {

enum Kind : char { kPtr, kInt, kI64, kSize, kFloat, kU64, kU32, kStream };

struct Arg {
    const char* name;
    Kind kind;
};

constexpr int kMaxArgs = 17;

struct Function {
    const char* name;
    int nargs;
    Arg args[kMaxArgs];
    void* address;
};

union Value {
    void* p;
    int64_t i;
    uint64_t u;
    float f;
};

const Arg kGrad{"d_grad", kPtr}, kOff{"d_off", kPtr}, kT{"T", kInt}, kN{"total_elems", kI64}, kLevels{"d_levels", kPtr},
    kStatus{"d_status", kPtr}, kThresh{"d_thresh", kPtr}, kTau{"d_tau", kPtr}, kWs{"d_ws", kPtr}, kWsBytes{"ws_bytes", kSize},
    kS{"s", kInt}, kScheme{"scheme", kInt}, kVariant{"variant", kInt}, kLloyd{"lloyd_iters", kInt}, kSeed{"seed", kU64},
    kStreamId{"stream_id", kU32}, kPackedOff{"d_packed_off", kPtr}, kPacked{"d_packed", kPtr}, kPackedK{"d_packed_k", kPtr},
    kLevelsK{"d_levels_k", kPtr}, kK{"K", kInt}, kScale{"scale", kFloat}, kOut{"d_out", kPtr}, kErr{"d_err", kPtr}, kD{"d", kInt},
    kStr{"stream", kStream};

Function g_functions[] = {
    {"ogq_levels_bingrad", 12, {kGrad, kOff, kT, kN, kVariant, kLloyd, kLevels, kThresh, kStatus, kWs, kWsBytes, kStr}, nullptr},
    {"ogq_levels_bingrad_b_noalloc", 9, {kGrad, kOff, kT, kN, kLloyd, kLevels, kThresh, kStatus, kStr}, nullptr},
    {"ogq_levels_orq", 10, {kGrad, kOff, kT, kN, kS, kLevels, kStatus, kWs, kWsBytes, kStr}, nullptr},
    {"ogq_quantize_pack", 13, {kGrad, kOff, kT, kN, kScheme, kS, kLevels, kThresh, kSeed, kStreamId, kPackedOff, kPacked, kStr}, nullptr},
    {"ogq_unpack_sum", 11, {kPackedK, kLevelsK, kK, kOff, kPackedOff, kT, kN, kS, kScale, kOut, kStr}, nullptr},
    {"ogq_clip_threshold", 10, {kGrad, kOff, kT, kN, {"c", kFloat}, kTau, kStatus, kWs, kWsBytes, kStr}, nullptr},
    {"ogq_levels_orq_clipped", 11, {kGrad, kOff, kT, kN, kS, kTau, kLevels, kStatus, kWs, kWsBytes, kStr}, nullptr},
    {"ogq_levels_bingrad_clipped", 13, {kGrad, kOff, kT, kN, kVariant, kLloyd, kTau, kLevels, kThresh, kStatus, kWs, kWsBytes, kStr}, nullptr},
    {"ogq_quant_error", 10, {kGrad, kOff, kT, kN, kS, kLevels, kPackedOff, kPacked, kErr, kStr}, nullptr},
    {"ogq_expected_error", 8, {kGrad, kOff, kT, kN, kS, kLevels, kErr, kStr}, nullptr},
    {"ogq_quantize_pack_dense", 11, {kGrad, kOff, kT, kN, kS, kLevels, kSeed, kStreamId, kPackedOff, kPacked, kStr}, nullptr},
    {"ogq_unpack_sum_dense", 11, {kPackedK, kLevelsK, kK, kOff, kPackedOff, kT, kN, kS, kScale, kOut, kStr}, nullptr},
    {"ogq_quantize_pack_clipped", 14, {kGrad, kOff, kT, kN, kScheme, kS, kLevels, kThresh, kTau, kSeed, kStreamId, kPackedOff, kPacked, kStr}, nullptr},
    {"ogq_bucket_encode", 14, {kGrad, kN, kD, kScheme, kS, {"iters", kInt}, {"clip_c", kFloat}, kSeed, kStreamId, kLevels, kThresh, kStatus, kPacked, kStr}, nullptr},
    {"ogq_bucket_decode_sum", 9, {kPackedK, kLevelsK, kK, kN, kD, kS, kScale, kOut, kStr}, nullptr},
};
constexpr int kFunctions = sizeof(g_functions) / sizeof(g_functions[0]);

PyObject *g_attach, *g_raise, *g_device, *g_raw_stream;  // set by binding.py
PyObject *g_str_data_ptr, *g_str_cuda_stream;

// An address: None, an integer, or an object with data_ptr() (a torch tensor).
bool to_address(PyObject* o, void** out)
{
    if (o == Py_None) { *out = nullptr; return true; }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return !(*out == nullptr && PyErr_Occurred());
    }
    PyObject* r = PyObject_CallMethodNoArgs(o, g_str_data_ptr);
    if (!r) return false;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return !(*out == nullptr && PyErr_Occurred());
}

// A stream: None (torch's current stream on its current device), an integer handle, or a torch stream.
bool to_stream(PyObject* o, void** out)
{
    if (o == nullptr || o == Py_None) {
        PyObject* d = PyObject_CallNoArgs(g_device);
        if (!d) return false;
        PyObject* r = PyObject_CallOneArg(g_raw_stream, d);
        Py_DECREF(d);
        if (!r) return false;
        *out = PyLong_AsVoidPtr(r);
        Py_DECREF(r);
    } else if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
    } else {
        PyObject* r = PyObject_GetAttr(o, g_str_cuda_stream);
        if (!r) return false;
        *out = PyLong_AsVoidPtr(r);
        Py_DECREF(r);
    }
    return !(*out == nullptr && PyErr_Occurred());
}

bool to_integer(PyObject* o, bool wrap, Value* v)
{
    PyObject* n = PyNumber_Index(o);
    if (!n) {  // what int() accepts beyond that (a float)
        PyErr_Clear();
        n = PyNumber_Long(o);
        if (!n) return false;
    }
    if (wrap) v->u = PyLong_AsUnsignedLongLongMask(n);
    else v->i = PyLong_AsLongLong(n);
    Py_DECREF(n);
    return !PyErr_Occurred();
}

template <class A> A as(const Value& v);
template <> void* as<void*>(const Value& v) { return v.p; }
template <> int as<int>(const Value& v) { return (int)v.i; }
template <> int64_t as<int64_t>(const Value& v) { return v.i; }
template <> uint64_t as<uint64_t>(const Value& v) { return v.u; }  // size_t too
template <> uint32_t as<uint32_t>(const Value& v) { return (uint32_t)v.u; }
template <> float as<float>(const Value& v) { return v.f; }

template <class... A, size_t... I>
int invoke(void* f, const Value* v, std::index_sequence<I...>)
{
    return ((int (*)(A...))f)(as<A>(v[I])...);
}
template <class... A>
int invoke(void* f, const Value* v)
{
    return invoke<A...>(f, v, std::index_sequence_for<A...>());
}

// The call itself, with the C types of the arguments listed above.
int call(int which, const Value* v)
{
    typedef void* P;
    typedef int I;
    typedef int64_t L;
    typedef uint64_t U;
    typedef uint32_t W;
    typedef float F;
    void* f = g_functions[which].address;
    switch (which) {
        case 0: return invoke<P, P, I, L, I, I, P, P, P, P, U, P>(f, v);
        case 1: return invoke<P, P, I, L, I, P, P, P, P>(f, v);
        case 2: return invoke<P, P, I, L, I, P, P, P, U, P>(f, v);
        case 3: return invoke<P, P, I, L, I, I, P, P, U, W, P, P, P>(f, v);
        case 4:
        case 11: return invoke<P, P, I, P, P, I, L, I, F, P, P>(f, v);
        case 5: return invoke<P, P, I, L, F, P, P, P, U, P>(f, v);
        case 6: return invoke<P, P, I, L, I, P, P, P, P, U, P>(f, v);
        case 7: return invoke<P, P, I, L, I, I, P, P, P, P, P, U, P>(f, v);
        case 8: return invoke<P, P, I, L, I, P, P, P, P, P>(f, v);
        case 9: return invoke<P, P, I, L, I, P, P, P>(f, v);
        case 10: return invoke<P, P, I, L, I, P, U, W, P, P, P>(f, v);
        case 12: return invoke<P, P, I, L, I, I, P, P, P, U, W, P, P, P>(f, v);
        case 13: return invoke<P, L, I, I, I, I, F, U, W, P, P, P, P, P>(f, v);
        default: return invoke<P, P, I, L, I, I, F, P, P>(f, v);
    }
}

template <int I>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames)
{
    Function& f = g_functions[I];
    if (!f.address) {
        if (!g_attach) return PyErr_Format(PyExc_RuntimeError, "the module has not been set up"), nullptr;
        PyObject* r = PyObject_CallNoArgs(g_attach);
        if (!r) return nullptr;
        Py_DECREF(r);
        if (!f.address) return PyErr_Format(PyExc_RuntimeError, "%s is not in the library", f.name), nullptr;
    }
    PyObject* given[kMaxArgs] = {};
    if (nargs > f.nargs)
        return PyErr_Format(PyExc_TypeError, "%s() takes %d arguments but %zd were given", f.name, f.nargs, nargs), nullptr;
    for (Py_ssize_t i = 0; i < nargs; ++i) given[i] = args[i];
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        const char* name = PyUnicode_AsUTF8(PyTuple_GET_ITEM(kwnames, k));
        if (!name) return nullptr;
        int i = 0;
        while (i < f.nargs && strcmp(f.args[i].name, name) != 0) ++i;
        if (i == f.nargs) return PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%s'", f.name, name), nullptr;
        if (given[i]) return PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", f.name, name), nullptr;
        given[i] = args[nargs + k];
    }
    Value v[kMaxArgs];
    for (int i = 0; i < f.nargs; ++i) {
        PyObject* o = given[i];
        const Kind kind = f.args[i].kind;
        v[i].u = 0;
        if (!o && kind != kStream)
            return PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", f.name, f.args[i].name), nullptr;
        bool ok = true;
        switch (kind) {
            case kPtr: ok = to_address(o, &v[i].p); break;
            case kStream: ok = to_stream(o, &v[i].p); break;
            case kFloat: {
                const double d = PyFloat_AsDouble(o);
                ok = !(d == -1.0 && PyErr_Occurred());
                v[i].f = (float)d;
                break;
            }
            default: ok = to_integer(o, kind == kU64 || kind == kU32, &v[i]); break;
        }
        if (!ok) return nullptr;
    }
    int code;
    Py_BEGIN_ALLOW_THREADS
    code = call(I, v);
    Py_END_ALLOW_THREADS
    if (code != 0) {
        PyObject* r = PyObject_CallFunction(g_raise, "is", code, f.name);
        Py_XDECREF(r);
        if (r) PyErr_Format(PyExc_RuntimeError, "%s failed: %d", f.name, code);
        return nullptr;
    }
    Py_RETURN_NONE;
}

// setup(attach, raise, device, raw_stream): attach() is called before the first entry point runs and calls
// set_addresses; raise(code, name) raises; device() is the current device and raw_stream(device) its
// current stream's handle.
PyObject* setup(PyObject*, PyObject* args)
{
    PyObject *a, *r, *d, *s;
    if (!PyArg_ParseTuple(args, "OOOO", &a, &r, &d, &s)) return nullptr;
    Py_XSETREF(g_attach, Py_NewRef(a));
    Py_XSETREF(g_raise, Py_NewRef(r));
    Py_XSETREF(g_device, Py_NewRef(d));
    Py_XSETREF(g_raw_stream, Py_NewRef(s));
    Py_RETURN_NONE;
}

// set_addresses(dict): the library's functions by name.
PyObject* set_addresses(PyObject*, PyObject* d)
{
    if (!PyDict_Check(d)) return PyErr_Format(PyExc_TypeError, "a dict is wanted"), nullptr;
    for (int i = 0; i < kFunctions; ++i) {
        PyObject* o = PyDict_GetItemString(d, g_functions[i].name);
        void* p = nullptr;
        if (o && !to_address(o, &p)) return nullptr;
        g_functions[i].address = p;
    }
    Py_RETURN_NONE;
}

#define ENTRY(I, NAME, SIGNATURE, DOC) \
    {NAME, (PyCFunction)(void (*)(void))(PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t, PyObject*))entry<I>, \
     METH_FASTCALL | METH_KEYWORDS, NAME SIGNATURE "\n--\n\n" DOC}

PyMethodDef g_methods[] = {
    ENTRY(0, "ogq_levels_bingrad", "(d_grad, d_off, T, total_elems, variant, lloyd_iters, d_levels, d_thresh, d_status, d_ws, ws_bytes, stream=None)", "BinGrad-b or BinGrad-pb levels."),
    ENTRY(1, "ogq_levels_bingrad_b_noalloc", "(d_grad, d_off, T, total_elems, lloyd_iters, d_levels, d_thresh, d_status, stream=None)",
          "BinGrad-b levels with the solver's scratch held inside the library (no workspace argument).\n\nFor callers that may not allocate "
          "device memory; at most 1024 tensors per call, and calls that\noverlap on the GPU must be ordered because they share the one built-in scratch array."),
    ENTRY(2, "ogq_levels_orq", "(d_grad, d_off, T, total_elems, s, d_levels, d_status, d_ws, ws_bytes, stream=None)", "ORQ levels."),
    ENTRY(3, "ogq_quantize_pack", "(d_grad, d_off, T, total_elems, scheme, s, d_levels, d_thresh, seed, stream_id, d_packed_off, d_packed, stream=None)", "Quantize and pack."),
    ENTRY(4, "ogq_unpack_sum", "(d_packed_k, d_levels_k, K, d_off, d_packed_off, T, total_elems, s, scale, d_out, stream=None)", "Unpack, dequantize and sum over K workers."),
    ENTRY(5, "ogq_clip_threshold", "(d_grad, d_off, T, total_elems, c, d_tau, d_status, d_ws, ws_bytes, stream=None)", "Clipping thresholds."),
    ENTRY(6, "ogq_levels_orq_clipped", "(d_grad, d_off, T, total_elems, s, d_tau, d_levels, d_status, d_ws, ws_bytes, stream=None)", "ORQ levels of the clipped gradient."),
    ENTRY(7, "ogq_levels_bingrad_clipped", "(d_grad, d_off, T, total_elems, variant, lloyd_iters, d_tau, d_levels, d_thresh, d_status, d_ws, ws_bytes, stream=None)", "BinGrad levels of the clipped gradient."),
    ENTRY(8, "ogq_quant_error", "(d_grad, d_off, T, total_elems, s, d_levels, d_packed_off, d_packed, d_err, stream=None)", "Realised quantization error."),
    ENTRY(9, "ogq_expected_error", "(d_grad, d_off, T, total_elems, s, d_levels, d_err, stream=None)", "Expected quantization error."),
    ENTRY(10, "ogq_quantize_pack_dense", "(d_grad, d_off, T, total_elems, s, d_levels, seed, stream_id, d_packed_off, d_packed, stream=None)", "Quantize and pack to base-s words."),
    ENTRY(11, "ogq_unpack_sum_dense", "(d_packed_k, d_levels_k, K, d_off, d_packed_off, T, total_elems, s, scale, d_out, stream=None)", "Unpack base-s words, dequantize and sum over K workers."),
    ENTRY(12, "ogq_quantize_pack_clipped", "(d_grad, d_off, T, total_elems, scheme, s, d_levels, d_thresh, d_tau, seed, stream_id, d_packed_off, d_packed, stream=None)", "Quantize and pack the clipped gradient."),
    ENTRY(13, "ogq_bucket_encode", "(d_grad, total_elems, d, scheme, s, iters, clip_c, seed, stream_id, d_levels, d_thresh, d_status, d_packed, stream=None)", "Levels, quantize and pack of fixed-length buckets."),
    ENTRY(14, "ogq_bucket_decode_sum", "(d_packed_k, d_levels_k, K, total_elems, d, s, scale, d_out, stream=None)", "Unpack, dequantize and sum of fixed-length buckets."),
    {"setup", setup, METH_VARARGS, nullptr},
    {"set_addresses", set_addresses, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", "Data-path calls of libogq.so.", -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    g_str_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_str_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!g_str_data_ptr || !g_str_cuda_stream) return nullptr;
    return PyModule_Create(&g_module);
}
