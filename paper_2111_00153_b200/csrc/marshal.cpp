// Argument marshalling of the calls that a program makes per layer and pass, as a CPython extension: the same Python
// signatures that binding.py gives the rest, converted and handed to librmsmp without ctypes.  A small layer's call is
// all host time (launch 2.1 us), and the generic route -- Python wrapper, one ctypes conversion object per argument --
// cost as much again (rmsmp_gemm 4.7 us, rmsmp_quantize_act 5.6 us).  Nothing is kept between calls.
//
// A device pointer is a torch tensor (its data_ptr() is called), an int, or None; a layer descriptor or plan is the
// ctypes structure of binding.py, read through the buffer protocol; stream None is the current torch stream.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <cstdint>
#include <initializer_list>
#include <type_traits>
#include "../../include/rmsmp.h"

namespace {

// the library's entry points (filled by setup() with the addresses that binding.py's loader found)
struct Api {
    decltype(&rmsmp_quantize_act) quantize_act;
    decltype(&rmsmp_gemm) gemm;
    decltype(&rmsmp_gemm_variant) gemm_variant;
    decltype(&rmsmp_gemm_workspace) gemm_workspace;
    decltype(&rmsmp_gemm_workspace_requant) gemm_workspace_requant;
    decltype(&rmsmp_conv_implicit) conv_implicit;
    decltype(&rmsmp_conv_implicit_variant) conv_implicit_variant;
    decltype(&rmsmp_conv_implicit_workspace) conv_implicit_workspace;
    decltype(&rmsmp_conv_implicit_workspace_requant) conv_implicit_workspace_requant;
    decltype(&rmsmp_conv_depthwise) conv_depthwise;
    decltype(&rmsmp_im2col_codes) im2col_codes;
    decltype(&rmsmp_expand_weights) expand_weights;
    decltype(&rmsmp_assign_quantize_pack) assign_quantize_pack;
    decltype(&rmsmp_quantize_pack) quantize_pack;
    decltype(&rmsmp_gemm_grouped_launch) gemm_grouped_launch;
} api;

PyObject* g_stream;          // callable: the current stream's handle
PyObject *g_raw, *g_device;  // torch's accessors, once CUDA has been started up: g_raw(g_device()) is that handle
PyObject* g_error;           // callable(status, where): raises RmsmpError
PyObject* g_array;           // callable(object, format): a contiguous array of bytes ('B') or floats ('f') with its values
PyObject *s_data_ptr, *s_numel, *s_element_size, *s_cuda_stream;

// Arguments of one call, positions filled from positional and keyword arguments; conversions record the first failure.
struct Call {
    static constexpr int kMax = 16;
    PyObject* a[kMax] = {};
    bool ok = true;

    Call(const char* where, const char* const* names, int n, int required, PyObject* const* args, Py_ssize_t nargs, PyObject* kw)
    {
        if (nargs > n) {
            PyErr_Format(PyExc_TypeError, "%s takes at most %d arguments (%zd given)", where, n, nargs);
            ok = false;
            return;
        }
        for (Py_ssize_t i = 0; i < nargs; ++i) a[i] = args[i];
        const Py_ssize_t nkw = kw ? PyTuple_GET_SIZE(kw) : 0;
        for (Py_ssize_t i = 0; i < nkw; ++i) {
            PyObject* key = PyTuple_GET_ITEM(kw, i);
            int at = 0;
            while (at < n && PyUnicode_CompareWithASCIIString(key, names[at]) != 0) ++at;
            if (at == n || a[at]) {
                PyErr_Format(PyExc_TypeError, at == n ? "%s got an unexpected keyword argument '%U'" : "%s got multiple values for argument '%U'", where, key);
                ok = false;
                return;
            }
            a[at] = args[nargs + i];
        }
        for (int i = 0; i < required; ++i)
            if (!a[i]) {
                PyErr_Format(PyExc_TypeError, "%s is missing argument '%s'", where, names[i]);
                ok = false;
                return;
            }
    }
    bool none(int i) const { return !a[i] || a[i] == Py_None; }
    long long i64(int i, long long dflt = 0)
    {
        if (!ok || !a[i]) return dflt;
        long long v;
        if (PyLong_Check(a[i])) {
            v = PyLong_AsLongLong(a[i]);
        } else {
            PyObject* x = PyNumber_Index(a[i]);
            if (!x) { ok = false; return dflt; }
            v = PyLong_AsLongLong(x);
            Py_DECREF(x);
        }
        if (v == -1 && PyErr_Occurred()) ok = false;
        return v;
    }
    int i32(int i, int dflt = 0)
    {
        const long long v = i64(i, dflt);
        if (ok && (v < INT32_MIN || v > INT32_MAX)) {
            PyErr_SetString(PyExc_OverflowError, "argument does not fit a C int");
            ok = false;
        }
        return (int)v;
    }
    size_t size(int i) { return (size_t)i64(i); }
    float f32(int i)
    {
        if (!ok) return 0.0f;
        const double v = PyFloat_AsDouble(a[i]);
        if (v == -1.0 && PyErr_Occurred()) ok = false;
        return (float)v;
    }
    void* address(PyObject* o)                                  // the value of an int, or what a method returned
    {
        void* p = PyLong_AsVoidPtr(o);
        if (!p && PyErr_Occurred()) ok = false;
        return p;
    }
    void* ptr(int i)
    {
        if (!ok || none(i)) return nullptr;
        if (PyLong_Check(a[i])) return address(a[i]);
        PyObject* r = PyObject_CallMethodNoArgs(a[i], s_data_ptr);
        if (!r) { ok = false; return nullptr; }
        void* p = address(r);
        Py_DECREF(r);
        return p;
    }
    size_t bytes_of(int i)                                      // numel() * element_size() of a tensor
    {
        if (!ok) return 0;
        size_t n = 1;
        for (PyObject* m : {s_numel, s_element_size}) {
            PyObject* r = PyObject_CallMethodNoArgs(a[i], m);
            if (!r) { ok = false; return 0; }
            n *= PyLong_AsSize_t(r);
            Py_DECREF(r);
            if (PyErr_Occurred()) { ok = false; return 0; }
        }
        return n;
    }
    template <typename T> const T* structure(int i)
    {
        if (!ok) return nullptr;
        Py_buffer b;
        if (PyObject_GetBuffer(a[i], &b, PyBUF_SIMPLE) != 0) { ok = false; return nullptr; }
        const T* p = static_cast<const T*>(b.buf);
        if (b.len != (Py_ssize_t)sizeof(T)) {
            PyErr_SetString(PyExc_TypeError, "not the structure this call takes");
            ok = false;
        }
        PyBuffer_Release(&b);                                   // the caller holds the object for the length of the call
        return p;
    }
    void* stream(int i)
    {
        if (!ok) return nullptr;
        if (!none(i) && PyLong_Check(a[i])) return address(a[i]);
        PyObject* r;
        if (!none(i)) {
            r = PyObject_GetAttr(a[i], s_cuda_stream);
        } else if (g_raw) {
            PyObject* device = PyObject_CallNoArgs(g_device);
            r = device ? PyObject_CallOneArg(g_raw, device) : nullptr;
            Py_XDECREF(device);
        } else {
            r = PyObject_CallNoArgs(g_stream);
        }
        if (!r) { ok = false; return nullptr; }
        void* p = address(r);
        Py_DECREF(r);
        return p;
    }
};

bool failed(rmsmp_status st, const char* where)
{
    if (st == RMSMP_OK) return false;
    PyObject* r = PyObject_CallFunction(g_error, "is", (int)st, where);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
    return true;
}

#define ARGS(where, required, ...)                                                                                      \
    static const char* const names[] = {__VA_ARGS__};                                                                   \
    constexpr int kCount = (int)(sizeof(names) / sizeof(names[0]));                                                     \
    static_assert(kCount <= Call::kMax, "room for every argument");                                                     \
    Call c(where, names, kCount, required, args, nargs, kw);                                                            \
    if (!c.ok) return nullptr;
// calls the library without the interpreter lock (a launch can wait for room in the stream's queue)
#define RUN(where, expr)                                                                                                \
    if (!c.ok) return nullptr;                                                                                          \
    rmsmp_status st;                                                                                                    \
    Py_BEGIN_ALLOW_THREADS st = (expr);                                                                                 \
    Py_END_ALLOW_THREADS if (failed(st, where)) return nullptr;
#define DEF(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw)

DEF(quantize_act)
{
    ARGS("rmsmp_quantize_act", 5, "d_X", "count", "alpha_a", "kind", "d_codes", "stream")
    const float* x = (const float*)c.ptr(0);
    const size_t n = c.size(1);
    const float alpha = c.f32(2);
    const int kind = c.i32(3);
    int8_t* codes = (int8_t*)c.ptr(4);
    void* s = c.stream(5);
    float step = 0.0f;
    RUN("rmsmp_quantize_act", api.quantize_act(x, n, alpha, (rmsmp_act_kind)kind, codes, &step, s))
    return PyFloat_FromDouble((double)step);
}

DEF(gemm)
{
    ARGS("rmsmp_gemm", 8, "layer", "d_packed", "d_act", "N", "ld_act", "act_step", "d_out", "ld_out", "out_layout", "d_acc", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *act = c.ptr(2);
    const long long N = c.i64(3), ld = c.i64(4);
    const float step = c.f32(5);
    void* out = c.ptr(6);
    const long long ld_out = c.i64(7);
    const int layout = c.i32(8);
    void *acc = c.ptr(9), *s = c.stream(10);
    RUN("rmsmp_gemm", api.gemm(L, pk, (const int8_t*)act, N, ld, step, (float*)out, ld_out, (rmsmp_out_layout)layout, (int32_t*)acc, s))
    Py_RETURN_NONE;
}

DEF(gemm_variant)
{
    ARGS("rmsmp_gemm_variant", 11, "layer", "d_packed", "d_act", "N", "ld_act", "act_step", "d_out", "ld_out", "out_layout", "d_acc", "variant", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *act = c.ptr(2);
    const long long N = c.i64(3), ld = c.i64(4);
    const float step = c.f32(5);
    void* out = c.ptr(6);
    const long long ld_out = c.i64(7);
    const int layout = c.i32(8);
    void* acc = c.ptr(9);
    const int variant = c.i32(10);
    void* s = c.stream(11);
    RUN("rmsmp_gemm_variant", api.gemm_variant(L, pk, (const int8_t*)act, N, ld, step, (float*)out, ld_out, (rmsmp_out_layout)layout, (int32_t*)acc,
                                               (rmsmp_variant)variant, s))
    Py_RETURN_NONE;
}

DEF(gemm_workspace)
{
    ARGS("rmsmp_gemm_workspace", 9, "layer", "d_packed", "d_workspace", "d_act", "N", "ld_act", "act_step", "d_out", "ld_out", "out_layout", "d_acc", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *ws = c.ptr(2), *act = c.ptr(3);
    const long long N = c.i64(4), ld = c.i64(5);
    const float step = c.f32(6);
    void* out = c.ptr(7);
    const long long ld_out = c.i64(8);
    const int layout = c.i32(9);
    void *acc = c.ptr(10), *s = c.stream(11);
    RUN("rmsmp_gemm_workspace", api.gemm_workspace(L, pk, ws, (const int8_t*)act, N, ld, step, (float*)out, ld_out, (rmsmp_out_layout)layout, (int32_t*)acc, s))
    Py_RETURN_NONE;
}

DEF(gemm_workspace_requant)
{
    ARGS("rmsmp_gemm_workspace_requant", 11, "layer", "d_packed", "d_workspace", "d_act", "N", "ld_act", "act_step", "next_alpha", "next_kind",
         "d_next_codes", "ld_codes", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *ws = c.ptr(2), *act = c.ptr(3);
    const long long N = c.i64(4), ld = c.i64(5);
    const float step = c.f32(6), alpha = c.f32(7);
    const int kind = c.i32(8);
    void* codes = c.ptr(9);
    const long long ld_codes = c.i64(10);
    void* s = c.stream(11);
    float next = 0.0f;
    RUN("rmsmp_gemm_workspace_requant", api.gemm_workspace_requant(L, pk, ws, (const int8_t*)act, N, ld, step, alpha, (rmsmp_act_kind)kind, (int8_t*)codes,
                                                                  ld_codes, &next, s))
    return PyFloat_FromDouble((double)next);
}

DEF(conv_implicit)
{
    ARGS("rmsmp_conv_implicit", 10, "layer", "d_packed", "d_act", "B", "H", "W", "stride", "pad", "act_step", "d_out", "out_layout", "d_acc", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *act = c.ptr(2);
    const int B = c.i32(3), H = c.i32(4), W = c.i32(5), stride = c.i32(6), pad = c.i32(7);
    const float step = c.f32(8);
    void* out = c.ptr(9);
    const int layout = c.i32(10);
    void *acc = c.ptr(11), *s = c.stream(12);
    RUN("rmsmp_conv_implicit", api.conv_implicit(L, pk, (const int8_t*)act, B, H, W, stride, pad, step, (float*)out, (rmsmp_out_layout)layout, (int32_t*)acc, s))
    Py_RETURN_NONE;
}

DEF(conv_implicit_variant)
{
    ARGS("rmsmp_conv_implicit_variant", 13, "layer", "d_packed", "d_act", "B", "H", "W", "stride", "pad", "act_step", "d_out", "out_layout", "d_acc",
         "variant", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *act = c.ptr(2);
    const int B = c.i32(3), H = c.i32(4), W = c.i32(5), stride = c.i32(6), pad = c.i32(7);
    const float step = c.f32(8);
    void* out = c.ptr(9);
    const int layout = c.i32(10);
    void* acc = c.ptr(11);
    const int variant = c.i32(12);
    void* s = c.stream(13);
    RUN("rmsmp_conv_implicit_variant", api.conv_implicit_variant(L, pk, (const int8_t*)act, B, H, W, stride, pad, step, (float*)out, (rmsmp_out_layout)layout,
                                                                 (int32_t*)acc, (rmsmp_variant)variant, s))
    Py_RETURN_NONE;
}

DEF(conv_implicit_workspace)
{
    ARGS("rmsmp_conv_implicit_workspace", 11, "layer", "d_packed", "d_workspace", "d_act", "B", "H", "W", "stride", "pad", "act_step", "d_out", "out_layout",
         "d_acc", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *ws = c.ptr(2), *act = c.ptr(3);
    const int B = c.i32(4), H = c.i32(5), W = c.i32(6), stride = c.i32(7), pad = c.i32(8);
    const float step = c.f32(9);
    void* out = c.ptr(10);
    const int layout = c.i32(11);
    void *acc = c.ptr(12), *s = c.stream(13);
    RUN("rmsmp_conv_implicit_workspace", api.conv_implicit_workspace(L, pk, ws, (const int8_t*)act, B, H, W, stride, pad, step, (float*)out,
                                                                     (rmsmp_out_layout)layout, (int32_t*)acc, s))
    Py_RETURN_NONE;
}

DEF(conv_implicit_workspace_requant)
{
    ARGS("rmsmp_conv_implicit_workspace_requant", 13, "layer", "d_packed", "d_workspace", "d_act", "B", "H", "W", "stride", "pad", "act_step", "next_alpha",
         "next_kind", "d_next_codes", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *ws = c.ptr(2), *act = c.ptr(3);
    const int B = c.i32(4), H = c.i32(5), W = c.i32(6), stride = c.i32(7), pad = c.i32(8);
    const float step = c.f32(9), alpha = c.f32(10);
    const int kind = c.i32(11);
    void *codes = c.ptr(12), *s = c.stream(13);
    float next = 0.0f;
    RUN("rmsmp_conv_implicit_workspace_requant", api.conv_implicit_workspace_requant(L, pk, ws, (const int8_t*)act, B, H, W, stride, pad, step, alpha,
                                                                                     (rmsmp_act_kind)kind, (int8_t*)codes, &next, s))
    return PyFloat_FromDouble((double)next);
}

DEF(conv_depthwise)
{
    ARGS("rmsmp_conv_depthwise", 10, "layer", "d_packed", "d_act", "B", "H", "W", "stride", "pad", "act_step", "d_out", "d_acc", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *act = c.ptr(2);
    const int B = c.i32(3), H = c.i32(4), W = c.i32(5), stride = c.i32(6), pad = c.i32(7);
    const float step = c.f32(8);
    void *out = c.ptr(9), *acc = c.ptr(10), *s = c.stream(11);
    RUN("rmsmp_conv_depthwise", api.conv_depthwise(L, pk, (const int8_t*)act, B, H, W, stride, pad, step, (float*)out, (int32_t*)acc, s))
    Py_RETURN_NONE;
}

DEF(im2col_codes)
{
    ARGS("rmsmp_im2col_codes", 12, "d_act", "B", "H", "W", "Cc", "pix_pitch", "kh", "kw", "stride", "pad", "d_cols", "ld_cols", "stream")
    const void* act = c.ptr(0);
    const int B = c.i32(1), H = c.i32(2), W = c.i32(3), C = c.i32(4);
    const long long pitch = c.i64(5);
    const int kh = c.i32(6), kw_ = c.i32(7), stride = c.i32(8), pad = c.i32(9);
    void* cols = c.ptr(10);
    const long long ld = c.i64(11);
    void* s = c.stream(12);
    RUN("rmsmp_im2col_codes", api.im2col_codes((const int8_t*)act, B, H, W, C, pitch, kh, kw_, stride, pad, (int8_t*)cols, ld, s))
    Py_RETURN_NONE;
}

DEF(expand_weights)
{
    ARGS("rmsmp_expand_weights", 3, "layer", "d_packed", "d_workspace", "workspace_bytes", "stream")
    const rmsmp_layer* L = c.structure<rmsmp_layer>(0);
    void *pk = c.ptr(1), *ws = c.ptr(2);
    const size_t n = c.none(3) ? c.bytes_of(2) : c.size(3);
    void* s = c.stream(4);
    RUN("rmsmp_expand_weights", api.expand_weights(L, pk, ws, n, s))
    Py_RETURN_NONE;
}

DEF(assign_quantize_pack)
{
    ARGS("rmsmp_assign_quantize_pack", 8, "d_W", "w_layout", "layer", "ratio", "d_alpha", "pot_mode", "d_packed", "d_scratch", "d_scheme", "d_bits", "stream")
    void* W = c.ptr(0);
    const int w_layout = c.i32(1);
    const rmsmp_layer* L = c.structure<rmsmp_layer>(2);
    int r[3] = {0, 0, 0};
    for (int i = 0; c.ok && i < 3; ++i) {
        PyObject* item = PySequence_GetItem(c.a[3], i);
        PyObject* whole = item ? PyNumber_Long(item) : nullptr;
        Py_XDECREF(item);
        if (!whole) return nullptr;
        r[i] = (int)PyLong_AsLong(whole);
        Py_DECREF(whole);
        if (PyErr_Occurred()) return nullptr;
    }
    void* alpha = c.ptr(4);
    const int mode = c.i32(5);
    void* pk = c.ptr(6);
    const size_t pk_bytes = c.bytes_of(6);
    void* scratch = c.ptr(7);
    const size_t scratch_bytes = c.bytes_of(7);
    void *scheme = c.ptr(8), *bits = c.ptr(9), *s = c.stream(10);
    RUN("rmsmp_assign_quantize_pack", api.assign_quantize_pack((const float*)W, (rmsmp_w_layout)w_layout, L, r[0], r[1], r[2], (const float*)alpha,
                                                               (rmsmp_pot_mode)mode, pk, pk_bytes, scratch, scratch_bytes, (uint8_t*)scheme, (uint8_t*)bits, s))
    Py_RETURN_NONE;
}

// A host array: the object's own memory where it is contiguous and of the type asked for, otherwise a converted copy.
struct HostArray {
    Py_buffer b{};
    bool held = false;
    ~HostArray() { if (held) PyBuffer_Release(&b); }
    bool take(PyObject* o, char format)
    {
        if (PyObject_GetBuffer(o, &b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) { PyErr_Clear(); return false; }
        held = true;
        if (b.format && b.format[0] == format && b.format[1] == 0) return true;
        PyBuffer_Release(&b);
        held = false;
        return false;
    }
    const void* get(Call& c, int i, char format)
    {
        if (!c.ok) return nullptr;
        if (take(c.a[i], format)) return b.buf;
        PyObject* copy = PyObject_CallFunction(g_array, "OC", c.a[i], (int)format);
        if (copy && !take(copy, format)) PyErr_SetString(PyExc_TypeError, "not an array of numbers");
        Py_XDECREF(copy);                                       // (the buffer holds it)
        if (!held) c.ok = false;
        return held ? b.buf : nullptr;
    }
    Py_ssize_t count() const { return b.itemsize ? b.len / b.itemsize : 0; }
};

DEF(quantize_pack)
{
    ARGS("rmsmp_quantize_pack", 8, "d_W", "w_layout", "layer", "h_scheme", "h_bits", "h_alpha", "pot_mode", "d_packed", "packed_bytes", "stream")
    void* W = c.ptr(0);
    const int w_layout = c.i32(1);
    const rmsmp_layer* L = c.structure<rmsmp_layer>(2);
    HostArray scheme, bits, alpha;
    const void *hs = scheme.get(c, 3, 'B'), *hb = bits.get(c, 4, 'B'), *ha = alpha.get(c, 5, 'f');
    if (c.ok && (scheme.count() != L->M || bits.count() != L->M || alpha.count() != L->M)) {
        PyErr_SetString(PyExc_ValueError, "scheme/bits/alpha need M entries");
        c.ok = false;
    }
    const int mode = c.i32(6);
    void* pk = c.ptr(7);
    const size_t pk_bytes = c.none(8) ? c.bytes_of(7) : c.size(8);
    void* s = c.stream(9);
    RUN("rmsmp_quantize_pack", api.quantize_pack((const float*)W, (rmsmp_w_layout)w_layout, L, (const uint8_t*)hs, (const uint8_t*)hb, (const float*)ha,
                                                 (rmsmp_pot_mode)mode, pk, pk_bytes, s))
    Py_RETURN_NONE;
}

DEF(gemm_grouped_launch)
{
    ARGS("rmsmp_gemm_grouped_launch", 1, "plan", "stream")
    const rmsmp_grouped_plan* plan = c.structure<rmsmp_grouped_plan>(0);
    void* s = c.stream(1);
    RUN("rmsmp_gemm_grouped_launch", api.gemm_grouped_launch(plan, s))
    Py_RETURN_NONE;
}

// setup(addresses: {name: int}, stream: callable, error: callable, array: callable)
PyObject* setup(PyObject*, PyObject* args)
{
    PyObject *addr, *stream, *error, *array;
    if (!PyArg_ParseTuple(args, "O!OOO", &PyDict_Type, &addr, &stream, &error, &array)) return nullptr;
    auto get = [&](const char* name, auto& fn) -> bool {
        PyObject* v = PyDict_GetItemString(addr, name);
        if (!v) { PyErr_SetString(PyExc_KeyError, name); return false; }
        void* p = PyLong_AsVoidPtr(v);
        if (!p) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, name); return false; }
        fn = reinterpret_cast<std::remove_reference_t<decltype(fn)>>(p);
        return true;
    };
    if (!get("rmsmp_quantize_act", api.quantize_act) || !get("rmsmp_gemm", api.gemm) || !get("rmsmp_gemm_variant", api.gemm_variant) ||
        !get("rmsmp_gemm_workspace", api.gemm_workspace) || !get("rmsmp_gemm_workspace_requant", api.gemm_workspace_requant) ||
        !get("rmsmp_conv_implicit", api.conv_implicit) || !get("rmsmp_conv_implicit_variant", api.conv_implicit_variant) ||
        !get("rmsmp_conv_implicit_workspace", api.conv_implicit_workspace) ||
        !get("rmsmp_conv_implicit_workspace_requant", api.conv_implicit_workspace_requant) || !get("rmsmp_conv_depthwise", api.conv_depthwise) ||
        !get("rmsmp_im2col_codes", api.im2col_codes) || !get("rmsmp_expand_weights", api.expand_weights) ||
        !get("rmsmp_assign_quantize_pack", api.assign_quantize_pack) || !get("rmsmp_gemm_grouped_launch", api.gemm_grouped_launch) ||
        !get("rmsmp_quantize_pack", api.quantize_pack))
        return nullptr;
    Py_INCREF(stream); Py_XSETREF(g_stream, stream);
    Py_INCREF(error); Py_XSETREF(g_error, error);
    Py_INCREF(array); Py_XSETREF(g_array, array);
    Py_RETURN_NONE;
}

PyObject* stream_accessors(PyObject*, PyObject* args)
{
    PyObject *raw, *device;
    if (!PyArg_ParseTuple(args, "OO", &raw, &device)) return nullptr;
    Py_INCREF(device); Py_XSETREF(g_device, device);
    Py_INCREF(raw); Py_XSETREF(g_raw, raw);
    Py_RETURN_NONE;
}

#define METHOD(name, doc) {"rmsmp_" #name, (PyCFunction)(void (*)(void))name, METH_FASTCALL | METH_KEYWORDS, doc}
PyMethodDef methods[] = {
    {"setup", setup, METH_VARARGS, "entry points, current-stream callable, error callable, array callable"},
    {"stream_accessors", stream_accessors, METH_VARARGS, "callable(device) and callable(): the current stream's handle without a Python frame"},
    METHOD(quantize_act, "Returns the activation step (alpha_a/15 or alpha_a/7) as a Python float (fp32 value)."),
    METHOD(gemm, "Linear layer."),
    METHOD(gemm_variant, "Linear layer by a chosen kernel."),
    METHOD(gemm_workspace, "Linear layer on expanded weights."),
    METHOD(gemm_workspace_requant, "Linear layer whose epilogue writes the next layer's 4-bit activation codes; returns their step."),
    METHOD(conv_implicit, "Convolution layer."),
    METHOD(conv_implicit_variant, "Convolution layer by a chosen kernel."),
    METHOD(conv_implicit_workspace, "Convolution layer on expanded weights."),
    METHOD(conv_implicit_workspace_requant, "Convolution layer whose epilogue writes the next layer's codes; returns their step."),
    METHOD(conv_depthwise, "Depthwise convolution."),
    METHOD(im2col_codes, "Patch matrix of a convolution's activation codes."),
    METHOD(expand_weights, "Expands a layer's packed codes into its workspace."),
    METHOD(assign_quantize_pack, "Row assignment on the device + quantize + pack, from the ratio alone."),
    METHOD(quantize_pack, "Quantize + group + pack by a given scheme, precision and scale per row."),
    METHOD(gemm_grouped_launch, "One launch of a prepared grouped plan."),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_marshal", "Argument marshalling of librmsmp's per-layer calls.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module_def);
}
