// Python entry points for the calls that are made once per layer and pass.  They take plain integers (addresses, pitches, sizes)
// and hand them to libcrisp's C ABI.  ctypes converts eight arguments in 1.7 us, these in 0.2, of the 4 to 5 us that
// such a call takes on the host.  The library runs without the interpreter's lock, as under ctypes: a launch may have to wait
// for room in a stream.  bind() says which loaded library they call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>

#include "crisp.h"

namespace {

struct {
    decltype(&crisp_spmm) spmm;
    decltype(&crisp_spmm_conv) spmm_conv;
    decltype(&crisp_decode) decode;
    decltype(&crisp_build_mask) build_mask;
    decltype(&crisp_encode_sizes) encode_sizes;
    decltype(&crisp_encode) encode;
    decltype(&crisp_mask_destroy) mask_destroy;
    decltype(&crisp_destroy) destroy;
} lib;

// args[0 .. n) as 64-bit integers; false with an exception set if one is not an integer or does not fit.
bool integers(const char *name, PyObject *const *args, Py_ssize_t given, Py_ssize_t n, long long *out) {
    if (given != n) {
        PyErr_Format(PyExc_TypeError, "%s takes %zd arguments (%zd given)", name, n, given);
        return false;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        out[i] = PyLong_AsLongLong(args[i]);
        if (out[i] == -1 && PyErr_Occurred()) return false;
    }
    return true;
}
template <typename T> T *address(long long v) { return reinterpret_cast<T *>((uintptr_t)v); }
template <typename H> H handle(long long v) { return reinterpret_cast<H>((uintptr_t)v); }

// spmm(handle, x, ldx, ncols, y, ldy, y_dtype, stream) -> status
PyObject *spmm(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[8];
    if (!integers("spmm", args, n, 8, v)) return nullptr;
    crisp_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = lib.spmm(handle<crisp_handle_t>(v[0]), address<const uint16_t>(v[1]), v[2], v[3], address<void>(v[4]), v[5], (int32_t)v[6], address<void>(v[7]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)s);
}

// spmm_conv(handle, activation, batch, height, width, channels, kernel_h, kernel_w, pad, y_layout, y, ldy, y_dtype, stream) -> status
PyObject *spmm_conv(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[14];
    if (!integers("spmm_conv", args, n, 14, v)) return nullptr;
    for (int i = 2; i < 10; ++i)
        if (v[i] != (int32_t)v[i]) return PyLong_FromLong((long)CRISP_BAD_SHAPE);
    const crisp_conv_desc_t conv = {(int32_t)v[2], (int32_t)v[3], (int32_t)v[4], (int32_t)v[5], (int32_t)v[6], (int32_t)v[7], (int32_t)v[8], (int32_t)v[9]};
    crisp_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = lib.spmm_conv(handle<crisp_handle_t>(v[0]), address<const uint16_t>(v[1]), &conv, address<void>(v[10]), v[11], (int32_t)v[12], address<void>(v[13]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)s);
}

// decode(handle, w, ld, stream) -> status
PyObject *decode(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[4];
    if (!integers("decode", args, n, 4, v)) return nullptr;
    crisp_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = lib.decode(handle<crisp_handle_t>(v[0]), address<uint16_t>(v[1]), v[2], address<void>(v[3]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)s);
}

// build_mask(saliency, ld, descriptor, mask buffer, workspace, stream, replaced mask) -> (status, mask)
PyObject *build_mask(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[7];
    if (!integers("build_mask", args, n, 7, v)) return nullptr;
    crisp_status_t s;
    crisp_mask_t mask = nullptr;
    Py_BEGIN_ALLOW_THREADS
    lib.mask_destroy(handle<crisp_mask_t>(v[6]));
    s = lib.build_mask(address<const float>(v[0]), v[1], address<const crisp_layer_desc_t>(v[2]), address<void>(v[3]), address<void>(v[4]), address<void>(v[5]), &mask);
    Py_END_ALLOW_THREADS
    return Py_BuildValue("lK", (long)s, (unsigned long long)(uintptr_t)mask);
}

// encode_sizes(mask) -> (status, canonical bytes, execution bytes)
PyObject *encode_sizes(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[1];
    if (!integers("encode_sizes", args, n, 1, v)) return nullptr;
    size_t canonical = 0, exec = 0;
    const crisp_status_t s = lib.encode_sizes(handle<crisp_mask_t>(v[0]), &canonical, &exec);
    return Py_BuildValue("lKK", (long)s, (unsigned long long)canonical, (unsigned long long)exec);
}

// encode(w, ld, mask, canonical buffer, execution buffer, stream, replaced handle) -> (status, handle)
PyObject *encode(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[7];
    if (!integers("encode", args, n, 7, v)) return nullptr;
    crisp_status_t s;
    crisp_handle_t h = nullptr;
    Py_BEGIN_ALLOW_THREADS
    lib.destroy(handle<crisp_handle_t>(v[6]));
    s = lib.encode(address<const uint16_t>(v[0]), v[1], handle<crisp_mask_t>(v[2]), address<void>(v[3]), address<void>(v[4]), address<void>(v[5]), &h);
    Py_END_ALLOW_THREADS
    return Py_BuildValue("lK", (long)s, (unsigned long long)(uintptr_t)h);
}

// bind(addresses of the functions in the order of `lib`)
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long v[8];
    if (!integers("bind", args, n, 8, v)) return nullptr;
    lib = {handle<decltype(&crisp_spmm)>(v[0]), handle<decltype(&crisp_spmm_conv)>(v[1]), handle<decltype(&crisp_decode)>(v[2]),
           handle<decltype(&crisp_build_mask)>(v[3]), handle<decltype(&crisp_encode_sizes)>(v[4]), handle<decltype(&crisp_encode)>(v[5]),
           handle<decltype(&crisp_mask_destroy)>(v[6]), handle<decltype(&crisp_destroy)>(v[7])};
    Py_RETURN_NONE;
}

#define CRISP_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {CRISP_METHOD(bind), CRISP_METHOD(spmm), CRISP_METHOD(spmm_conv), CRISP_METHOD(decode), CRISP_METHOD(build_mask),
                         CRISP_METHOD(encode_sizes), CRISP_METHOD(encode), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, 0, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
