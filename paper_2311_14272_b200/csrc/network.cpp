// The parts of a pruning iteration that go over all layers and gradients of a network in Python: the table of the layers, and the tensors that
// decode returns.  They take torch's tensors themselves.  Asking a tensor for its address and pitch from Python takes 0.4 us, a layer's entry of
// the table 3 us and a tensor made by torch.empty_strided 1.6, of an iteration of 35 layers and 140 gradients that waits for all of it.  What they
// cannot do as the Python code beside their callers does (tensor subclasses, other containers, types and shapes) they leave to it by returning None.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty_strided.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

#include <cstdint>
#include <cstring>

#include "crisp.h"

namespace {

decltype(&crisp_decode) lib_decode;

// The names of attributes, made once.
struct {
    PyObject *desc, *mask_buf, *workspace, *canonical_buf, *exec_buf, *mask, *handle, *kkeep;
} names;

struct Ref {                             // an owned reference
    PyObject *p;
    explicit Ref(PyObject *o = nullptr) : p(o) {}
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

// A plain tensor (or parameter) of two dimensions on a GPU, or nullptr.
const at::Tensor *plain(PyObject *o) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(o);
    return t.is_cuda() && t.layout() == at::kStrided && t.dim() == 2 ? &t : nullptr;
}
// The address of a buffer that the object owns; false with an exception, or true and *out null where the attribute is no plain tensor.
bool buffer(PyObject *owner, PyObject *name, void **out, int64_t *numel) {
    Ref o(PyObject_GetAttr(owner, name));
    if (!o.p) return false;
    *out = nullptr;
    if (THPVariable_CheckExact(o.p)) {
        const at::Tensor &t = THPVariable_Unpack(o.p);
        *out = t.data_ptr();
        if (numel) *numel = t.numel();
    }
    return true;
}
// Whether it holds the layer's rows of consecutive elements.
bool holds(const at::Tensor &t, const crisp_layer_desc_t &d) {
    return t.size(0) >= d.rows && t.size(1) >= d.k && (t.stride(1) == 1 || d.k == 1);
}
bool descriptor(PyObject *layer, crisp_layer_desc_t *copy, double *keep_ratio) {        // reads it, or sets its keep ratio
    Ref o(PyObject_GetAttr(layer, names.desc));
    if (!o.p) return false;
    Py_buffer view;
    if (PyObject_GetBuffer(o.p, &view, PyBUF_WRITABLE) != 0) return false;
    const bool ok = view.len == (Py_ssize_t)sizeof(crisp_layer_desc_t);
    if (ok && copy) std::memcpy(copy, view.buf, sizeof *copy);
    if (ok && keep_ratio) static_cast<crisp_layer_desc_t *>(view.buf)->keep_ratio = *keep_ratio;
    PyBuffer_Release(&view);
    if (!ok) PyErr_SetString(PyExc_TypeError, "a layer's descriptor has another size");
    return ok;
}
template <typename T> T *address(PyObject *o) { return reinterpret_cast<T *>(PyLong_AsVoidPtr(o)); }
bool arguments(const char *name, Py_ssize_t given, Py_ssize_t n) {
    if (given == n) return true;
    PyErr_Format(PyExc_TypeError, "%s takes %zd arguments (%zd given)", name, n, given);
    return false;
}

// table(layers, weights, gradients, saliencies, array of crisp_prune_layer_t) -> bytes that the array's entries point into, or None: not filled in.
// All four are lists; an entry of `gradients` is a list or tuple.
PyObject *table(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arguments("table", n, 5)) return nullptr;
    for (int i = 0; i < 4; ++i)
        if (!PyList_CheckExact(args[i])) Py_RETURN_NONE;
    const Py_ssize_t count = PyList_GET_SIZE(args[1]);
    crisp_prune_layer_t *arr = address<crisp_prune_layer_t>(args[4]);
    if (!arr) return PyErr_Occurred() ? nullptr : Py_NewRef(Py_None);
    if (PyList_GET_SIZE(args[0]) < count || PyList_GET_SIZE(args[2]) < count || PyList_GET_SIZE(args[3]) < count) Py_RETURN_NONE;
    Py_ssize_t total = 0;
    for (Py_ssize_t l = 0; l < count; ++l) {
        PyObject *gs = PyList_GET_ITEM(args[2], l);
        if (!PyList_CheckExact(gs) && !PyTuple_CheckExact(gs)) Py_RETURN_NONE;
        total += PySequence_Fast_GET_SIZE(gs);
    }
    Ref held(PyBytes_FromStringAndSize(nullptr, total * (Py_ssize_t)(sizeof(void *) + sizeof(int64_t) + sizeof(int32_t)) + 8));
    if (!held.p) return nullptr;
    uintptr_t at = (reinterpret_cast<uintptr_t>(PyBytes_AS_STRING(held.p)) + 7) & ~(uintptr_t)7;
    const void **ptrs = reinterpret_cast<const void **>(at);
    int64_t *lds = reinterpret_cast<int64_t *>(ptrs + total);
    int32_t *dtypes = reinterpret_cast<int32_t *>(lds + total);
    for (Py_ssize_t l = 0; l < count; ++l) {
        crisp_prune_layer_t &P = arr[l];
        PyObject *layer = PyList_GET_ITEM(args[0], l), *gs = PyList_GET_ITEM(args[2], l);
        const at::Tensor *w = plain(PyList_GET_ITEM(args[1], l)), *s = plain(PyList_GET_ITEM(args[3], l));
        if (!w || !s || w->element_size() != 2 || w->stride(1) != 1) Py_RETURN_NONE;
        if (!descriptor(layer, &P.desc, nullptr) || !buffer(layer, names.mask_buf, &P.d_mask_buf, nullptr) ||
            !buffer(layer, names.workspace, &P.d_workspace, nullptr))
            return nullptr;
        if (!P.d_mask_buf || !P.d_workspace || !holds(*w, P.desc)) Py_RETURN_NONE;
        P.d_w_bf16 = static_cast<const uint16_t *>(w->data_ptr()); P.ld_w = w->stride(0);
        P.d_saliency = static_cast<float *>(s->data_ptr()); P.ld_s = s->stride(0);
        P.d_grads = ptrs; P.ld_grads = lds; P.grad_dtypes = dtypes;
        P.samples = (int32_t)PySequence_Fast_GET_SIZE(gs);
        PyObject **items = PySequence_Fast_ITEMS(gs);
        for (int32_t h = 0; h < P.samples; ++h) {
            const at::Tensor *g = plain(items[h]);
            if (!g || (g->scalar_type() != at::kBFloat16 && g->scalar_type() != at::kFloat) || !holds(*g, P.desc)) Py_RETURN_NONE;
            *ptrs++ = g->data_ptr(); *lds++ = g->stride(0);
            *dtypes++ = g->scalar_type() == at::kBFloat16 ? 0 : 1;
        }
    }
    return Py_NewRef(held.p);
    END_HANDLE_TH_ERRORS
}

// encodings(layers, array of crisp_prune_layer_t, size_t canonical capacities, size_t execution capacities, old masks, old handles): what the encodings
// need whatever the counts are, and the masks and handles that they will take the place of.
PyObject *encodings(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arguments("encodings", n, 6)) return nullptr;
    if (!PyList_CheckExact(args[0])) Py_RETURN_FALSE;
    crisp_prune_layer_t *arr = address<crisp_prune_layer_t>(args[1]);
    size_t *canonical = address<size_t>(args[2]), *execution = address<size_t>(args[3]);
    void **masks = address<void *>(args[4]), **handles = address<void *>(args[5]);
    if (!arr || !canonical || !execution || !masks || !handles) return PyErr_Occurred() ? nullptr : Py_NewRef(Py_False);
    for (Py_ssize_t l = 0; l < PyList_GET_SIZE(args[0]); ++l) {
        PyObject *layer = PyList_GET_ITEM(args[0], l);
        int64_t have_c = 0, have_e = 0;
        if (!buffer(layer, names.canonical_buf, &arr[l].d_canonical_buf, &have_c) || !buffer(layer, names.exec_buf, &arr[l].d_exec_buf, &have_e)) return nullptr;
        canonical[l] = (size_t)have_c; execution[l] = (size_t)have_e;
        Ref mask(PyObject_GetAttr(layer, names.mask)), handle(PyObject_GetAttr(layer, names.handle));
        if (!mask.p || !handle.p) return nullptr;
        masks[l] = PyLong_AsVoidPtr(mask.p); handles[l] = PyLong_AsVoidPtr(handle.p);
        if (PyErr_Occurred()) return nullptr;
    }
    Py_RETURN_TRUE;
    END_HANDLE_TH_ERRORS
}

// encoded(layers, counts, blocks, masks, handles): the layers take their new masks and handles; blocks: int32 blocks of a row tile.
PyObject *encoded(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arguments("encoded", n, 5)) return nullptr;
    const int32_t *blocks = address<int32_t>(args[2]);
    void **masks = address<void *>(args[3]), **handles = address<void *>(args[4]);
    if (!PyList_CheckExact(args[0]) || !PyList_CheckExact(args[1]) || PyList_GET_SIZE(args[1]) < PyList_GET_SIZE(args[0]) || !blocks || !masks || !handles) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "encoded(layers, counts, blocks, masks, handles)");
        return nullptr;
    }
    for (Py_ssize_t l = 0; l < PyList_GET_SIZE(args[0]); ++l) {
        PyObject *layer = PyList_GET_ITEM(args[0], l), *c = PyList_GET_ITEM(args[1], l);
        Ref mask(PyLong_FromVoidPtr(masks[l])), handle(PyLong_FromVoidPtr(handles[l]));
        if (!mask.p || !handle.p || PyObject_SetAttr(layer, names.mask, mask.p) || PyObject_SetAttr(layer, names.handle, handle.p) ||
            PyObject_SetAttr(layer, names.kkeep, c))
            return nullptr;
        double ratio = (double)PyLong_AsLong(c) / (double)blocks[l];                // floor(ratio * blocks + 0.5) gives the count back
        if (PyErr_Occurred() || !descriptor(layer, nullptr, &ratio)) return nullptr;
    }
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// decode(handle, rows, k, GPU, stream) -> (status, bf16 tensor [rows, k])
PyObject *decode(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arguments("decode", n, 5)) return nullptr;
    long long v[5];
    for (int i = 0; i < 5; ++i) {
        v[i] = PyLong_AsLongLong(args[i]);
        if (v[i] == -1 && PyErr_Occurred()) return nullptr;
    }
    at::Tensor w = at::empty_strided({v[1], v[2]}, {v[2], 1}, at::TensorOptions().dtype(at::kBFloat16).device(at::Device(at::kCUDA, (at::DeviceIndex)v[3])));
    crisp_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = lib_decode(reinterpret_cast<crisp_handle_t>((uintptr_t)v[0]), static_cast<uint16_t *>(w.data_ptr()), v[2], reinterpret_cast<void *>((uintptr_t)v[4]));
    Py_END_ALLOW_THREADS
    Ref out(THPVariable_Wrap(std::move(w)));
    return out.p ? Py_BuildValue("lO", (long)s, out.p) : nullptr;
    END_HANDLE_TH_ERRORS
}

// bind(address of crisp_decode)
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (!arguments("bind", n, 1)) return nullptr;
    lib_decode = reinterpret_cast<decltype(&crisp_decode)>(PyLong_AsVoidPtr(args[0]));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

#define CRISP_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {CRISP_METHOD(bind), CRISP_METHOD(table), CRISP_METHOD(encodings), CRISP_METHOD(encoded), CRISP_METHOD(decode), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_network", nullptr, 0, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__network(void) {
    names = {PyUnicode_InternFromString("desc"), PyUnicode_InternFromString("mask_buf"), PyUnicode_InternFromString("workspace"),
             PyUnicode_InternFromString("canonical_buf"), PyUnicode_InternFromString("exec_buf"), PyUnicode_InternFromString("mask"),
             PyUnicode_InternFromString("handle"), PyUnicode_InternFromString("kkeep")};
    PyObject *m = PyModule_Create(&module);
    // what the binding compares: the layout of torch's tensors and of Python's objects is that of the headers
#define CRISP_TEXT2(x) #x
#define CRISP_TEXT(x) CRISP_TEXT2(x)
    if (m && PyModule_AddStringConstant(m, "built_for", CRISP_TEXT(TORCH_VERSION_MAJOR) "." CRISP_TEXT(TORCH_VERSION_MINOR) "." CRISP_TEXT(TORCH_VERSION_PATCH)
                                        " " CRISP_TEXT(PY_MAJOR_VERSION) "." CRISP_TEXT(PY_MINOR_VERSION)) != 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
