// Descriptors of LayerBuffers objects (binding.py), written straight into an array of squant_layer: in
// Python this takes about 2 us a layer, longer than the GPU needs for the layers of a small model.
// fill(list, start, address) writes descriptors from element `start` on and returns the index of the first
// element it leaves to the Python code: one that is not made of plain tensors, or that the Python code
// would reject.  It neither keeps nor caches anything.
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstddef>
#include <limits>

#include "squant.h"

namespace {

PyObject *s_names[8];   // w, codes, scales, kernel_err, channel_err, dequant, dequant_bf16, scales_in

// A reference that goes with its scope, also when data_ptr() throws.
struct Held {
    PyObject *p = nullptr;
    Held() = default;
    Held(const Held &) = delete;
    Held &operator=(const Held &) = delete;
    ~Held() { Py_XDECREF(p); }
};

// The tensor behind attribute i of o: 1 found, 0 None, -1 not a plain tensor (or no such attribute).
int tensor_of(PyObject *o, int i, const at::Tensor *&t, Held &held)
{
    held.p = PyObject_GetAttr(o, s_names[i]);
    if (!held.p) {
        PyErr_Clear();
        return -1;
    }
    if (held.p == Py_None) return 0;
    if (!THPVariable_CheckExact(held.p)) return -1;   // subclasses may have their own idea of data_ptr()
    t = &THPVariable_Unpack(held.p);
    return 1;
}

// One descriptor.  False: left to the Python code.
bool descriptor(PyObject *o, squant_layer &l)
{
    void *ptr[8] = {};
    bool ok = true;
    const at::Tensor *w = nullptr;
    Held held[8];
    for (int i = 0; i < 8 && ok; ++i) {
        const at::Tensor *t = nullptr;
        const int kind = tensor_of(o, i, t, held[i]);
        if (kind < 0 || (i == 0 && kind == 0)) { ok = false; break; }
        if (kind == 0) continue;
        ptr[i] = t->data_ptr();
        if (i == 0) {
            w = t;
            const auto s = w->sizes();
            if (s.size() < 2 || s.size() > 4) { ok = false; break; }
            int32_t d[4] = {1, 1, 1, 1};
            for (size_t k = 0; k < s.size(); ++k) {
                if (s[k] > std::numeric_limits<int32_t>::max()) ok = false;
                d[k] = static_cast<int32_t>(s[k]);
            }
            l.cout = d[0]; l.cin = d[1]; l.kh = d[2]; l.kw = d[3];
        } else if (i == 7) {
            ok = t->scalar_type() == at::kFloat && t->numel() == l.cout && t->is_contiguous() && t->device() == w->device();
        }
    }
    if (ok) {
        l.w = static_cast<const float *>(ptr[0]);
        l.codes = static_cast<int8_t *>(ptr[1]);
        l.scales = static_cast<float *>(ptr[2]);
        l.kernel_err = static_cast<float *>(ptr[3]);
        l.channel_err = static_cast<float *>(ptr[4]);
        l.dequant = static_cast<float *>(ptr[5]);
        l.dequant_bf16 = static_cast<uint16_t *>(ptr[6]);
        l.scales_in = static_cast<const float *>(ptr[7]);
    }
    return ok;
}

PyObject *fill(PyObject *, PyObject *args)
{
    PyObject *list = nullptr;
    Py_ssize_t start = 0;
    unsigned long long address = 0;
    if (!PyArg_ParseTuple(args, "O!nK", &PyList_Type, &list, &start, &address)) return nullptr;
    squant_layer *out = reinterpret_cast<squant_layer *>(static_cast<uintptr_t>(address));
    Py_ssize_t i = start;
    if (!at::impl::torch_function_mode_enabled()) {
        for (; i < PyList_GET_SIZE(list); ++i) {
            bool ok = false;
            try {
                ok = descriptor(PyList_GET_ITEM(list, i), out[i]);
            } catch (const std::exception &) {   // a tensor without storage: the Python code raises its error
                ok = false;
            }
            if (!ok) break;
        }
    }
    return PyLong_FromSsize_t(i);
}

PyMethodDef methods[] = {{"fill", fill, METH_VARARGS, "fill(list, start, address) -> index of the first element left out"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
    const char *names[8] = {"w", "codes", "scales", "kernel_err", "channel_err", "dequant", "dequant_bf16", "scales_in"};
    for (int i = 0; i < 8; ++i) {
        s_names[i] = PyUnicode_InternFromString(names[i]);
        if (!s_names[i]) return nullptr;
    }
    PyObject *m = PyModule_Create(&module);
    if (!m) return nullptr;
    // Size of a descriptor and the places of its fields as this extension was built with them, in the order of
    // squant.h: the Python code compares them with its own before it hands over an array.
    using L = squant_layer;
    PyObject *layout = Py_BuildValue("(nnnnnnnnnnnnn)", sizeof(L), offsetof(L, w), offsetof(L, cout), offsetof(L, cin), offsetof(L, kh), offsetof(L, kw),
                                     offsetof(L, codes), offsetof(L, scales), offsetof(L, kernel_err), offsetof(L, channel_err),
                                     offsetof(L, dequant), offsetof(L, dequant_bf16), offsetof(L, scales_in));
    if (!layout || PyModule_AddObject(m, "layout", layout) != 0) {
        Py_XDECREF(layout);
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
