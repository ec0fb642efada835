// The calls a program makes once per layer and step, from torch tensors to the C ABI without Python
// in between: argument checks, the output's allocation, the current stream and the call itself.
//
// What bounds it: at batch 1 a layer is about 7 us of GPU time, and the same call through Python and
// ctypes took 12.9 us of host time (torch.cuda.current_stream() 3.2, torch.empty 2.5, shape checks and
// attribute look-ups 2.6, ctypes 1.1, the C call itself 2.5-3.6), so small layers waited for the host.
//
// Every function returns an int where it cannot do the call: the library's status code when the
// C ABI returned one, or -1 when the arguments do not fit, upon which the Python wrapper goes through its own
// checks and raises with a message.  So it does when torch throws here, as it does for tensors without a storage (under a
// transform such as vmap, say): nothing C++ may leave a function that Python called.
#define PY_SSIZE_T_CLEAN
#include <cstring>
#include <Python.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "asx.h"

namespace {

PyObject* refuse() { return PyLong_FromLong(-1); }

const at::Tensor* tensor_or_null(PyObject* o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

// The stream argument of the wrappers: None is the current stream of the current device, else its cudaStream_t as an int.
bool stream_of(PyObject* o, void** st)
{
    if (o == Py_None) {
        try {
            *st = c10::cuda::getCurrentCUDAStream().stream();
            return true;
        } catch (const std::exception&) {
            return false;                          // no driver: the wrapper raises torch's own error
        }
    }
    *st = PyLong_AsVoidPtr(o);
    return !(*st == nullptr && PyErr_Occurred());
}

at::Tensor empty_on(const at::Tensor& like, at::IntArrayRef sizes, at::ScalarType type)
{
    return at::detail::empty_cuda(sizes, type, like.device(), c10::nullopt);
}

// run(geometry, x, w, bias, out, flags, stream) with geometry = (handle, C_in, C_out, kh, kw, stride, pad)
PyObject* run(PyObject* const* args, Py_ssize_t nargs)
{
    if (nargs != 7 || !PyTuple_Check(args[0]) || PyTuple_GET_SIZE(args[0]) != 7) return refuse();
    PyObject* g = args[0];
    asx_layer* layer = static_cast<asx_layer*>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(g, 0)));
    int64_t d[6];
    for (int i = 0; i < 6; ++i) d[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(g, i + 1));
    const int64_t C_in = d[0], C_out = d[1], kh = d[2], kw = d[3], stride = d[4], pad = d[5];
    const at::Tensor *x = tensor_or_null(args[1]), *w = tensor_or_null(args[2]);
    const long flags = PyLong_AsLong(args[5]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return refuse();
    }
    if (x == nullptr || w == nullptr || layer == nullptr) return refuse();
    const at::ScalarType type = (flags & ASX_F32) ? at::kFloat : at::kBFloat16;
    if (x->scalar_type() != type || w->scalar_type() != type || !x->is_cuda() || !w->is_cuda() || !x->is_contiguous() ||
        !w->is_contiguous() || x->dim() != 4 || w->dim() != 4)
        return refuse();
    const at::IntArrayRef xs = x->sizes(), ws = w->sizes();
    if (xs[3] != C_in || ws[0] != C_out || ws[1] != kh || ws[2] != kw || ws[3] != C_in) return refuse();
    const int64_t Nb = xs[0], H = xs[1], W = xs[2];
    if (Nb < 1 || H + 2 * pad < kh || W + 2 * pad < kw) return refuse();
    const int64_t size[4] = {Nb, (H + 2 * pad - kh) / stride + 1, (W + 2 * pad - kw) / stride + 1, C_out};
    const float* bias = nullptr;
    if (args[3] != Py_None) {
        const at::Tensor* b = tensor_or_null(args[3]);
        if (b == nullptr || b->scalar_type() != at::kFloat || !b->is_cuda() || b->numel() != C_out) return refuse();
        bias = static_cast<const float*>(b->data_ptr());
    }
    const void *xp = x->data_ptr(), *wp = w->data_ptr();
    void* st = nullptr;
    if (!stream_of(args[6], &st)) {
        PyErr_Clear();
        return refuse();
    }
    PyObject* out = args[4];
    void* y = nullptr;
    if (out == Py_None) {
        try {
            at::Tensor t = empty_on(*x, size, type);
            y = t.data_ptr();
            out = THPVariable_Wrap(std::move(t));
        } catch (const std::exception&) {
            return refuse();                       // out of memory: the wrapper's own allocation raises torch's error
        }
        if (out == nullptr) return nullptr;
    } else {
        const at::Tensor* t = tensor_or_null(out);
        if (t == nullptr || t->scalar_type() != type || !t->is_contiguous() || t->sizes() != at::IntArrayRef(size, 4)) return refuse();
        y = t->data_ptr();
        Py_INCREF(out);
    }
    asx_status s;
    Py_BEGIN_ALLOW_THREADS
    s = asx_run(layer, xp, (int)Nb, (int)H, (int)W, wp, bias, y, (int)flags, st);
    Py_END_ALLOW_THREADS
    if (s == ASX_OK) return out;
    Py_DECREF(out);
    return PyLong_FromLong(s);
}

// set_mask(handle, mask, stream): a contiguous uint8 tensor on either side, or a contiguous numpy array of bytes (through Python's own
// conversions and ctypes that took 6.5 us more)
PyObject* set_mask(PyObject* const* args, Py_ssize_t nargs)
{
    if (nargs != 3) return refuse();
    asx_layer* layer = static_cast<asx_layer*>(PyLong_AsVoidPtr(args[0]));
    const at::Tensor* m = tensor_or_null(args[1]);
    void* st = nullptr;
    if (PyErr_Occurred() || (m != nullptr && (m->scalar_type() != at::kByte || !m->is_contiguous())) || !stream_of(args[2], &st)) {
        PyErr_Clear();
        return refuse();
    }
    Py_buffer view;
    if (m == nullptr) {
        if (std::strcmp(Py_TYPE(args[1])->tp_name, "numpy.ndarray") != 0) return refuse();
        if (PyObject_GetBuffer(args[1], &view, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
            PyErr_Clear();
            return refuse();
        }
        if (view.itemsize != 1 || view.format == nullptr || std::strcmp(view.format, "B") != 0) {
            PyBuffer_Release(&view);
            return refuse();
        }
    }
    const uint8_t* p = m != nullptr ? static_cast<const uint8_t*>(m->data_ptr()) : static_cast<const uint8_t*>(view.buf);
    const int64_t rows = m != nullptr ? m->numel() : (int64_t)view.len;
    asx_status s;
    Py_BEGIN_ALLOW_THREADS
    s = asx_set_mask(layer, p, rows, st);
    Py_END_ALLOW_THREADS
    if (m == nullptr) PyBuffer_Release(&view);
    return PyLong_FromLong(s);
}

// mask_from_activation(x, stream) -> uint8 mask, one entry per row
PyObject* mask_from_activation(PyObject* const* args, Py_ssize_t nargs)
{
    if (nargs != 2) return refuse();
    const at::Tensor* x = tensor_or_null(args[0]);
    void* st = nullptr;
    if (x == nullptr || x->scalar_type() != at::kBFloat16 || !x->is_cuda() || !x->is_contiguous() || x->dim() < 1 ||
        x->size(-1) < 1 || x->size(-1) > (1 << 20) || !stream_of(args[1], &st)) {
        PyErr_Clear();
        return refuse();
    }
    const int64_t C = x->size(-1), rows = x->numel() / C;
    at::Tensor mask;
    try {
        mask = empty_on(*x, {rows}, at::kByte);
    } catch (const std::exception&) {
        return refuse();
    }
    const void* xp = x->data_ptr();
    uint8_t* mp = static_cast<uint8_t*>(mask.data_ptr());
    asx_status s;
    Py_BEGIN_ALLOW_THREADS
    s = asx_mask_from_activation(xp, rows, (int)C, mp, st);
    Py_END_ALLOW_THREADS
    return s == ASX_OK ? THPVariable_Wrap(std::move(mask)) : PyLong_FromLong(s);
}

// compact_mask(mask, stream) -> (kept, count, scratch)
PyObject* compact_mask(PyObject* const* args, Py_ssize_t nargs)
{
    if (nargs != 2) return refuse();
    const at::Tensor* m = tensor_or_null(args[0]);
    void* st = nullptr;
    if (m == nullptr || m->element_size() != 1 || !m->is_cuda() || !m->is_contiguous() || !stream_of(args[1], &st)) {
        PyErr_Clear();
        return refuse();
    }
    const int64_t rows = m->numel(), bytes = asx_compact_scratch_bytes(rows);
    at::Tensor kept, count, scratch;
    try {
        kept = empty_on(*m, {std::max<int64_t>(rows, 1)}, at::kInt);
        count = empty_on(*m, {1}, at::kInt);
        scratch = empty_on(*m, {(bytes + 7) / 8}, at::kLong);
    } catch (const std::exception&) {
        return refuse();
    }
    const uint8_t* mp = static_cast<const uint8_t*>(m->data_ptr());
    int32_t *kp = static_cast<int32_t*>(kept.data_ptr()), *cp = static_cast<int32_t*>(count.data_ptr());
    void* sp = scratch.data_ptr();
    asx_status s;
    Py_BEGIN_ALLOW_THREADS
    s = asx_compact(mp, rows, kp, cp, sp, bytes, st);
    Py_END_ALLOW_THREADS
    if (s != ASX_OK) return PyLong_FromLong(s);
    PyObject* all = PyTuple_New(3);
    if (all == nullptr) return nullptr;
    PyTuple_SET_ITEM(all, 0, THPVariable_Wrap(std::move(kept)));
    PyTuple_SET_ITEM(all, 1, THPVariable_Wrap(std::move(count)));
    PyTuple_SET_ITEM(all, 2, THPVariable_Wrap(std::move(scratch)));
    return all;
}

template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* args, Py_ssize_t nargs)
{
    try {
        return F(args, nargs);
    } catch (const std::exception&) {
        PyErr_Clear();
        return refuse();
    }
}
template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyCFunction entry()
{
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<F>));
}

PyMethodDef methods[] = {
    {"run", entry<run>(), METH_FASTCALL, nullptr},
    {"set_mask", entry<set_mask>(), METH_FASTCALL, nullptr},
    {"mask_from_activation", entry<mask_from_activation>(), METH_FASTCALL, nullptr},
    {"compact_mask", entry<compact_mask>(), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_asx_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__asx_torch() { return PyModule_Create(&module); }
