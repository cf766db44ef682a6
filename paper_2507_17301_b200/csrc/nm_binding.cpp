// CPython extension behind nm.py: the per-call work of the convolution and pooling entry points and of those that make and export a handle (type
// checks, output allocation, pointers, current stream) in native code.  A layer of a batch-1 network runs for a few microseconds; the
// same steps in Python with ctypes cost more than that: 12.8 us per nm_conv2d call before, 3.2 of them for
// torch.cuda.current_stream() alone.
//
// It links against torch only and calls the C-ABI library through the addresses nm.py hands to bind(), so that the library
// nm.py has loaded (NM_LIBRARY included) is the one that runs.
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/nm.h"

namespace {

decltype(&nm_conv2d) p_conv2d = nullptr;
decltype(&nm_conv2d_res) p_conv2d_res = nullptr;
decltype(&nm_maxpool2d) p_maxpool2d = nullptr;
decltype(&nm_prune) p_prune = nullptr;
decltype(&nm_weights_import) p_import = nullptr;
decltype(&nm_weights_export) p_export = nullptr;
decltype(&nm_weights_dims) p_dims = nullptr;

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// A contiguous float32 CUDA tensor, or NULL with a TypeError set.
const at::Tensor* dev_f32(PyObject* obj, const char* what)
{
    if (THPVariable_Check(obj)) {
        const at::Tensor& t = THPVariable_Unpack(obj);
        if (t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous()) return &t;
    }
    PyErr_Format(PyExc_TypeError, "%s must be a contiguous float32 CUDA tensor", what);
    return nullptr;
}

// An int, or a pair of them.
bool pair_of(PyObject* obj, int out[2])
{
    if (PyLong_Check(obj)) {
        out[0] = out[1] = static_cast<int>(PyLong_AsLong(obj));
        return !PyErr_Occurred();
    }
    for (int i = 0; i < 2; ++i) {
        PyObject* v = PySequence_GetItem(obj, i);
        if (!v) return false;
        PyObject* n = PyNumber_Long(v);
        Py_DECREF(v);
        if (!n) return false;
        out[i] = static_cast<int>(PyLong_AsLong(n));
        Py_DECREF(n);
        if (PyErr_Occurred()) return false;
    }
    return true;
}

bool rank4(const at::Tensor& t, const char* what)
{
    if (t.dim() == 4) return true;
    PyErr_Format(PyExc_ValueError, "%s must have four dimensions (got %d)", what, static_cast<int>(t.dim()));
    return false;
}

// Output positions along one axis, at least one (the library rejects a window that does not fit).
int64_t out_extent(int64_t in, int pad, int window, int stride)
{
    const int64_t room = in + 2 * static_cast<int64_t>(pad) - window;
    const int64_t n = (room >= 0 ? room / stride : -((-room + stride - 1) / stride)) + 1;
    return n > 1 ? n : 1;
}

// conv2d(handle, c_out, x, kh, kw, stride, pad, dil, bias, relu, y, plan address, residual) -> y, or the status as an int
PyObject* conv2d(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 13) {
        PyErr_SetString(PyExc_TypeError, "conv2d takes 13 arguments");
        return nullptr;
    }
    const auto* w = static_cast<const nm_weights_t*>(PyLong_AsVoidPtr(a[0]));
    const long c_out = PyLong_AsLong(a[1]);
    const auto* plan = static_cast<const nm_plan_t*>(PyLong_AsVoidPtr(a[11]));
    if (PyErr_Occurred()) return nullptr;
    int stride[2], pad[2], dil[2];
    if (!pair_of(a[5], stride) || !pair_of(a[6], pad) || !pair_of(a[7], dil)) return nullptr;
    const at::Tensor* x = dev_f32(a[2], "x");
    if (!x || !rank4(*x, "x")) return nullptr;
    const int64_t b = x->size(0), h = x->size(1), wd = x->size(2);
    at::Tensor made;
    const at::Tensor* y;
    if (a[10] == Py_None) {   // (the window's extent is looked at for the output's shape only: the handle knows it)
        const long kh = PyLong_AsLong(a[3]), kw = PyLong_AsLong(a[4]);
        if (PyErr_Occurred()) return nullptr;
        if (stride[0] < 1 || stride[1] < 1 || dil[0] < 1 || dil[1] < 1) {   // the library reports it
            made = at::empty({4}, x->options());
        } else {
            made = at::empty({b > 1 ? b : 1, out_extent(h, pad[0], dil[0] * (static_cast<int>(kh) - 1) + 1, stride[0]),
                              out_extent(wd, pad[1], dil[1] * (static_cast<int>(kw) - 1) + 1, stride[1]), c_out > 1 ? c_out : 1},
                             x->options());
        }
        y = &made;
    } else {
        y = dev_f32(a[10], "y");
        if (!y) return nullptr;
    }
    const float* bias = nullptr;
    if (a[8] != Py_None) {
        const at::Tensor* t = dev_f32(a[8], "bias");
        if (!t) return nullptr;
        bias = t->const_data_ptr<float>();
    }
    const int relu = PyObject_IsTrue(a[9]);
    if (relu < 0) return nullptr;
    const float* residual = nullptr;
    if (a[12] != Py_None) {
        const at::Tensor* t = dev_f32(a[12], "residual");
        if (!t) return nullptr;
        if (t->sizes() != y->sizes()) {
            PyErr_SetString(PyExc_TypeError, "residual must have the output's shape");
            return nullptr;
        }
        residual = t->const_data_ptr<float>();
    }
    const float* xp = x->const_data_ptr<float>();
    float* yp = y->mutable_data_ptr<float>();
    void* st = current_stream();
    const int bi = static_cast<int>(b), hi = static_cast<int>(h), wi = static_cast<int>(wd);
    nm_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = residual ? p_conv2d_res(w, xp, bi, hi, wi, stride[0], stride[1], pad[0], pad[1], dil[0], dil[1], bias, residual, relu, yp, plan, st)
                 : p_conv2d(w, xp, bi, hi, wi, stride[0], stride[1], pad[0], pad[1], dil[0], dil[1], bias, relu, yp, plan, st);
    Py_END_ALLOW_THREADS
    if (s != NM_OK) return PyLong_FromLong(s);
    if (a[10] == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(a[10]);
    return a[10];
}

// maxpool2d(x, kernel, stride, pad, y) -> y, or the status as an int
PyObject* maxpool2d(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 5) {
        PyErr_SetString(PyExc_TypeError, "maxpool2d takes 5 arguments");
        return nullptr;
    }
    int k[2], stride[2], pad[2];
    if (!pair_of(a[1], k) || !pair_of(a[2], stride) || !pair_of(a[3], pad)) return nullptr;
    const at::Tensor* x = dev_f32(a[0], "x");
    if (!x || !rank4(*x, "x")) return nullptr;
    const int64_t b = x->size(0), h = x->size(1), wd = x->size(2), c = x->size(3);
    at::Tensor made;
    const at::Tensor* y;
    if (a[4] == Py_None) {
        const int sh = stride[0] > 0 ? stride[0] : 1, sw = stride[1] > 0 ? stride[1] : 1;   // the library reports a bad one
        made = at::empty({b, out_extent(h, pad[0], k[0], sh), out_extent(wd, pad[1], k[1], sw), c}, x->options());
        y = &made;
    } else {
        y = dev_f32(a[4], "y");
        if (!y) return nullptr;
    }
    const float* xp = x->const_data_ptr<float>();
    float* yp = y->mutable_data_ptr<float>();
    void* st = current_stream();
    nm_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = p_maxpool2d(xp, static_cast<int>(b), static_cast<int>(h), static_cast<int>(wd), static_cast<int>(c), k[0], k[1], stride[0],
                    stride[1], pad[0], pad[1], yp, st);
    Py_END_ALLOW_THREADS
    if (s != NM_OK) return PyLong_FromLong(s);
    if (a[4] == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(a[4]);
    return a[4];
}

// `n` ints from `a` on; false with an exception set
bool ints_of(PyObject* const* a, int n, int* out)
{
    for (int i = 0; i < n; ++i) out[i] = static_cast<int>(PyLong_AsLong(a[i]));
    return !PyErr_Occurred();
}

// (handle, c_out, k, kk, n_tiles, tile_t) of a new handle, or the status as an int
PyObject* made_handle(nm_status_t s, nm_weights_t* w)
{
    int dims[5] = {0, 0, 0, 0, 0};
    if (s == NM_OK) s = p_dims(w, dims, dims + 1, dims + 2, dims + 3, dims + 4);
    if (s != NM_OK) return PyLong_FromLong(s);
    return Py_BuildValue("(Niiiii)", PyLong_FromVoidPtr(w), dims[0], dims[1], dims[2], dims[3], dims[4]);
}

// prune(w_dense, n_keep, m_group, tile_t)
PyObject* prune(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 4) {
        PyErr_SetString(PyExc_TypeError, "prune takes 4 arguments");
        return nullptr;
    }
    const at::Tensor* w = dev_f32(a[0], "w_dense");
    if (!w) return nullptr;
    if (w->dim() != 4) {
        PyErr_SetString(PyExc_TypeError, "w_dense must be [c_out, kh, kw, c_in]");
        return nullptr;
    }
    int v[3];
    if (!ints_of(a + 1, 3, v)) return nullptr;
    const float* ptr = w->const_data_ptr<float>();
    const int c_out = static_cast<int>(w->size(0)), kh = static_cast<int>(w->size(1)), kw = static_cast<int>(w->size(2)), c_in = static_cast<int>(w->size(3));
    void* st = current_stream();
    nm_weights_t* out = nullptr;
    nm_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = p_prune(ptr, c_out, kh, kw, c_in, v[0], v[1], v[2], st, &out);
    Py_END_ALLOW_THREADS
    return made_handle(s, out);
}

// weights_import(values, indices, kh, kw, c_in, n_keep, m_group, tile_t)
PyObject* weights_import(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 8) {
        PyErr_SetString(PyExc_TypeError, "weights_import takes 8 arguments");
        return nullptr;
    }
    const at::Tensor* values = dev_f32(a[0], "values");
    if (!values) return nullptr;
    const at::Tensor* indices = THPVariable_Check(a[1]) ? &THPVariable_Unpack(a[1]) : nullptr;
    if (!indices || !indices->is_cuda() || indices->scalar_type() != at::kUInt16 || !indices->is_contiguous()) {
        PyErr_SetString(PyExc_TypeError, "indices must be a contiguous uint16 CUDA tensor");
        return nullptr;
    }
    if (values->dim() < 1) {
        PyErr_SetString(PyExc_IndexError, "values has no rows");
        return nullptr;
    }
    int v[6];
    if (!ints_of(a + 2, 6, v)) return nullptr;
    const float* vp = values->const_data_ptr<float>();
    const auto* ip = static_cast<const uint16_t*>(indices->const_data_ptr());
    const int c_out = static_cast<int>(values->size(0));
    void* st = current_stream();
    nm_weights_t* out = nullptr;
    nm_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = p_import(vp, ip, c_out, v[0], v[1], v[2], v[3], v[4], v[5], st, &out);
    Py_END_ALLOW_THREADS
    return made_handle(s, out);
}

// weights_export(handle, c_out, kk, n_tiles) -> (values, indices), or the status as an int
PyObject* weights_export(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 4) {
        PyErr_SetString(PyExc_TypeError, "weights_export takes 4 arguments");
        return nullptr;
    }
    const auto* w = static_cast<const nm_weights_t*>(PyLong_AsVoidPtr(a[0]));
    int v[3];
    if (PyErr_Occurred() || !ints_of(a + 1, 3, v)) return nullptr;
    at::Tensor values = at::empty({v[0], v[1]}, at::TensorOptions().dtype(at::kFloat).device(at::kCUDA));
    at::Tensor indices = at::empty({v[2], v[1]}, at::TensorOptions().dtype(at::kUInt16).device(at::kCUDA));
    float* vp = values.mutable_data_ptr<float>();
    auto* ip = static_cast<uint16_t*>(indices.mutable_data_ptr());
    void* st = current_stream();
    nm_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = p_export(w, vp, ip, st);
    Py_END_ALLOW_THREADS
    if (s != NM_OK) return PyLong_FromLong(s);
    PyObject* vo = THPVariable_Wrap(std::move(values));
    PyObject* io = vo ? THPVariable_Wrap(std::move(indices)) : nullptr;
    if (!io) {
        Py_XDECREF(vo);
        return nullptr;
    }
    return Py_BuildValue("(NN)", vo, io);
}

PyObject* stream_ptr(PyObject*, PyObject* const*, Py_ssize_t n)
{
    if (n != 0) {
        PyErr_SetString(PyExc_TypeError, "stream_ptr takes no arguments");
        return nullptr;
    }
    return PyLong_FromVoidPtr(current_stream());
}

PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 7) {
        PyErr_SetString(PyExc_TypeError, "bind takes 7 addresses");
        return nullptr;
    }
    p_conv2d = reinterpret_cast<decltype(p_conv2d)>(PyLong_AsVoidPtr(a[0]));
    p_conv2d_res = reinterpret_cast<decltype(p_conv2d_res)>(PyLong_AsVoidPtr(a[1]));
    p_maxpool2d = reinterpret_cast<decltype(p_maxpool2d)>(PyLong_AsVoidPtr(a[2]));
    p_prune = reinterpret_cast<decltype(p_prune)>(PyLong_AsVoidPtr(a[3]));
    p_import = reinterpret_cast<decltype(p_import)>(PyLong_AsVoidPtr(a[4]));
    p_export = reinterpret_cast<decltype(p_export)>(PyLong_AsVoidPtr(a[5]));
    p_dims = reinterpret_cast<decltype(p_dims)>(PyLong_AsVoidPtr(a[6]));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

// C++ exceptions of torch (an allocation that fails, a process without a usable device) become Python exceptions.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    try {
        return F(self, a, n);
    } catch (const c10::OutOfMemoryError& e) {
        PyObject* torch = PyImport_ImportModule("torch");
        PyObject* type = torch ? PyObject_GetAttrString(torch, "OutOfMemoryError") : nullptr;
        if (type) PyErr_SetString(type, e.what_without_backtrace());
        Py_XDECREF(type);
        Py_XDECREF(torch);
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
    }
    return nullptr;
}

PyMethodDef methods[] = {
    {"conv2d", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<conv2d>)), METH_FASTCALL, nullptr},
    {"maxpool2d", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<maxpool2d>)), METH_FASTCALL, nullptr},
    {"prune", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<prune>)), METH_FASTCALL, nullptr},
    {"weights_import", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<weights_import>)), METH_FASTCALL, nullptr},
    {"weights_export", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<weights_export>)), METH_FASTCALL, nullptr},
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bind)), METH_FASTCALL, nullptr},
    {"stream_ptr", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<stream_ptr>)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_nm_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__nm_binding() { return PyModule_Create(&module_def); }
