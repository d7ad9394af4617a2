// Python side of the calls a program makes per activation map: argument checks on torch tensors, the output tensor and the
// call into libdivision.so, without a Python interpreter step in between.  (The ctypes route costs 2.3 us of marshalling per
// compress call and 5 us per decompress call, 2.8 us of it to parse the arguments of torch.empty: more than the 2.5 us that
// the launch itself takes.)  Plain CPython extension, vector calls; all arithmetic stays in the CUDA library.
#include <torch/csrc/Device.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>

#include <cstring>

#include "../../include/division.h"

namespace {

bool tensor_arg(PyObject* o, const at::Tensor** out) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a tensor");
        return false;
    }
    *out = &THPVariable_Unpack(o);
    return true;
}
// the descriptor's fields, copied: the object may be replaced or changed while the interpreter is released
bool desc_arg(PyObject* o, div_desc* out) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    const bool ok = view.len == (Py_ssize_t)sizeof(*out);
    if (ok) memcpy(out, view.buf, sizeof(*out));
    PyBuffer_Release(&view);
    if (!ok) PyErr_SetString(PyExc_TypeError, "expected a DivDesc");
    return ok;
}
at::ScalarType scalar(const div_desc& d) { return d.x_dtype == DIV_F32 ? at::kFloat : at::kBFloat16; }
void* stream() { return reinterpret_cast<void*>(c10::cuda::getCurrentCUDAStream().stream()); }
bool matches(const at::Tensor& x, const div_desc& d) {
    return x.is_cuda() && x.scalar_type() == scalar(d) && x.dim() == 4 && x.size(0) == d.n && x.size(1) == d.c && x.size(2) == d.h &&
           x.size(3) == d.w && x.is_contiguous();
}

// compress(descriptor, x, blob, workspace or None (per-plane groups), seed, flags) -> status, or -1: x does not match
// (What a tensor may answer with an exception, its sizes, layout and storage, is asked before the interpreter is released.)
PyObject* compress(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 6) {
        PyErr_SetString(PyExc_TypeError, "compress takes 6 arguments");
        return nullptr;
    }
    div_desc d;
    const at::Tensor *x, *blob, *ws = nullptr;
    if (!desc_arg(a[0], &d) || !tensor_arg(a[1], &x) || !tensor_arg(a[2], &blob) || (a[3] != Py_None && !tensor_arg(a[3], &ws))) return nullptr;
    const uint64_t seed = PyLong_AsUnsignedLongLongMask(a[4]);
    PyObject* whole = PyNumber_Long(a[5]);                 // whatever int() takes
    if (!whole) return nullptr;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(whole);
    Py_DECREF(whole);
    if (PyErr_Occurred()) return nullptr;
    if (!matches(*x, d)) return PyLong_FromLong(-1);
    const void* from = x->data_ptr();
    void *to = blob->data_ptr(), *scratch = ws ? ws->data_ptr() : nullptr, *st = stream();
    const size_t room = (size_t)blob->numel(), scratch_room = ws ? (size_t)ws->numel() : 0;
    div_status got;
    Py_BEGIN_ALLOW_THREADS              // a full launch queue blocks
    got = ws ? div_compress_ex(&d, from, to, room, scratch, scratch_room, seed, st, flags) : div_planegroup_compress(&d, from, to, room, seed, st, flags);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)got);
    END_HANDLE_TH_ERRORS
}

// decompress(descriptor, blob, out or None, device, per-plane groups?) -> the output tensor (where out is None a new one on
// the device: the blob may be elsewhere, in pinned host memory for instance), or a status
PyObject* decompress(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 5) {
        PyErr_SetString(PyExc_TypeError, "decompress takes 5 arguments");
        return nullptr;
    }
    div_desc d;
    const at::Tensor *blob, *given = nullptr;
    if (!desc_arg(a[0], &d) || !tensor_arg(a[1], &blob) || (a[2] != Py_None && !tensor_arg(a[2], &given))) return nullptr;
    if (!THPDevice_Check(a[3])) {
        PyErr_SetString(PyExc_TypeError, "expected a device");
        return nullptr;
    }
    at::Tensor made;
    if (!given) {
        made = at::empty({d.n, d.c, d.h, d.w}, at::TensorOptions(reinterpret_cast<THPDevice*>(a[3])->device).dtype(scalar(d)));
        given = &made;
    }
    const auto call = a[4] == Py_True ? div_planegroup_decompress : div_decompress;
    const void* from = blob->data_ptr();
    void *to = given->data_ptr(), *st = stream();
    const size_t bytes = (size_t)blob->numel();
    div_status got;
    Py_BEGIN_ALLOW_THREADS
    got = call(&d, from, bytes, to, st);
    Py_END_ALLOW_THREADS
    if (got != DIV_OK) return PyLong_FromLong((long)got);
    if (made.defined()) return THPVariable_Wrap(std::move(made));
    Py_INCREF(a[2]);
    return a[2];
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"compress", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(compress)), METH_FASTCALL, nullptr},
    {"decompress", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decompress)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
