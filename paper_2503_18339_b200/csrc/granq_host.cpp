// The binding's calls in native code: takes the tensors apart, allocates what is missing and calls the library, all without the
// interpreter.  A call that Python marshals argument by argument costs the host 8 us with its buffers at hand and up to 20 us with
// everything to allocate, of which the library takes 3 to 5; small layers are paced by that.  Host time, us, Python / here: fused call with its
// buffers 7.9 / 4.3, forward with packed mask and everything to allocate 18.0 / 9.1, codes 19.7 / 10.1, range 13.9 / 9.3.
//
// Only the plain case is handled: CUDA tensors of the exact tensor type, contiguous, of the shapes and types that go together, on the
// current stream.  For anything else a function returns None, has done nothing, and binding.py goes its own way, errors included.
#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#include "../../include/granq.h"

namespace {

// entry points of the loaded library, in the order of kEntries
struct Library {
    decltype(&granq_num_groups) num_groups;
    decltype(&granq_workspace_bytes) workspace_bytes;
    decltype(&granq_range) range;
    decltype(&granq_fakequant_fused) fused;
    decltype(&granq_fakequant_fused_fwd_packmask) fused_fwd_packmask;
    decltype(&granq_fakequant_fused_stats) fused_stats;
    decltype(&granq_quantize_packed_fused) quantize_packed_fused;
    decltype(&granq_fakequant_fwd_packmask) fwd_packmask;
    decltype(&granq_fakequant_bwd_packmask) bwd_packmask;
    decltype(&granq_dequantize_packed) dequantize_packed;
    decltype(&granq_accumulate_codes) accumulate_codes;
    decltype(&granq_accumulate_workspace_bytes) accumulate_workspace_bytes;
    decltype(&granq_packmask_bytes) packmask_bytes;
    decltype(&granq_packed_codes_bytes) packed_codes_bytes;
};
constexpr const char* kEntries[] = {
    "granq_num_groups", "granq_workspace_bytes", "granq_range", "granq_fakequant_fused", "granq_fakequant_fused_fwd_packmask",
    "granq_fakequant_fused_stats", "granq_quantize_packed_fused", "granq_fakequant_fwd_packmask", "granq_fakequant_bwd_packmask",
    "granq_dequantize_packed", "granq_accumulate_codes", "granq_accumulate_workspace_bytes", "granq_packmask_bytes",
    "granq_packed_codes_bytes"};
static_assert(sizeof(Library) == sizeof(kEntries), "one address each");

Library lib{};
PyObject* out_class = nullptr;       // binding.FakeQuantOut
PyObject* error_class = nullptr;     // binding.GranqError

enum Field { Y, GX, LO, HI, S, Z, CODES, MASK, WORKSPACE, PACKED_MASK, SUMS, PACKED_CODES, kFields };
constexpr const char* kFieldNames[kFields] = {"y", "gx", "lo", "hi", "s", "z", "codes", "mask", "workspace", "packed_mask", "sums", "packed_codes"};
PyObject* field_names[kFields];

// a tensor as it was passed, or as it was made here
struct Buffer {
    at::Tensor t;
    bool made = false;
    void* ptr() const { return t.defined() ? t.data_ptr() : nullptr; }
};

// A tensor that the library can take as it is: false for anything else.  None leaves the buffer empty.
bool take(PyObject* o, Buffer& b) {
    if (o == Py_None) return true;
    if (!THPVariable_CheckExact(o)) return false;
    b.t = THPVariable_Unpack(o);
    return b.t.is_cuda() && b.t.is_contiguous();
}

bool number(PyObject* o, long& v) {
    if (!PyLong_CheckExact(o)) return false;
    v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) PyErr_Clear();
    else return v >= INT32_MIN && v <= INT32_MAX;
    return false;
}

int dtype_of(const at::Tensor& t) { return t.scalar_type() == at::kFloat ? 0 : t.scalar_type() == at::kBFloat16 ? 1 : -1; }

// x: four dims, a type the library knows
bool activation(PyObject* o, Buffer& x) { return o != Py_None && take(o, x) && x.t.dim() == 4 && dtype_of(x.t) >= 0; }

bool dims_of(PyObject* shape, int64_t (&dims)[4]) {
    if (!PyTuple_Check(shape) || PyTuple_GET_SIZE(shape) != 4) return false;
    for (int i = 0; i < 4; ++i) {
        long v;
        if (!number(PyTuple_GET_ITEM(shape, i), v)) return false;
        dims[i] = v;
    }
    return true;
}

void make(Buffer& b, at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
    b.t = at::empty(sizes, like.options().dtype(type).requires_grad(false));
    b.made = true;
}

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* failed(int rc, const char* what) {
    PyObject* e = PyObject_CallFunction(error_class, "is", rc, what);
    if (e) {
        PyErr_SetObject(error_class, e);
        Py_DECREF(e);
    }
    return nullptr;
}

// wraps what was made here into `out`; a new record where none was passed
PyObject* hand_back(PyObject* out, Buffer (&f)[kFields]) {
    PyObject* o = out == Py_None ? PyObject_CallNoArgs(out_class) : Py_NewRef(out);
    if (!o) return nullptr;
    for (int i = 0; i < kFields; ++i) {
        if (!f[i].made) continue;
        PyObject* t = THPVariable_Wrap(std::move(f[i].t));
        const int bad = t ? PyObject_SetAttr(o, field_names[i], t) : -1;
        Py_XDECREF(t);
        if (bad) {
            Py_DECREF(o);
            return nullptr;
        }
    }
    return o;
}

bool plain_now() { return !at::impl::torch_function_mode_enabled(); }

// call(kind, x, bits, gy, channel_axis, group, out, want_params, flags)
// kind 0: fused, 1: fused_fwd_packmask, 2: fused_stats, 3: quantize_packed_fused
PyObject* fused_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 9 || !plain_now()) Py_RETURN_NONE;
    long kind, bits, axis, group, want, flags;
    Buffer x, gy, f[kFields];
    if (!number(a[0], kind) || !activation(a[1], x) || !number(a[2], bits) || !take(a[3], gy) || !number(a[4], axis) || !number(a[5], group) ||
        !number(a[7], want) || !number(a[8], flags))
        Py_RETURN_NONE;
    if (gy.t.defined() && (gy.t.scalar_type() != x.t.scalar_type() || gy.t.sizes() != x.t.sizes())) Py_RETURN_NONE;
    PyObject* out = a[6];
    if (out != Py_None) {
        if (Py_TYPE(out) != (PyTypeObject*)out_class) Py_RETURN_NONE;
        for (int i = 0; i < kFields; ++i) {
            PyObject* t = PyObject_GetAttr(out, field_names[i]);
            if (!t) return nullptr;
            const bool ok = take(t, f[i]);
            Py_DECREF(t);           // the record keeps it
            if (!ok) Py_RETURN_NONE;
        }
        if (f[CODES].t.defined() || f[MASK].t.defined()) Py_RETURN_NONE;
    }
    const int64_t* dims = x.t.sizes().data();
    const int dt = dtype_of(x.t);
    const int64_t G = lib.num_groups(dims, (int)axis, (int)group);
    if (G < 0) Py_RETURN_NONE;
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        auto missing = [&](Field i) { return !f[i].t.defined(); };
        if (kind != 3 && missing(Y)) make(f[Y], x.t.sizes(), x.t.scalar_type(), x.t);
        if (kind == 0 && gy.t.defined() && missing(GX)) make(f[GX], x.t.sizes(), x.t.scalar_type(), x.t);
        if (kind == 1 && missing(PACKED_MASK)) make(f[PACKED_MASK], {(int64_t)lib.packmask_bytes(dims) / 4}, at::kInt, x.t);
        if (kind == 2 && missing(SUMS)) make(f[SUMS], {4}, at::kDouble, x.t);
        if (missing(LO)) make(f[LO], {G}, at::kFloat, x.t);
        if (missing(HI)) make(f[HI], {G}, at::kFloat, x.t);
        if (kind == 3) {
            if (missing(S)) make(f[S], {G}, at::kFloat, x.t);
            if (missing(Z)) make(f[Z], {G}, at::kFloat, x.t);
        } else if (want && missing(S)) {
            make(f[S], {G}, at::kFloat, x.t);
            make(f[Z], {G}, at::kFloat, x.t);
        }
        if (kind == 3 && missing(PACKED_CODES)) make(f[PACKED_CODES], {(int64_t)lib.packed_codes_bytes(dims, (int)bits) / 4}, at::kInt, x.t);
        if (missing(WORKSPACE)) make(f[WORKSPACE], {(int64_t)lib.workspace_bytes(dt, dims, (int)axis, (int)group)}, at::kByte, x.t);
        float *lo = (float*)f[LO].ptr(), *hi = (float*)f[HI].ptr(), *s = (float*)f[S].ptr(), *z = (float*)f[Z].ptr();
        void* ws = f[WORKSPACE].ptr();
        const size_t wsb = (size_t)f[WORKSPACE].t.numel();
        void* st = current_stream();
        switch (kind) {
            case 0:
                rc = lib.fused(x.ptr(), gy.ptr(), dt, dims, (int)axis, (int)group, (int)bits, f[Y].ptr(), gy.t.defined() ? f[GX].ptr() : nullptr,
                               lo, hi, nullptr, nullptr, s, z, ws, wsb, (uint32_t)flags, st);
                break;
            case 1:
                rc = lib.fused_fwd_packmask(x.ptr(), dt, dims, (int)axis, (int)group, (int)bits, f[Y].ptr(), (uint32_t*)f[PACKED_MASK].ptr(), lo,
                                            hi, s, z, ws, wsb, (uint32_t)flags, st);
                break;
            case 2:
                rc = lib.fused_stats(x.ptr(), dt, dims, (int)axis, (int)group, (int)bits, f[Y].ptr(), lo, hi, s, z, (double*)f[SUMS].ptr(), ws,
                                     wsb, (uint32_t)flags, st);
                break;
            default:
                rc = lib.quantize_packed_fused(x.ptr(), dt, dims, (int)axis, (int)group, (int)bits, (uint32_t*)f[PACKED_CODES].ptr(), lo, hi, s,
                                               z, ws, wsb, (uint32_t)flags, st);
        }
    }
    constexpr const char* names[] = {"granq_fakequant_fused", "granq_fakequant_fused_fwd_packmask", "granq_fakequant_fused_stats",
                                     "granq_quantize_packed_fused"};
    if (rc != GRANQ_OK) return failed(rc, names[kind]);
    return hand_back(out, f);
    END_HANDLE_TH_ERRORS
}

// range_call(x, channel_axis, group, lo, hi, workspace, flags) -> (lo, hi)
PyObject* range_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 7 || !plain_now()) Py_RETURN_NONE;
    long axis, group, flags;
    Buffer x, lo, hi, ws;
    if (!activation(a[0], x) || !number(a[1], axis) || !number(a[2], group) || !take(a[3], lo) || !take(a[4], hi) || !take(a[5], ws) ||
        !number(a[6], flags))
        Py_RETURN_NONE;
    const int64_t* dims = x.t.sizes().data();
    const int dt = dtype_of(x.t);
    const int64_t G = lib.num_groups(dims, (int)axis, (int)group);
    if (G < 0) Py_RETURN_NONE;
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        if (!lo.t.defined()) make(lo, {G}, at::kFloat, x.t);
        if (!hi.t.defined()) make(hi, {G}, at::kFloat, x.t);
        if (!ws.t.defined()) make(ws, {(int64_t)lib.workspace_bytes(dt, dims, (int)axis, (int)group)}, at::kByte, x.t);
        rc = lib.range(x.ptr(), dt, dims, (int)axis, (int)group, (float*)lo.ptr(), (float*)hi.ptr(), ws.ptr(), (size_t)ws.t.numel(),
                       (uint32_t)flags, current_stream());
    }
    if (rc != GRANQ_OK) return failed(rc, "granq_range");
    PyObject* l = lo.made ? THPVariable_Wrap(lo.t) : Py_NewRef(a[3]);
    PyObject* h = hi.made ? THPVariable_Wrap(hi.t) : Py_NewRef(a[4]);
    PyObject* r = l && h ? PyTuple_Pack(2, l, h) : nullptr;
    Py_XDECREF(l);
    Py_XDECREF(h);
    return r;
    END_HANDLE_TH_ERRORS
}

// fwd_packmask_call(x, bits, lo, hi, channel_axis, group, y, packed_mask, want_params, flags)
PyObject* fwd_packmask_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 10 || !plain_now()) Py_RETURN_NONE;
    long bits, axis, group, want, flags;
    Buffer x, f[kFields];
    if (!activation(a[0], x) || !number(a[1], bits) || a[2] == Py_None || !take(a[2], f[LO]) || a[3] == Py_None || !take(a[3], f[HI]) ||
        !number(a[4], axis) || !number(a[5], group) || !take(a[6], f[Y]) || !take(a[7], f[PACKED_MASK]) || !number(a[8], want) ||
        !number(a[9], flags))
        Py_RETURN_NONE;
    const int64_t* dims = x.t.sizes().data();
    const int dt = dtype_of(x.t);
    const int64_t G = lib.num_groups(dims, (int)axis, (int)group);
    if (G < 0) Py_RETURN_NONE;
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        if (!f[Y].t.defined()) make(f[Y], x.t.sizes(), x.t.scalar_type(), x.t);
        if (!f[PACKED_MASK].t.defined()) make(f[PACKED_MASK], {(int64_t)lib.packmask_bytes(dims) / 4}, at::kInt, x.t);
        if (want) {
            make(f[S], {G}, at::kFloat, x.t);
            make(f[Z], {G}, at::kFloat, x.t);
        }
        rc = lib.fwd_packmask(x.ptr(), dt, dims, (int)axis, (int)group, (int)bits, (const float*)f[LO].ptr(), (const float*)f[HI].ptr(),
                              f[Y].ptr(), (uint32_t*)f[PACKED_MASK].ptr(), (float*)f[S].ptr(), (float*)f[Z].ptr(), (uint32_t)flags,
                              current_stream());
    }
    if (rc != GRANQ_OK) return failed(rc, "granq_fakequant_fwd_packmask");
    PyObject* o = hand_back(Py_None, f);
    // what the caller passed comes back in the record
    const struct {
        Field field;
        PyObject* given;
    } passed[] = {{LO, a[2]}, {HI, a[3]}, {Y, a[6]}, {PACKED_MASK, a[7]}};
    for (const auto& p : passed)
        if (o && p.given != Py_None && PyObject_SetAttr(o, field_names[p.field], p.given)) Py_CLEAR(o);
    return o;
    END_HANDLE_TH_ERRORS
}

// bwd_packmask_call(gy, packed_mask, gx, flags)
PyObject* bwd_packmask_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 4 || !plain_now()) Py_RETURN_NONE;
    long flags;
    Buffer gy, mask, gx;
    if (!activation(a[0], gy) || a[1] == Py_None || !take(a[1], mask) || !take(a[2], gx) || !number(a[3], flags)) Py_RETURN_NONE;
    const int64_t* dims = gy.t.sizes().data();
    if ((size_t)mask.t.nbytes() < lib.packmask_bytes(dims)) Py_RETURN_NONE;
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        if (!gx.t.defined()) make(gx, gy.t.sizes(), gy.t.scalar_type(), gy.t);
        rc = lib.bwd_packmask(gy.ptr(), (const uint32_t*)mask.ptr(), dtype_of(gy.t), dims, gx.ptr(), (uint32_t)flags, current_stream());
    }
    if (rc != GRANQ_OK) return failed(rc, "granq_fakequant_bwd_packmask");
    return gx.made ? THPVariable_Wrap(gx.t) : Py_NewRef(a[2]);
    END_HANDLE_TH_ERRORS
}

// dequantize_call(packed_codes, shape, dtype, bits, s, z, channel_axis, group, y)
PyObject* dequantize_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 9 || !plain_now()) Py_RETURN_NONE;
    long bits, axis, group;
    int64_t dims[4];
    Buffer codes, s, z, y;
    if (a[0] == Py_None || !take(a[0], codes) || !dims_of(a[1], dims) || !THPDtype_Check(a[2]) || !number(a[3], bits) || a[4] == Py_None ||
        !take(a[4], s) || a[5] == Py_None || !take(a[5], z) || !number(a[6], axis) || !number(a[7], group) || !take(a[8], y))
        Py_RETURN_NONE;
    for (int64_t d : dims)
        if (d < 0) Py_RETURN_NONE;
    const at::ScalarType type = y.t.defined() ? y.t.scalar_type() : reinterpret_cast<THPDtype*>(a[2])->scalar_type;
    if (type != at::kFloat && type != at::kBFloat16) Py_RETURN_NONE;
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        if (!y.t.defined()) make(y, dims, type, codes.t);
        rc = lib.dequantize_packed((const uint32_t*)codes.ptr(), dtype_of(y.t), dims, (int)axis, (int)group, (int)bits, (const float*)s.ptr(),
                                   (const float*)z.ptr(), y.ptr(), 0, current_stream());
    }
    if (rc != GRANQ_OK) return failed(rc, "granq_dequantize_packed");
    return y.made ? THPVariable_Wrap(y.t) : Py_NewRef(a[8]);
    END_HANDLE_TH_ERRORS
}

// accumulate_call(packed_codes, shape, bits, s, z, weights, channel_axis, y, workspace, flags) -> (y, workspace)
PyObject* accumulate_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 10 || !plain_now()) Py_RETURN_NONE;
    long bits, axis, flags;
    int64_t dims[4];
    Buffer codes, s, z, w, y, ws;
    if (a[0] == Py_None || !take(a[0], codes) || !dims_of(a[1], dims) || !number(a[2], bits) || a[3] == Py_None || !take(a[3], s) ||
        a[4] == Py_None || !take(a[4], z) || a[5] == Py_None || !take(a[5], w) || !number(a[6], axis) || !take(a[7], y) || !take(a[8], ws) ||
        !number(a[9], flags))
        Py_RETURN_NONE;
    if ((axis != 1 && axis != 3) || w.t.scalar_type() != at::kFloat || w.t.dim() != 2 || w.t.size(1) != dims[axis]) Py_RETURN_NONE;
    for (int64_t d : dims)
        if (d < 0) Py_RETURN_NONE;
    const int64_t o = w.t.size(0);
    int rc;
    {
        pybind11::gil_scoped_release free_others;
        if (!y.t.defined()) {
            const int64_t nchw[4] = {dims[0], o, dims[2], dims[3]}, nhwc[4] = {dims[0], dims[1], dims[2], o};
            make(y, axis == 1 ? at::IntArrayRef(nchw) : at::IntArrayRef(nhwc), at::kFloat, codes.t);
        }
        if (!ws.t.defined()) make(ws, {(int64_t)lib.accumulate_workspace_bytes(dims, (int)axis, o)}, at::kByte, codes.t);
        rc = lib.accumulate_codes((const uint32_t*)codes.ptr(), dims, (int)axis, (int)bits, (const float*)s.ptr(), (const float*)z.ptr(),
                                  (const float*)w.ptr(), o, (float*)y.ptr(), ws.ptr(), (size_t)ws.t.numel(), (uint32_t)flags, current_stream());
    }
    if (rc != GRANQ_OK) return failed(rc, "granq_accumulate_codes");
    PyObject* py = y.made ? THPVariable_Wrap(y.t) : Py_NewRef(a[7]);
    PyObject* pw = ws.made ? THPVariable_Wrap(ws.t) : Py_NewRef(a[8]);
    PyObject* r = py && pw ? PyTuple_Pack(2, py, pw) : nullptr;
    Py_XDECREF(py);
    Py_XDECREF(pw);
    return r;
    END_HANDLE_TH_ERRORS
}

// setup({entry point: address}, FakeQuantOut, GranqError)
PyObject* setup(PyObject*, PyObject* args) {
    PyObject *addresses, *out, *error;
    if (!PyArg_ParseTuple(args, "O!OO", &PyDict_Type, &addresses, &out, &error)) return nullptr;
    void* at[sizeof(kEntries) / sizeof(*kEntries)];
    for (size_t i = 0; i < sizeof(kEntries) / sizeof(*kEntries); ++i) {
        PyObject* v = PyDict_GetItemString(addresses, kEntries[i]);
        if (!v) return PyErr_Format(PyExc_KeyError, "%s", kEntries[i]);
        at[i] = PyLong_AsVoidPtr(v);
        if (!at[i]) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "%s", kEntries[i]);
    }
    memcpy(&lib, at, sizeof(lib));
    for (int i = 0; i < kFields; ++i)
        if (!field_names[i] && !(field_names[i] = PyUnicode_InternFromString(kFieldNames[i]))) return nullptr;
    Py_XSETREF(out_class, Py_NewRef(out));
    Py_XSETREF(error_class, Py_NewRef(error));
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"setup", setup, METH_VARARGS, nullptr},
                         {"fused_call", (PyCFunction)(void*)fused_call, METH_FASTCALL, nullptr},
                         {"range_call", (PyCFunction)(void*)range_call, METH_FASTCALL, nullptr},
                         {"fwd_packmask_call", (PyCFunction)(void*)fwd_packmask_call, METH_FASTCALL, nullptr},
                         {"bwd_packmask_call", (PyCFunction)(void*)bwd_packmask_call, METH_FASTCALL, nullptr},
                         {"dequantize_call", (PyCFunction)(void*)dequantize_call, METH_FASTCALL, nullptr},
                         {"accumulate_call", (PyCFunction)(void*)accumulate_call, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods};

}  // namespace

// built_for: the versions whose objects are taken apart here, which binding.py compares before it calls anything
PyMODINIT_FUNC PyInit__host() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", GRANQ_HOST_RECORD)) Py_CLEAR(m);
    return m;
}
