// The short calls of binding.py without ctypes: tensors to addresses and strides, the current stream, the call.
//
// A decode step or a prompt of a thousand tokens takes the GPU 15 to 30 us, and marshalling the arguments of its three or four
// calls through ctypes took the host as long: 8 us a focus_assign and 16 a focus_decode_step on a slow core.  A decode step over
// 2049 keys in a row of them: 33.0 -> 21.4 us (30.6 -> 19.4 on a faster host); from the call until the GPU is done, with the GPU
// idle before: 45.5 -> 34.3, and a prompt of 1024 tokens in buffers not used before 65 -> 48.
//
// The functions take what binding.py's take.  They answer None when an argument is none that they know how to read (a tensor
// subclass, a shape that is no focus_shape, ...), before anything has been enqueued; binding.py then goes through ctypes as for
// its other entry points.
#include <Python.h>

#include <optional>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "focus.h"

namespace {

PyObject* shape_type;                // binding.focus_shape

// The entry points, from the library that binding.py has loaded: linked against, the loader might find another copy of it.
decltype(&focus_assign) p_assign;
decltype(&focus_assign_hidden) p_assign_hidden;
decltype(&focus_build_tiles) p_build_tiles;
decltype(&focus_attn_fwd) p_attn_fwd;
decltype(&focus_decode_step) p_decode_step;

struct Args {
    PyObject* const* a;
    bool known = true;               // every argument so far was of a kind that is read here
    bool failed = false;             // a Python error is set

    const focus_shape* shape(int i) {
        Py_buffer b;
        if (!known || failed || (PyObject*)Py_TYPE(a[i]) != shape_type) { known = false; return nullptr; }
        if (PyObject_GetBuffer(a[i], &b, PyBUF_SIMPLE)) { failed = true; return nullptr; }
        const focus_shape* s = b.len == (Py_ssize_t)sizeof(focus_shape) ? static_cast<const focus_shape*>(b.buf) : nullptr;
        PyBuffer_Release(&b);        // (the caller's reference keeps the object, and with it the memory)
        if (!s) known = false;
        return s;
    }
    const at::Tensor* tensor(int i) {
        if (!known || failed || !THPVariable_CheckExact(a[i])) { known = false; return nullptr; }
        return &THPVariable_Unpack(a[i]);
    }
    // address of a tensor, or of nothing
    void* ptr(int i) {
        if (!known || failed || a[i] == Py_None) return nullptr;
        const at::Tensor* t = tensor(i);
        return t ? t->data_ptr() : nullptr;
    }
    // [H, n, D] or [batch, H, n, D] bf16 CUDA tensor with D contiguous; `vector`: [H, D] or [batch, H, D]
    focus_tensor bf16(int i, bool vector) {
        focus_tensor out = {};
        const at::Tensor* t = tensor(i);
        if (!t) return out;
        const int dims = (int)t->dim(), outer = vector ? 1 : 2;
        if (!t->is_cuda() || t->scalar_type() != at::kBFloat16 || (dims != outer + 1 && dims != outer + 2) || t->stride(dims - 1) != 1) {
            known = false;           // binding.py says what is wrong with it
            return out;
        }
        const int h = dims - outer - 1;                  // dimension of the heads
        out.ptr = t->data_ptr();
        out.stride_h = t->stride(h);
        out.stride_b = h == 0 ? out.stride_h * t->size(0) : t->stride(0);
        out.stride_n = vector ? t->size(dims - 1) : t->stride(h + 1);
        return out;
    }
    size_t bytes(int i) {
        const at::Tensor* t = tensor(i);
        return t ? (size_t)t->numel() * t->element_size() : 0;
    }
    int32_t integer(int i) {
        if (!known || failed) return 0;
        if (!PyLong_CheckExact(a[i])) { known = false; return 0; }
        int over = 0;
        const long v = PyLong_AsLongAndOverflow(a[i], &over);
        if (over || v != (int32_t)v) known = false;
        return (int32_t)v;
    }
    float number(int i) {
        if (!known || failed) return 0.f;
        if (!PyFloat_CheckExact(a[i])) { known = false; return 0.f; }
        return (float)PyFloat_AS_DOUBLE(a[i]);
    }
    void* stream(int i) {
        if (!known || failed) return nullptr;
        if (a[i] != Py_None) { known = false; return nullptr; }
        return c10::cuda::getCurrentCUDAStream().stream();
    }
};

// `read` reads the arguments and returns the call to make
template <class Read>
PyObject* enter(PyObject* const* args, Py_ssize_t got, Py_ssize_t want, Read read) {
    if (got != want) return PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", got, want);
    Args a{args};
    auto guarded = [&]() -> decltype(std::make_optional(read(a))) {
        try {
            return read(a);
        } catch (const std::exception&) {                // a tensor without storage, no driver, ...: binding.py meets it again
            a.known = false;
            return std::nullopt;
        }
    };
    auto call = guarded();
    if (a.failed) return nullptr;
    if (!a.known || !call) Py_RETURN_NONE;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (*call)();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyObject* assign(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return enter(args, n, 8, [](Args& a) {
        auto s = a.shape(0);
        auto x = a.bf16(1, false);
        auto H = a.integer(2);
        auto c = static_cast<const float*>(a.ptr(3));
        auto m = static_cast<uint32_t*>(a.ptr(4));
        auto near = static_cast<unsigned long long*>(a.ptr(5));
        auto eps = a.number(6);
        auto st = a.stream(7);
        return [=] { return p_assign(s, x, H, c, m, near, eps, st); };
    });
}

PyObject* assign_hidden(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return enter(args, n, 11, [](Args& a) {
        auto s = a.shape(0);
        focus_tensor h = {};                             // [n, d_model] or [batch, n, d_model]
        int32_t d = 0, dg = 0;
        if (const at::Tensor* t = a.tensor(1)) {
            if (t->is_cuda() && t->scalar_type() == at::kBFloat16 && (t->dim() == 2 || t->dim() == 3) && t->stride(-1) == 1) {
                h.ptr = t->data_ptr();
                h.stride_n = t->stride(-2);
                h.stride_b = t->dim() == 3 ? t->stride(0) : t->stride(0) * t->size(0);
                d = (int32_t)t->size(-1);
            } else {
                a.known = false;
            }
        }
        if (const at::Tensor* t = a.tensor(2)) {
            if (t->dim() == 2) dg = (int32_t)t->size(1);
            else a.known = false;
        }
        auto Wg = static_cast<const float*>(a.ptr(2)), Cg = static_cast<const float*>(a.ptr(3)), bias = static_cast<const float*>(a.ptr(4));
        auto folded = static_cast<float*>(a.ptr(5));
        auto mq = static_cast<uint32_t*>(a.ptr(6)), mk = static_cast<uint32_t*>(a.ptr(7));
        auto near = static_cast<unsigned long long*>(a.ptr(8));
        auto eps = a.number(9);
        auto st = a.stream(10);
        return [=] { return p_assign_hidden(s, h.ptr, h.stride_b, h.stride_n, d, dg, Wg, Cg, bias, folded, mq, mk, near, eps, st); };
    });
}

PyObject* build_tiles(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return enter(args, n, 6, [](Args& a) {
        auto s = a.shape(0);
        auto mq = static_cast<const uint32_t*>(a.ptr(1));
        auto mk = static_cast<const uint32_t*>(a.ptr(2));
        auto layout = a.integer(3);
        auto ws = a.ptr(4);
        auto bytes = a.bytes(4);
        auto st = a.stream(5);
        return [=] { return p_build_tiles(s, mq, mk, layout, ws, bytes, st); };
    });
}

PyObject* attn_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return enter(args, n, 12, [](Args& a) {
        auto s = a.shape(0);
        auto q = a.bf16(1, false), k = a.bf16(2, false), v = a.bf16(3, false);
        auto mq = static_cast<const uint32_t*>(a.ptr(4));
        auto mk = static_cast<const uint32_t*>(a.ptr(5));
        auto ws = a.ptr(6);
        auto layout = a.integer(7);
        auto o = a.bf16(8, false);
        auto lse = static_cast<float*>(a.ptr(9));
        auto status = static_cast<int32_t*>(a.ptr(10));
        auto st = a.stream(11);
        return [=] { return p_attn_fwd(s, q, k, v, mq, mk, ws, layout, o, lse, status, st); };
    });
}

PyObject* decode_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return enter(args, n, 10, [](Args& a) {
        auto s = a.shape(0);
        auto q = a.bf16(1, true);
        auto k = a.bf16(2, false), v = a.bf16(3, false);
        auto mq = static_cast<const uint32_t*>(a.ptr(4));
        auto mk = static_cast<const uint32_t*>(a.ptr(5));
        auto o = a.bf16(6, true);
        auto lse = static_cast<float*>(a.ptr(7));
        auto ws = a.ptr(8);
        auto bytes = a.bytes(8);
        auto st = a.stream(9);
        return [=] { return p_decode_step(s, q, k, v, mq, mk, o, lse, ws, bytes, st); };
    });
}

// init(type of a shape, addresses of the entry points in the order above)
PyObject* init(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 6) return PyErr_Format(PyExc_TypeError, "%zd arguments, not 6", n);
    void* at[5];
    for (int i = 0; i < 5; ++i) {
        at[i] = PyLong_AsVoidPtr(args[1 + i]);
        if (!at[i]) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "no address");
    }
    p_assign = reinterpret_cast<decltype(p_assign)>(at[0]);
    p_assign_hidden = reinterpret_cast<decltype(p_assign_hidden)>(at[1]);
    p_build_tiles = reinterpret_cast<decltype(p_build_tiles)>(at[2]);
    p_attn_fwd = reinterpret_cast<decltype(p_attn_fwd)>(at[3]);
    p_decode_step = reinterpret_cast<decltype(p_decode_step)>(at[4]);
    Py_INCREF(args[0]);
    Py_XSETREF(shape_type, args[0]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"init", (PyCFunction)(void*)init, METH_FASTCALL, nullptr},
    {"assign", (PyCFunction)(void*)assign, METH_FASTCALL, nullptr},
    {"assign_hidden", (PyCFunction)(void*)assign_hidden, METH_FASTCALL, nullptr},
    {"build_tiles", (PyCFunction)(void*)build_tiles, METH_FASTCALL, nullptr},
    {"attn_fwd", (PyCFunction)(void*)attn_fwd, METH_FASTCALL, nullptr},
    {"decode_step", (PyCFunction)(void*)decode_step, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "short calls of binding.py", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
    PyObject* m = PyModule_Create(&module);
    // the torch and the Python whose objects the code above reads; binding.py compares before it passes it any
    if (m && PyModule_AddStringConstant(m, "built_for", FOCUS_BUILT_FOR)) Py_CLEAR(m);
    return m;
}
