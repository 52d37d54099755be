// The attention calls of the Python binding in native code: argument checks, output allocation and the C ABI call of
// include/terra.h in one go.  The small calls (one 8 x 8-window block on a regional grid) take the GPU a few microseconds; the same
// marshalling in Python and ctypes took 15 to 40 microseconds a call, this takes about 2.
//
// No function of the library is linked: binding.py hands over the entry points of the library that it loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/terra.h"

namespace {

decltype(&terra_swin_workspace_bytes) f_workspace = nullptr;
decltype(&terra_swin_attn_fwd) f_fwd = nullptr;
decltype(&terra_swin_attn_bwd) f_bwd = nullptr;
decltype(&terra_swin_attn_fwd_packed) f_fwd_packed = nullptr;
decltype(&terra_swin_attn_bwd_packed) f_bwd_packed = nullptr;
decltype(&terra_swin_attn_fwd_noalloc) f_fwd_noalloc = nullptr;
PyObject* on_status = nullptr;          // binding._check: raises the TerraError of a status

struct Failed {};                       // a Python error is set

// Other Python threads run while this one allocates or launches: both wait for the GPU at times (a new segment of the caching
// allocator, a full launch queue).
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};

// The descriptor is a ctypes structure; its bytes are read through the buffer protocol.
struct Desc {
    Py_buffer view{};
    const terra_swin_desc* d = nullptr;
    explicit Desc(PyObject* o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE)) throw Failed{};
        if (view.len < (Py_ssize_t)sizeof(terra_swin_desc)) {
            PyBuffer_Release(&view);
            PyErr_SetString(PyExc_TypeError, "terra: the descriptor must be a terra_swin_desc");
            throw Failed{};
        }
        d = static_cast<const terra_swin_desc*>(view.buf);
    }
    ~Desc() { if (d) PyBuffer_Release(&view); }
    int64_t rows() const { return (int64_t)d->B * d->H * d->W * d->heads; }
    int64_t table() const { return (int64_t)(2 * d->window - 1) * (2 * d->window - 1) * d->heads; }
    at::ScalarType act() const { return d->dtype == TERRA_DTYPE_F16 ? at::kHalf : at::kBFloat16; }
};

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "terra: %s must be a tensor", name);
        throw Failed{};
    }
    return THPVariable_Unpack(o);
}

const char* dtype_name(at::ScalarType t) {
    switch (t) {
        case at::kBFloat16: return "torch.bfloat16";
        case at::kHalf: return "torch.float16";
        case at::kFloat: return "torch.float32";
        default: return c10::toString(t);
    }
}

void expect(const at::Tensor& t, at::ScalarType dtype, int64_t numel, const char* name) {
    if (t.scalar_type() == dtype && t.numel() == numel) return;
    PyErr_Format(PyExc_ValueError, "terra: %s must be %s with %lld elements, got %s x %lld", name, dtype_name(dtype), (long long)numel,
                 dtype_name(t.scalar_type()), (long long)t.numel());
    throw Failed{};
}

void* ptr(const at::Tensor& t) {
    if (!t.is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "terra: tensors must be CUDA tensors (the library has no CPU path)");
        throw Failed{};
    }
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "terra: tensors must be contiguous");
        throw Failed{};
    }
    // the library launches on the current device (its stream, SM count and built-in scratch are that device's)
    const int current = c10::cuda::current_device();
    if (t.device().index() != current) {
        PyErr_Format(PyExc_ValueError, "terra: tensor lives on cuda:%d but the current device is cuda:%d; make the tensors' device current "
                     "(torch.cuda.device(...)) around the call", (int)t.device().index(), current);
        throw Failed{};
    }
    return t.data_ptr();
}

void check(int status) {
    if (status == TERRA_OK) return;
    PyObject* r = PyObject_CallFunction(on_status, "i", status);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_Format(PyExc_RuntimeError, "terra status %d", status);
    throw Failed{};
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The library call (its pointers are taken before: that may raise).
template <class F, class... A>
void launch(F f, A... args) {
    int status;
    {
        NoGil no_gil;
        status = f(args...);
    }
    check(status);
}

// The caller's tensor, or a new one.
at::Tensor output(PyObject* o, const char* name, at::ScalarType dtype, at::IntArrayRef shape, const at::Tensor& like) {
    if (o != Py_None) return tensor(o, name);
    NoGil no_gil;
    return at::detail::empty_cuda(shape, dtype, like.device(), std::nullopt);
}

// The caller's workspace, or a new one of the size the call wants (an undefined tensor where it wants none).
at::Tensor workspace(PyObject* o, const Desc& desc, bool backward, const at::Tensor& like, size_t& bytes) {
    at::Tensor t;
    if (o != Py_None) {
        t = tensor(o, "workspace");
    } else {
        size_t need = 0;
        check(f_workspace(desc.d, backward, &need));
        if (need) {
            NoGil no_gil;
            t = at::detail::empty_cuda({(int64_t)need}, at::kByte, like.device(), std::nullopt);
        }
    }
    bytes = t.defined() ? t.nbytes() : 0;
    return t;
}
void* opt_ptr(const at::Tensor& t) { return t.defined() ? ptr(t) : nullptr; }

PyObject* tuple(std::initializer_list<at::Tensor> ts) {
    PyObject* r = PyTuple_New((Py_ssize_t)ts.size());
    if (!r) throw Failed{};
    Py_ssize_t i = 0;
    for (const at::Tensor& t : ts) PyTuple_SET_ITEM(r, i++, THPVariable_Wrap(t));
    return r;
}

template <class F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F body) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "terra: %zd arguments, %zd wanted", n, want);
        return nullptr;
    }
    try {
        return body();
    } catch (const Failed&) {
        return nullptr;
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// desc, q, k, v, bias_table, o, lse, workspace -> (o, lse)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&] {
        Desc d(a[0]);
        const at::Tensor &q = tensor(a[1], "q"), &k = tensor(a[2], "k"), &v = tensor(a[3], "v"), &b = tensor(a[4], "bias_table");
        const int64_t rows = d.rows(), all = rows * d.d->head_dim;
        expect(q, d.act(), all, "q"); expect(k, d.act(), all, "k"); expect(v, d.act(), all, "v");
        expect(b, at::kFloat, d.table(), "bias_table");
        void *pq = ptr(q), *pk = ptr(k), *pv = ptr(v), *pb = ptr(b);
        at::Tensor o = output(a[5], "o", d.act(), q.sizes(), q);
        at::Tensor lse = output(a[6], "lse", at::kFloat, {d.d->B, d.d->H, d.d->W, d.d->heads}, q);
        expect(o, d.act(), all, "o"); expect(lse, at::kFloat, rows, "lse");
        size_t bytes;
        at::Tensor ws = workspace(a[7], d, false, q, bytes);
        launch(f_fwd, d.d, pq, pk, pv, (const float*)pb, ptr(o), (float*)ptr(lse), opt_ptr(ws), bytes, stream());
        return tuple({o, lse});
    });
}

// desc, qkv, bias_table, o, lse, workspace -> (o, lse)
PyObject* fwd_packed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 6, [&] {
        Desc d(a[0]);
        const at::Tensor &x = tensor(a[1], "qkv"), &b = tensor(a[2], "bias_table");
        const int64_t rows = d.rows(), all = rows * d.d->head_dim;
        expect(x, d.act(), 3 * all, "qkv");
        expect(b, at::kFloat, d.table(), "bias_table");
        void *px = ptr(x), *pb = ptr(b);
        at::Tensor o = output(a[3], "o", d.act(), {d.d->B, d.d->H, d.d->W, d.d->heads, d.d->head_dim}, x);
        at::Tensor lse = output(a[4], "lse", at::kFloat, {d.d->B, d.d->H, d.d->W, d.d->heads}, x);
        expect(o, d.act(), all, "o"); expect(lse, at::kFloat, rows, "lse");
        size_t bytes;
        at::Tensor ws = workspace(a[5], d, false, x, bytes);
        launch(f_fwd_packed, d.d, px, (const float*)pb, ptr(o), (float*)ptr(lse), opt_ptr(ws), bytes, stream());
        return tuple({o, lse});
    });
}

// desc, q, k, v, bias_table, o, lse -> (o, lse)
PyObject* fwd_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        Desc d(a[0]);
        const at::Tensor &q = tensor(a[1], "q"), &k = tensor(a[2], "k"), &v = tensor(a[3], "v"), &b = tensor(a[4], "bias_table");
        const at::Tensor &o = tensor(a[5], "o"), &lse = tensor(a[6], "lse");
        const int64_t rows = d.rows(), all = rows * d.d->head_dim;
        expect(q, d.act(), all, "q"); expect(k, d.act(), all, "k"); expect(v, d.act(), all, "v"); expect(o, d.act(), all, "o");
        expect(b, at::kFloat, d.table(), "bias_table"); expect(lse, at::kFloat, rows, "lse");
        launch(f_fwd_noalloc, d.d, ptr(q), ptr(k), ptr(v), (const float*)ptr(b), ptr(o), (float*)ptr(lse), stream());
        return tuple({o, lse});
    });
}

// desc, q, k, v, bias_table, o, lse, d_o, dq, dk, dv, dbias, workspace -> (dq, dk, dv, dbias)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&] {
        Desc d(a[0]);
        const at::Tensor &q = tensor(a[1], "q"), &k = tensor(a[2], "k"), &v = tensor(a[3], "v"), &b = tensor(a[4], "bias_table");
        const at::Tensor &o = tensor(a[5], "o"), &lse = tensor(a[6], "lse"), &g = tensor(a[7], "d_o");
        const int64_t rows = d.rows(), all = rows * d.d->head_dim;
        expect(q, d.act(), all, "q"); expect(k, d.act(), all, "k"); expect(v, d.act(), all, "v"); expect(o, d.act(), all, "o"); expect(g, d.act(), all, "d_o");
        expect(lse, at::kFloat, rows, "lse"); expect(b, at::kFloat, d.table(), "bias_table");
        void *pq = ptr(q), *pk = ptr(k), *pv = ptr(v), *pb = ptr(b), *po = ptr(o), *pl = ptr(lse), *pg = ptr(g);
        at::Tensor dq = output(a[8], "dq", d.act(), q.sizes(), q), dk = output(a[9], "dk", d.act(), q.sizes(), q), dv = output(a[10], "dv", d.act(), q.sizes(), q);
        at::Tensor db = output(a[11], "dbias", at::kFloat, b.sizes(), q);
        expect(dq, d.act(), all, "dq"); expect(dk, d.act(), all, "dk"); expect(dv, d.act(), all, "dv"); expect(db, at::kFloat, b.numel(), "dbias");
        size_t bytes;
        at::Tensor ws = workspace(a[12], d, true, q, bytes);
        launch(f_bwd, d.d, pq, pk, pv, (const float*)pb, po, (const float*)pl, pg, ptr(dq), ptr(dk), ptr(dv), (float*)ptr(db), opt_ptr(ws), bytes, stream());
        return tuple({dq, dk, dv, db});
    });
}

// desc, qkv, bias_table, o, lse, d_o, dqkv, dbias, workspace -> (dqkv, dbias)
PyObject* bwd_packed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        Desc d(a[0]);
        const at::Tensor &x = tensor(a[1], "qkv"), &b = tensor(a[2], "bias_table"), &o = tensor(a[3], "o"), &lse = tensor(a[4], "lse"), &g = tensor(a[5], "d_o");
        const int64_t rows = d.rows(), all = rows * d.d->head_dim;
        expect(x, d.act(), 3 * all, "qkv"); expect(o, d.act(), all, "o"); expect(g, d.act(), all, "d_o");
        expect(lse, at::kFloat, rows, "lse"); expect(b, at::kFloat, d.table(), "bias_table");
        void *px = ptr(x), *pb = ptr(b), *po = ptr(o), *pl = ptr(lse), *pg = ptr(g);
        at::Tensor dx = output(a[6], "dqkv", d.act(), x.sizes(), x), db = output(a[7], "dbias", at::kFloat, b.sizes(), x);
        expect(dx, d.act(), 3 * all, "dqkv"); expect(db, at::kFloat, b.numel(), "dbias");
        size_t bytes;
        at::Tensor ws = workspace(a[8], d, true, x, bytes);
        launch(f_bwd_packed, d.d, px, (const float*)pb, po, (const float*)pl, pg, ptr(dx), (float*)ptr(db), opt_ptr(ws), bytes, stream());
        return tuple({dx, db});
    });
}

// The library's entry points (addresses, in this order) and the callable that raises for a status.
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 7, [&]() -> PyObject* {
        void* p[6];
        for (int i = 0; i < 6; ++i) {
            p[i] = PyLong_AsVoidPtr(a[i]);
            if (PyErr_Occurred()) throw Failed{};
        }
        f_workspace = (decltype(f_workspace))p[0];
        f_fwd = (decltype(f_fwd))p[1];
        f_bwd = (decltype(f_bwd))p[2];
        f_fwd_packed = (decltype(f_fwd_packed))p[3];
        f_bwd_packed = (decltype(f_bwd_packed))p[4];
        f_fwd_noalloc = (decltype(f_fwd_noalloc))p[5];
        Py_INCREF(a[6]);
        Py_XDECREF(on_status);
        on_status = a[6];
        Py_RETURN_NONE;
    });
}

#define FN(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FN(bind), FN(fwd), FN(bwd), FN(fwd_packed), FN(bwd_packed), FN(fwd_noalloc), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() { return PyModule_Create(&module); }
