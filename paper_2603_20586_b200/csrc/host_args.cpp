// Host side of the binding: the levels of a call as the array of 64-bit words that mka_level[3], mka_level_grad[3] and
// mka_paged_level[3] are, the call's small outputs, and the calls of the library that short steps consist of.  Asked for one by one from Python, the
// pointers, shapes and strides of the six tensors of a call took longer than a short decode takes on the GPU (6.3 us; 0.2 us here); the
// rest of a call's arguments through ctypes took 1.7 us of a router's 4.6, and of a forward's 12.2 (a short prompt is over in 17) 7.7.
#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <torch/csrc/autograd/python_variable.h>

#include <Python.h>
#include <stdint.h>
#include <string.h>

#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include "mka.h"

namespace {

constexpr char kLevelsWanted[] = "levels: tensors [batch, head, row, column] with dense columns, K and V alike; tables and row counts int32";
constexpr char kTensorWanted[] = "a tensor (or None where an argument may be left out) is expected";
constexpr char kCountWanted[] = "wrong number of arguments";
struct Bad { const char* what = kLevelsWanted; };    // what an assertion of the binding would have refused
struct PyErrSet {};                                  // the Python error is set

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) throw Bad{kTensorWanted};
    return THPVariable_Unpack(o);
}

struct Held {                                        // a reference of our own
    PyObject* o;
    explicit Held(PyObject* x) : o(x) { if (!o) throw PyErrSet(); }
    ~Held() { Py_XDECREF(o); }
    Held(const Held&) = delete;
    Held& operator=(const Held&) = delete;
};
// Entries of a list or tuple, or of whatever else answers x[i] (then held as long as this is).
class Seq {
    PyObject* x_;
    const bool plain_;
    std::vector<PyObject*> held_;

  public:
    explicit Seq(PyObject* x) : x_(x), plain_(PyList_Check(x) || PyTuple_Check(x)) { Py_INCREF(x_); }
    ~Seq() {
        for (PyObject* h : held_) Py_DECREF(h);
        Py_DECREF(x_);
    }
    Seq(const Seq&) = delete;
    Seq& operator=(const Seq&) = delete;
    PyObject* at(Py_ssize_t i) {
        if (plain_ && i < PySequence_Fast_GET_SIZE(x_)) return PySequence_Fast_GET_ITEM(x_, i);
        const Held at(PyLong_FromSsize_t(i));
        PyObject* item = PyObject_GetItem(x_, at.o);
        if (!item) throw PyErrSet();
        held_.push_back(item);
        return item;
    }
    const at::Tensor* tensor_at(Py_ssize_t i) {               // nullptr for None
        PyObject* x = at(i);
        return x == Py_None ? nullptr : &tensor(x);
    }
};

int64_t address(const at::Tensor& t) { return static_cast<int64_t>(reinterpret_cast<intptr_t>(t.data_ptr())); }
int64_t integer(PyObject* o) {                       // int(o)
    int64_t v;
    if (PyLong_CheckExact(o)) {
        v = PyLong_AsLongLong(o);
    } else {
        const Held whole(PyNumber_Long(o));
        v = PyLong_AsLongLong(whole.o);
    }
    if (v == -1 && PyErr_Occurred()) throw PyErrSet();
    return v;
}
template <size_t N> PyObject* bytes(const int64_t (&w)[N]) { return PyBytes_FromStringAndSize(reinterpret_cast<const char*>(w), sizeof(w)); }

// Four dimensions, the last one dense, and V laid out as K.
void check_layout(const at::Tensor& k, const at::Tensor& v) {
    if (k.dim() != 4 || k.stride(3) != 1 || v.strides() != k.strides()) throw Bad{};
}
void check_pair(const at::Tensor& k, const at::Tensor& v) {
    check_layout(k, v);
    if (v.sizes() != k.sizes()) throw Bad{};
}

template <typename F>
PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const Bad& bad) {
        PyErr_SetString(PyExc_AssertionError, bad.what);
        return nullptr;
    } catch (const PyErrSet&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// Words of a level: k, v, n, stride_b, stride_h, stride_n; zeros where keys are None or have no rows.
void put_level(int64_t* o, const at::Tensor& k, const at::Tensor& v) {
    o[0] = address(k); o[1] = address(v); o[2] = k.size(2);
    for (int i = 0; i < 3; ++i) o[3 + i] = k.stride(i);
}
PyObject* levels(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 2) throw Bad{kCountWanted};
        Seq K(a[0]), V(a[1]);
        int64_t w[18] = {};
        for (int l = 0; l < 3; ++l) {
            const at::Tensor* k = K.tensor_at(l);
            if (!k || k->size(2) == 0) continue;
            const at::Tensor* v = V.tensor_at(l);
            if (!v) throw Bad{};
            check_pair(*k, *v);
            put_level(w + 6 * l, *k, *v);
        }
        return bytes(w);
    });
}
PyObject* grads(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 3) throw Bad{kCountWanted};
        Seq K(a[0]), dK(a[1]), dV(a[2]);
        int64_t w[18] = {};
        for (int l = 0; l < 3; ++l) {
            const at::Tensor* k = K.tensor_at(l);
            if (!k || k->size(2) == 0) continue;
            const at::Tensor *dk = dK.tensor_at(l), *dv = dV.tensor_at(l);
            if (!dk || !dv) throw Bad{};
            check_layout(*dk, *dv);
            put_level(w + 6 * l, *dk, *dv);
        }
        return bytes(w);
    });
}

PyObject* paged_levels(PyObject*, PyObject* const* a, Py_ssize_t n_args) {
    return guarded([&]() -> PyObject* {
        if (n_args != 5) throw Bad{kCountWanted};
        Seq K(a[0]), V(a[1]), tabs(a[2]), rows(a[3]), n(a[4]);
        const bool counted = a[3] != Py_None;
        int64_t w[36] = {};
        for (int l = 0; l < 3; ++l) {
            int64_t* o = w + 12 * l;
            o[7] = 1;
            const at::Tensor* k = K.tensor_at(l);
            if (!k) continue;
            const int64_t most = integer(n.at(l));
            if (most == 0) continue;
            const at::Tensor *v = V.tensor_at(l), *tab = tabs.tensor_at(l), *r = counted ? rows.tensor_at(l) : nullptr;
            if (!v || !tab) throw Bad{};
            check_pair(*k, *v);
            // [B, pages]: one table per sequence; [B, H_kv, pages]: one per (sequence, KV head)
            if (tab->scalar_type() != at::kInt || (tab->dim() != 2 && tab->dim() != 3) || tab->stride(tab->dim() - 1) != 1) throw Bad{};
            if (r && (r->scalar_type() != at::kInt || !r->is_contiguous())) throw Bad{};
            o[0] = address(*k); o[1] = address(*v); o[2] = address(*tab); o[3] = r ? address(*r) : 0;
            o[4] = most; o[5] = tab->stride(0); o[6] = tab->dim() == 3 ? tab->stride(1) : 0; o[7] = k->size(2);
            for (int i = 0; i < 3; ++i) o[8 + i] = k->stride(i);
            o[11] = k->size(0);
        }
        return bytes(w);
    });
}

PyObject* paged_level(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 3) throw Bad{kCountWanted};
        const at::Tensor &k = tensor(a[0]), &v = tensor(a[1]), &tab = tensor(a[2]);
        check_layout(k, v);
        if (tab.scalar_type() != at::kInt || tab.dim() != 2 || tab.stride(1) != 1) throw Bad{};
        const int64_t w[12] = {address(k), address(v), address(tab), 0, tab.size(1) * k.size(2), tab.stride(0), 0, k.size(2),
                               k.stride(0), k.stride(1), k.stride(2), k.size(0)};
        return bytes(w);
    });
}

PyObject* empties_like(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 1) throw Bad{kCountWanted};
        const Held in(PySequence_Fast(a[0], "a sequence of tensors is expected"));
        const Py_ssize_t size = PySequence_Fast_GET_SIZE(in.o);
        Held out(PyList_New(size));
        for (Py_ssize_t i = 0; i < size; ++i) {
            PyObject* x = PySequence_Fast_GET_ITEM(in.o, i);
            PyObject* o = x == Py_None ? Py_None : THPVariable_Wrap(at::empty_like(tensor(x)));
            if (x == Py_None) Py_INCREF(o);
            PyList_SET_ITEM(out.o, i, o);
        }
        Py_INCREF(out.o);
        return out.o;
    });
}

PyObject* empty_f32(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 3) throw Bad{kCountWanted};
        const at::Tensor& t = tensor(a[0]);
        const int64_t keep = integer(a[1]), extra = integer(a[2]);
        if (keep < 0 || keep > t.dim()) throw Bad{"as many dimensions as the tensor has, at most"};
        std::vector<int64_t> size(t.sizes().begin(), t.sizes().begin() + keep);
        if (extra) size.push_back(extra);
        return THPVariable_Wrap(at::empty(size, at::TensorOptions().device(t.device()).dtype(at::kFloat)));
    });
}

// A C argument from a Python object; what was taken out of the object lives as long as this.
template <typename P> struct Arg;
template <> struct Arg<int64_t> {
    int64_t v;
    explicit Arg(PyObject* o) : v(0) {                // an int or what answers __index__ as one (numpy's, a tensor's); no float
        const Held whole(PyNumber_Index(o));
        v = PyLong_AsLongLong(whole.o);
        if (v == -1 && PyErr_Occurred()) throw PyErrSet();
    }
};
template <> struct Arg<int32_t> {
    int32_t v;
    explicit Arg(PyObject* o) : v(static_cast<int32_t>(Arg<int64_t>(o).v)) {}
};
template <> struct Arg<size_t> {
    size_t v;
    explicit Arg(PyObject* o) : v(static_cast<size_t>(Arg<int64_t>(o).v)) {}
};
void* pointer(PyObject* o) {                         // an int, or None for null
    if (o == Py_None) return nullptr;
    if (!PyLong_Check(o)) throw Bad{"an address is expected: an int or None"};
    void* const v = PyLong_AsVoidPtr(o);
    if (!v && PyErr_Occurred()) throw PyErrSet();
    return v;
}
// A tensor's memory, or that of whatever else has a data_ptr(), as a storage has, or None; no int, as True in an output's place would be address 1.
template <typename T> struct Arg<T*> {
    T* v;
    explicit Arg(PyObject* o) : v(nullptr) {
        if (o == Py_None) return;
        if (THPVariable_Check(o)) {
            v = static_cast<T*>(tensor(o).data_ptr());
            return;
        }
        if (!PyObject_HasAttrString(o, "data_ptr")) throw Bad{kTensorWanted};
        const Held at(PyObject_CallMethod(o, "data_ptr", nullptr));
        v = static_cast<T*>(pointer(at.o));
    }
};
struct Address {                                     // of a function, or a stream's handle: an int, or what holds one as a c_void_p does
    void* v;
    explicit Address(PyObject* o) : v(nullptr) {
        if (o == Py_None || PyLong_Check(o) || !PyObject_HasAttrString(o, "value")) {
            v = pointer(o);
            return;
        }
        const Held at(PyObject_GetAttrString(o, "value"));
        v = pointer(at.o);
    }
};
template <typename T> struct Levels {                // three levels as `levels`, `grads` or `paged_levels` returned them
    const T* v;
    explicit Levels(PyObject* o) : v(nullptr) {
        if (!PyBytes_Check(o) || PyBytes_GET_SIZE(o) != static_cast<Py_ssize_t>(3 * sizeof(T))) throw Bad{};
        v = reinterpret_cast<const T*>(PyBytes_AS_STRING(o));
    }
};
template <> struct Arg<const mka_level*> : Levels<mka_level> { using Levels::Levels; };
template <> struct Arg<const mka_level_grad*> : Levels<mka_level_grad> { using Levels::Levels; };
template <> struct Arg<const mka_paged_level*> : Levels<mka_paged_level> { using Levels::Levels; };
PyObject* shape_class = nullptr;                     // the binding's mka_shape: other buffers of its size are no shapes
PyObject* shape_type(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 1 || !PyType_Check(a[0])) {
        PyErr_SetString(PyExc_TypeError, "a class is expected");
        return nullptr;
    }
    Py_INCREF(a[0]);
    Py_XDECREF(shape_class);
    shape_class = a[0];
    Py_RETURN_NONE;
}
template <> struct Arg<const mka_shape*> {
    mka_shape copy;
    const mka_shape* v;
    explicit Arg(PyObject* o) : v(&copy) {
        if (!shape_class || !PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(shape_class))) {
            PyErr_SetString(PyExc_TypeError, "an mka_shape is expected");
            throw PyErrSet();
        }
        Py_buffer view;
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw PyErrSet();
        const bool fits = view.len == static_cast<Py_ssize_t>(sizeof(mka_shape));
        if (fits) memcpy(&copy, view.buf, sizeof(mka_shape));
        PyBuffer_Release(&view);
        if (!fits) {
            PyErr_SetString(PyExc_TypeError, "an mka_shape is expected");
            throw PyErrSet();
        }
    }
    Arg(const Arg&) = delete;
};

// The library's function at address a[0] (of the type of the declaration named) with the other arguments, the last of which is the stream; its
// status.  Other threads run meanwhile.
template <typename R, typename... P, size_t... I>
PyObject* invoke(R (*)(P...), PyObject* const* a, std::index_sequence<I...>) {
    const auto f = reinterpret_cast<R (*)(P...)>(Address(a[0]).v);
    if (!f) throw Bad{"the address of a function is expected"};
    const std::tuple<std::conditional_t<I + 1 == sizeof...(P), Address, Arg<P>>...> args{a[1 + I]...};
    R status;
    Py_BEGIN_ALLOW_THREADS
    status = f(std::get<I>(args).v...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLongLong(static_cast<long long>(status));
}
template <typename R, typename... P>
PyObject* call(R (*declared)(P...), PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != static_cast<Py_ssize_t>(1 + sizeof...(P))) throw Bad{kCountWanted};
        return invoke(declared, a, std::index_sequence_for<P...>());
    });
}
#define MKA_CALL(name) \
    PyObject* call_##name(PyObject*, PyObject* const* a, Py_ssize_t n) { return call(static_cast<decltype(&mka_##name)>(nullptr), a, n); }
MKA_CALL(router)
MKA_CALL(fwd_with_scratch)
MKA_CALL(fwd_paged_with_scratch)
MKA_CALL(decode)
MKA_CALL(decode_paged)
MKA_CALL(bwd)
#undef MKA_CALL

PyObject* empty_like(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 1) throw Bad{kCountWanted};
        return THPVariable_Wrap(at::empty_like(tensor(a[0])));
    });
}
PyObject* row_counts(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 1) throw Bad{kCountWanted};
        Seq K(a[0]);
        int64_t rows[3];
        for (int l = 0; l < 3; ++l) {
            const at::Tensor* k = K.tensor_at(l);
            rows[l] = k ? k->size(2) : 0;
        }
        return Py_BuildValue("LLL", static_cast<long long>(rows[0]), static_cast<long long>(rows[1]), static_cast<long long>(rows[2]));
    });
}

template <typename F> PyMethodDef method(const char* name, F f, const char* doc) {
    return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, doc};
}
PyMethodDef methods[] = {
    method("levels", levels, "levels(K, V) -> mka_level[3] as bytes; None or no rows: an absent level"),
    method("grads", grads, "grads(K, dK, dV) -> mka_level_grad[3] as bytes; a level absent from K is absent"),
    method("paged_levels", paged_levels, "paged_levels(pools_k, pools_v, tables, rows or None, n) -> mka_paged_level[3] as bytes"),
    method("paged_level", paged_level, "paged_level(pool_k, pool_v, table) -> one mka_paged_level over the table's width as bytes"),
    method("empties_like", empties_like, "empties_like(tensors) -> list of empty_like, None for None"),
    method("empty_f32", empty_f32, "empty_f32(t, keep, extra) -> fp32 tensor of t's first `keep` dimensions, then `extra` if not 0"),
    method("shape_type", shape_type, "shape_type(cls): the class whose instances are shapes"),
    method("empty_like", empty_like, "empty_like(t)"),
    method("row_counts", row_counts, "row_counts(K) -> the rows of three levels, 0 for None"),
    method("call_router", call_router, "call_router(address, arguments of mka_router...) -> its status"),
    method("call_fwd", call_fwd_with_scratch, "the same for mka_fwd_with_scratch"),
    method("call_fwd_paged", call_fwd_paged_with_scratch, "the same for mka_fwd_paged_with_scratch"),
    method("call_decode", call_decode, "the same for mka_decode"),
    method("call_decode_paged", call_decode_paged, "the same for mka_decode_paged"),
    method("call_bwd", call_bwd, "the same for mka_bwd"),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_args", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_args() { return PyModule_Create(&module); }
