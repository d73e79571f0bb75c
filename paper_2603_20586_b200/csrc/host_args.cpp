// Host side of the binding: the levels of a call as the array of 64-bit words that mka_level[3], mka_level_grad[3] and
// mka_paged_level[3] are, and the call's small outputs.  Asked for one by one from Python, the pointers, shapes and strides of the
// six tensors of a call took longer than a short decode takes on the GPU (6.3 us; 0.2 us here).
#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <torch/csrc/autograd/python_variable.h>

#include <Python.h>
#include <stdint.h>

#include <vector>

namespace {

struct Bad {};                                       // what an assertion of the binding would have refused
struct PyErrSet {};                                  // the Python error is set

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) throw Bad();
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
    if (k.dim() != 4 || k.stride(3) != 1 || v.strides() != k.strides()) throw Bad();
}
void check_pair(const at::Tensor& k, const at::Tensor& v) {
    check_layout(k, v);
    if (v.sizes() != k.sizes()) throw Bad();
}

template <typename F>
PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const Bad&) {
        PyErr_SetString(PyExc_AssertionError, "levels: tensors [batch, head, row, column] with dense columns, K and V alike; tables and row counts int32");
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
        if (n != 2) throw Bad();
        Seq K(a[0]), V(a[1]);
        int64_t w[18] = {};
        for (int l = 0; l < 3; ++l) {
            const at::Tensor* k = K.tensor_at(l);
            if (!k || k->size(2) == 0) continue;
            const at::Tensor* v = V.tensor_at(l);
            if (!v) throw Bad();
            check_pair(*k, *v);
            put_level(w + 6 * l, *k, *v);
        }
        return bytes(w);
    });
}
PyObject* grads(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 3) throw Bad();
        Seq K(a[0]), dK(a[1]), dV(a[2]);
        int64_t w[18] = {};
        for (int l = 0; l < 3; ++l) {
            const at::Tensor* k = K.tensor_at(l);
            if (!k || k->size(2) == 0) continue;
            const at::Tensor *dk = dK.tensor_at(l), *dv = dV.tensor_at(l);
            if (!dk || !dv) throw Bad();
            check_layout(*dk, *dv);
            put_level(w + 6 * l, *dk, *dv);
        }
        return bytes(w);
    });
}

PyObject* paged_levels(PyObject*, PyObject* const* a, Py_ssize_t n_args) {
    return guarded([&]() -> PyObject* {
        if (n_args != 5) throw Bad();
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
            if (!v || !tab) throw Bad();
            check_pair(*k, *v);
            // [B, pages]: one table per sequence; [B, H_kv, pages]: one per (sequence, KV head)
            if (tab->scalar_type() != at::kInt || (tab->dim() != 2 && tab->dim() != 3) || tab->stride(tab->dim() - 1) != 1) throw Bad();
            if (r && (r->scalar_type() != at::kInt || !r->is_contiguous())) throw Bad();
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
        if (n != 3) throw Bad();
        const at::Tensor &k = tensor(a[0]), &v = tensor(a[1]), &tab = tensor(a[2]);
        check_layout(k, v);
        if (tab.scalar_type() != at::kInt || tab.dim() != 2 || tab.stride(1) != 1) throw Bad();
        const int64_t w[12] = {address(k), address(v), address(tab), 0, tab.size(1) * k.size(2), tab.stride(0), 0, k.size(2),
                               k.stride(0), k.stride(1), k.stride(2), k.size(0)};
        return bytes(w);
    });
}

PyObject* empties_like(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        if (n != 1) throw Bad();
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
        if (n != 3) throw Bad();
        const at::Tensor& t = tensor(a[0]);
        const int64_t keep = integer(a[1]), extra = integer(a[2]);
        if (keep < 0 || keep > t.dim()) throw Bad();
        std::vector<int64_t> size(t.sizes().begin(), t.sizes().begin() + keep);
        if (extra) size.push_back(extra);
        return THPVariable_Wrap(at::empty(size, at::TensorOptions().device(t.device()).dtype(at::kFloat)));
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
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_args", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_args() { return PyModule_Create(&module); }
