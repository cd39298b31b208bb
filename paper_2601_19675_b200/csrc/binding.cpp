// Argument marshalling of the per-call entry points as a CPython extension: tensors and descriptors in, addresses and
// strides out, one call of the C ABI.  Through ctypes a forward cost 7.2 us of host time besides its launches (the
// conversion of every argument to an object and the stream lookup in Python), more than a small layer takes on the GPU;
// through here 0.35 us.
//
// The functions take positional arguments only, return the status code and raise AssertionError for what is no device
// tensor of the expected kind; keywords, defaults and allocation stay in lopro.py.  The C ABI's addresses come from
// there too (bind), so that both sides use the same copy of the library.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "lopro.h"
#include "lopro_block.h"
#include "lopro_vq.h"

namespace {

struct Api {
    decltype(&lopro_linear_fwd) linear_fwd;
    decltype(&lopro_linear_fwd_host) linear_fwd_host;
    decltype(&lopro_linear_fwd_noalloc) linear_fwd_noalloc;
    decltype(&lopro_linear_fwd_group) linear_fwd_group;
    decltype(&lopro_linear_fwd_experts) linear_fwd_experts;
    decltype(&lopro_vq_linear_fwd) vq_linear_fwd;
    decltype(&lopro_rotate) rotate;
    decltype(&lopro_block_add_rmsnorm) add_rmsnorm;
    decltype(&lopro_block_rope_append) rope_append;
    decltype(&lopro_block_attention_decode) attention_decode;
    decltype(&lopro_block_silu_mul) silu_mul;
} api;

constexpr Py_ssize_t kMaxList = 4096;  // layers of a group or experts of a call

struct Raised {};  // a Python exception is set

void require(bool ok, const char* what) {
    if (ok) return;
    PyErr_SetString(PyExc_AssertionError, what);
    throw Raised{};
}

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expects a torch tensor");
        throw Raised{};
    }
    return THPVariable_Unpack(o);
}
void* address(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
void* contiguous_device(PyObject* o, size_t item) {
    const at::Tensor& t = tensor(o);
    require(t.is_cuda() && t.is_contiguous() && t.element_size() == item, "expects a contiguous device tensor");
    return t.data_ptr();
}
long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
int32_t int32(PyObject* o) {
    const long long v = integer(o);
    if (v < INT32_MIN || v > INT32_MAX) {
        PyErr_SetString(PyExc_OverflowError, "a 32-bit integer is expected");
        throw Raised{};
    }
    return (int32_t)v;
}
double number(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised{};
    return v;
}

// Row-major activations: device tensor of 16-bit entries, rows may be strided.
const at::Tensor& activations(PyObject* o) {
    const at::Tensor& t = tensor(o);
    require(t.is_cuda() && t.dim() == 2 && t.element_size() == 2 && t.stride(1) == 1,
            "x: a two-dimensional device tensor of 16-bit entries with unit stride along a row");
    return t;
}
// Leading dimension of T rows: the stride means nothing for a single row.
int64_t leading(const at::Tensor& t, int64_t T, int64_t width) {
    const int64_t ld = t.stride(0);
    return T > 1 || ld > width ? ld : width;
}

// The memory of a ctypes structure.
template <typename T>
struct Struct {
    Py_buffer view;
    explicit Struct(PyObject* o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised{};
        if (view.len != (Py_ssize_t)sizeof(T)) {
            PyBuffer_Release(&view);
            PyErr_SetString(PyExc_TypeError, "not a descriptor of this library");
            throw Raised{};
        }
    }
    Struct(const Struct&) = delete;
    ~Struct() { PyBuffer_Release(&view); }
    const T* operator->() const { return static_cast<const T*>(view.buf); }
    const T* get() const { return static_cast<const T*>(view.buf); }
};

// A list or tuple for the length of a call.
struct Sequence {
    PyObject* fast;
    explicit Sequence(PyObject* o) : fast(PySequence_Fast(o, "expects a sequence")) {
        if (fast == nullptr) throw Raised{};
    }
    Sequence(const Sequence&) = delete;
    ~Sequence() { Py_DECREF(fast); }
    Py_ssize_t size() const { return PySequence_Fast_GET_SIZE(fast); }
    PyObject* operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Calls into the library with the interpreter lock released: a launch may wait for room in the driver's queue.  Nothing but
// the call runs in there: a tensor's address may be refused with an exception (a batched or a fake tensor has none), and
// whoever catches that needs the lock.
template <typename F, typename... Args>
PyObject* status_of(F* call, Args... args) {
    struct Unlocked {
        PyThreadState* state = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(state); }
    };
    lopro_status st;
    {
        Unlocked unlocked;
        st = call(args...);
    }
    return PyLong_FromLong((long)st);
}

template <typename F>
PyObject* guarded(F&& body) {
    try {
        return body();
    } catch (const Raised&) {
        return nullptr;
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

bool expects(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, got);
    return false;
}

// (desc, packed, x, out_dtype, workspace, y)
PyObject* linear_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 6)) return nullptr;
    return guarded([&] {
        Struct<lopro_desc> d(a[0]);
        const at::Tensor &x = activations(a[2]), &ws = tensor(a[4]), &y = tensor(a[5]);
        const int32_t T = (int32_t)x.size(0), out = int32(a[3]);
        const void* packed = address(a[1]);
        void* s = current_stream();
        return status_of(api.linear_fwd, d.get(), packed, (const uint16_t*)x.data_ptr(), leading(x, T, d->d_in),
                         y.data_ptr(), leading(y, T, d->d_out), out, T, ws.data_ptr(), (size_t)ws.numel(), s);
    });
}

// (desc, packed, x_host, out_dtype, workspace, y_host)
PyObject* linear_fwd_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 6)) return nullptr;
    return guarded([&] {
        Struct<lopro_desc> d(a[0]);
        const at::Tensor &x = tensor(a[2]), &ws = tensor(a[4]), &y = tensor(a[5]);
        require(!x.is_cuda() && !y.is_cuda() && x.is_contiguous() && y.is_contiguous(), "x_host, y_host: contiguous host tensors");
        const int32_t T = (int32_t)x.size(0), out = int32(a[3]);
        const void* packed = address(a[1]);
        void* s = current_stream();
        return status_of(api.linear_fwd_host, d.get(), packed, (const uint16_t*)x.data_ptr(), y.data_ptr(), out, T,
                         ws.data_ptr(), (size_t)ws.numel(), s);
    });
}

// (desc, packed, x, out_dtype, y)
PyObject* linear_fwd_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 5)) return nullptr;
    return guarded([&] {
        Struct<lopro_desc> d(a[0]);
        const at::Tensor &x = activations(a[2]), &y = tensor(a[4]);
        const int32_t T = (int32_t)x.size(0), out = int32(a[3]);
        const void* packed = address(a[1]);
        void* s = current_stream();
        return status_of(api.linear_fwd_noalloc, d.get(), packed, (const uint16_t*)x.data_ptr(), leading(x, T, d->d_in),
                         y.data_ptr(), leading(y, T, d->d_out), out, T, s);
    });
}

// (descs, packed, x, out_dtype, workspace, ys)
PyObject* linear_fwd_group(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 6)) return nullptr;
    return guarded([&] {
        Sequence descs(a[0]), packed(a[1]), ys(a[5]);
        const at::Tensor &x = activations(a[2]), &ws = tensor(a[4]);
        const int32_t T = (int32_t)x.size(0), out = int32(a[3]);
        const Py_ssize_t k = descs.size();
        require(k >= 1 && k <= kMaxList && packed.size() == k && ys.size() == k, "descs, packed and ys: one entry per layer");
        std::vector<lopro_desc> d((size_t)k);
        std::vector<const lopro_desc*> dp((size_t)k);
        std::vector<const void*> blobs((size_t)k);
        std::vector<void*> outs((size_t)k);
        std::vector<int64_t> ldy((size_t)k);
        for (Py_ssize_t i = 0; i < k; ++i) {
            d[i] = *Struct<lopro_desc>(descs[i]).operator->();
            dp[i] = &d[i];
            blobs[i] = address(packed[i]);
            const at::Tensor& y = tensor(ys[i]);
            outs[i] = y.data_ptr();
            ldy[i] = leading(y, T, d[i].d_out);
        }
        void* s = current_stream();
        return status_of(api.linear_fwd_group, (int32_t)k, dp.data(), blobs.data(), (const uint16_t*)x.data_ptr(),
                         leading(x, T, d[0].d_in), outs.data(), ldy.data(), out, T, ws.data_ptr(), (size_t)ws.numel(),
                         s);
    });
}

// (desc, blobs, row_offsets, x, out_dtype, workspace, y)
PyObject* linear_fwd_experts(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 7)) return nullptr;
    return guarded([&] {
        Struct<lopro_desc> d(a[0]);
        Sequence blobs(a[1]), rows(a[2]);
        const at::Tensor &x = tensor(a[3]), &ws = tensor(a[5]), &y = tensor(a[6]);
        const int32_t out = int32(a[4]);
        const Py_ssize_t k = blobs.size();
        require(k >= 1 && k <= kMaxList && rows.size() == k + 1, "row_offsets: one entry more than there are experts");
        std::vector<const void*> ptrs((size_t)k);
        std::vector<int32_t> offs((size_t)k + 1);
        for (Py_ssize_t i = 0; i < k; ++i) ptrs[i] = address(blobs[i]);
        for (Py_ssize_t i = 0; i <= k; ++i) offs[i] = int32(rows[i]);
        void* s = current_stream();
        return status_of(api.linear_fwd_experts, d.get(), (int32_t)k, ptrs.data(), offs.data(),
                         (const uint16_t*)x.data_ptr(), x.stride(0), y.data_ptr(), y.stride(0), out, ws.data_ptr(),
                         (size_t)ws.numel(), s);
    });
}

// (desc, packed, x, out_dtype, workspace, y)
PyObject* vq_linear_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 6)) return nullptr;
    return guarded([&] {
        Struct<lopro_vq_desc> d(a[0]);
        const at::Tensor &x = tensor(a[2]), &ws = tensor(a[4]), &y = tensor(a[5]);
        const int32_t T = (int32_t)x.size(0), out = int32(a[3]);
        const void* packed = address(a[1]);
        void* s = current_stream();
        return status_of(api.vq_linear_fwd, d.get(), packed, (const uint16_t*)x.data_ptr(), leading(x, T, d->d_in),
                         y.data_ptr(), leading(y, T, d->d_out), out, T, ws.data_ptr(), (size_t)ws.numel(), s);
    });
}

// (desc, perm, x, out)
PyObject* rotate(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 4)) return nullptr;
    return guarded([&] {
        Struct<lopro_desc> d(a[0]);
        const at::Tensor &x = activations(a[2]), &out = tensor(a[3]);
        const int32_t T = (int32_t)x.size(0);
        const void* perm = address(a[1]);
        void* s = current_stream();
        return status_of(api.rotate, d.get(), (const int32_t*)perm, (const uint16_t*)x.data_ptr(), leading(x, T, d->d_in),
                         (uint16_t*)out.data_ptr(), leading(out, T, d->d_in), T, s);
    });
}

// (h, y or None, w, eps, out)
PyObject* block_add_rmsnorm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 5)) return nullptr;
    return guarded([&] {
        const at::Tensor &h = tensor(a[0]), &out = tensor(a[4]);
        require(h.dim() == 2, "h: two dimensions");
        const at::Tensor* y = a[1] == Py_None ? nullptr : &tensor(a[1]);
        const void* w = contiguous_device(a[2], 2);
        const float eps = (float)number(a[3]);
        void* s = current_stream();
        return status_of(api.add_rmsnorm, (uint16_t*)h.data_ptr(), h.stride(0),
                         y ? (const uint16_t*)y->data_ptr() : nullptr, y ? y->stride(0) : 0, (const uint16_t*)w, eps,
                         (uint16_t*)out.data_ptr(), out.stride(0), (int32_t)h.size(0), (int32_t)h.size(1), s);
    });
}

// (q, k, v, pos, k_cache, v_cache, theta, status)
PyObject* block_rope_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 8)) return nullptr;
    return guarded([&] {
        const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &kc = tensor(a[4]);
        require(kc.dim() == 4, "k_cache: four dimensions");
        const void* pos = contiguous_device(a[3], 4);
        void *kp = contiguous_device(a[4], 2), *vp = contiguous_device(a[5], 2), *status = address(a[7]);
        const float theta = (float)number(a[6]);
        void* s = current_stream();
        return status_of(api.rope_append, (uint16_t*)q.data_ptr(), q.stride(0), (const uint16_t*)k.data_ptr(),
                         k.stride(0), (const uint16_t*)v.data_ptr(), v.stride(0), (const int32_t*)pos, (uint16_t*)kp,
                         (uint16_t*)vp, (int32_t)kc.size(0), (int32_t)kc.size(1), (int32_t)kc.size(3),
                         (int32_t)kc.size(2), theta, status, s);
    });
}

// (q, k_cache, v_cache, ctx, scale, workspace, status, out)
PyObject* block_attention_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 8)) return nullptr;
    return guarded([&] {
        const at::Tensor &q = tensor(a[0]), &kc = tensor(a[1]), &ws = tensor(a[5]), &out = tensor(a[7]);
        require(kc.dim() == 4, "k_cache: four dimensions");
        const void *kp = contiguous_device(a[1], 2), *vp = contiguous_device(a[2], 2), *ctx = contiguous_device(a[3], 4);
        void* status = address(a[6]);
        const float scale = (float)number(a[4]);
        void* s = current_stream();
        return status_of(api.attention_decode, (const uint16_t*)q.data_ptr(), q.stride(0), (const uint16_t*)kp,
                         (const uint16_t*)vp, (const int32_t*)ctx, (uint16_t*)out.data_ptr(), out.stride(0),
                         (int32_t)kc.size(0), (int32_t)kc.size(1), (int32_t)kc.size(3), (int32_t)kc.size(2), scale,
                         ws.data_ptr(), (size_t)ws.numel(), status, s);
    });
}

// (gate, up, out)
PyObject* block_silu_mul(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expects(n, 3)) return nullptr;
    return guarded([&] {
        const at::Tensor &g = tensor(a[0]), &u = tensor(a[1]), &out = tensor(a[2]);
        require(g.dim() == 2, "gate: two dimensions");
        void* s = current_stream();
        return status_of(api.silu_mul, (const uint16_t*)g.data_ptr(), g.stride(0), (const uint16_t*)u.data_ptr(),
                         u.stride(0), (uint16_t*)out.data_ptr(), out.stride(0), (int32_t)g.size(0),
                         (int32_t)g.size(1), s);
    });
}

// bind({symbol: address}): the C ABI entry points of the loaded library
PyObject* bind(PyObject*, PyObject* table) {
    struct Entry {
        const char* name;
        void** slot;
    };
    const Entry entries[] = {
        {"lopro_linear_fwd", (void**)&api.linear_fwd},
        {"lopro_linear_fwd_host", (void**)&api.linear_fwd_host},
        {"lopro_linear_fwd_noalloc", (void**)&api.linear_fwd_noalloc},
        {"lopro_linear_fwd_group", (void**)&api.linear_fwd_group},
        {"lopro_linear_fwd_experts", (void**)&api.linear_fwd_experts},
        {"lopro_vq_linear_fwd", (void**)&api.vq_linear_fwd},
        {"lopro_rotate", (void**)&api.rotate},
        {"lopro_block_add_rmsnorm", (void**)&api.add_rmsnorm},
        {"lopro_block_rope_append", (void**)&api.rope_append},
        {"lopro_block_attention_decode", (void**)&api.attention_decode},
        {"lopro_block_silu_mul", (void**)&api.silu_mul},
    };
    for (const Entry& e : entries) {
        PyObject* v = PyDict_GetItemString(table, e.name);
        if (v == nullptr) {
            PyErr_SetString(PyExc_KeyError, e.name);
            return nullptr;
        }
        void* p = PyLong_AsVoidPtr(v);
        if (p == nullptr) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, e.name);
            return nullptr;
        }
        *e.slot = p;
    }
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST(linear_fwd), FAST(linear_fwd_host), FAST(linear_fwd_noalloc), FAST(linear_fwd_group), FAST(linear_fwd_experts),
    FAST(vq_linear_fwd), FAST(rotate), FAST(block_add_rmsnorm), FAST(block_rope_append), FAST(block_attention_decode),
    FAST(block_silu_mul), {"bind", bind, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
