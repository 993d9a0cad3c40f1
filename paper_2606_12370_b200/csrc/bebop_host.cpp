// Argument marshalling of the Python binding, in native code: tensors in, device pointers to the C ABI
// (include/bebop.h), tensors out.  Nothing is computed here.
//
// Small calls take 4 to 16 us on the device, so what the host does per call is part of their time.  In Python the
// thirty-odd tensor queries, the 23 converted arguments and the stream look-up took 15 us of a call's 23; here a whole call
// costs the host 2.8 us with given buffers, launch included.  The library's functions come as addresses (init), so that the library itself is loaded, and
// looked for, in one place.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/bebop.h"

namespace {

decltype(&bebop_verify) f_verify;
decltype(&bebop_tv) f_tv;
decltype(&bebop_tv_static) f_tv_static;
decltype(&bebop_greedy_verify) f_greedy;
decltype(&bebop_workspace_bytes) f_bytes;
PyObject *k_accept_len, *k_out_tokens, *k_tv, *k_p_draft, *k_q_draft, *k_row_status, *k_workspace, *k_s_aux;

// What goes wrong is a C++ exception here and becomes a Python one at the boundary: a status code (negative: found here,
// before the call) is returned as a number, for the binding to raise.
struct Code { long v; };
struct Bad { const char* what; };      // AssertionError
struct Raised {};                      // a Python error is set
struct Shape { const char* what; };    // ValueError
constexpr long kNotCuda = -8, kBadDtype = -3;

inline void need(bool ok, const char* what) { if (!ok) throw Bad{what}; }
inline const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "a tensor is expected"); throw Raised(); }
    return THPVariable_Unpack(o);
}
inline void need_rank(const at::Tensor& t, int64_t n, const char* what) { if (t.dim() != n) throw Shape{what}; }
inline bool given(PyObject* o) { return o != Py_None; }
inline bool truth(PyObject* o) {
    if (o == Py_True) return true;
    if (o == Py_False) return false;
    const int t = PyObject_IsTrue(o);
    if (t < 0) throw Raised();
    return t != 0;
}
inline float number(PyObject* o) {
    if (PyFloat_CheckExact(o)) return (float)PyFloat_AS_DOUBLE(o);
    PyObject* const f = PyNumber_Float(o);                  // what float() takes
    if (!f) throw Raised();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return (float)v;
}
inline bebop_dtype_t dtype_of(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return BEBOP_F32;
    if (t.scalar_type() == at::kBFloat16) return BEBOP_BF16;
    throw Code{kBadDtype};
}
// distance between consecutive rows of a [.., R, V] tensor whose rows are equally spaced
inline int64_t row_distance(const at::Tensor& t, int64_t ndim) {
    if (!t.is_cuda()) throw Code{kNotCuda};
    need(t.dim() == ndim && t.stride(-1) == 1, "vocabulary must be contiguous");
    const int64_t ld = t.stride(-2);
    if (ndim == 3 && t.size(0) > 1) need(t.stride(0) == t.size(1) * ld, "rows of the batch must be equally spaced");
    return ld;
}
inline void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// New outputs, on the inputs' device, each with a storage of its own, straight from the allocator.  (As pieces of one block they
// cost 0.45 us less apiece -- a greedy call of the smallest size 4.1 us instead of 5.0, bebop_verify without given buffers
// 4.9 instead of 7.6 -- but then a resize_() of one runs into the next, saving one saves all, and holding one holds all.
// Building the tensors by hand on the allocator's blocks is no faster than empty_cuda.)
struct Maker {
    at::Device dev;
    bool poison;                        // filled with a value no call leaves (tests)
    at::Tensor make(at::IntArrayRef shape, at::ScalarType type) const {       // (int32 or float32)
        if (poison) return at::full(shape, -77, at::TensorOptions().dtype(type).device(dev));
        return at::Tensor(at::detail::empty_cuda(shape, type, dev, c10::nullopt));
    }
};
// a result dictionary that owns what is put into it
struct Dict {
    PyObject* d = PyDict_New();
    Dict() { if (!d) throw Raised(); }
    ~Dict() { Py_XDECREF(d); }
    void put(PyObject* key, PyObject* value) {      // (steals value)
        if (!value) throw Raised();
        const int rc = PyDict_SetItem(d, key, value);
        Py_DECREF(value);
        if (rc < 0) throw Raised();
    }
    void put(PyObject* key, const at::Tensor& t) { put(key, THPVariable_Wrap(t)); }
    void none(PyObject* key) { Py_INCREF(Py_None); put(key, Py_None); }
    PyObject* release() { PyObject* r = d; d = nullptr; return r; }
};
// the caller's buffer for an output, a new one, or none
void* output(Dict& d, PyObject* out, PyObject* key, const Maker& m, at::IntArrayRef shape, at::ScalarType type, bool want) {
    if (given(out)) {
        PyObject* o = PyDict_GetItemWithError(out, key);
        if (!o && PyErr_Occurred()) throw Raised();
        if (o && given(o)) {
            void* p = tensor(o).data_ptr();
            Py_INCREF(o);
            d.put(key, o);
            return p;
        }
    }
    if (!want) { d.none(key); return nullptr; }
    const at::Tensor t = m.make(shape, type);
    d.put(key, t);
    return t.data_ptr();
}
struct Space { void* p; size_t bytes; at::Tensor made; };
Space workspace_of(PyObject* o, int B, int K, int V, bebop_dtype_t dt, at::Device dev) {
    Space s;
    if (given(o)) { const at::Tensor& t = tensor(o); s.p = t.data_ptr(); s.bytes = t.nbytes(); return s; }
    const int64_t need = (int64_t)f_bytes(B, K, V, dt);
    s.made = at::zeros({need < 256 ? 256 : need}, at::TensorOptions().dtype(at::kByte).device(dev));
    s.p = s.made.data_ptr(); s.bytes = s.made.nbytes();
    return s;
}
template <typename T> inline const T* ptr_or_null(PyObject* o) {
    return given(o) ? static_cast<const T*>(tensor(o).data_ptr()) : nullptr;
}
template <typename F> inline void call(F&& f) {
    bebop_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = f();
    Py_END_ALLOW_THREADS
    if (s != BEBOP_OK) throw Code{(long)s};
}
template <typename F> PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& f) {
    if (n != want) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    try { return f(); }
    catch (const Code& c) { return PyLong_FromLong(c.v); }
    catch (const Bad& b) { PyErr_SetString(PyExc_AssertionError, b.what); return nullptr; }
    catch (const Shape& b) { PyErr_SetString(PyExc_ValueError, b.what); return nullptr; }
    catch (const Raised&) { return nullptr; }
    catch (...) { torch::translate_exception_to_python(std::current_exception()); return nullptr; }      // torch's own types: OutOfMemoryError and the like
}

// target, draft, draft_tokens, u_accept, u_final, draft_len, temperature, temperature_all, out, workspace, want_tv,
// want_probs, want_status, poison
PyObject* py_verify(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 14, [&]() -> PyObject* {
        const at::Tensor& tg = tensor(a[0]);
        const at::Tensor& dr = tensor(a[1]);
        need_rank(tg, 3, "target_logits must be [B, K+1, V]");
        const int B = (int)tg.size(0), K = (int)tg.size(1) - 1, V = (int)tg.size(2);
        const bebop_dtype_t dt = dtype_of(tg);
        need(dr.scalar_type() == tg.scalar_type() && dr.dim() == 3 && dr.size(0) == B && dr.size(1) == K && dr.size(2) == V,
             "draft_logits must be [B, K, V] of the target's type");
        const int64_t ldt = row_distance(tg, 3), ldd = row_distance(dr, 3);
        const Maker m{tg.device(), truth(a[13])};
        const bool want_tv = truth(a[10]), want_probs = truth(a[11]), want_status = truth(a[12]);
        Dict d;
        int32_t* acc = (int32_t*)output(d, a[8], k_accept_len, m, {B}, at::kInt, true);
        int32_t* tok = (int32_t*)output(d, a[8], k_out_tokens, m, {B, K + 1}, at::kInt, true);
        float* tv = (float*)output(d, a[8], k_tv, m, {B, K}, at::kFloat, want_tv);
        float* pd = (float*)output(d, a[8], k_p_draft, m, {B, K}, at::kFloat, want_probs);
        float* qd = (float*)output(d, a[8], k_q_draft, m, {B, K}, at::kFloat, want_probs);
        int32_t* st = (int32_t*)output(d, a[8], k_row_status, m, {B}, at::kInt, want_status);
        const Space ws = workspace_of(a[9], B, K, V, dt, m.dev);
        for (int i = 2; i < 5; ++i) need(tensor(a[i]).is_cuda() && tensor(a[i]).is_contiguous(), "draft_tokens, u_accept and u_final must be contiguous CUDA tensors");
        need(tensor(a[2]).scalar_type() == at::kInt && tensor(a[3]).scalar_type() == at::kFloat && tensor(a[4]).scalar_type() == at::kFloat,
             "draft_tokens must be int32, u_accept and u_final float32");
        if (given(a[5])) need(tensor(a[5]).scalar_type() == at::kInt && tensor(a[5]).is_contiguous(), "draft_len must be contiguous int32");
        if (given(a[6])) need(tensor(a[6]).scalar_type() == at::kFloat && tensor(a[6]).is_contiguous(), "temperature must be contiguous float32");
        const float tau = number(a[7]);
        const int32_t* dt_tok = (const int32_t*)tensor(a[2]).data_ptr();
        const int32_t* dlen = ptr_or_null<int32_t>(a[5]);
        const float* temp = ptr_or_null<float>(a[6]);
        const float* ua = (const float*)tensor(a[3]).data_ptr();
        const float* uf = (const float*)tensor(a[4]).data_ptr();
        const void* tp = tg.data_ptr();
        const void* dp = dr.data_ptr();
        void* const s = stream();
        call([&] { return f_verify(tp, ldt, dp, ldd, dt_tok, dlen, temp, tau, ua, uf, B, K, V, dt, acc, tok, tv, pd, qd, st, ws.p, ws.bytes, s); });
        if (given(a[9])) { Py_INCREF(a[9]); d.put(k_workspace, a[9]); } else d.put(k_workspace, ws.made);
        return d.release();
    });
}

// target, draft, temperature, temperature_all, workspace, want_s_aux, want_status, poison, whether the built-in scratch takes the workspace's place
PyObject* py_tv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&]() -> PyObject* {
        const at::Tensor& tg = tensor(a[0]);
        const at::Tensor& dr = tensor(a[1]);
        need_rank(tg, 2, "target_logits must be [N, V]");
        const int N = (int)tg.size(0), V = (int)tg.size(1);
        const bebop_dtype_t dt = dtype_of(tg);
        need(dr.scalar_type() == tg.scalar_type() && dr.dim() == 2 && dr.size(0) == N && dr.size(1) == V, "draft_logits must be as target_logits");
        const int64_t ldt = row_distance(tg, 2), ldd = row_distance(dr, 2);
        const Maker m{tg.device(), truth(a[7])};
        Dict d;
        float* tv = (float*)output(d, Py_None, k_tv, m, {N}, at::kFloat, true);
        float* sx = (float*)output(d, Py_None, k_s_aux, m, {N}, at::kFloat, truth(a[5]));
        int32_t* st = (int32_t*)output(d, Py_None, k_row_status, m, {N}, at::kInt, truth(a[6]));
        const float tau = number(a[3]);
        const float* temp = ptr_or_null<float>(a[2]);
        const void* tp = tg.data_ptr();
        const void* dp = dr.data_ptr();
        void* const s = stream();
        if (truth(a[8])) {
            call([&] { return f_tv_static(tp, ldt, dp, ldd, temp, tau, N, V, dt, tv, sx, st, s); });
        } else {
            const Space ws = workspace_of(a[4], N, 1, V, dt, m.dev);
            call([&] { return f_tv(tp, ldt, dp, ldd, temp, tau, N, V, dt, tv, sx, st, ws.p, ws.bytes, s); });
        }
        return d.release();
    });
}

// target, draft_tokens, draft_len, workspace, poison
PyObject* py_greedy(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 5, [&]() -> PyObject* {
        const at::Tensor& tg = tensor(a[0]);
        need_rank(tg, 3, "target_logits must be [B, K+1, V]");
        const int B = (int)tg.size(0), K = (int)tg.size(1) - 1, V = (int)tg.size(2);
        const bebop_dtype_t dt = dtype_of(tg);
        const int64_t ldt = row_distance(tg, 3);
        const at::Tensor& tok = tensor(a[1]);
        need(tok.scalar_type() == at::kInt && tok.is_contiguous() && tok.is_cuda(), "draft_tokens must be contiguous int32 on the device");
        const Maker m{tg.device(), truth(a[4])};
        Dict d;
        int32_t* acc = (int32_t*)output(d, Py_None, k_accept_len, m, {B}, at::kInt, true);
        int32_t* out = (int32_t*)output(d, Py_None, k_out_tokens, m, {B, K + 1}, at::kInt, true);
        int32_t* st = (int32_t*)output(d, Py_None, k_row_status, m, {B}, at::kInt, true);
        const Space ws = workspace_of(a[3], B, K, V, dt, m.dev);
        const int32_t* tokp = (const int32_t*)tok.data_ptr();
        const int32_t* dlen = ptr_or_null<int32_t>(a[2]);
        const void* tp = tg.data_ptr();
        void* const s = stream();
        call([&] { return f_greedy(tp, ldt, tokp, dlen, B, K, V, dt, acc, out, st, ws.p, ws.bytes, s); });
        return d.release();
    });
}

// addresses of bebop_verify, bebop_tv, bebop_tv_static, bebop_greedy_verify, bebop_workspace_bytes
PyObject* py_init(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 5, [&]() -> PyObject* {
        void* p[5];
        for (int i = 0; i < 5; ++i) {
            p[i] = PyLong_AsVoidPtr(a[i]);
            if (!p[i] && PyErr_Occurred()) throw Raised();
        }
        f_verify = (decltype(f_verify))p[0]; f_tv = (decltype(f_tv))p[1]; f_tv_static = (decltype(f_tv_static))p[2];
        f_greedy = (decltype(f_greedy))p[3]; f_bytes = (decltype(f_bytes))p[4];
        Py_RETURN_NONE;
    });
}

#define FAST(f) (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"init", FAST(py_init)}, {"verify", FAST(py_verify)}, {"tv", FAST(py_tv)}, {"greedy_verify", FAST(py_greedy)},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_bebop_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__bebop_host(void) {
    struct { PyObject** k; const char* s; } const names[] = {
        {&k_accept_len, "accept_len"}, {&k_out_tokens, "out_tokens"}, {&k_tv, "tv"}, {&k_p_draft, "p_draft"}, {&k_q_draft, "q_draft"},
        {&k_row_status, "row_status"}, {&k_workspace, "workspace"}, {&k_s_aux, "s_aux"}};
    for (const auto& x : names) if (!(*x.k = PyUnicode_InternFromString(x.s))) return nullptr;
    return PyModule_Create(&module);
}
