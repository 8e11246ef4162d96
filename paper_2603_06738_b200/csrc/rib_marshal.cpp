// Argument marshalling of the binding's hot calls in native code: checks the tensors, allocates the results, calls the C ABI.
//
// What a call costs on the host is what bounds the smallest maps and the feature generator: their kernels take 5 to 20 us, the
// Python form of the checks, allocations and ctypes conversions 12 to 20 (one 64 x 64 map 15.7 -> 10.2 us per pass, both generator
// calls 40.0 -> 20.5).  Every function here returns None for anything it does not know to be plain (another type, shape, device, a
// tensor subclass or wrapper, an active dispatch or function mode, a number that is no int): the caller then takes the Python
// form of the same call, which raises what it always raised.  An int is the status of the C call, a tuple its results.
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>

#include <type_traits>

#include "../../include/rib_window_attn.h"

namespace {

// The tensor behind a plain torch.Tensor of the given type: dense CUDA memory of its own, contiguous; else null.
const at::Tensor* plain(PyObject* o, at::ScalarType type, int dim)
{
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || t.is_nested() || t.layout() != at::kStrided || !t.is_cuda() || t.scalar_type() != type || t.dim() != dim || !t.has_storage() || !t.is_contiguous()) return nullptr;
    const auto keys = t.key_set();
    if (keys.has_any(c10::DispatchKeySet({c10::DispatchKey::Python, c10::DispatchKey::FuncTorchBatched, c10::DispatchKey::FuncTorchGradWrapper,
                                          c10::DispatchKey::Functionalize, c10::DispatchKey::Conjugate, c10::DispatchKey::Negative, c10::DispatchKey::ZeroTensor}))) return nullptr;
    return &t;
}

// Is something between this thread's calls and the kernels of torch: a dispatch or function mode, a transform, a trace?  (Its own
// handlers may be in Python; what is there on every thread, and autocast, is not.)
bool modes_active()
{
    const c10::DispatchKeySet usual = c10::default_included_set | c10::autocast_dispatch_keyset;
    return c10::impl::TorchDispatchModeTLS::any_modes_set() || at::impl::PythonTorchFunctionTLS::stack_len() > 0 ||
           !(c10::impl::tls_local_dispatch_key_set().included_ - usual).empty();
}

bool get_int(PyObject* o, int* v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long long x = PyLong_AsLongLongAndOverflow(o, &overflow);
    if (overflow || x < -(1ll << 30) || x > (1ll << 30)) return false;
    *v = (int)x;
    return true;
}
void* address(PyObject* o) { return PyLong_AsVoidPtr(o); }

// the current stream, or the `cuda_stream` of the one given
bool get_stream(PyObject* o, void** s)
{
    if (o == Py_None) { *s = (void*)c10::cuda::getCurrentCUDAStream().stream(); return true; }
    PyObject* p = PyObject_GetAttrString(o, "cuda_stream");
    if (!p) { PyErr_Clear(); return false; }
    if (PyLong_Check(p)) *s = PyLong_AsVoidPtr(p);
    const bool ok = PyLong_Check(p) && !PyErr_Occurred();
    Py_DECREF(p);
    PyErr_Clear();
    return ok;
}

struct Image { const at::Tensor *q, *k, *v, *pq, *pk; int B, H, W, heads, d, r, n, window, shift; long long stride; };

// q, k, v of one shape [B, H, W, heads, d] and the tables [n, r] (tables: 1), [heads, n, r] (2) or either (3)
bool get_image(PyObject* const* a, int tables, PyObject* window, PyObject* shift, Image* m)
{
    m->q = plain(a[0], at::kBFloat16, 5); m->k = plain(a[1], at::kBFloat16, 5); m->v = plain(a[2], at::kBFloat16, 5);
    if (!m->q || !m->k || !m->v || m->k->sizes() != m->q->sizes() || m->v->sizes() != m->q->sizes()) return false;
    if (!get_int(window, &m->window) || !get_int(shift, &m->shift) || m->window < 1 || m->window > 32768) return false;
    const auto s = m->q->sizes();
    for (int i = 0; i < 5; ++i) if (s[i] > (1ll << 30)) return false;
    m->B = (int)s[0]; m->H = (int)s[1]; m->W = (int)s[2]; m->heads = (int)s[3]; m->d = (int)s[4];
    m->n = m->window * m->window;
    for (int dim = 2; dim <= 3; ++dim) {
        if (!(tables & (dim - 1))) continue;
        m->pq = plain(a[3], at::kBFloat16, dim); m->pk = plain(a[4], at::kBFloat16, dim);
        if (!m->pq || !m->pk) continue;
        if (m->pq->size(dim - 2) != m->n || m->pk->size(dim - 2) != m->n) return false;
        if (dim == 3 && (m->pq->size(0) != m->heads || m->pk->size(0) != m->heads)) return false;
        if (m->pq->size(dim - 1) > (1 << 20) || m->pq->size(dim - 1) != m->pk->size(dim - 1)) return false;
        m->r = (int)m->pq->size(dim - 1);
        m->stride = dim == 3 ? (long long)m->n * m->r : 0;
        return true;
    }
    return false;
}

// The types of the C calls, from their header: a signature that changes there does not compile here.
using Fwd = decltype(&rib_window_attn_fwd_headwise);
using Bwd = decltype(&rib_window_attn_bwd_headwise);
using GenFwd = decltype(&rib_generate_features);
using GenBwd = decltype(&rib_generate_features_bwd);
static_assert(std::is_same_v<Fwd, decltype(&rib_window_attn_fwd_padded)> && std::is_same_v<Fwd, decltype(&rib_window_attn_fwd_masked)>);
static_assert(std::is_same_v<Bwd, decltype(&rib_window_attn_bwd_padded)> && std::is_same_v<Bwd, decltype(&rib_window_attn_bwd_masked)>);

// The body of a call.  No C++ exception may leave through the C frames of the interpreter (a tensor of an unusual kind may throw
// wherever it is asked for its sizes or its memory): the Python form meets the same condition and raises it.
template <class Body>
PyObject* guarded(Body&& body) noexcept
{
    try {
        return body();
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// No lock of the interpreter while this lives, an exception or not.  The allocations are made without it, too, as torch.empty makes
// them: one that finds no cached memory waits for the device, and a host function on some stream may be waiting for the lock.
struct Unlocked {
    PyThreadState* const state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked&) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};

PyObject* status(int rc) { return PyLong_FromLong(rc); }

// the results of a call, None in the place of an undefined one
PyObject* results(std::initializer_list<at::Tensor*> tensors)
{
    PyObject* res = PyTuple_New((Py_ssize_t)tensors.size());
    if (!res) return nullptr;
    Py_ssize_t i = 0;
    for (at::Tensor* t : tensors) {
        PyObject* o = t->defined() ? THPVariable_Wrap(std::move(*t)) : Py_NewRef(Py_None);
        if (!o) { Py_DECREF(res); return nullptr; }
        PyTuple_SET_ITEM(res, i++, o);
    }
    return res;
}

// fwd(address, q, k, v, pq, pk, tables, window, shift, want_lse, stream)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t count)
{
    return guarded([&]() -> PyObject* {
        Image m;
        int tables = 0;
        void* stream;
        if (count != 11 || modes_active() || !get_int(a[6], &tables) || !get_image(a + 1, tables, a[7], a[8], &m) || !PyBool_Check(a[9]) || !get_stream(a[10], &stream)) Py_RETURN_NONE;
        const Fwd fn = reinterpret_cast<Fwd>(address(a[0]));
        const bool want_lse = a[9] == Py_True;
        at::Tensor out, lse;
        int rc;
        {
            const Unlocked unlocked;
            out = at::empty_like(*m.q);
            if (want_lse) lse = at::empty({m.B, m.heads, m.H, m.W}, m.q->options().dtype(at::kFloat));
            rc = fn(m.q->const_data_ptr(), m.k->const_data_ptr(), m.v->const_data_ptr(), m.pq->const_data_ptr(), m.pk->const_data_ptr(), m.stride, m.B, m.H, m.W, m.heads,
                    m.d, m.r, m.window, m.shift, out.mutable_data_ptr(), lse.defined() ? lse.mutable_data_ptr<float>() : nullptr, stream);
        }
        if (rc) return status(rc);
        return results({&out, &lse});
    });
}

// bwd(address, q, k, v, pq, pk, out, lse, dout, tables, window, shift, workspace, stream)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t count)
{
    return guarded([&]() -> PyObject* {
        Image m;
        int tables = 0;
        void* stream;
        if (count != 14 || modes_active() || !get_int(a[9], &tables) || !get_image(a + 1, tables, a[10], a[11], &m) || !get_stream(a[13], &stream)) Py_RETURN_NONE;
        const at::Tensor *out = plain(a[6], at::kBFloat16, 5), *lse = plain(a[7], at::kFloat, 4), *dout = plain(a[8], at::kBFloat16, 5);
        const at::Tensor* ws = plain(a[12], at::kByte, 1);
        if (!out || !lse || !dout || !ws || out->sizes() != m.q->sizes() || dout->sizes() != m.q->sizes() ||
            lse->size(0) != m.B || lse->size(1) != m.heads || lse->size(2) != m.H || lse->size(3) != m.W) Py_RETURN_NONE;
        const Bwd fn = reinterpret_cast<Bwd>(address(a[0]));
        const auto f32 = m.q->options().dtype(at::kFloat);
        at::Tensor dq, dk, dv, dpq, dpk;
        int rc;
        {
            const Unlocked unlocked;
            dq = at::empty_like(*m.q); dk = at::empty_like(*m.q); dv = at::empty_like(*m.q);
            dpq = at::empty(m.pq->sizes(), f32); dpk = at::empty(m.pq->sizes(), f32);
            rc = fn(m.q->const_data_ptr(), m.k->const_data_ptr(), m.v->const_data_ptr(), m.pq->const_data_ptr(), m.pk->const_data_ptr(), m.stride, out->const_data_ptr(),
                    lse->const_data_ptr<float>(), dout->const_data_ptr(), m.B, m.H, m.W, m.heads, m.d, m.r, m.window, m.shift, dq.mutable_data_ptr(), dk.mutable_data_ptr(),
                    dv.mutable_data_ptr(), dpq.mutable_data_ptr<float>(), dpk.mutable_data_ptr<float>(), ws->mutable_data_ptr(), (size_t)ws->numel(), stream);
        }
        if (rc) return status(rc);
        return results({&dq, &dk, &dv, &dpq, &dpk});
    });
}

struct Generator { const at::Tensor *w_h, *b_h, *w_pq, *w_pk; int window, L, dh, r; void* stream; };

bool get_generator(PyObject* const* w, PyObject* window, PyObject* stream, Generator* g)
{
    g->w_h = plain(w[0], at::kFloat, 2); g->b_h = plain(w[1], at::kFloat, 1); g->w_pq = plain(w[2], at::kFloat, 2); g->w_pk = plain(w[3], at::kFloat, 2);
    if (!g->w_h || !g->b_h || !g->w_pq || !g->w_pk || !get_int(window, &g->window) || g->window < 1 || g->window > 32768 || !get_stream(stream, &g->stream)) return false;
    const int64_t rows = g->w_h->size(0), dh = g->w_h->size(1), r = g->w_pq->size(1);
    if (rows < 2 || (rows - 2) % 4 || rows > 4096 || dh > 4096 || r > 4096 || g->b_h->size(0) != dh || g->w_pq->size(0) != dh || g->w_pk->size(0) != dh || g->w_pk->size(1) != r) return false;
    g->L = (int)((rows - 2) / 4); g->dh = (int)dh; g->r = (int)r;
    return true;
}

// generate(address, w_h, b_h, w_pq, w_pk, window, stream)
PyObject* generate(PyObject*, PyObject* const* a, Py_ssize_t count)
{
    return guarded([&]() -> PyObject* {
        Generator g;
        if (count != 7 || modes_active() || !get_generator(a + 1, a[5], a[6], &g)) Py_RETURN_NONE;
        const GenFwd fn = reinterpret_cast<GenFwd>(address(a[0]));
        const auto options = g.w_h->options().dtype(at::kBFloat16);
        at::Tensor pq, pk;
        int rc;
        {
            const Unlocked unlocked;
            pq = at::empty({g.window * g.window, g.r}, options); pk = at::empty({g.window * g.window, g.r}, options);
            rc = fn(g.w_h->const_data_ptr<float>(), g.b_h->const_data_ptr<float>(), g.w_pq->const_data_ptr<float>(), g.w_pk->const_data_ptr<float>(), g.window, g.L, g.dh, g.r,
                    pq.mutable_data_ptr(), pk.mutable_data_ptr(), g.stream);
        }
        if (rc) return status(rc);
        return results({&pq, &pk});
    });
}

// generate_bwd(address, w_h, b_h, w_pq, w_pk, dpq, dpk, window, stream)
PyObject* generate_bwd(PyObject*, PyObject* const* a, Py_ssize_t count)
{
    return guarded([&]() -> PyObject* {
        Generator g;
        if (count != 9 || modes_active() || !get_generator(a + 1, a[7], a[8], &g)) Py_RETURN_NONE;
        const at::Tensor *dpq = plain(a[5], at::kFloat, 2), *dpk = plain(a[6], at::kFloat, 2);
        const int64_t n = (int64_t)g.window * g.window;
        if (!dpq || !dpk || dpq->size(0) != n || dpk->size(0) != n || dpq->size(1) != g.r || dpk->size(1) != g.r) Py_RETURN_NONE;
        const GenBwd fn = reinterpret_cast<GenBwd>(address(a[0]));
        at::Tensor out[4];
        int rc;
        {
            const Unlocked unlocked;
            out[0] = at::empty_like(*g.w_h); out[1] = at::empty_like(*g.b_h); out[2] = at::empty_like(*g.w_pq); out[3] = at::empty_like(*g.w_pk);
            rc = fn(g.w_h->const_data_ptr<float>(), g.b_h->const_data_ptr<float>(), g.w_pq->const_data_ptr<float>(), g.w_pk->const_data_ptr<float>(),
                    dpq->const_data_ptr<float>(), dpk->const_data_ptr<float>(), g.window, g.L, g.dh, g.r, out[0].mutable_data_ptr<float>(), out[1].mutable_data_ptr<float>(),
                    out[2].mutable_data_ptr<float>(), out[3].mutable_data_ptr<float>(), g.stream);
        }
        if (rc) return status(rc);
        return results({&out[0], &out[1], &out[2], &out[3]});
    });
}

PyMethodDef methods[] = {
    {"fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(fwd)), METH_FASTCALL, nullptr},
    {"bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bwd)), METH_FASTCALL, nullptr},
    {"generate", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(generate)), METH_FASTCALL, nullptr},
    {"generate_bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(generate_bwd)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_rib_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rib_marshal()
{
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", RIB_BUILT_FOR) < 0) { Py_DECREF(m); return nullptr; }      // the binding compares it
    return m;
}
