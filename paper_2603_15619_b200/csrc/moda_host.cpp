// Host path of the calls that a program makes once per layer or token, as a CPython extension: arguments, output tensors, the
// C entry points of libmoda_b200.so, and the autograd node of moda_attention.
//
// It serves the plain case alone: torch.Tensor (or Parameter) objects on the device, contiguous, of the documented types and
// sizes, on the current stream, with no mode, transform or tracer active.  For anything else a function returns None and the
// caller goes on with its own code (binding.py, autograd.py), which has the same checks and says what is wrong.  A call through here
// makes the same C call with the same arguments.
//
// Why: at the sizes of a decode step or of a small layer the device waits for the host.  Microseconds a call in a loop, through
// Python and ctypes -> through here: decode of one sequence over 8192 keys 15.9 -> 12.3 (10 on the device); T = 256, 2 heads, l = 4:
// forward 12.7 -> 8.5, backward 31.3 -> 20.5, moda_attention and its gradients 137 -> 86 (what is left is the engine's hand-over
// to its device thread and back).
#include <Python.h>
#include <dlfcn.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/cuda/CUDAContext.h>
#include <c10/core/DispatchKeySet.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/PyInterpreter.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <climits>
#include <initializer_list>

#include "../../include/moda.h"

namespace {

using at::Tensor;

// ---- the library: addresses from the handle that the binding has opened -----------------------------------------------
#define MODA_HOST_CALLS(X)                                                                                              \
    X(moda_attn_fwd_gqa) X(moda_attn_fwd_append) X(moda_attn_bwd_gqa) X(moda_attn_bwd_gqa_stages) X(moda_attn_bwd_gqa_slot) \
    X(moda_bwd_workspace_bytes_gqa) X(moda_depth_cache_bytes) X(moda_attn_decode) X(moda_attn_decode_varlen)            \
    X(moda_attn_decode_paged) X(moda_decode_workspace_bytes)
struct Library {
#define X(name) decltype(&::name) name = nullptr;
    MODA_HOST_CALLS(X)
#undef X
} lib;
PyObject* check_fn = nullptr;                                  // binding._check: raises ModaError

[[noreturn]] void fail(int rc, const char* what) {
    PyGILState_STATE gil = PyGILState_Ensure();
    PyObject* r = PyObject_CallFunction(check_fn, "is", rc, what);
    Py_XDECREF(r);
    if (r != nullptr) PyErr_Format(PyExc_RuntimeError, "%s failed: [%d]", what, rc);
    python_error e;
    e.persist();
    PyGILState_Release(gil);
    throw e;
}

struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};

// ---- what counts as plain --------------------------------------------------------------------------------------------
// Keys of an ordinary CUDA tensor; wrappers, views that conjugate or negate, fake and batched tensors carry others.
uint64_t plain_keys() {
    static const uint64_t keys = (c10::DispatchKeySet(c10::DispatchKey::CUDA) |
                                  c10::getAutogradRelatedKeySetFromBackend(c10::BackendComponent::CUDABit) |
                                  c10::getAutocastRelatedKeySetFromBackend(c10::BackendComponent::CUDABit) |
                                  c10::DispatchKeySet(c10::DispatchKey::ADInplaceOrView)).raw_repr();
    return keys;
}
// A torch-function mode sees the torch calls of the Python form.  Not so the one of a default device (torch.set_default_device): it
// fills in a device where none is given, and these calls give one.
PyObject* device_mode = nullptr;                               // torch.utils._device.DeviceContext
bool function_mode() {
    using TLS = at::impl::PythonTorchFunctionTLS;
    if (!at::impl::torch_function_mode_enabled()) return false;
    for (int64_t i = 0; i < TLS::stack_len(); ++i)
        if (reinterpret_cast<PyObject*>(Py_TYPE(TLS::get_stack_at(i)->ptr(getPyInterpreter()))) != device_mode) return true;
    return false;
}
// No mode, functorch transform, functionalisation or tracer: but for torch-function modes their keys would be in the thread's included set.
bool plain_thread() {
    if (function_mode()) return false;
    static const uint64_t keys = (c10::DispatchKeySet(c10::DispatchKey::BackendSelect) | c10::DispatchKeySet(c10::DispatchKey::ADInplaceOrView)).raw_repr();
    return (c10::impl::tls_local_dispatch_key_set().included_.raw_repr() & ~keys) == 0;
}
const Tensor* plain(PyObject* o) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || (t.key_set().raw_repr() & ~plain_keys()) != 0) return nullptr;
    return &t;
}
const Tensor* dense(PyObject* o, at::ScalarType type, int64_t dim) {
    const Tensor* t = plain(o);
    return t != nullptr && t->scalar_type() == type && t->dim() == dim && t->is_contiguous() ? t : nullptr;
}
// An argument that may be None: a null tensor, or a contiguous one.  False: neither.
bool optional_dense(PyObject* o, const Tensor*& t) {
    t = nullptr;
    if (o == Py_None) return true;
    t = plain(o);
    return t != nullptr && t->is_contiguous();
}
bool shape_is(const Tensor& t, std::initializer_list<int64_t> want) { return t.sizes() == at::IntArrayRef(want); }
bool int_arg(PyObject* o, int& v) {
    if (!PyLong_CheckExact(o)) return false;
    int over = 0;
    const long x = PyLong_AsLongAndOverflow(o, &over);
    if (over != 0 || x < INT_MIN || x > INT_MAX) return false;
    v = int(x);
    return true;
}
bool float_arg(PyObject* o, float& v) {
    if (!PyFloat_CheckExact(o)) return false;
    v = float(PyFloat_AS_DOUBLE(o));
    return true;
}
bool small(const Tensor& t) {                                   // every extent fits the int of the C calls
    for (int64_t n : t.sizes())
        if (n > INT_MAX) return false;
    return true;
}

void* ptr(const Tensor* t) { return t != nullptr ? t->data_ptr() : nullptr; }
void* stream() { return at::cuda::getCurrentCUDAStream().stream(); }
size_t bytes_of(const Tensor& t) { return size_t(t.numel()) * t.element_size(); }
Tensor like(const Tensor& t) { return at::empty(t.sizes(), t.options().requires_grad(false)); }
Tensor fresh(std::initializer_list<int64_t> shape, at::ScalarType type, const Tensor& on) {
    return at::empty(at::IntArrayRef(shape), on.options().dtype(type).requires_grad(false));
}
// A tensor that a kernel reads or writes n elements of, where it is given.
bool holds(const Tensor* t, at::ScalarType type, int64_t n) { return t == nullptr || (t->scalar_type() == type && t->numel() >= n); }
// A given tensor's own object, or the new tensor.
PyObject* out(PyObject* given, const Tensor& made) { return given != Py_None ? Py_NewRef(given) : THPVariable_Wrap(made); }
PyObject* none() { Py_RETURN_NONE; }

// ---- attention: shapes, forward, backward ----------------------------------------------------------------------------
struct Shape { int B, T, H, Hk, d; };
bool shapes(const Tensor& Q, const Tensor& K, const Tensor& V, Shape& s) {
    if (Q.dim() != 4 || K.dim() != 4 || Q.scalar_type() != at::kBFloat16 || K.scalar_type() != at::kBFloat16 || V.scalar_type() != at::kBFloat16) return false;
    if (!small(Q) || !small(K)) return false;
    s = {int(Q.size(0)), int(Q.size(1)), int(Q.size(2)), int(K.size(2)), int(Q.size(3))};
    return K.size(0) == s.B && K.size(1) == s.T && K.size(3) == s.d && V.sizes() == K.sizes();
}
// Whether a depth cache, or its gradient, has n slots (a number that no cache has is the C call's to refuse).
bool holds_slots(const Tensor* t, const Shape& s, int n) { return t == nullptr || bytes_of(*t) >= lib.moda_depth_cache_bytes(s.B, s.T, s.Hk, s.d, n); }
bool holds_slot(const Tensor* t, const Shape& s, int slot) { return holds_slots(t, s, std::min(slot, MODA_MAX_DEPTH) + 1); }
int64_t rows(const Shape& s) { return int64_t(s.B) * s.H * s.T; }
void forward(const Shape& s, const Tensor& Q, const Tensor& K, const Tensor& V, const Tensor* depth, int l, float scale,
             const Tensor* cache, int slot, Tensor& O, Tensor& LSE) {
    if (!O.defined()) O = like(Q);
    if (!LSE.defined()) LSE = fresh({s.B, s.H, s.T}, at::kFloat, Q);
    const int rc = cache == nullptr
        ? lib.moda_attn_fwd_gqa(Q.data_ptr(), K.data_ptr(), V.data_ptr(), l > 0 ? ptr(depth) : nullptr, s.B, s.T, s.H, s.Hk, s.d, l, scale,
                                O.data_ptr(), static_cast<float*>(LSE.data_ptr()), stream())
        : lib.moda_attn_fwd_append(Q.data_ptr(), K.data_ptr(), V.data_ptr(), l > 0 ? ptr(depth) : nullptr, s.B, s.T, s.H, s.Hk, s.d, l, scale,
                                   O.data_ptr(), static_cast<float*>(LSE.data_ptr()), cache->data_ptr(), slot, stream());
    if (rc != 0) fail(rc, cache == nullptr ? "moda_attn_fwd_gqa" : "moda_attn_fwd_append");
}
// mode: moda_attn_bwd_gqa, the call with a mask, or the call with a slot
enum Mode { kWhole, kMask, kSlot };
void backward(const Shape& s, const Tensor& Q, const Tensor& K, const Tensor& V, const Tensor* depth, const Tensor& O, const Tensor& dO,
              const Tensor& LSE, int l, float scale, Mode mode, int arg, Tensor& dQ, Tensor& dK, Tensor& dV, Tensor& dcache, Tensor& ws) {
    if (!dQ.defined()) dQ = like(Q);
    if (!dK.defined()) dK = like(K);
    if (!dV.defined()) dV = like(V);
    if (l > 0 && !dcache.defined()) {
        dcache = fresh({int64_t(lib.moda_depth_cache_bytes(s.B, s.T, s.Hk, s.d, l) / 2)}, at::kBFloat16, Q);
    }
    if (!ws.defined()) ws = fresh({int64_t(lib.moda_bwd_workspace_bytes_gqa(s.B, s.T, s.H, s.Hk, s.d, l))}, at::kByte, Q);
    const void* dep = l > 0 ? ptr(depth) : nullptr;
    void* dc = l > 0 ? dcache.data_ptr() : nullptr;
    const float* lse = static_cast<const float*>(LSE.data_ptr());
    if (mode == kSlot) {
        const int rc = lib.moda_attn_bwd_gqa_slot(Q.data_ptr(), K.data_ptr(), V.data_ptr(), dep, O.data_ptr(), dO.data_ptr(), lse, s.B, s.T, s.H, s.Hk, s.d, l,
                                                  scale, dQ.data_ptr(), dK.data_ptr(), dV.data_ptr(), dcache.data_ptr(), ws.data_ptr(), bytes_of(ws), arg, stream());
        if (rc != 0) fail(rc, "moda_attn_bwd_gqa_slot");
        return;
    }
    const int rc = mode == kWhole
        ? lib.moda_attn_bwd_gqa(Q.data_ptr(), K.data_ptr(), V.data_ptr(), dep, O.data_ptr(), dO.data_ptr(), lse, s.B, s.T, s.H, s.Hk, s.d, l,
                                scale, dQ.data_ptr(), dK.data_ptr(), dV.data_ptr(), dc, ws.data_ptr(), bytes_of(ws), stream())
        : lib.moda_attn_bwd_gqa_stages(Q.data_ptr(), K.data_ptr(), V.data_ptr(), dep, O.data_ptr(), dO.data_ptr(), lse, s.B, s.T, s.H, s.Hk,
                                       s.d, l, scale, dQ.data_ptr(), dK.data_ptr(), dV.data_ptr(), dc, ws.data_ptr(), bytes_of(ws), arg,
                                       stream());
    if (rc != 0) fail(rc, mode == kWhole ? "moda_attn_bwd_gqa" : "moda_attn_bwd_gqa_stages");
}

// attn_fwd(Q, K, V, depth, l, scale, cache, slot, O, LSE) -> (O, LSE)
PyObject* attn_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    int l, slot = 0;
    float scale;
    if (n != 10 || !plain_thread() || !int_arg(a[4], l) || l < 0 || !float_arg(a[5], scale) || !int_arg(a[7], slot)) return none();
    const Tensor *Q = dense(a[0], at::kBFloat16, 4), *K = dense(a[1], at::kBFloat16, 4), *V = dense(a[2], at::kBFloat16, 4);
    const Tensor *depth, *cache, *O, *LSE;
    Shape s;
    if (Q == nullptr || K == nullptr || V == nullptr || !shapes(*Q, *K, *V, s) || !optional_dense(a[3], depth) || !optional_dense(a[6], cache) ||
        !optional_dense(a[8], O) || !optional_dense(a[9], LSE)) return none();
    if (!holds(O, at::kBFloat16, Q->numel()) || !holds(LSE, at::kFloat, rows(s)) || (l > 0 && !holds_slots(depth, s, l)) || !holds_slot(cache, s, slot)) return none();
    Tensor o = O != nullptr ? *O : Tensor(), lse = LSE != nullptr ? *LSE : Tensor();
    {
        NoGil nogil;
        forward(s, *Q, *K, *V, depth, l, scale, cache, slot, o, lse);
    }
    return Py_BuildValue("NN", out(a[8], o), out(a[9], lse));
    END_HANDLE_TH_ERRORS
}

// attn_bwd(Q, K, V, depth, O, dO, LSE, l, scale, dQ, dK, dV, dcache, workspace, stages or None) -> (dQ, dK, dV, dcache); with one argument more: the one before it is a slot
PyObject* attn_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    int l, arg = -1;
    float scale;
    if (n < 15 || n > 16 || !plain_thread() || !int_arg(a[7], l) || l < 0 || !float_arg(a[8], scale)) return none();
    if (a[14] != Py_None && (!int_arg(a[14], arg) || arg < 0)) return none();
    const Mode mode = n == 16 ? kSlot : a[14] == Py_None ? kWhole : kMask;
    if (mode == kSlot && (a[12] == Py_None || a[14] == Py_None)) return none();
    const Tensor *Q = dense(a[0], at::kBFloat16, 4), *K = dense(a[1], at::kBFloat16, 4), *V = dense(a[2], at::kBFloat16, 4);
    const Tensor *depth, *O, *dO, *LSE, *g[5];
    Shape s;
    if (Q == nullptr || K == nullptr || V == nullptr || !shapes(*Q, *K, *V, s) || !optional_dense(a[3], depth)) return none();
    if (!optional_dense(a[4], O) || !optional_dense(a[5], dO) || !optional_dense(a[6], LSE) || O == nullptr || dO == nullptr || LSE == nullptr) return none();
    for (int i = 0; i < 5; ++i)
        if (!optional_dense(a[9 + i], g[i])) return none();
    const int64_t nq = Q->numel(), nk = K->numel();
    if (!holds(O, at::kBFloat16, nq) || !holds(dO, at::kBFloat16, nq) || !holds(LSE, at::kFloat, rows(s)) || !holds(g[0], at::kBFloat16, nq) ||
        !holds(g[1], at::kBFloat16, nk) || !holds(g[2], at::kBFloat16, nk)) return none();
    if ((l > 0 && (!holds_slots(depth, s, l) || !holds_slots(g[3], s, l))) || (mode == kSlot && !holds_slot(g[3], s, arg))) return none();
    // no gradient cache can be made for this width or so many slots: the Python form says so
    if (l > 0 && g[3] == nullptr && lib.moda_depth_cache_bytes(s.B, s.T, s.Hk, s.d, l) == 0) return none();
    Tensor t[5];
    for (int i = 0; i < 5; ++i)
        if (g[i] != nullptr) t[i] = *g[i];
    {
        NoGil nogil;
        backward(s, *Q, *K, *V, depth, *O, *dO, *LSE, l, scale, mode, arg, t[0], t[1], t[2], t[3], t[4]);
    }
    return Py_BuildValue("NNNN", out(a[9], t[0]), out(a[10], t[1]), out(a[11], t[2]), t[3].defined() ? out(a[12], t[3]) : none());
    END_HANDLE_TH_ERRORS
}

// ---- the differentiable call ------------------------------------------------------------------------------------------
constexpr const char* kBadShapes = "K and V must be bf16 [B, T, H_kv, d] tensors matching Q's B, T and d";
void addressable(const Tensor& t) {
    TORCH_CHECK_VALUE(t.defined() && t.is_cuda(), "device (CUDA) tensors required");
    TORCH_CHECK_VALUE(t.is_contiguous(), "contiguous tensors required");
}
struct Attention : torch::autograd::Function<Attention> {
    static torch::autograd::variable_list forward(torch::autograd::AutogradContext* ctx, const Tensor& Q_, const Tensor& K_, const Tensor& V_,
                                                  const std::optional<Tensor>& depth_, int64_t l, double scale) {
        const Tensor Q = Q_.contiguous(), K = K_.contiguous(), V = V_.contiguous(), depth = l > 0 ? *depth_ : Tensor();
        Shape s;
        TORCH_CHECK_VALUE(shapes(Q, K, V, s), kBadShapes);
        Tensor O, LSE;
        ::forward(s, Q, K, V, l > 0 ? &depth : nullptr, int(l), float(scale), nullptr, 0, O, LSE);
        ctx->save_for_backward({Q, K, V, depth, O, LSE});
        ctx->saved_data["l"] = l;
        ctx->saved_data["scale"] = scale;
        if (l > 0) ctx->saved_data["type"] = int64_t(depth.scalar_type());
        ctx->mark_non_differentiable({LSE});
        ctx->set_materialize_grads(false);                     // nothing to fill for LSE
        return {O, LSE};
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, const torch::autograd::variable_list& grads) {
        const auto saved = ctx->get_saved_variables();
        const Tensor &Q = saved[0], &K = saved[1], &V = saved[2], &depth = saved[3], &O = saved[4], &LSE = saved[5];
        const int l = int(ctx->saved_data["l"].toInt());
        const float scale = float(ctx->saved_data["scale"].toDouble());
        const Tensor dO = grads[0].defined() ? grads[0].contiguous() : at::zeros_like(O);
        // Saved-tensor hooks may hand back anything, and torch does not look at it: every tensor again, before a kernel gets its address.
        Shape s;
        for (const Tensor* t : {&Q, &K, &V, &O, &LSE, &dO}) addressable(*t);
        TORCH_CHECK_VALUE(shapes(Q, K, V, s), kBadShapes);
        TORCH_CHECK_VALUE(holds(&O, at::kBFloat16, Q.numel()) && holds(&dO, at::kBFloat16, Q.numel()),
                          "O and its gradient must be bf16 tensors of Q's size");
        TORCH_CHECK_VALUE(holds(&LSE, at::kFloat, rows(s)), "LSE must be an fp32 tensor of B H T elements");
        if (l > 0) {
            addressable(depth);
            TORCH_CHECK_VALUE(int64_t(depth.scalar_type()) == ctx->saved_data["type"].toInt(), "depth_kv has changed its type");
            TORCH_CHECK_VALUE(holds_slots(&depth, s, l), "depth_kv holds fewer than l slots");
        }
        Tensor dQ, dK, dV, dcache, ws;
        if (l > 0) {
            // the kernels write every element of slots < l; later slots of the caller's cache get no gradient
            dcache = at::empty_like(depth);
            const int64_t slots = int64_t(lib.moda_depth_cache_bytes(s.B, s.T, s.Hk, s.d, l) / 2);
            if (slots < depth.numel()) dcache.view({-1}).slice(0, slots).zero_();
        }
        ::backward(s, Q, K, V, l > 0 ? &depth : nullptr, O, dO, LSE, l, scale, kWhole, 0, dQ, dK, dV, dcache, ws);
        return {dQ, dK, dV, dcache, Tensor(), Tensor()};
    }
};

bool dual(const Tensor& t) { return t._fw_grad(0).defined(); }

// attention(Q, K, V, depth or None, l, scale) -> (O, LSE)
PyObject* attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    int l;
    float scale;
    if (n != 6 || !plain_thread() || !int_arg(a[4], l) || l < 0 || !float_arg(a[5], scale)) return none();
    const Tensor *Q = plain(a[0]), *K = plain(a[1]), *V = plain(a[2]), *depth;
    Shape s;
    if (Q == nullptr || K == nullptr || V == nullptr || !shapes(*Q, *K, *V, s) || !optional_dense(a[3], depth) || (l > 0 && (depth == nullptr || !holds_slots(depth, s, l)))) return none();
    if (dual(*Q) || dual(*K) || dual(*V) || (depth != nullptr && dual(*depth))) return none();
    const Tensor q = *Q, k = *K, v = *V;
    const std::optional<Tensor> dep = depth != nullptr ? std::optional<Tensor>(*depth) : std::nullopt;
    torch::autograd::variable_list r;
    {
        NoGil nogil;
        r = Attention::apply(q, k, v, dep, int64_t(l), PyFloat_AS_DOUBLE(a[5]));
    }
    return Py_BuildValue("NN", THPVariable_Wrap(r[0]), THPVariable_Wrap(r[1]));
    END_HANDLE_TH_ERRORS
}

// ---- decode steps -----------------------------------------------------------------------------------------------------
// decode(q, K, V, table or None, seq_lens or None, depth, T_kv, l, scale, O, LSE, workspace) -> (O, LSE): one length for all
// sequences, a length for each, or pages
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    int T_kv, l;
    float scale;
    if (n != 12 || !plain_thread() || !int_arg(a[6], T_kv) || !int_arg(a[7], l) || l < 0 || !float_arg(a[8], scale)) return none();
    const Tensor *q = dense(a[0], at::kBFloat16, 3), *K = dense(a[1], at::kBFloat16, 4), *V = dense(a[2], at::kBFloat16, 4);
    if (q == nullptr || K == nullptr || V == nullptr || !small(*q) || !small(*K) || V->sizes() != K->sizes() || K->size(3) != q->size(2)) return none();
    const int B = int(q->size(0)), H = int(q->size(1)), d = int(q->size(2)), Hk = int(K->size(2));
    const bool varlen = a[4] != Py_None, paged = a[3] != Py_None;
    const Tensor *lens = nullptr, *table = nullptr, *depth = nullptr, *O, *LSE, *ws;
    if (varlen && ((lens = dense(a[4], at::kInt, 1)) == nullptr || lens->size(0) != B)) return none();
    if (paged) {
        if (!varlen || (table = dense(a[3], at::kInt, 2)) == nullptr || table->size(0) != B || !small(*table)) return none();
    } else if (K->size(0) != B) {
        return none();
    }
    if (l > 0 && ((depth = dense(a[5], at::kBFloat16, 5)) == nullptr || !shape_is(*depth, {l, B, Hk, 2, d}))) return none();
    if (!optional_dense(a[9], O) || !optional_dense(a[10], LSE) || !optional_dense(a[11], ws)) return none();
    if (!holds(O, at::kBFloat16, q->numel()) || !holds(LSE, at::kFloat, int64_t(B) * H)) return none();
    Tensor o = O != nullptr ? *O : Tensor(), lse = LSE != nullptr ? *LSE : Tensor(), w = ws != nullptr ? *ws : Tensor();
    {
        NoGil nogil;
        if (!o.defined()) o = like(*q);
        if (!lse.defined()) lse = fresh({B, H}, at::kFloat, *q);
        if (!w.defined()) w = fresh({int64_t(lib.moda_decode_workspace_bytes(B, H, d))}, at::kByte, *q);
        float* lse_p = static_cast<float*>(lse.data_ptr());
        const int* lens_p = varlen ? static_cast<const int*>(lens->data_ptr()) : nullptr;
        int rc;
        if (paged)
            rc = lib.moda_attn_decode_paged(q->data_ptr(), K->data_ptr(), V->data_ptr(), static_cast<const int*>(table->data_ptr()), lens_p,
                                            ptr(depth), B, T_kv, int(K->size(1)), int(K->size(0)), int(table->size(1)), H, Hk, d, l, scale,
                                            o.data_ptr(), lse_p, w.data_ptr(), bytes_of(w), stream());
        else if (varlen)
            rc = lib.moda_attn_decode_varlen(q->data_ptr(), K->data_ptr(), V->data_ptr(), lens_p, ptr(depth), B, T_kv, int(K->size(1)), H, Hk,
                                             d, l, scale, o.data_ptr(), lse_p, w.data_ptr(), bytes_of(w), stream());
        else
            rc = lib.moda_attn_decode(q->data_ptr(), K->data_ptr(), V->data_ptr(), ptr(depth), B, T_kv, int(K->size(1)), H, Hk, d, l, scale,
                                      o.data_ptr(), lse_p, w.data_ptr(), bytes_of(w), stream());
        if (rc != 0) fail(rc, paged ? "moda_attn_decode_paged" : varlen ? "moda_attn_decode_varlen" : "moda_attn_decode");
    }
    return Py_BuildValue("NN", out(a[9], o), out(a[10], lse));
    END_HANDLE_TH_ERRORS
}

// ---- module -----------------------------------------------------------------------------------------------------------
// bind(handle of libmoda_b200.so, check, DeviceContext): must come first
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 3) return PyErr_Format(PyExc_TypeError, "bind(handle, check, device_mode)");
    void* handle = PyLong_AsVoidPtr(a[0]);
    if (PyErr_Occurred()) return nullptr;
#define X(name)                                                                                            \
    lib.name = reinterpret_cast<decltype(&::name)>(dlsym(handle, #name));                                  \
    if (lib.name == nullptr) return PyErr_Format(PyExc_ImportError, "libmoda_b200.so has no %s", #name);
    MODA_HOST_CALLS(X)
#undef X
    Py_XSETREF(check_fn, Py_NewRef(a[1]));
    Py_XSETREF(device_mode, Py_NewRef(a[2]));
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f))
PyMethodDef methods[] = {
    {"bind", FAST(bind), METH_FASTCALL, nullptr},         {"attn_fwd", FAST(attn_fwd), METH_FASTCALL, nullptr},
    {"attn_bwd", FAST(attn_bwd), METH_FASTCALL, nullptr}, {"attention", FAST(attention), METH_FASTCALL, nullptr},
    {"decode", FAST(decode), METH_FASTCALL, nullptr},     {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() { return PyModule_Create(&module); }
