// The hot half of the Python binding: argument checks, output and workspace tensors, and the calls into
// libs2a.so (include/s2a.h), plus the differentiable front end as a C++ autograd function.  A small
// problem takes the GPU 40 to 100 us for a forward and a backward; marshalled through ctypes and Python's
// autograd.Function the host took 160 us for them.
//
// Errors stay Python's business: where an argument is not what the kernels would take it for, a function
// returns None and binding.py finds out what to say about it; where the library refuses, it returns the status.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/extension.h>

#include <ATen/cuda/CUDAContext.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>

#include <cmath>
#include <limits>
#include <optional>

#include "../../include/s2a.h"

namespace {

using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

struct Sizes {
    int64_t B, N, H, Hkv, d;
};

bool is_dense(const Tensor& t, at::ScalarType type) { return t.defined() && t.is_cuda() && t.scalar_type() == type && t.is_contiguous(); }
bool same_shape(const Tensor& t, at::IntArrayRef shape, const Tensor& like, at::ScalarType type) {
    return is_dense(t, type) && t.sizes() == shape && t.device() == like.device();
}

bool fits_int(int64_t x) { return x >= 0 && x <= std::numeric_limits<int>::max(); }

// q [B, N, H, d] and k, v [B, N, Hkv, d]: bf16, contiguous, on one CUDA device
std::optional<Sizes> sizes_of(const Tensor& q, const Tensor& k, const Tensor& v) {
    if (!is_dense(q, at::kBFloat16) || q.dim() != 4 || !is_dense(k, at::kBFloat16) || k.dim() != 4 || k.device() != q.device()) return {};
    const Sizes s{q.size(0), q.size(1), q.size(2), k.size(2), q.size(3)};
    if (k.size(0) != s.B || k.size(1) != s.N || k.size(3) != s.d) return {};
    if (!same_shape(v, k.sizes(), q, at::kBFloat16)) return {};
    for (int64_t x : {s.B, s.N, s.H, s.Hkv, s.d})
        if (!fits_int(x)) return {};
    return s;
}

bool is_stats(const Tensor& lse, const Sizes& s, const Tensor& like) { return same_shape(lse, {s.B, s.H, s.N}, like, at::kFloat); }
Tensor new_stats(const Sizes& s, const Tensor& like) { return at::empty({s.B, s.H, s.N}, like.options().dtype(at::kFloat)); }
Tensor new_like(const Tensor& t) { return at::empty(t.sizes(), t.options()); }

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The stream of a call of binding.py: the one it was given, or torch's current one.  What is made for a call on another
// stream than the current one (the workspace, outputs that were not given) belongs to that stream in the caching
// allocator.  From the current stream's memory it could take a block that work still queued there uses, and the
// workspace, which goes back when the call returns, could be handed out and overwritten before the kernels ran.
class CallStream {
public:
    CallStream(std::optional<int64_t> given, const Tensor& like)
        : stream_(given ? reinterpret_cast<cudaStream_t>(*given) : c10::cuda::getCurrentCUDAStream().stream()) {
        const auto current = c10::cuda::getCurrentCUDAStream(like.device().index());
        if (given && stream_ != current.stream()) {
            caller_ = current;
            guard_.reset_stream(c10::cuda::getStreamFromExternal(stream_, like.device().index()));
        }
    }
    // an output: the caller will go on with it on the current stream
    Tensor output(Tensor t) const {
        if (caller_) t.record_stream(*caller_);
        return t;
    }
    // to be called when everything has been made
    void* begin() {
        guard_.reset();
        return stream_;
    }

private:
    cudaStream_t stream_;
    std::optional<c10::cuda::CUDAStream> caller_;
    c10::cuda::OptionalCUDAStreamGuard guard_;
};

// Bytes that the caching allocator has from the device, and how many of them are not in use.
struct Held {
    int64_t all, unused;
    explicit Held(const Tensor& like) {
        const auto stats = c10::cuda::CUDACachingAllocator::getDeviceStats(like.device().index());
        const auto total = static_cast<size_t>(c10::CachingDeviceAllocator::StatType::AGGREGATE);
        all = stats.reserved_bytes[total].current, unused = all - stats.allocated_bytes[total].current;
    }
};

// Workspace for a call that was given none: the fast size, of which no more than half of the free device memory comes
// from the device, or the minimum.  The driver takes 70 to 220 us and more to say how much is free while the GPU is busy,
// longer than the whole backward of a small problem, so it is asked only where the caching allocator has to go to the
// device: not where it finds the workspace in what it holds, as from the second backward of a program on.
Tensor new_workspace(const Sizes& s, int G, const Tensor& like, bool fast) {
    const auto options = like.options().dtype(at::kByte);
    const int B = s.B, N = s.N, H = s.H, Hkv = s.Hkv, d = s.d;
    const size_t least = std::max<size_t>(s2a_bwd_workspace_bytes(B, N, H, Hkv, d, G), 256);
    auto make = [&](size_t bytes) { return at::empty({static_cast<int64_t>(std::max(bytes, least))}, options); };
    if (!fast) return make(least);
    const size_t need = s2a_bwd_workspace_bytes_fast(B, N, H, Hkv, d, G, size_t(1) << 62);
    size_t free_bytes = 0, total = 0;
    const Held before(like);
    if (static_cast<int64_t>(need) <= before.unused && c10::cuda::currentStreamCaptureStatusMayInitCtx() == c10::cuda::CaptureStatus::None) {
        try {
            Tensor t = make(need);
            const int64_t taken = Held(like).all - before.all;
            if (taken <= 0) return t;
            // the unused bytes were in pieces, or another stream's
            if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) free_bytes = 0;
            if (need <= (free_bytes + taken) / 2) return t;
        } catch (const c10::OutOfMemoryError&) {
        }
        c10::cuda::CUDACachingAllocator::emptyCache();  // what was taken goes back
    }
    if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) free_bytes = 0;
    return make(s2a_bwd_workspace_bytes_fast(B, N, H, Hkv, d, G, free_bytes / 2));
}

// What distinguishes the generalised entry points from the default ones.
struct Options {
    std::optional<double> scale;
    std::optional<int64_t> n_unshifted, shift;
    unsigned flags = 0;
};
struct Resolved {
    float scale;
    int n_unshifted, shift;
};
Resolved resolve(const Options& o, const Sizes& s, int G) {
    return {static_cast<float>(o.scale ? *o.scale : 1.0 / std::sqrt(static_cast<double>(s.d))),
            static_cast<int>(o.n_unshifted ? *o.n_unshifted : s.H / 2), static_cast<int>(o.shift ? *o.shift : G / 2)};
}

int call_fwd(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& o, const Tensor& lse, const Sizes& s, int G,
             const Options* ex, void* stream) {
    float* l = static_cast<float*>(lse.data_ptr());
    if (!ex) return s2a_fwd(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), l, s.B, s.N, s.H, s.Hkv, s.d, G, stream);
    const Resolved r = resolve(*ex, s, G);
    return s2a_fwd_ex(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), l, s.B, s.N, s.H, s.Hkv, s.d, G, r.scale, r.n_unshifted,
                      r.shift, ex->flags, stream);
}

int call_bwd(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& o, const Tensor& lse, const Tensor& dO, const Tensor& dq,
             const Tensor& dk, const Tensor& dv, const Tensor& ws, const Sizes& s, int G, const Options* ex, void* stream) {
    const float* l = static_cast<const float*>(lse.data_ptr());
    const size_t bytes = static_cast<size_t>(ws.numel());
    if (!ex)
        return s2a_bwd(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), l, dO.data_ptr(), dq.data_ptr(), dk.data_ptr(), dv.data_ptr(),
                       s.B, s.N, s.H, s.Hkv, s.d, G, ws.data_ptr(), bytes, stream);
    const Resolved r = resolve(*ex, s, G);
    return s2a_bwd_ex(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), l, dO.data_ptr(), dq.data_ptr(), dk.data_ptr(), dv.data_ptr(),
                      s.B, s.N, s.H, s.Hkv, s.d, G, r.scale, r.n_unshifted, r.shift, ex->flags, ws.data_ptr(), bytes, stream);
}

// ---------------------------------------------------------------------------------------------
// functions of binding.py
// ---------------------------------------------------------------------------------------------
// An argument that may be a tensor, None (= make one) or something that binding.py will refuse.
struct Arg {
    Tensor t;
    bool given = false, bad = false;
    explicit Arg(py::handle h) {
        if (h.is_none()) return;
        given = true;
        if (THPVariable_Check(h.ptr())) t = THPVariable_Unpack(h.ptr());
        else bad = true;
    }
};

py::object fwd_any(py::handle q_, py::handle k_, py::handle v_, int G, py::handle o_, py::handle lse_, const Options* ex,
                   std::optional<int64_t> stream) {
    Arg q(q_), k(k_), v(v_), o(o_), lse(lse_);
    if (q.bad || k.bad || v.bad || o.bad || lse.bad) return py::none();
    const auto s = sizes_of(q.t, k.t, v.t);
    if (!s) return py::none();
    CallStream on(stream, q.t);
    if (!o.given) o.t = on.output(new_like(q.t));
    else if (!same_shape(o.t, q.t.sizes(), q.t, at::kBFloat16)) return py::none();
    if (!lse.given) lse.t = on.output(new_stats(*s, q.t));
    else if (!is_stats(lse.t, *s, q.t)) return py::none();
    void* st = on.begin();
    int rc;
    {
        py::gil_scoped_release nogil;
        rc = call_fwd(q.t, k.t, v.t, o.t, lse.t, *s, G, ex, st);
    }
    if (rc != S2A_OK) return py::int_(rc);
    return py::make_tuple(o.t, lse.t);
}

py::object fwd(py::handle q, py::handle k, py::handle v, int G, py::handle o, py::handle lse, std::optional<int64_t> stream) {
    return fwd_any(q, k, v, G, o, lse, nullptr, stream);
}
py::object fwd_ex(py::handle q, py::handle k, py::handle v, int G, std::optional<double> scale, std::optional<int64_t> n_unshifted,
                  std::optional<int64_t> shift, unsigned flags, py::handle o, py::handle lse, std::optional<int64_t> stream) {
    const Options ex{scale, n_unshifted, shift, flags};
    return fwd_any(q, k, v, G, o, lse, &ex, stream);
}

py::object bwd_any(py::handle q_, py::handle k_, py::handle v_, py::handle o_, py::handle lse_, py::handle dO_, int G, py::handle dq_,
                   py::handle dk_, py::handle dv_, py::handle ws_, bool fast, bool noalloc, const Options* ex, std::optional<int64_t> stream) {
    Arg q(q_), k(k_), v(v_), o(o_), lse(lse_), dO(dO_), dq(dq_), dk(dk_), dv(dv_), ws(ws_);
    for (const Arg* a : {&q, &k, &v, &o, &lse, &dO, &dq, &dk, &dv, &ws})
        if (a->bad) return py::none();
    const auto s = sizes_of(q.t, k.t, v.t);
    if (!s || !same_shape(o.t, q.t.sizes(), q.t, at::kBFloat16) || !is_stats(lse.t, *s, q.t) ||
        !same_shape(dO.t, q.t.sizes(), q.t, at::kBFloat16))
        return py::none();
    CallStream on(stream, q.t);
    const struct {
        Arg* out;
        const Tensor* like;
    } outs[] = {{&dq, &q.t}, {&dk, &k.t}, {&dv, &v.t}};
    for (const auto& x : outs) {
        if (!x.out->given) {
            if (noalloc) return py::none();
            x.out->t = on.output(new_like(*x.like));
        } else if (!same_shape(x.out->t, x.like->sizes(), q.t, at::kBFloat16)) {
            return py::none();
        }
    }
    if (!noalloc) {
        if (!ws.given) ws.t = new_workspace(*s, G, q.t, fast);
        else if (!is_dense(ws.t, at::kByte) || ws.t.device() != q.t.device()) return py::none();
    }
    void* st = on.begin();
    int rc;
    {
        py::gil_scoped_release nogil;
        if (noalloc)
            rc = s2a_bwd_noalloc(q.t.data_ptr(), k.t.data_ptr(), v.t.data_ptr(), o.t.data_ptr(), static_cast<const float*>(lse.t.data_ptr()),
                                 dO.t.data_ptr(), dq.t.data_ptr(), dk.t.data_ptr(), dv.t.data_ptr(), s->B, s->N, s->H, s->Hkv, s->d, G, st);
        else
            rc = call_bwd(q.t, k.t, v.t, o.t, lse.t, dO.t, dq.t, dk.t, dv.t, ws.t, *s, G, ex, st);
    }
    if (rc != S2A_OK) return py::int_(rc);
    return py::make_tuple(dq.t, dk.t, dv.t);
}

py::object bwd(py::handle q, py::handle k, py::handle v, py::handle o, py::handle lse, py::handle dO, int G, py::handle dq, py::handle dk,
               py::handle dv, py::handle ws, bool fast, std::optional<int64_t> stream) {
    return bwd_any(q, k, v, o, lse, dO, G, dq, dk, dv, ws, fast, false, nullptr, stream);
}
py::object bwd_ex(py::handle q, py::handle k, py::handle v, py::handle o, py::handle lse, py::handle dO, int G, std::optional<double> scale,
                  std::optional<int64_t> n_unshifted, std::optional<int64_t> shift, unsigned flags, py::handle dq, py::handle dk,
                  py::handle dv, py::handle ws, bool fast, std::optional<int64_t> stream) {
    const Options ex{scale, n_unshifted, shift, flags};
    return bwd_any(q, k, v, o, lse, dO, G, dq, dk, dv, ws, fast, false, &ex, stream);
}
py::object bwd_noalloc(py::handle q, py::handle k, py::handle v, py::handle o, py::handle lse, py::handle dO, int G, py::handle dq,
                       py::handle dk, py::handle dv, std::optional<int64_t> stream) {
    return bwd_any(q, k, v, o, lse, dO, G, dq, dk, dv, py::none(), false, true, nullptr, stream);
}

// qkv [B, N, 3, H, d]
std::optional<Sizes> packed_sizes(const Tensor& qkv) {
    if (!is_dense(qkv, at::kBFloat16) || qkv.dim() != 5 || qkv.size(2) != 3) return {};
    const Sizes s{qkv.size(0), qkv.size(1), qkv.size(3), qkv.size(3), qkv.size(4)};
    for (int64_t x : {s.B, s.N, s.H, s.d})
        if (!fits_int(x)) return {};
    return s;
}

py::object fwd_packed(py::handle qkv_, int G, py::handle o_, py::handle lse_, std::optional<int64_t> stream) {
    Arg qkv(qkv_), o(o_), lse(lse_);
    if (qkv.bad || o.bad || lse.bad) return py::none();
    const auto s = packed_sizes(qkv.t);
    if (!s) return py::none();
    CallStream on(stream, qkv.t);
    if (!o.given) o.t = on.output(at::empty({s->B, s->N, s->H, s->d}, qkv.t.options()));
    else if (!same_shape(o.t, {s->B, s->N, s->H, s->d}, qkv.t, at::kBFloat16)) return py::none();
    if (!lse.given) lse.t = on.output(new_stats(*s, qkv.t));
    else if (!is_stats(lse.t, *s, qkv.t)) return py::none();
    void* st = on.begin();
    int rc;
    {
        py::gil_scoped_release nogil;
        rc = s2a_fwd_packed(qkv.t.data_ptr(), o.t.data_ptr(), static_cast<float*>(lse.t.data_ptr()), s->B, s->N, s->H, s->d, G, st);
    }
    if (rc != S2A_OK) return py::int_(rc);
    return py::make_tuple(o.t, lse.t);
}

py::object bwd_packed(py::handle qkv_, py::handle o_, py::handle lse_, py::handle dO_, int G, py::handle dqkv_, py::handle ws_, bool fast,
                      std::optional<int64_t> stream) {
    Arg qkv(qkv_), o(o_), lse(lse_), dO(dO_), dqkv(dqkv_), ws(ws_);
    for (const Arg* a : {&qkv, &o, &lse, &dO, &dqkv, &ws})
        if (a->bad) return py::none();
    const auto s = packed_sizes(qkv.t);
    if (!s || !same_shape(o.t, {s->B, s->N, s->H, s->d}, qkv.t, at::kBFloat16) || !is_stats(lse.t, *s, qkv.t) ||
        !same_shape(dO.t, {s->B, s->N, s->H, s->d}, qkv.t, at::kBFloat16))
        return py::none();
    CallStream on(stream, qkv.t);
    if (!dqkv.given) dqkv.t = on.output(new_like(qkv.t));
    else if (!same_shape(dqkv.t, qkv.t.sizes(), qkv.t, at::kBFloat16)) return py::none();
    if (!ws.given) ws.t = new_workspace(*s, G, qkv.t, fast);
    else if (!is_dense(ws.t, at::kByte) || ws.t.device() != qkv.t.device()) return py::none();
    void* st = on.begin();
    int rc;
    {
        py::gil_scoped_release nogil;
        rc = s2a_bwd_packed(qkv.t.data_ptr(), o.t.data_ptr(), static_cast<const float*>(lse.t.data_ptr()), dO.t.data_ptr(), dqkv.t.data_ptr(), s->B,
                            s->N, s->H, s->d, G, ws.t.data_ptr(), static_cast<size_t>(ws.t.numel()), st);
    }
    if (rc != S2A_OK) return py::int_(rc);
    return py::cast(dqkv.t);
}

// ---------------------------------------------------------------------------------------------
// differentiable front end
// ---------------------------------------------------------------------------------------------
// Raises binding.S2AError; callable from the threads of the autograd engine.
[[noreturn]] void raise_status(int rc, const char* what) {
    py::gil_scoped_acquire gil;
    py::object type = py::module_::import("paper_2309_12307_b200.binding").attr("S2AError");
    py::object err = type(rc, what);
    PyErr_SetObject(type.ptr(), err.ptr());
    python_error e;
    e.persist();
    throw e;
}

struct S2Attn : public torch::autograd::Function<S2Attn> {
    static Tensor forward(AutogradContext* ctx, const Tensor& q, const Tensor& k, const Tensor& v, int64_t G, std::optional<double> scale,
                          std::optional<int64_t> n_unshifted, std::optional<int64_t> shift, int64_t flags, bool fast) {
        const Options ex{scale, n_unshifted, shift, static_cast<unsigned>(flags)};
        const auto s = sizes_of(q, k, v);
        TORCH_CHECK_VALUE(s, "q, k, v");  // checked by s2_attn
        Tensor o = new_like(q), lse = new_stats(*s, q);
        const int rc = call_fwd(q, k, v, o, lse, *s, static_cast<int>(G), &ex, current_stream());
        if (rc != S2A_OK) raise_status(rc, "s2a_fwd_ex");
        ctx->save_for_backward({q, k, v, o, lse});
        ctx->saved_data["G"] = G;
        ctx->saved_data["scale"] = scale;
        ctx->saved_data["n_unshifted"] = n_unshifted;
        ctx->saved_data["shift"] = shift;
        ctx->saved_data["flags"] = flags;
        ctx->saved_data["fast"] = fast;
        return o;
    }
    static variable_list backward(AutogradContext* ctx, variable_list grads) {
        const variable_list saved = ctx->get_saved_variables();
        const Tensor &q = saved[0], &k = saved[1], &v = saved[2], &o = saved[3], &lse = saved[4];
        const Options ex{ctx->saved_data["scale"].toOptional<double>(), ctx->saved_data["n_unshifted"].toOptional<int64_t>(),
                         ctx->saved_data["shift"].toOptional<int64_t>(), static_cast<unsigned>(ctx->saved_data["flags"].toInt())};
        const int G = static_cast<int>(ctx->saved_data["G"].toInt());
        const Tensor dO = grads[0].contiguous();
        const auto s = sizes_of(q, k, v);
        // saved-tensor hooks decide what comes back
        TORCH_CHECK_VALUE(s && same_shape(o, q.sizes(), q, at::kBFloat16) && is_stats(lse, *s, q),
                          "the saved q, k, v, o and lse have come back with another type, shape, layout or device");
        TORCH_CHECK_VALUE(same_shape(dO, q.sizes(), q, at::kBFloat16), "dO must be a bf16 CUDA tensor of the shape of q");
        at::NoGradGuard no_grad;
        Tensor dq = new_like(q), dk = new_like(k), dv = new_like(v);
        const Tensor ws = new_workspace(*s, G, q, ctx->saved_data["fast"].toBool());
        const int rc = call_bwd(q, k, v, o, lse, dO, dq, dk, dv, ws, *s, G, &ex, current_stream());
        if (rc != S2A_OK) raise_status(rc, "s2a_bwd_ex");
        return {dq, dk, dv, Tensor(), Tensor(), Tensor(), Tensor(), Tensor(), Tensor()};
    }
};

// o, or None where q, k, v are not what the kernels take
py::object s2_attn(py::handle q_, py::handle k_, py::handle v_, int G, std::optional<double> scale, std::optional<int64_t> n_unshifted,
                   std::optional<int64_t> shift, unsigned flags, bool fast) {
    Arg q(q_), k(k_), v(v_);
    if (!q.given || !k.given || !v.given || q.bad || k.bad || v.bad) return py::none();
    Tensor o;
    {
        py::gil_scoped_release nogil;
        q.t = q.t.contiguous(), k.t = k.t.contiguous(), v.t = v.t.contiguous();
        if (sizes_of(q.t, k.t, v.t)) o = S2Attn::apply(q.t, k.t, v.t, G, scale, n_unshifted, shift, flags, fast);
    }
    return o.defined() ? py::cast(o) : py::none();
}

}  // namespace

PYBIND11_MODULE(_s2a_torch, m) {
    m.doc() = "Hot path of the Python binding of libs2a.so; called by binding.py and autograd.py.";
    m.attr("torch_version") = S2A_TORCH_VERSION;
    m.def("fwd", &fwd);
    m.def("fwd_ex", &fwd_ex);
    m.def("fwd_packed", &fwd_packed);
    m.def("bwd", &bwd);
    m.def("bwd_ex", &bwd_ex);
    m.def("bwd_packed", &bwd_packed);
    m.def("bwd_noalloc", &bwd_noalloc);
    m.def("s2_attn", torch::wrap_pybind_function(&s2_attn));
}
