// Argument marshalling of the hot entry points as a Python extension module: checks the tensors, allocates the results and calls
// the C functions of include/tlin.h, nothing else.  A small call is over on the device in about ten microseconds; the same checks
// and calls through Python attributes and ctypes took sixteen.
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/utils/pybind.h>
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <optional>
#include <vector>
#include "../../include/tlin.h"

namespace py = pybind11;
using at::Tensor;

namespace {

[[noreturn]] void bad(const std::string& what) { throw py::value_error(what); }

void check(const Tensor& t, at::ScalarType dtype, at::IntArrayRef shape, const char* name) {
    if (t.is_cuda() && t.scalar_type() == dtype && t.sizes() == shape && t.is_contiguous()) return;
    if (!t.is_cuda()) bad(std::string(name) + " must be a CUDA tensor");
    std::ostringstream s;
    s << name << " must be contiguous " << dtype << " of shape " << shape << ", got " << t.scalar_type() << " " << t.sizes();
    bad(s.str());
}
const Tensor& four_dims(const Tensor& t, const char* name) {
    if (t.dim() != 4) bad(std::string(name) + " must have four dimensions");
    return t;
}
int as_int(int64_t x) {
    if (x > INT32_MAX) bad("a dimension exceeds 2^31 - 1");
    return (int)x;
}
// Asked for once the tensors have been checked: without a device there is no current stream, and a CPU tensor is the caller's error.
tlin_stream_t current_stream() { return (tlin_stream_t)c10::cuda::getCurrentCUDAStream().stream(); }
tlin_stream_t stream_of(const py::object& stream) {
    return stream.is_none() ? current_stream() : reinterpret_cast<tlin_stream_t>(stream.attr("cuda_stream").cast<uintptr_t>());
}
Tensor fresh(at::IntArrayRef shape, at::ScalarType dtype, const Tensor& like) {
    return at::detail::empty_cuda(shape, dtype, like.device(), std::nullopt);
}
using Opt = std::optional<Tensor>;
Tensor given_or_fresh(const Opt& t, at::IntArrayRef shape, at::ScalarType dtype, const Tensor& like, const char* name, bool checked = true) {
    if (!t.has_value()) return fresh(shape, dtype, like);
    if (checked) check(*t, dtype, shape, name);
    return *t;
}
template <class F>
int without_gil(F&& f) {                 // called with the lock held (from Python) or without it (from autograd's threads)
    if (!PyGILState_Check()) return f();
    py::gil_scoped_release release;
    return f();
}
using Result = std::tuple<int, Tensor, Tensor>;

// Whether `t` lies in memory that a graph's capture keeps for it (or in another pool of its own): what PyTorch allocates under its own
// captures.
bool in_a_pool(const Tensor& t) {
    const size_t at = (size_t)t.data_ptr();
    for (const auto& s : c10::cuda::CUDACachingAllocator::snapshot({0, 0}, false).segments)
        if (s.device == t.device().index() && at >= s.address && at < s.address + s.total_size)
            return s.owner_private_pool_id != c10::MempoolId_t{0, 0};
    return false;
}
// Scratch of one call, from PyTorch's allocator on the call's stream: its memory is not given out again before the call is over there.
// Undefined where none is wanted or there is no memory for it, and under a capture that PyTorch does not know of (cudaStreamBeginCapture
// by the caller): there the memory would be given out again while the graph still writes to it at every launch.
Tensor scratch_for(size_t bytes, const Tensor& like, tlin_stream_t st) {
    if (bytes == 0) return Tensor();
    try {
        const c10::cuda::CUDAStreamGuard guard(c10::cuda::getStreamFromExternal((cudaStream_t)st, like.device().index()));
        const Tensor t = at::detail::empty_cuda({(int64_t)bytes}, at::kByte, like.device(), std::nullopt);
        if (c10::cuda::currentStreamCaptureStatusMayInitCtx() != c10::cuda::CaptureStatus::None && !in_a_pool(t)) return Tensor();
        return t;
    } catch (const c10::OutOfMemoryError&) {
        return Tensor();
    }
}
size_t workspace_forward(const Tensor& q, const Tensor& k, int64_t n_keys, int causal) {
    four_dims(q, "q");
    four_dims(k, "k");
    return tlin_workspace_bytes_forward(as_int(q.size(0)), as_int(q.size(1)), as_int(n_keys < 0 ? k.size(2) : n_keys), as_int(q.size(2)),
                                        as_int(q.size(3)), causal);
}
// kind: 0 bf16, 1 fp32, 2 bf16 over the first n_keys rows of a cache
template <class StreamFn>
Result run_forward(int kind, const Tensor& q, const Tensor& k, const Tensor& v, int64_t n_keys, const Opt& out_, const Opt& lse_, int causal,
                   StreamFn&& stream) {
    const int64_t B = four_dims(q, "q").size(0), H = q.size(1), W = q.size(2), d = q.size(3), N = four_dims(k, "k").size(2);
    const at::ScalarType dt = kind == 1 ? at::kFloat : at::kBFloat16;
    check(q, dt, {B, H, W, d}, "q");
    check(k, dt, {B, H, N, d}, kind == 2 ? "k_cache" : "k");
    check(v, dt, {B, H, N, d}, kind == 2 ? "v_cache" : "v");
    const Tensor out = given_or_fresh(out_, {B, H, W, d}, dt, q, "out"), lse = given_or_fresh(lse_, {B, H, W}, at::kFloat, q, "lse");
    const int b = as_int(B), h = as_int(H), n = as_int(N), w = as_int(W), dd = as_int(d), nk = as_int(n_keys);
    const tlin_stream_t st = stream();
    const size_t bytes = kind == 1 ? tlin_scratch_bytes_forward_f32(b, h, n, w, dd, causal) : 0;
    const Tensor scratch = scratch_for(bytes, q, st);
    const int rc = without_gil([&] {
        const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
        float* lp = (float*)lse.data_ptr();
        if (kind == 0) return tlin_attn_forward(qp, kp, vp, out.data_ptr(), lp, b, h, n, w, dd, causal, st);
        if (kind == 1)
            return tlin_attn_forward_f32_scratch((const float*)qp, (const float*)kp, (const float*)vp, (float*)out.data_ptr(), lp, b, h, n, w, dd, causal,
                                                 scratch.defined() ? scratch.data_ptr() : nullptr, scratch.defined() ? bytes : 0, st);
        return tlin_attn_forward_cache(qp, kp, vp, out.data_ptr(), lp, b, h, n, nk, w, dd, causal, st);
    });
    return {rc, out, lse};
}

Result forward(int kind, const Tensor& q, const Tensor& k, const Tensor& v, int64_t n_keys, const Opt& out, const Opt& lse, int causal,
               const py::object& stream) {
    return run_forward(kind, q, k, v, n_keys, out, lse, causal, [&] { return stream_of(stream); });
}

using Gradients = std::tuple<int, Tensor, Tensor, Tensor>;
template <class StreamFn>
Gradients run_backward(bool f32, const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& out, const Tensor& lse, const Tensor& dout,
                       const Opt& dq_, const Opt& dk_, const Opt& dv_, int causal, StreamFn&& stream) {
    const int64_t B = four_dims(q, "q").size(0), H = q.size(1), W = q.size(2), d = q.size(3), N = four_dims(k, "k").size(2);
    const at::ScalarType dt = f32 ? at::kFloat : at::kBFloat16;
    check(q, dt, {B, H, W, d}, "q");
    check(k, dt, {B, H, N, d}, "k");
    check(v, dt, {B, H, N, d}, "v");
    check(out, dt, {B, H, W, d}, "out");
    check(dout, dt, {B, H, W, d}, "dout");
    check(lse, at::kFloat, {B, H, W}, "lse");
    const Tensor dq = given_or_fresh(dq_, {B, H, W, d}, dt, q, "dq"), dk = given_or_fresh(dk_, {B, H, N, d}, dt, q, "dk"),
                 dv = given_or_fresh(dv_, {B, H, N, d}, dt, q, "dv");
    const int b = as_int(B), h = as_int(H), n = as_int(N), w = as_int(W), dd = as_int(d);
    const tlin_stream_t st = stream();
    const size_t bytes = f32 ? tlin_scratch_bytes_backward_f32(b, h, n, w, dd, causal) : 0;
    const Tensor scratch = scratch_for(bytes, q, st);
    const int rc = without_gil([&] {
        if (f32)
            return tlin_attn_backward_f32_scratch((const float*)q.data_ptr(), (const float*)k.data_ptr(), (const float*)v.data_ptr(), (const float*)out.data_ptr(),
                                          (const float*)lse.data_ptr(), (const float*)dout.data_ptr(), (float*)dq.data_ptr(), (float*)dk.data_ptr(),
                                          (float*)dv.data_ptr(), b, h, n, w, dd, causal, scratch.defined() ? scratch.data_ptr() : nullptr,
                                                  scratch.defined() ? bytes : 0, st);
        return tlin_attn_backward(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), (const float*)lse.data_ptr(), dout.data_ptr(), dq.data_ptr(),
                                  dk.data_ptr(), dv.data_ptr(), b, h, n, w, dd, causal, st);
    });
    return {rc, dq, dk, dv};
}

Gradients backward(bool f32, const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& out, const Tensor& lse, const Tensor& dout, const Opt& dq,
                   const Opt& dk, const Opt& dv, int causal, const py::object& stream) {
    return run_backward(f32, q, k, v, out, lse, dout, dq, dk, dv, causal, [&] { return stream_of(stream); });
}
size_t workspace_backward(const Tensor& q, const Tensor& k) {
    four_dims(q, "q");
    four_dims(k, "k");
    return tlin_workspace_bytes_backward(as_int(q.size(0)), as_int(q.size(1)), as_int(k.size(2)), as_int(q.size(2)), as_int(q.size(3)));
}

// ---- autograd: the forward and the backward entry point as one differentiable operation (nothing is computed here)
// The Python side owns the workspace and the exception type.
void raise(int rc, const char* where) {
    if (rc == TLIN_OK) return;
    py::gil_scoped_acquire lock;
    const py::object type = py::module_::import("paper_2508_20407_b200.binding").attr("TlinError");
    PyErr_SetObject(type.ptr(), type(rc, where).ptr());
    throw py::error_already_set();
}
void ensure_workspace(size_t bytes, const Tensor& like) {
    py::gil_scoped_acquire lock;
    py::module_::import("paper_2508_20407_b200.binding").attr("ensure_workspace")(bytes, like.device());
}

struct Attention : public torch::autograd::Function<Attention> {
    static torch::autograd::variable_list forward(torch::autograd::AutogradContext* ctx, const Tensor& q_in, const Tensor& k_in, const Tensor& v_in,
                                                  int64_t causal) {
        const Tensor q = q_in.contiguous(), k = k_in.contiguous(), v = v_in.contiguous();
        const bool f32 = q.scalar_type() == at::kFloat;
        if (!f32 && q.is_cuda()) ensure_workspace(workspace_forward(q, k, -1, (int)causal), q);
        const auto [rc, out, lse] = run_forward(f32 ? 1 : 0, q, k, v, 0, std::nullopt, std::nullopt, (int)causal, current_stream);
        raise(rc, f32 ? "tlin_attn_forward_f32" : "tlin_attn_forward");
        ctx->save_for_backward({q, k, v, out, lse});
        ctx->saved_data["causal"] = causal;
        ctx->mark_non_differentiable({lse});
        return {out, lse};
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads) {
        const auto saved = ctx->get_saved_variables();
        const Tensor &q = saved[0], &k = saved[1];
        const bool f32 = q.scalar_type() == at::kFloat;
        const Tensor dout = grads[0].defined() ? grads[0].contiguous() : at::zeros_like(saved[3]);
        const int causal = (int)ctx->saved_data["causal"].toInt();
        auto [rc, dq, dk, dv] = run_backward(f32, q, k, saved[2], saved[3], saved[4], dout, std::nullopt, std::nullopt, std::nullopt, causal, current_stream);
        if (rc == TLIN_ERR_WORKSPACE) {      // too small so far: asking first would cost this thread a turn of the interpreter (20 us)
            ensure_workspace(workspace_backward(q, k), q);
            std::tie(rc, dq, dk, dv) = run_backward(f32, q, k, saved[2], saved[3], saved[4], dout, dq, dk, dv, causal, current_stream);
        }
        raise(rc, f32 ? "tlin_attn_backward_f32" : "tlin_attn_backward");
        return {dq, dk, dv, Tensor()};
    }
};
std::tuple<Tensor, Tensor> attention(const Tensor& q, const Tensor& k, const Tensor& v, int64_t causal) {
    const auto r = Attention::apply(q, k, v, causal);
    return {r[0], r[1]};
}

size_t workspace_decode(const Tensor& k_cache) {
    four_dims(k_cache, "k_cache");
    return tlin_workspace_bytes_decode(as_int(k_cache.size(0)), as_int(k_cache.size(1)), as_int(k_cache.size(2)), as_int(k_cache.size(3)));
}
// kind: 0 one position, 1 8-bit cache (a, b: the scales), 2 ragged (a: the positions, pos: their upper bound)
Result decode(int kind, const Tensor& q, const Tensor& kn, const Tensor& vn, const Tensor& kc, const Tensor& vc, const Opt& a, const Opt& b2, int64_t pos,
              const Opt& out_, const Opt& lse_, const py::object& stream) {
    const int64_t B = four_dims(kc, "k_cache").size(0), H = kc.size(1), N = kc.size(2), d = kc.size(3);
    check(q, at::kBFloat16, {B, H, 1, d}, "q_new");
    check(kn, at::kBFloat16, {B, H, 1, d}, "k_new");
    check(vn, at::kBFloat16, {B, H, 1, d}, "v_new");
    const at::ScalarType ct = kind == 1 ? at::kByte : at::kBFloat16;
    check(kc, ct, {B, H, N, d}, "k_cache");
    check(vc, ct, {B, H, N, d}, "v_cache");
    if (kind == 1) {
        check(*a, at::kFloat, {B, H}, "k_scale");
        check(*b2, at::kFloat, {B, H}, "v_scale");
    }
    if (kind == 2) check(*a, at::kInt, {B}, "pos");
    const Tensor out = given_or_fresh(out_, {B, H, 1, d}, at::kBFloat16, q, "out", false), lse = given_or_fresh(lse_, {B, H}, at::kFloat, q, "lse", false);
    const tlin_stream_t st = stream_of(stream);
    const int b = as_int(B), h = as_int(H), n = as_int(N), dd = as_int(d);
    if (pos < INT32_MIN || pos > INT32_MAX) bad("pos out of range");
    const int p = (int)pos;
    const int rc = without_gil([&] {
        const void *qp = q.data_ptr(), *knp = kn.data_ptr(), *vnp = vn.data_ptr();
        void *kp = kc.data_ptr(), *vp = vc.data_ptr(), *op = out.data_ptr();
        float* lp = (float*)lse.data_ptr();
        if (kind == 0) return tlin_decode_step(qp, knp, vnp, kp, vp, op, lp, b, h, n, p, dd, st);
        if (kind == 1) return tlin_decode_step_fp8(qp, knp, vnp, kp, vp, (const float*)a->data_ptr(), (const float*)b2->data_ptr(), op, lp, b, h, n, p, dd, st);
        return tlin_decode_step_ragged(qp, knp, vnp, kp, vp, op, lp, b, h, n, (const int32_t*)a->data_ptr(), p, dd, st);
    });
    return {rc, out, lse};
}

// problems: a sequence of (q, k, v, out, lse, n_keys, causal_window), each any iterable; the numbers whatever int() takes
int64_t number(const py::handle& x) { return py::int_(py::reinterpret_borrow<py::object>(x)).cast<int64_t>(); }
int forward_batched(const py::sequence& problems, const py::object& stream) {
    if (problems.size() == 0) throw py::index_error("a table needs at least one problem");
    std::vector<tlin_problem> table;
    table.reserve(problems.size());
    int d_first = 0, i = 0;
    for (const py::handle item : problems) {
        const py::tuple pr(py::reinterpret_borrow<py::object>(item));
        if (pr.size() != 7) bad("problem " + std::to_string(i) + ": expected (q, k, v, out, lse, n_keys, causal_window)");
        const Tensor q = pr[0].cast<Tensor>(), k = pr[1].cast<Tensor>(), v = pr[2].cast<Tensor>(), out = pr[3].cast<Tensor>();
        const Tensor* all[4] = {&q, &k, &v, &out};
        const char* names[4] = {"q", "k", "v", "out"};
        const std::string here = "problem " + std::to_string(i);
        for (int x = 0; x < 4; ++x)
            if (!all[x]->is_cuda() || all[x]->scalar_type() != at::kBFloat16 || !all[x]->is_contiguous()) bad(here + ": " + names[x] + " must be a contiguous bf16 CUDA tensor");
        if (q.dim() < 2 || k.dim() < 2) bad(here + ": shape mismatch");
        const int64_t d = q.size(-1), W = q.size(-2), rows = k.size(-2), bh = W * d > 0 ? q.numel() / (W * d) : 0;
        const int64_t n_keys = pr[5].is_none() ? rows : number(pr[5]);
        if (k.numel() != bh * rows * d || !v.sizes().equals(k.sizes()) || !out.sizes().equals(q.sizes())) bad(here + ": shape mismatch");
        tlin_problem t = {};
        t.q = q.data_ptr(); t.k = k.data_ptr(); t.v = v.data_ptr(); t.out = out.data_ptr();
        if (!pr[4].is_none()) {
            const Tensor lse = pr[4].cast<Tensor>();
            if (lse.scalar_type() != at::kFloat || lse.numel() != bh * W || !lse.is_contiguous()) bad(here + ": lse must be contiguous fp32 of " + std::to_string(bh * W) + " elements");
            t.lse = (float*)lse.data_ptr();
        }
        t.BH = as_int(bh); t.n_keys = as_int(n_keys); t.kv_rows = rows != n_keys ? as_int(rows) : 0; t.n_queries = as_int(W);
        t.causal_window = (int)number(pr[6]);
        table.push_back(t);
        if (i++ == 0) d_first = as_int(d);
    }
    const tlin_stream_t st = stream_of(stream);
    return without_gil([&] { return tlin_attn_forward_batched(table.data(), (int)table.size(), d_first, st); });
}

}  // namespace

PYBIND11_MODULE(_fastcall, m) {
    m.def("workspace_forward", &workspace_forward);
    m.def("forward", &forward);
    m.def("backward", &backward);
    m.def("workspace_backward", &workspace_backward);
    m.def("attention", &attention);
    m.def("workspace_decode", &workspace_decode);
    m.def("decode", &decode);
    m.def("forward_batched", &forward_batched);
}
