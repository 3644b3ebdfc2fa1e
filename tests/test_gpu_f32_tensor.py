"""fp32 calls on the tensor cores, three bf16 parts per number: sizes at the edges of their tiles, results against 64-bit sums, and the
numbers that the parts do not hold."""
import ctypes
import math
import os
import subprocess
import sys

import pytest
import torch

from guards import Guarded
from paper_2508_20407_b200 import binding as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def normal(seed, *shape):
    return torch.randn(*shape, generator=torch.Generator(device="cpu").manual_seed(seed)).to(DEV)


def scratch(n):
    return torch.empty(n, dtype=torch.uint8, device=DEV) if n else None


def pointers(*tensors):
    return [t.data_ptr() for t in tensors]


def both_sides(q, k, v, dout, causal, chunks=False):
    """(out, lse, dq, dk, dv) of the call with scratch and of the call without, which the CUDA cores serve."""
    B, H, W, d = q.shape
    N, lib, stream = k.shape[2], tl.lib(), torch.cuda.current_stream().cuda_stream
    sizes = (B, H, N, W, d, causal)
    tl.ensure_workspace(tl.workspace_bytes_backward(*sizes[:5]))
    results = []
    for with_scratch in (True, False):
        out, lse = torch.empty_like(q), torch.empty(B, H, W, device=DEV)
        grads = [torch.empty_like(t) for t in (q, k, v)]
        fwd = lib.tlin_scratch_bytes_forward_f32(*sizes) if with_scratch else 0
        bwd = lib.tlin_scratch_bytes_backward_f32(*sizes) if with_scratch else 0
        s, s2 = scratch(fwd), scratch(bwd)
        assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out, lse), *sizes, s.data_ptr() if fwd else None, fwd, stream) == 0
        launches = tl.tlin_last_launch_count()
        assert not fwd or (launches > 3 if chunks else launches == 3)
        assert lib.tlin_attn_backward_f32_scratch(*pointers(q, k, v, out, lse, dout, *grads), *sizes, s2.data_ptr() if bwd else None, bwd, stream) == 0
        results.append(([out, lse] + grads, bool(fwd), bool(bwd)))
    assert tl.tlin_get_status() == 0
    return results


def exact(q, k, v, dout, causal):
    q, k, v, dout = (t.double() for t in (q, k, v, dout))
    W, N, d = q.shape[2], k.shape[2], q.shape[3]
    s = q @ k.transpose(-1, -2) / math.sqrt(d)
    if causal:
        s.masked_fill_(torch.arange(N, device=DEV)[None] > (N - W + torch.arange(W, device=DEV))[:, None], -math.inf)
    lse = torch.logsumexp(s, -1)
    p = torch.exp(s - lse[..., None])
    ds = p * (dout @ v.transpose(-1, -2) - (p * (dout @ v.transpose(-1, -2))).sum(-1, keepdim=True)) / math.sqrt(d)
    return p @ v, lse, ds @ k, ds.transpose(-1, -2) @ q, p.transpose(-1, -2) @ dout


# one row beyond, at and below the tiles of 64 and 128; shared keys in clusters of 2 to 8; one and several pieces of dq; d at and off the
# multiples of 16 and 64
SHAPES = [(2, 16, 385, 129, 36, 1), (2, 16, 384, 128, 64, 0), (4, 16, 257, 257, 40, 1), (1, 40, 1000, 127, 20, 0), (1, 12, 1537, 513, 64, 1),
          (1, 3, 3000, 700, 128, 0), (1, 2, 8192, 300, 100, 1), (1, 5, 2100, 640, 68, 1), (1, 30, 700, 700, 52, 1), (1, 64, 300, 200, 4, 0)]


# against 64 bits no further off than the CUDA cores' sums, with a fifth for the chance in both, and 4 units of 2^-24 where those are that good
@pytest.mark.parametrize("B,H,N,W,d,causal", SHAPES)
def test_as_exact_as_the_cuda_cores(B, H, N, W, d, causal):
    q, dout, k, v = normal(1, B, H, W, d), normal(2, B, H, W, d), normal(3, B, H, N, d), normal(4, B, H, N, d)
    (got, fwd, bwd), (ref, _, _) = both_sides(q, k, v, dout, causal)
    assert fwd or bwd
    for a, b, x in zip(got, ref, exact(q, k, v, dout, causal)):
        size = float(x.norm())
        assert float((a - x).norm()) <= max(1.2 * float((b - x).norm()), 4 * 2.0 ** -24 * size)


def forward(q, k, v, causal, with_scratch=True, out=None):
    """(out, lse) of the C entry point: on the tensor cores, which the sizes have to be for, or without scratch on the CUDA cores."""
    (B, H, W, d), N, lib = q.shape, k.shape[2], tl.lib()
    need = lib.tlin_scratch_bytes_forward_f32(B, H, N, W, d, causal) if with_scratch else 0
    assert not with_scratch or need
    s, out, lse = scratch(need), torch.empty_like(q) if out is None else out, torch.empty(B, H, W, device=DEV)
    assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out, lse), B, H, N, W, d, causal, s.data_ptr() if need else None, need,
                                             torch.cuda.current_stream().cuda_stream) == 0
    return out, lse


def backward(q, k, v, out, lse, dout, causal, with_scratch=True, grads=None):
    (B, H, W, d), N, lib = q.shape, k.shape[2], tl.lib()
    tl.ensure_workspace(tl.workspace_bytes_backward(B, H, N, W, d))
    need = lib.tlin_scratch_bytes_backward_f32(B, H, N, W, d, causal) if with_scratch else 0
    assert not with_scratch or need
    s, grads = scratch(need), [torch.empty_like(t) for t in (q, k, v)] if grads is None else grads
    assert lib.tlin_attn_backward_f32_scratch(*pointers(q, k, v, out, lse, dout, *grads), B, H, N, W, d, causal, s.data_ptr() if need else None, need,
                                              torch.cuda.current_stream().cuda_stream) == 0
    return grads


def same(a, b):
    return torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(), b.nan_to_num())


def check_that_one_head_goes_to_the_cuda_cores(t, what, head, value, causal=1, in_place=False):
    """`value` in one (b,h) of t[what]: that one as the CUDA cores compute it, all others as without it, bit for bit.  dq of more than one
    addition in any order (the CUDA cores', and the tensor cores' over more than 1536 keys) to the rounding of its sums."""
    clean = forward(t["q"], t["k"], t["v"], causal)
    clean_grads = backward(t["q"], t["k"], t["v"], *clean, t["dout"], causal)
    t = dict(t)
    t[what] = t[what].clone()
    t[what][head][min(17, t[what].shape[2] - 1), 3] = value
    q, k, v, dout = (t[x] for x in ("q", "k", "v", "dout"))
    others = torch.ones(q.shape[:2], dtype=torch.bool, device=DEV)
    others[head] = False
    got, cores = forward(q, k, v, causal, out=q.clone() if in_place else None), forward(q, k, v, causal, False)
    if in_place:
        over = q.clone()
        assert all(same(x, y) for x, y in zip(forward(over, k, v, causal, out=over), got))
    for x, y, z in zip(got, cores, clean):
        assert torch.equal(x[others], z[others])
        assert same(x[head], y[head]) if what != "dout" else torch.equal(x, z)
    cores_grads = backward(q, k, v, *got, dout, causal, False)
    if in_place:
        over = [q.clone(), k.clone(), v.clone()]
        grads = backward(*over, *got, dout, causal, grads=over)
    else:
        grads = backward(q, k, v, *got, dout, causal)
    for x, y, z, name in zip(grads, cores_grads, clean_grads, ("dq", "dk", "dv")):
        if name == "dq":
            ok = torch.isfinite(y[head])
            assert torch.equal(torch.isfinite(x[head]), ok)
            if not (what in ("q", "k") and abs(value) > 1):           # one key takes all there: ds is 0, and its rounding is multiplied by the value
                assert float((x[head] - y[head])[ok].double().norm()) <= 1e-6 * float(y[head][ok].double().norm())
        else:
            assert same(x[head], y[head])
        if name == "dq" and k.shape[2] > 1536:
            assert float((x[others] - z[others]).double().norm()) <= 1e-6 * float(z[others].double().norm())
        else:
            assert torch.equal(x[others], z[others])
    assert tl.tlin_get_status() == 0


def tensors(B, H, N, W, d):
    return dict(q=normal(1, B, H, W, d), dout=normal(2, B, H, W, d), k=normal(3, B, H, N, d), v=normal(4, B, H, N, d))


@pytest.mark.parametrize("what", ["q", "k", "v", "dout"])
@pytest.mark.parametrize("value", [math.inf, -3e38, 1e-35, 2e9])
def test_numbers_that_the_parts_do_not_hold_go_to_the_cuda_cores(what, value):
    check_that_one_head_goes_to_the_cuda_cores(tensors(2, 16, 500, 300, 36), what, (1, 3), value)


# keys shared in a cluster (forward) and dq in several pieces; several pieces without clusters; several launches, the head in the last and in
# the first; results over inputs
@pytest.mark.parametrize("B,H,N,W,d,head,in_place", [(1, 3, 3000, 200, 64, (0, 1), False), (1, 40, 2100, 640, 36, (0, 39), False), (2, 160, 2000, 300, 64, (1, 159), False),
                                                     (2, 160, 2000, 300, 64, (0, 0), False), (2, 16, 500, 500, 36, (1, 3), True), (1, 3, 3000, 200, 64, (0, 2), True)])
@pytest.mark.parametrize("what,value", [("v", math.nan), ("k", math.inf)])
def test_one_head_on_the_cuda_cores_in_every_form(B, H, N, W, d, head, in_place, what, value):
    check_that_one_head_goes_to_the_cuda_cores(tensors(B, H, N, W, d), what, head, value, in_place=in_place)


def test_one_head_on_one_warp_per_row():
    """A call that the CUDA cores compute with the kernel of one warp per row, when they compute all of it."""
    q, k, v = (normal(i, 1, 1000, rows, 128) for i, rows in enumerate((19, 27, 27)))
    clean = forward(q, k, v, 1)
    v[0, 501, 20, 7] = math.nan
    got, cores = forward(q, k, v, 1), forward(q, k, v, 1, False)
    for x, y, z in zip(got, cores, clean):
        assert same(x[0, 501], y[0, 501]) and torch.equal(x[0, :501], z[0, :501]) and torch.equal(x[0, 502:], z[0, 502:])
    assert tl.tlin_get_status() == 0


def test_results_over_inputs_and_too_little_scratch():
    B, H, N, W, d = 2, 16, 500, 500, 36
    q, dout, k, v = normal(1, B, H, W, d), normal(2, B, H, W, d), normal(3, B, H, N, d), normal(4, B, H, N, d)
    out, lse = tl.tlin_attn_forward_f32(q, k, v)
    want = tl.tlin_attn_backward_f32(q, k, v, out, lse, dout)
    q2, k2, v2 = q.clone(), k.clone(), v.clone()
    got = tl.tlin_attn_backward_f32(q2, k2, v2, out, lse, dout, dq=q2, dk=k2, dv=v2)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    lib, stream, sizes = tl.lib(), torch.cuda.current_stream().cuda_stream, (B, H, N, W, d, 1)
    need = lib.tlin_scratch_bytes_forward_f32(*sizes)
    s, out2, plain = scratch(need), torch.empty_like(out), torch.empty_like(out)
    assert lib.tlin_attn_forward_f32(*pointers(q, k, v, plain, lse), *sizes, stream) == 0
    assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out2, lse), *sizes, s.data_ptr(), need - 1, stream) == 0
    assert torch.equal(out2, plain)
    assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out2, lse), *sizes, s.data_ptr(), need, stream) == 0
    assert torch.equal(out2, out) and tl.tlin_get_status() == 0


def test_one_call_in_several_launches():
    """More parts than L2 holds: the call goes through in chunks of (b,h)."""
    B, H, N, W, d = 2, 160, 2000, 300, 64
    q, dout, k, v = normal(1, B, H, W, d), normal(2, B, H, W, d), normal(3, B, H, N, d), normal(4, B, H, N, d)
    (got, fwd, bwd), (ref, _, _) = both_sides(q, k, v, dout, 1, chunks=True)
    assert fwd and bwd
    for a, b in zip(got, ref):
        assert float((a - b).double().norm()) <= 2e-6 * float(b.double().norm())


def test_a_long_history_goes_in_chunks_of_no_more_than_the_bound():
    """24 heads of 131072 keys are 2.3 GiB of parts for one query tile each: several launches, the last of fewer heads or not."""
    B, H, N, W, d = 1, 24, 131072, 20, 64
    lib, sizes, stream = tl.lib(), (B, H, N, W, d, 1), torch.cuda.current_stream().cuda_stream
    need = lib.tlin_scratch_bytes_forward_f32(*sizes)
    assert 0 < need <= 2 << 30
    g = torch.Generator(device=DEV).manual_seed(1)
    q, k, v = (torch.randn(B, H, rows, d, generator=g, device=DEV) for rows in (W, N, N))
    results = []
    for s in (scratch(need), None):
        out, lse = torch.empty_like(q), torch.empty(B, H, W, device=DEV)
        assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out, lse), *sizes, s.data_ptr() if s is not None else None, need if s is not None else 0, stream) == 0
        results.append((out, lse, tl.tlin_last_launch_count()))
    assert tl.tlin_get_status() == 0 and results[0][2] > 3
    scores = q.double() @ k.double().transpose(-1, -2) / math.sqrt(d)
    scores.masked_fill_(torch.arange(N, device=DEV)[None] > (N - W + torch.arange(W, device=DEV))[:, None], -math.inf)
    lse = torch.logsumexp(scores, -1)
    out = scores.sub_(lse[..., None]).exp_() @ v.double()
    for x, a, b in zip((out, lse), results[0], results[1]):      # as test_as_exact_as_the_cuda_cores
        assert float((a - x).norm()) <= max(1.2 * float((b - x).norm()), 4 * 2.0 ** -24 * float(x.norm()))


def forward_lse(q, k):
    """lse of the tensor cores for values that do not matter, and the 64-bit scores."""
    B, H, W, d = q.shape
    N, lib = k.shape[2], tl.lib()
    need = lib.tlin_scratch_bytes_forward_f32(B, H, N, W, d, 0)
    assert need > 0
    s, out, lse = scratch(need), torch.empty_like(q), torch.empty(B, H, W, device=DEV)
    assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, k, out, lse), B, H, N, W, d, 0, s.data_ptr(), need, torch.cuda.current_stream().cuda_stream) == 0
    assert tl.tlin_get_status() == 0
    return lse, q.double() @ k.double().transpose(-1, -2) / math.sqrt(d)


# what the tensor pipe cuts off a score is put back only where something was cut off: the mean of 7200 roundings to nearest is far below an
# eighth of 2^-24
@pytest.mark.parametrize("d", [36, 64, 100, 128])
@pytest.mark.parametrize("sign", [0, -1])
def test_lse_of_whole_scores(d, sign):
    q, k = (torch.randint(-8, 9, (2, 12, rows, d), generator=torch.Generator().manual_seed(rows)).float().to(DEV) for rows in (300, 1500))
    if sign:
        q, k = -q.abs(), k.abs()
    lse, scores = forward_lse(q, k)
    want = torch.logsumexp(scores, -1)
    assert abs(float(((lse - want) / want.abs()).mean())) <= 2.0 ** -27


# and it is put back in the direction it was cut, towards zero.  With products of one sign the partial sums of a score grow evenly over its
# n products of 16 columns, each cut by half of a last place, 2^-24.5 of it on average, at most: (n + 1) / 2 * 2^-24.5 of the
# score less the 0.94e-8 n that are put back
@pytest.mark.parametrize("d", [36, 64, 100, 128])
@pytest.mark.parametrize("sign", [1, -1])
def test_lse_of_scores_of_one_sign(d, sign):
    q, k = sign * normal(1, 2, 12, 300, d).abs(), normal(2, 2, 12, 1500, d).abs()
    lse, scores = forward_lse(q, k)
    want, n = torch.logsumexp(scores, -1), (d + 15) // 16
    size = float((torch.softmax(scores, -1) * scores.abs()).sum(-1).mean())
    assert abs(float((lse - want).mean())) <= ((n + 1) / 2 * 2.0 ** -24.5 - 0.94e-8 * n) * size


# ds is split into parts as well: gradients of the same accuracy wherever dout and v lie inside the range, here with products down to 2^-116
# (fp32 itself has less than 24 bits left below 2^-126).  dq of the CUDA cores is no measure there: their additions in memory flush to zero
@pytest.mark.parametrize("of_dout,of_v", [(-96, -20), (-90, -20), (-60, -50), (-96, 0), (19, 28), (0, 0)])
def test_gradients_at_the_ends_of_the_range(of_dout, of_v):
    B, H, N, W, d = 2, 12, 1500, 300, 36
    q, k, v, dout = normal(1, B, H, W, d), normal(2, B, H, N, d), normal(3, B, H, N, d), normal(4, B, H, W, d)
    v, dout = (t.sign() * t.abs().clamp(0.25, 2.0) * 2.0 ** e for t, e in ((v, of_v), (dout, of_dout - 1)))
    out, lse = forward(q, k, v, 1)
    got, cores = backward(q, k, v, out, lse, dout, 1), backward(q, k, v, out, lse, dout, 1, False)
    for x, a, b in zip(exact(q, k, v, dout, 1)[2:], got, cores):
        size = float(x.norm())
        assert float((a - x).norm()) <= max(min(1.2 * float((b - x).norm()), 2.0 ** -20 * size), 4 * 2.0 ** -24 * size)
    assert tl.tlin_get_status() == 0


def test_replay_of_a_capture():
    """PyTorch's captures keep the scratch for the graph: the tensor cores serve the call there too."""
    t = tensors(2, 16, 500, 300, 36)
    other = {x: normal(7 + i, *t[x].shape) for i, x in enumerate(t)}

    def call():
        out, lse = tl.tlin_attn_forward_f32(t["q"], t["k"], t["v"])
        return [out, lse] + list(tl.tlin_attn_backward_f32(t["q"], t["k"], t["v"], out, lse, t["dout"]))

    call()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        recorded = call()
    for values in (other, tensors(2, 16, 500, 300, 36)):
        for x in t:
            t[x].copy_(values[x])
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(recorded, call()))
    assert tl.tlin_get_status() == 0


def test_a_capture_that_pytorch_does_not_know_of_takes_no_scratch():
    """Its memory would be given out again while the graph still writes to it: the call is recorded on the CUDA cores."""
    rt = ctypes.CDLL("libcudart.so.12")
    t = tensors(2, 16, 500, 300, 36)
    q, k, v, dout = (t[x] for x in ("q", "k", "v", "dout"))
    stream = torch.cuda.Stream()
    out, lse, grads = torch.empty_like(q), torch.empty(2, 16, 300, device=DEV), [torch.empty_like(x) for x in (q, k, v)]
    need = max(tl.lib().tlin_scratch_bytes_forward_f32(2, 16, 500, 300, 36, 1), tl.lib().tlin_scratch_bytes_backward_f32(2, 16, 500, 300, 36, 1))

    def call():
        tl.tlin_attn_forward_f32(q, k, v, out, lse, stream=stream)
        tl.tlin_attn_backward_f32(q, k, v, out, lse, dout, *grads, stream=stream)

    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        call()
        torch.cuda.synchronize()
        handle, graph, run = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(handle, 1) == 0              # of this thread
        call()
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
        assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0
        taken = [torch.zeros(need, dtype=torch.uint8, device=DEV) for _ in range(4)]        # what the warm call's scratch left
        for x in [out, lse] + grads:
            x.zero_()
        assert rt.cudaGraphLaunch(run, handle) == 0
        torch.cuda.synchronize()
    assert rt.cudaGraphExecDestroy(run) == 0 and rt.cudaGraphDestroy(graph) == 0
    assert not any(bool(x.any()) for x in taken)
    want = forward(q, k, v, 1, False)
    assert torch.equal(out, want[0]) and torch.equal(lse, want[1])
    want = backward(q, k, v, *want, dout, 1, False)
    assert torch.equal(grads[1], want[1]) and torch.equal(grads[2], want[2])
    assert float((grads[0] - want[0]).double().norm()) <= 1e-6 * float(want[0].double().norm())
    assert tl.tlin_get_status() == 0


_LOGGED = """
import torch
from paper_2508_20407_b200 import binding as tl
for d, dtype in ((36, torch.float32), (100, torch.float32), (64, torch.bfloat16), (96, torch.bfloat16), (128, torch.bfloat16)):
    q, k, v = (torch.randn(2, 16, n, d, device="cuda").to(dtype).requires_grad_() for n in (300, 500, 500))
    tl.attention(q, k, v)[0].sum().backward()
torch.cuda.synchronize()
"""


def test_the_plan_log_names_every_call():
    r = subprocess.run([sys.executable, "-c", _LOGGED], capture_output=True, text=True, timeout=300, env=dict(os.environ, TLIN_LOG="1"),
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr
    lines = [line for line in r.stderr.splitlines() if line.startswith("libtlin:")]
    assert [("forward" in line, "backward" in line) for line in lines] == [(True, False), (False, True)] * 5, r.stderr
    assert "three bf16 parts" in lines[0] and "three bf16 parts" in lines[1] and "CUDA cores" in lines[3] and "CUDA cores" in lines[7]


def test_calls_in_several_launches_whose_results_lie_over_inputs():
    """They go to the CUDA cores with nothing launched before."""
    B, H, N, W, d = 2, 160, 2000, 2000, 36
    t = tensors(B, H, N, W, d)
    q, k, v, dout = (t[x] for x in ("q", "k", "v", "dout"))
    assert tl.lib().tlin_scratch_bytes_forward_f32(B, H, N, W, d, 1) and tl.lib().tlin_scratch_bytes_backward_f32(B, H, N, W, d, 1)
    out, lse = forward(q, k, v, 1, False)
    over = q.clone()
    got = forward(over, k, v, 1, out=over)
    assert tl.tlin_last_launch_count() == 1 and torch.equal(got[0], out) and torch.equal(got[1], lse)
    want = backward(q, k, v, out, lse, dout, 1, False)
    launches = tl.tlin_last_launch_count()
    over = k.clone()
    dq, dk, dv = backward(q, over, v, out, lse, dout, 1, grads=[torch.empty_like(q), over, torch.empty_like(v)])
    assert tl.tlin_last_launch_count() == launches and torch.equal(dk, want[1]) and torch.equal(dv, want[2])
    assert float((dq - want[0]).double().norm()) <= 1e-6 * float(want[0].double().norm())          # summed in any order
    assert tl.tlin_get_status() == 0


def test_two_streams_at_once():
    sizes = [(2, 16, 500, 300, 36), (1, 12, 1500, 513, 64)]
    inputs = [tensors(*s) for s in sizes]

    def call(t):
        out, lse = tl.tlin_attn_forward_f32(t["q"], t["k"], t["v"])
        return [out, lse] + list(tl.tlin_attn_backward_f32(t["q"], t["k"], t["v"], out, lse, t["dout"]))

    want = [call(t) for t in inputs]
    torch.cuda.synchronize()
    streams, got = [torch.cuda.Stream(), torch.cuda.Stream()], []
    for _ in range(10):
        for s, t in zip(streams, inputs):
            with torch.cuda.stream(s):
                got.append(call(t))
    torch.cuda.synchronize()
    for i, results in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(results, want[i % 2]))
    assert tl.tlin_get_status() == 0


# in a cluster, in several launches, at one d8 beyond d, with more (b,h) than blocks of the split; some of them with a head for the CUDA cores
@pytest.mark.parametrize("B,H,N,W,d,special", [(1, 3, 3000, 200, 64, True), (2, 160, 2000, 300, 64, True), (1, 5, 2100, 640, 68, False), (8, 32, 520, 512, 20, False),
                                               (2, 500, 256, 200, 16, True), (2, 16, 385, 129, 36, True)])
def test_scratch_of_the_documented_size_between_guards(B, H, N, W, d, special):
    """Nothing is written beyond it and nothing in it is read before it is written: it starts as NaNs, and words that are set."""
    t = tensors(B, H, N, W, d)
    if special:
        t["v"][B - 1, H - 1, N // 2, 1] = math.inf
    q, k, v, dout = (t[x] for x in ("q", "k", "v", "dout"))
    lib, sizes, stream = tl.lib(), (B, H, N, W, d, 0), torch.cuda.current_stream().cuda_stream
    if lib.tlin_scratch_bytes_forward_f32(*sizes):
        want = forward(q, k, v, 0)
        s, out, lse = Guarded((lib.tlin_scratch_bytes_forward_f32(*sizes),), torch.uint8), torch.empty_like(q), torch.empty(B, H, W, device=DEV)
        assert lib.tlin_attn_forward_f32_scratch(*pointers(q, k, v, out, lse), *sizes, s.t.data_ptr(), s.nbytes, stream) == 0
        s.check("forward")
        assert same(out, want[0]) and same(lse, want[1])
    else:
        out, lse = tl.tlin_attn_forward_f32(q, k, v, causal_window=0)
    if lib.tlin_scratch_bytes_backward_f32(*sizes):
        want = backward(q, k, v, out, lse, dout, 0)
        s, grads = Guarded((lib.tlin_scratch_bytes_backward_f32(*sizes),), torch.uint8), [torch.empty_like(x) for x in (q, k, v)]
        assert lib.tlin_attn_backward_f32_scratch(*pointers(q, k, v, out, lse, dout, *grads), *sizes, s.t.data_ptr(), s.nbytes, stream) == 0
        s.check("backward")
        assert same(grads[1], want[1]) and same(grads[2], want[2])
        ok = torch.isfinite(want[0])                   # dq of several additions in any order
        assert torch.equal(torch.isfinite(grads[0]), ok)
        assert float((grads[0] - want[0])[ok].double().norm()) <= 1e-6 * float(want[0][ok].double().norm())
    assert tl.tlin_get_status() == 0
