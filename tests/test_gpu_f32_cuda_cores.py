"""fp32 on the CUDA cores, which serve small calls, calls without scratch and the (b,h) that the tensor cores leave to them: the fp32 cases of the forward
and the backward tests, which the library's own choice takes to the tensor cores, and the sizes of the tensor tests against 64 bits."""
import pytest
import torch

import test_gpu_backward as bwd
import test_gpu_f32_tensor as tensor
import test_gpu_forward as fwd
from paper_2508_20407_b200 import binding as tl
from paper_2508_20407_b200 import synth

pytestmark = pytest.mark.gpu


def cases(test):
    return [m for m in test.pytestmark if m.name == "parametrize"][0].args[1]


@pytest.fixture
def cuda_cores():
    prev = tl.tlin_set_forward_impl(1)
    assert tl.lib().tlin_scratch_bytes_forward_f32(8, 12, 1024, 512, 36, 1) == 0 and tl.lib().tlin_scratch_bytes_backward_f32(8, 12, 1024, 512, 36, 1) == 0
    yield
    tl.tlin_set_forward_impl(prev)


@pytest.mark.parametrize("B,H,N,W,d,causal", cases(fwd.test_fp32_path) + cases(fwd.test_fp32_tilings_and_key_sharing_clusters))
def test_forward(B, H, N, W, d, causal):
    fwd.full_compare(synth.Workload("f32 tiles", B, H, d, N, W, seed=40 + N + d, causal_window=causal), 1, kind="f32")


@pytest.mark.parametrize("B,H,N,W,d,causal", cases(bwd.test_backward_f32))
def test_backward(cuda_cores, B, H, N, W, d, causal):
    bwd.test_backward_f32(B, H, N, W, d, causal)


# the other side of test_as_exact_as_the_cuda_cores, and small heads, whose products take one or two MMAs of 16 columns.  A score is a chain of up to 128
# roundings, off by about 8 of 2^-24 of its size with what is done to it after, and a sum of n results rounds n times, a random walk
SMALL_HEADS = [(4, 32, 1100, 257, 8, 1), (1, 8, 3000, 513, 16, 1), (8, 32, 520, 512, 20, 0), (1, 64, 300, 200, 32, 1), (2, 64, 700, 385, 32, 1)]


@pytest.mark.parametrize("B,H,N,W,d,causal", tensor.SHAPES + SMALL_HEADS)
def test_both_sides_against_64_bits(B, H, N, W, d, causal):
    q, dout, k, v = tensor.normal(1, B, H, W, d), tensor.normal(2, B, H, W, d), tensor.normal(3, B, H, N, d), tensor.normal(4, B, H, N, d)
    (got, on_tensor_fwd, on_tensor_bwd), (ref, *on_cores) = tensor.both_sides(q, k, v, dout, causal)
    assert on_cores == [False, False] and on_tensor_fwd
    assert on_tensor_bwd == (d <= 64 and (d, W) not in [(20, 127), (4, 200)])
    for a, b, x in zip(got, ref, tensor.exact(q, k, v, dout, causal)):
        bound = 2.0 ** -24 * (8 + 0.3 * max(N, W) ** 0.5) * float(x.norm())
        assert float((a - x).norm()) <= bound and float((b - x).norm()) <= bound
