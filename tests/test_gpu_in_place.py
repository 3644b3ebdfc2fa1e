"""Results written over an input that the call has no further use for (the C ABI borrows buffers and says nothing against it)."""
import pytest
import torch

from paper_2508_20407_b200 import binding as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,H,N,W,d,dtype", [(2, 4, 700, 300, 36, torch.float32), (1, 3, 260, 130, 128, torch.float32), (1, 2, 200, 200, 192, torch.float32),
                                             (2, 4, 700, 300, 96, torch.bfloat16), (2, 4, 700, 300, 64, torch.bfloat16), (2, 4, 700, 300, 128, torch.bfloat16)])
def test_dq_over_q_dout_or_out(B, H, N, W, d, dtype):
    g = torch.Generator(device="cpu").manual_seed(d + N)
    q, k, v, dout = (torch.randn(B, H, rows, d, generator=g).to(dtype).to(DEV) for rows in (W, N, N, W))
    f32 = dtype == torch.float32
    out, lse = (tl.tlin_attn_forward_f32 if f32 else tl.tlin_attn_forward)(q, k, v)
    backward = tl.tlin_attn_backward_f32 if f32 else tl.tlin_attn_backward
    want = backward(q, k, v, out, lse, dout)
    # dq is a sum of up to N fp32 terms added in any order, then rounded to the result's type
    bound = (N * 2.0 ** -24 + (0 if f32 else 2.0 ** -8)) * float(want[0].float().abs().max())
    for over in range(3):
        args = [q.clone(), k, v, out.clone(), lse, dout.clone()]
        got = backward(*args, dq=(args[0], args[3], args[5])[over])
        assert tl.tlin_get_status() == 0
        assert float((got[0].float() - want[0].float()).abs().max()) <= bound
        assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
