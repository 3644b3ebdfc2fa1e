"""Wrong arguments of the binding are the caller's ValueError, TypeError or IndexError, with or without a device: the tensors are
looked at before a stream is asked for."""
import pytest
import torch

from paper_2508_20407_b200 import binding as tl

BF = torch.zeros(1, 2, 8, 64, dtype=torch.bfloat16)
F32 = BF.float()
ROW = BF[:, :, :1]
LSE = torch.zeros(1, 2, 8)
ENTRY = (BF, BF, BF, BF, None, None, 1)

CPU_TENSORS = {
    "forward": lambda: tl.tlin_attn_forward(BF, BF, BF),
    "forward, causal_window as a float": lambda: tl.tlin_attn_forward(BF, BF, BF, causal_window=1.0),
    "forward_f32": lambda: tl.tlin_attn_forward_f32(F32, F32, F32),
    "forward_cache": lambda: tl.tlin_attn_forward_cache(BF, BF, BF, 4),
    "backward": lambda: tl.tlin_attn_backward(BF, BF, BF, BF, LSE, BF),
    "backward_f32": lambda: tl.tlin_attn_backward_f32(F32, F32, F32, F32, LSE, F32),
    "attention": lambda: tl.attention(BF, BF, BF),
    "attention, with gradients": lambda: tl.attention(BF.clone().requires_grad_(), BF, BF),
    "decode": lambda: tl.tlin_decode_step(ROW, ROW, ROW, BF, BF, 3),
    "table": lambda: tl.tlin_attn_forward_batched([ENTRY]),
    "table, entries of another kind": lambda: tl.tlin_attn_forward_batched([iter(ENTRY), list(ENTRY)]),
}


@pytest.mark.parametrize("call", CPU_TENSORS.values(), ids=CPU_TENSORS.keys())
def test_cpu_tensors_are_a_value_error(call):
    with pytest.raises(ValueError, match="CUDA tensor"):
        call()


def test_other_wrong_arguments():
    for call in (lambda: tl.tlin_attn_forward(BF[0], BF, BF), lambda: tl.tlin_attn_backward(BF[0], BF, BF, BF, LSE, BF), lambda: tl.attention(BF, BF[0], BF)):
        with pytest.raises(ValueError):
            call()
    with pytest.raises(IndexError):
        tl.tlin_attn_forward_batched([])
    with pytest.raises(ValueError, match="expected"):
        tl.tlin_attn_forward_batched([ENTRY[:6]])
    with pytest.raises(TypeError):
        tl.tlin_attn_forward_batched(x for x in [ENTRY])


def test_transforms_that_pass_an_autograd_function_by_are_refused():
    x = torch.zeros(2, 1, 2, 8, 64)
    with pytest.raises(RuntimeError):
        torch.vmap(lambda t: tl.attention(t, t, t)[0])(x)
    with pytest.raises(RuntimeError):
        torch.func.grad(lambda t: tl.attention(t, t, t)[0].sum())(x[0])
