"""Forward calls of few query rows, or few keys, over many (b,h): one warp per row on the CUDA cores."""
import pytest
import torch

import oracle
import parity
from guards import Guarded
from paper_2508_20407_b200 import binding as tl
from paper_2508_20407_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"

# B, H, N, W, d, causal: one row and the ends of a CTA's eight, one key and the ends of a step's 32, columns below, at and beyond a
# warp's width, both masks; sizes at which the rows are several times cheaper than the tiles
FP32 = [(50, 40, 1, 1, 64, 1), (50, 40, 33, 1, 4, 0), (50, 40, 31, 7, 36, 1), (50, 32, 32, 8, 64, 1), (25, 32, 70, 9, 100, 1), (50, 40, 9, 9, 128, 1),
        (25, 40, 130, 3, 132, 0), (50, 32, 40, 4, 256, 1), (2, 8, 8, 8, 256, 0), (2, 8, 20, 30, 192, 0)]
BF16 = [(50, 40, 1, 1, 8, 1), (50, 40, 33, 3, 40, 0), (50, 32, 32, 8, 96, 1), (50, 40, 9, 9, 112, 1), (50, 40, 20, 2, 136, 0), (25, 40, 12, 4, 256, 1)]


def compare(wl, dtype, gate):
    q, k, v = synth.forward_inputs(wl, device=DEV, dtype=dtype)
    out, lse = Guarded(q.shape, dtype, DEV), Guarded((wl.B, wl.H, wl.W), torch.float32, DEV)
    fn = tl.tlin_attn_forward_f32 if dtype == torch.float32 else tl.tlin_attn_forward
    fn(q, k, v, out.t, lse.t, causal_window=wl.causal_window)
    torch.cuda.synchronize()
    assert tl.tlin_get_status() == 0 and tl.tlin_last_launch_count() == 1
    out.check("out")
    lse.check("lse")
    ref, ref_lse = oracle.attn_forward(q.cpu(), k.cpu(), v.cpu(), wl.causal_window)
    parity.check(out.t.float().cpu().numpy(), lse.t.cpu().numpy(), ref, ref_lse, gate, wl.name)
    return q, k, v, out.t, lse.t


@pytest.mark.parametrize("B,H,N,W,d,causal", FP32)
def test_fp32(B, H, N, W, d, causal):
    compare(synth.Workload("few rows", B, H, d, N, W, seed=7 + N + W, causal_window=causal), torch.float32, "f32")


@pytest.mark.parametrize("B,H,N,W,d,causal", BF16)
def test_bf16_at_other_head_sizes(B, H, N, W, d, causal):
    assert tl.tlin_plan_forward(B, H, N, W, d, causal).tensor_path == 0
    q, k, v, out, lse = compare(synth.Workload("few rows", B, H, d, N, W, seed=9 + N + W, causal_window=causal), torch.bfloat16, "bf16")
    # the first N rows of a longer cache, whose other rows are not read
    pad = torch.full((B, H, 5, d), float("nan"), dtype=torch.bfloat16, device=DEV)
    again, lse_again = tl.tlin_attn_forward_cache(q, torch.cat([k, pad], 2), torch.cat([v, pad], 2), N, causal_window=causal)
    assert tl.tlin_get_status() == 0 and torch.equal(out, again) and torch.equal(lse, lse_again)
