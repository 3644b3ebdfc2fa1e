"""lse against 64-bit arithmetic where P is kept to more than 8 bits: the kernels add no rounding that an fp32 value does not have."""
import pytest
import torch

from paper_2508_20407_b200 import binding as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"
EPS = 2.0 ** -24            # largest relative error of one rounding to fp32


def normal(seed, *shape):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return torch.randn(*shape, generator=g).to(torch.bfloat16).to(DEV)


def off_by(lse, scores):
    """Norm of the error over the norm of the value."""
    exact = torch.logsumexp(scores, -1)
    return float((lse.double() - exact).norm() / exact.norm())


# Rounding the result alone is off by EPS / sqrt(3) = 3.4e-8 at most (uniform over half a last place, at the lower end of a binade), and
# by 0.58 of that on the average over a binade; the sum of the exponentials (2 last places each, of random sign), its logarithm and the
# reference's part add less than another EPS / 3 here.  The two roundings of a sum in base-2 units, 1.44 times as large, come to 4.7e-8.
@pytest.mark.parametrize("B,H,N,W,d", [(8, 16, 561, 94, 96), (1, 4, 529, 106, 80), (8, 8, 300, 300, 40), (16, 16, 700, 260, 32), (2, 9, 3001, 517, 96)])
def test_forward_at_other_head_sizes(B, H, N, W, d):
    q, k, v = normal(1, B, H, W, d), normal(2, B, H, N, d), normal(3, B, H, N, d)
    _, lse = tl.tlin_attn_forward(q, k, v, causal_window=0)
    assert off_by(lse, q.double() @ k.double().transpose(2, 3) / d ** 0.5) <= 0.67 * EPS


@pytest.mark.parametrize("B,H,pos,d", [(8, 16, 600, 64), (8, 16, 600, 128), (4, 32, 360, 128), (6, 12, 1777, 64)])
def test_decode_step(B, H, pos, d):
    q, kn, vn = normal(1, B, H, 1, d), normal(2, B, H, 1, d), normal(3, B, H, 1, d)
    kc, vc = normal(4, B, H, pos + 1, d), normal(5, B, H, pos + 1, d)
    _, lse = tl.tlin_decode_step(q, kn, vn, kc, vc, pos)
    assert off_by(lse, (q.double() @ kc.double().transpose(2, 3) / d ** 0.5)[..., 0, :]) <= 0.67 * EPS
