"""Values at the ends of the formats through every form of the kernels: a NaN reaches what depends on it and nothing else."""
import pytest
import torch

from paper_2508_20407_b200 import binding as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"
NAN, INF = float("nan"), float("inf")


def normal(seed, *shape, dtype=torch.bfloat16):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return torch.randn(*shape, generator=g).to(dtype).to(DEV)


def forward(q, k, v, causal):
    fn = tl.tlin_attn_forward_f32 if q.dtype == torch.float32 else tl.tlin_attn_forward
    out, lse = fn(q, k, v, causal_window=causal)
    assert tl.tlin_get_status() == 0
    return out, lse


# keys shared in a cluster, split and merged by a second kernel (few and many parts), whole problems, one key tile
FORMS = [(1, 4, 1024, 128), (5, 16, 2048, 256), (1, 2, 60000, 64), (8, 16, 512, 300), (2, 3, 100, 60)]


@pytest.mark.parametrize("d,dtype", [(64, torch.bfloat16), (128, torch.bfloat16), (96, torch.bfloat16), (160, torch.bfloat16), (36, torch.float32)])
@pytest.mark.parametrize("B,H,N,W", FORMS)
def test_forward_passes_a_nan_on(B, H, N, W, d, dtype):
    q, k, v = normal(1, B, H, W, d, dtype=dtype), normal(2, B, H, N, d, dtype=dtype), normal(3, B, H, N, d, dtype=dtype)
    clean = forward(q, k, v, 0)
    assert all(bool(torch.isfinite(t).all()) for t in clean)
    hit = (B - 1, H - 1)

    def check(got, rows, with_lse):
        for t, ref, depends in zip(got, clean, (True, with_lse)):
            t, ref = t.clone(), ref.clone()
            if depends:
                assert bool(t[hit][rows].isnan().all())
                t[hit][rows] = ref[hit][rows] = 0
            assert torch.equal(t, ref)

    # single keys in columns that every form gives to the special-function unit: the cubic that d = 64 and 128 use for some of the
    # others takes a NaN for the lower end of its range, and that key then counts for nothing
    everywhere = slice(None)
    for keys in (slice(3, 4), slice(N // 10, N * 9 // 10), slice((N - 1) // 32 * 32, (N - 1) // 32 * 32 + 1)):
        bad = k.clone()
        bad[hit][keys] = NAN                        # every row's sum
        check(forward(q, bad, v, 0), everywhere, True)
        bad = v.clone()
        bad[hit][keys] = NAN                        # every row's result, not its sum
        check(forward(q, k, bad, 0), everywhere, False)
    bad = q.clone()
    bad[hit][W // 2] = NAN
    check(forward(bad, k, v, 0), slice(W // 2, W // 2 + 1), True)


# a score of -inf masks a key (an extra column of q at 1, of k at -inf); with every key masked there is nothing to attend to
@pytest.mark.parametrize("d", [36, 64])
@pytest.mark.parametrize("B,H,N,W", [(1, 4, 1024, 128), (8, 16, 512, 300)])
def test_fp32_rows_without_a_finite_score_have_a_sum_of_nothing(B, H, N, W, d):
    q, k, v = (normal(i, B, H, rows, d, dtype=torch.float32) for i, rows in enumerate((W, N, N)))
    q[..., 0] = 1
    k[..., 0] = -INF
    _, lse = forward(q, k, v, 0)
    assert bool((lse == -INF).all())
    k[:, :, N // 2:, 0] = 0                         # half of the keys are back, in the second shares only
    out, lse = forward(q, k, v, 0)
    alone, lse_alone = forward(q, k[:, :, N // 2:].contiguous(), v[:, :, N // 2:].contiguous(), 0)
    assert float((out - alone).abs().max()) <= 1e-5 and float((lse - lse_alone).abs().max()) <= 1e-5


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,pos", [(2, 4, 600), (2, 16, 1401), (1, 1, 30), (64, 32, 300), (4, 32, 8000)])
def test_decode_step_with_masked_scores(B, H, pos, d):
    q, kn, vn = normal(1, B, H, 1, d), normal(2, B, H, 1, d), normal(3, B, H, 1, d)
    kc, vc = normal(4, B, H, pos + 3, d), normal(5, B, H, pos + 3, d)
    q[..., 0] = 1
    kc[..., 0] = -INF
    kn[..., 0] = -INF
    at = torch.full((B,), pos, dtype=torch.int32, device=DEV)
    for out, lse in (tl.tlin_decode_step(q, kn, vn, kc, vc, pos), tl.tlin_decode_step_ragged(q, kn, vn, kc, vc, at, pos)):
        assert float(out.float().abs().max()) == 0.0 and bool((lse == -INF).all())
    kn[..., 0] = 0                                  # only the new row counts: the step returns its value
    for out, lse in (tl.tlin_decode_step(q, kn, vn, kc, vc, pos), tl.tlin_decode_step_ragged(q, kn, vn, kc, vc, at, pos)):
        assert torch.equal(out, vn)
        want = (q.float() * kn.float()).sum(-1)[..., 0] / d ** 0.5
        assert float((lse - want).abs().max()) <= 1e-5
    assert tl.tlin_get_status() == 0


# scores far beyond anything that a model has, as from keys masked with the lowest finite value instead of -inf: the forms that keep P
# beyond 8 bits (fp32, and bf16 at head sizes other than 64 and 128) stay exact there.  Forms: clusters, split and merged, whole
@pytest.mark.parametrize("d,dtype", [(40, torch.bfloat16), (96, torch.bfloat16), (160, torch.bfloat16), (36, torch.float32), (128, torch.float32)])
@pytest.mark.parametrize("B,H,N,W", [(1, 4, 1024, 128), (1, 2, 20000, 64), (8, 16, 512, 300), (2, 3, 100, 60)])
def test_scores_of_any_finite_size(B, H, N, W, d, dtype):
    q, k, v = (normal(i, B, H, rows, d, dtype=dtype) for i, rows in enumerate((W, N, N)))
    q[..., 0], k[..., 0] = 1, 0
    lowest = torch.finfo(torch.bfloat16).min
    tol = 2e-2 if dtype == torch.bfloat16 else 1e-4
    half = N // 2
    masked = k.clone()
    masked[:, :, :half, 0] = lowest
    out, lse = forward(q, masked, v, 0)
    alone, lse_alone = forward(q, k[:, :, half:].contiguous(), v[:, :, half:].contiguous(), 0)
    assert float((out.float() - alone.float()).abs().max()) <= tol and float((lse - lse_alone).abs().max()) <= 1e-4
    masked[..., 0] = lowest                         # every key alike: their mean
    out, lse = forward(q, masked, v, 0)
    mean = v.float().mean(2, keepdim=True)
    assert float((out.float() - mean).abs().max()) <= tol / 2 and bool(torch.isfinite(lse).all())
    huge = (k.float() * 1e12).to(dtype)             # one key takes all
    out, _ = forward(q, huge, v, 0)
    best = (q.double() @ huge.double().transpose(2, 3)).argmax(3)
    assert torch.equal(out, torch.gather(v, 2, best[..., None].expand(-1, -1, -1, d)))
