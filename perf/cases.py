"""What is timed: the attention calls a user of this library makes, through ``paper_2508_20407_b200.binding``.

The sizes are the library's own workloads (``synth.WORKLOADS``), the shapes of its tests, and what lies around them:
the smallest calls, where launches count, up to 131072 keys; head sizes 64 and 128 as well as the others; bf16, fp32 and
the 8-bit cache; ragged lengths; forward, forward plus backward, and the cached step.
"""
import math

import torch

from paper_2508_20407_b200 import binding as tl

DEV = "cuda"


def listed():
    return [
        # one short window over a short history: the first token of a small model, where launches are what counts
        dict(name="forward_tiny", kind="forward", dtype="bf16", B=1, H=4, N=1024, W=128, d=64, causal=1, cap=0, peaky=0),
        # a batch of middle-sized windows, head size 64
        dict(name="forward_mid", kind="forward", dtype="bf16", B=4, H=16, N=8192, W=256, d=64, causal=1, cap=0, peaky=0),
        # long history, a few dominant keys (attention sinks), recomputed in place over a decode cache after the window slid
        dict(name="forward_long_cache", kind="forward", dtype="bf16", B=1, H=32, N=32768, W=512, d=128, causal=1, cap=33024, peaky=1),
        # very long history: the summary queries and the window of the first token
        dict(name="forward_vlong", kind="forward", dtype="bf16", B=1, H=32, N=131072, W=1024, d=128, causal=1, cap=0, peaky=0),
        # another head size at ragged lengths: summary queries over a finished history (no mask)
        dict(name="forward_d96_ragged", kind="forward", dtype="bf16", B=2, H=9, N=3001, W=517, d=96, causal=0, cap=0, peaky=0),
        # the two inner layers (summary self-attention, window over [summary; window]) of four requests as one table
        dict(name="inner_table", kind="table", dtype="bf16", R=4, H=8, Ws=1024, Wg=1024, d=128),
        # short caches of different lengths in one served batch
        dict(name="decode_ragged_short", kind="decode", dtype="bf16", B=6, H=12, cap=2048, pos=1777, d=64, ragged=1),
        # one token over a long cache
        dict(name="decode_long", kind="decode", dtype="bf16", B=8, H=32, cap=65792, pos=65536, d=128, ragged=0),
        # the same step over an 8-bit cache, a smaller batch
        dict(name="decode_fp8", kind="decode", dtype="fp8", B=4, H=32, cap=16384, pos=15001, d=128, ragged=0),
        # training step (forward and backward) of the last window of a sliding-window pass
        dict(name="train_chunk", kind="train", dtype="bf16", B=4, H=32, N=8192, W=1024, d=128, causal=1),
        # training step at head size 64, ragged lengths, the whole sequence as one window
        dict(name="train_d64_ragged", kind="train", dtype="bf16", B=3, H=12, N=1999, W=1999, d=64, causal=1),
        # training step of the small fp32 model: 12 heads of size 36, 512-token windows over 1024 tokens
        dict(name="train_f32_d36", kind="train", dtype="f32", B=8, H=12, N=1024, W=512, d=36, causal=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["forward", "forward", "forward", "forward_other", "table", "decode", "decode", "train", "train", "train_f32"])
    if kind in ("forward", "train"):
        most = 1.5e12 if kind == "forward" else 6e11          # multiply-adds times two, kept below the largest listed case
        while True:
            c = dict(kind=kind, dtype="bf16", B=rng.choice([1, 1, 2, 3, 4, 8]), H=rng.choice([2, 4, 8, 12, 16, 32]),
                     N=_log_int(rng, 200, 131072 if kind == "forward" else 16384), W=_log_int(rng, 64, 4096), d=rng.choice([64, 128]),
                     causal=rng.choice([0, 1, 1]))
            c["W"] = min(c["W"], c["N"])
            if work(c)["flops"] <= most and c["B"] * c["H"] * c["N"] * c["d"] <= 1 << 29:
                break
        if kind == "forward":
            c["cap"] = c["N"] + rng.randrange(1, 300) if rng.random() < 0.3 else 0
            c["peaky"] = int(rng.random() < 0.3)
        return c
    if kind in ("forward_other", "train_f32"):
        f32 = kind == "train_f32"
        while True:
            c = dict(kind="train" if f32 else "forward", dtype="f32" if f32 else "bf16", B=rng.choice([1, 2, 4, 8]),
                     H=rng.choice([3, 4, 9, 12, 16]), N=_log_int(rng, 200, 8192), W=_log_int(rng, 64, 1024),
                     d=rng.choice([36, 64, 100, 128]) if f32 else rng.choice([32, 40, 80, 96, 112, 160, 256]), causal=rng.choice([0, 1, 1]))
            c["W"] = min(c["W"], c["N"])
            if work(c)["flops"] <= (1.8e10 if f32 else 1.2e10):
                break
        if not f32:
            c["cap"], c["peaky"] = 0, 0
        return c
    if kind == "table":
        return dict(kind="table", dtype="bf16", R=rng.randrange(1, 9), H=rng.choice([4, 8, 12, 16]), Ws=_log_int(rng, 128, 1024),
                    Wg=_log_int(rng, 128, 1024), d=rng.choice([64, 128]))
    while True:
        c = dict(kind="decode", dtype=rng.choice(["bf16", "bf16", "fp8"]), B=rng.choice([1, 2, 3, 4, 8, 16]), H=rng.choice([4, 8, 12, 16, 32]),
                 cap=_log_int(rng, 300, 65536), d=rng.choice([64, 128]), ragged=0)
        c["pos"] = rng.randrange(c["cap"] // 2, c["cap"])
        if c["dtype"] == "bf16":
            c["ragged"] = rng.choice([0, 1])
        if c["B"] * c["H"] * c["cap"] * c["d"] <= 1 << 30:
            return c


def _lengths(case):
    """Valid rows of every sequence before the step (ragged: between half of the longest and the longest)."""
    B, pos = case["B"], case["pos"]
    if not case["ragged"]:
        return [pos] * B
    return [pos - (b * 7919 % (pos // 2 + 1)) for b in range(B)]


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def normal(*shape, dtype=torch.bfloat16):
        return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)

    if case["kind"] == "forward":
        B, H, N, W, d = (case[k] for k in ("B", "H", "N", "W", "d"))
        rows = case["cap"] or N
        q, k, v = normal(B, H, W, d), normal(B, H, rows, d), normal(B, H, rows, d)
        if case["peaky"]:                                      # 1 % of the key rows are eight times as large
            k *= torch.where(torch.rand(B, H, rows, 1, generator=g, device=DEV) < 0.01, 8.0, 1.0).to(k.dtype)
        return dict(case=case, q=q, k=k, v=v)
    if case["kind"] == "table":
        R, H, Ws, Wg, d = (case[k] for k in ("R", "H", "Ws", "Wg", "d"))
        problems, outs = [], []
        for _ in range(R):
            for W, N, causal in ((Ws, Ws, 0), (Wg, Ws + Wg, 1)):
                q, k, v = normal(1, H, W, d), normal(1, H, N, d), normal(1, H, N, d)
                out, lse = torch.empty_like(q), torch.empty(1, H, W, device=DEV)
                problems.append((q, k, v, out, lse, N, causal))
                outs += [out, lse]
        return dict(case=case, problems=problems, outs=outs)
    if case["kind"] == "decode":
        B, H, cap, d = (case[k] for k in ("B", "H", "cap", "d"))
        s = dict(case=case, q=normal(B, H, 1, d), k_new=normal(B, H, 1, d), v_new=normal(B, H, 1, d))
        if case["dtype"] == "fp8":
            # codes of normal values at a scale that maps 4 standard deviations to the format's largest value
            for name in ("k", "v"):
                x = torch.empty(B, H, cap, d, dtype=torch.uint8, device=DEV)
                for b in range(B):
                    x[b] = (normal(H, cap, d) * (448.0 / 4.0)).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
                s[name] = x
                s[name + "_scale"] = torch.full((B, H), 4.0 / 448.0, device=DEV)
        else:
            s["k"], s["v"] = normal(B, H, cap, d), normal(B, H, cap, d)
        if case["ragged"]:
            s["pos"] = torch.tensor(_lengths(case), dtype=torch.int32, device=DEV)
        return s
    B, H, N, W, d = (case[k] for k in ("B", "H", "N", "W", "d"))
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    q, k, v = (normal(B, H, rows, d, dtype=dtype).requires_grad_() for rows in (W, N, N))
    return dict(case=case, q=q, k=k, v=v, dout=normal(B, H, W, d, dtype=dtype))


def run(state):
    c = state["case"]
    if c["kind"] == "forward":
        if c["cap"]:
            return tl.tlin_attn_forward_cache(state["q"], state["k"], state["v"], c["N"], causal_window=c["causal"])
        return tl.tlin_attn_forward(state["q"], state["k"], state["v"], causal_window=c["causal"])
    if c["kind"] == "table":
        tl.tlin_attn_forward_batched(state["problems"])
        return state["outs"]
    if c["kind"] == "decode":
        args = (state["q"], state["k_new"], state["v_new"], state["k"], state["v"])
        if c["dtype"] == "fp8":
            out, lse = tl.tlin_decode_step_fp8(*args, state["k_scale"], state["v_scale"], c["pos"])
        elif c["ragged"]:
            out, lse = tl.tlin_decode_step_ragged(*args, state["pos"], c["pos"])
        else:
            out, lse = tl.tlin_decode_step(*args, c["pos"])
        return out, lse, state["k"], state["v"]
    # one training step's attention: the loss gradient of `out` comes from the layers above
    q, k, v = state["q"], state["k"], state["v"]
    out, lse = tl.attention(q, k, v, c["causal"])
    dq, dk, dv = torch.autograd.grad(out, (q, k, v), state["dout"])
    return out.detach(), lse, dq, dk, dv


def _pairs(N, W, causal):
    return W * (N - W) + W * (W + 1) // 2 if causal else W * N


def work(case):
    d = case["d"]
    if case["kind"] == "table":
        R, H, Ws, Wg = (case[k] for k in ("R", "H", "Ws", "Wg"))
        pairs = _pairs(Ws, Ws, 0) + _pairs(Ws + Wg, Wg, 1)
        rows = (2 * Ws + 2 * Ws) + (2 * Wg + 2 * (Ws + Wg))                     # q and out, k and v of both layers
        return {"bytes": R * H * (rows * d * 2 + (Ws + Wg) * 4), "flops": 4 * d * R * H * pairs}
    if case["kind"] == "decode":
        B, H = case["B"], case["H"]
        size = 1 if case["dtype"] == "fp8" else 2
        cached, attended = sum(_lengths(case)), sum(_lengths(case)) + B
        new = B * H * (4 * d * 2 + 2 * d * size + 4)                            # q, k, v, out; the two appended rows; lse
        return {"bytes": 2 * H * cached * d * size + new, "flops": 4 * d * H * attended}
    B, H, N, W = (case[k] for k in ("B", "H", "N", "W"))
    size = 4 if case["dtype"] == "f32" else 2
    pairs = B * H * _pairs(N, W, case["causal"])
    if case["kind"] == "forward":
        return {"bytes": B * H * ((2 * W + 2 * N) * d * size + W * 4), "flops": 4 * d * pairs}
    # q, k, v, dout in; out, lse, dq, dk, dv out; two products forward and five backward
    return {"bytes": B * H * ((4 * W + 4 * N) * d * size + W * 4), "flops": 14 * d * pairs}


def tolerance(case):
    # about four times what the path differs by from the same computation in 64 bits: 1.6e-3 to 2.5e-3 in bf16 (and with the
    # 8-bit cache, whose codes are exact), 6e-7 in fp32 at the listed sizes, somewhat more over the longer sums of the range
    return {"rel": 5e-6 if case["dtype"] == "f32" else 1e-2}
