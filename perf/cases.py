"""Workloads of the attention-JVP path: what its users have it do, through the package's binding.

The path runs inside the attention layers of a diffusion transformer in training: the forward carries a tangent next
to the primal, the backward differentiates through both, and the QK normalisation in front of the attention does
the same.  Sizes are the ones of `paper_2511_19797_b200.inputs.WORKLOADS` (stand-ins for DiT-XL/2 layers on 256- and
512-pixel latents, a large-head model, the sequence sweep) and of the layout tests; bf16 throughout, which is the
training precision (the fp32 kernels are a checking aid).

A case: op    "fwd" | "bwd" | "step" (forward, then backward, as one training step of a layer calls them)
              | "bwd_detach" (backward for a loss that does not use the tangent output) | "norm_fwd" | "norm_bwd"
        B, H  batch and heads;  M queries against N keys;  d head dimension
        layout  "packed" (B, H, rows, d) or "token" (B, rows, H, d), the layout a projection leaves
        peaky   share of the rows of Q and K scaled by 4 (sharp softmax rows of a trained model)
"""
import math

import torch

from paper_2511_19797_b200 import binding

OPS = ("fwd", "bwd", "step", "bwd_detach", "norm_fwd", "norm_bwd")
EPS = 1e-6


def _case(name, op, B, H, M, N, d, layout="packed", peaky=0.0):
    return {"name": name, "op": op, "B": B, "H": H, "M": M, "N": N, "d": d, "layout": layout, "peaky": peaky}


def listed():
    return [
        # a toy model or a unit test of a training loop: a handful of blocks, so latency and host work are all there is
        _case("tiny_step", "step", 2, 2, 64, 64, 32),
        # one layer of DiT-XL/2 on 256-pixel latents: many short sequences, forward and backward
        _case("dit256_fwd", "fwd", 64, 16, 256, 256, 72),
        _case("dit256_bwd", "bwd", 64, 16, 256, 256, 72),
        # one layer of DiT-XL/2 on 512-pixel latents, the headline shape; detach is the cheaper training setting
        _case("dit512_fwd", "fwd", 16, 16, 1024, 1024, 72),
        _case("dit512_bwd", "bwd", 16, 16, 1024, 1024, 72),
        _case("dit512_bwd_detach", "bwd_detach", 16, 16, 1024, 1024, 72),
        # head dimension 128, long sequences, peaked attention rows
        _case("large_fwd", "fwd", 2, 24, 4096, 4096, 128, peaky=0.05),
        _case("large_bwd", "bwd", 2, 24, 4096, 4096, 128, peaky=0.05),
        # the longest sequence of the sweep: video or high-resolution tokens
        _case("sweep32768_bwd", "bwd", 2, 16, 32768, 32768, 64),
        # image tokens against a conditioning sequence, tensors in place as the projections left them; ragged tiles
        _case("cross_step", "step", 8, 12, 1000, 333, 64, "token"),
        # the QK normalisation in front of the attention, at the headline shape
        _case("dit512_norm_fwd", "norm_fwd", 16, 16, 1024, 1024, 72),
        _case("dit512_norm_bwd", "norm_bwd", 16, 16, 1024, 1024, 72),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: The most one drawn case may cost: multiply-adds per GEMM of the attention, and elements of one tensor.
_MOST_MACS, _MOST_ELEMENTS = 1.6e12, 7.0e7


def draw(rng):
    while True:
        op = rng.choice(OPS)
        # the attention of absent cotangents, strides and M != N takes head dimensions up to 80
        wide = op in ("fwd", "bwd", "step") and rng.random() < 0.3
        d = rng.choice((88, 96, 104, 112, 120, 128, 128) if wide else (32, 40, 48, 56, 64, 64, 72, 72, 80))
        layout = "packed" if wide or rng.random() < 0.5 else "token"
        N = _log(rng, 33, 16384)
        M = _log(rng, 33, 16384) if not wide and rng.random() < 0.3 else N
        H = rng.choice((1, 2, 4, 6, 8, 12, 16, 24))
        B = _log(rng, 1, 96)
        rows, macs = B * H * max(M, N), 1.0 * B * H * M * N * d
        if rows * d <= _MOST_ELEMENTS and macs <= _MOST_MACS:
            return {"op": op, "B": B, "H": H, "M": M, "N": N, "d": d, "layout": layout, "peaky": rng.choice((0.0, 0.0, 0.05))}


def _tensor(gen, B, H, rows, d, layout, std=1.0, scale=None):
    """N(0, std) values, rounded to bf16; `scale`: a factor for each row."""
    x = torch.randn((B, rows, H, d) if layout == "token" else (B, H, rows, d), generator=gen, device="cuda")
    x = x.mul_(std)
    x = x.permute(0, 2, 1, 3) if layout == "token" else x
    if scale is not None:
        x = x * scale
    return x.to(torch.bfloat16)


def prepare(case, seed):
    op, B, H, M, N, d, layout = (case[k] for k in ("op", "B", "H", "M", "N", "d", "layout"))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4000 + int(seed))

    def rows_scale(rows):
        if case["peaky"] <= 0.0:
            return None
        return torch.where(torch.rand((B, H, rows, 1), generator=gen, device="cuda") < case["peaky"], 4.0, 1.0)

    def q_side(std=1.0, scale=None):
        return _tensor(gen, B, H, M, d, layout, std, scale)

    def k_side(std=1.0, scale=None):
        return _tensor(gen, B, H, N, d, layout, std, scale)

    s = {"op": op, "Q": q_side(scale=rows_scale(M)), "K": k_side(scale=rows_scale(N)), "tQ": q_side(0.5), "tK": k_side(0.5)}
    if op in ("norm_fwd", "norm_bwd"):
        s["gQ"], s["gK"] = (1.0 + 0.3 * torch.randn(d, generator=gen, device="cuda") for _ in range(2))
        if op == "norm_bwd":
            s["cotangents"] = [q_side(), q_side(), k_side(), k_side()]
        return s
    s["V"], s["tV"] = k_side(), k_side(0.5)
    if op != "fwd":
        s["dO"], s["dtO"] = q_side(), None if op == "bwd_detach" else q_side()
    if op in ("bwd", "bwd_detach"):
        s["saved"] = binding.tvm_attn_jvp_fwd(s["Q"], s["K"], s["V"], s["tQ"], s["tK"], s["tV"])
    if op == "bwd_detach":
        # the three gradients there are; a training loop keeps these buffers
        s["out"] = [torch.empty_strided(t.shape, t.stride(), dtype=t.dtype, device=t.device) for t in (s["Q"], s["K"], s["V"])]
        s["out"] += [None, None, None]
    return s


def run(s):
    op = s["op"]
    if op == "norm_fwd":
        return binding.tvm_qk_rmsnorm_jvp_fwd(s["Q"], s["tQ"], s["K"], s["tK"], s["gQ"], s["gK"], eps=EPS)
    if op == "norm_bwd":
        return binding.tvm_qk_rmsnorm_jvp_bwd(s["Q"], s["tQ"], s["K"], s["tK"], s["gQ"], s["gK"], *s["cotangents"], eps=EPS)
    x = (s["Q"], s["K"], s["V"], s["tQ"], s["tK"], s["tV"])
    if op == "fwd":
        return binding.tvm_attn_jvp_fwd(*x)
    if op == "step":
        saved = binding.tvm_attn_jvp_fwd(*x)
        return tuple(saved) + tuple(binding.tvm_attn_jvp_bwd(*x, *saved, s["dO"], s["dtO"]))
    return tuple(binding.tvm_attn_jvp_bwd(*x, *s["saved"], s["dO"], s["dtO"], out=s.get("out")))


def work(case):
    """Every input read once and every output written once; GEMMs of the method (6 forward, 15 backward, 5 detached)."""
    op, B, H, M, N, d = (case[k] for k in ("op", "B", "H", "M", "N", "d"))
    q, k, stats = 2 * B * H * M * d, 2 * B * H * N * d, 4 * B * H * M
    gemm = 2 * B * H * M * N * d
    if op == "fwd":      # in Q tQ | K V tK tV, out O tO, lse and mu
        return {"bytes": 4 * q + 4 * k + 2 * stats, "flops": 6 * gemm}
    if op == "bwd":      # in Q tQ O tO dO dtO | K V tK tV, lse and mu, out dQ dtQ | dK dV dtK dtV
        return {"bytes": 8 * q + 8 * k + 2 * stats, "flops": 15 * gemm}
    if op == "step":     # in Q tQ dO dtO | K V tK tV, out O tO dQ dtQ | dK dV dtK dtV, lse and mu
        return {"bytes": 8 * q + 8 * k + 2 * stats, "flops": 21 * gemm}
    if op == "bwd_detach":   # in Q O dO | K V, lse, out dQ | dK dV
        return {"bytes": 4 * q + 4 * k + stats, "flops": 5 * gemm}
    if op == "norm_fwd":     # in Q tQ | K tK and the scales, out as many
        return {"bytes": 4 * q + 4 * k + 8 * d, "flops": 10 * B * H * (M + N) * d}
    # in Q tQ dQn dtQn | K tK dKn dtKn and the scales, out dQ dtQ | dK dtK and the scales' gradients
    return {"bytes": 6 * q + 6 * k + 16 * d, "flops": 40 * B * H * (M + N) * d}


def tolerance(case):
    """bf16 results of fp32 sums.  The attention also rounds the operands of its second GEMMs to bf16 (relative 2^-9
    in each term of a sum with random signs); the normalisation rounds only its results."""
    return {"rel": 4e-3, "max": 0.03} if case["op"] in ("norm_fwd", "norm_bwd") else {"rel": 1e-2, "max": 0.2}
