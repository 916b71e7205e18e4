"""Batched expert FFN (B > 1): which steps keep fp32 hidden states, and that no step leaves anything behind for the next."""
import numpy as np
import pytest
import torch

from oracle import apex_oracle as ao
from paper_2608_11688_b200 import synth

pytestmark = pytest.mark.gpu


def _problem(fmt, **shape):
    import harness
    return harness.Problem(synth.tiny_config(T=1, C=shape["N"], **shape), fp8=fmt == "fp8", fp4=fmt == "fp4")


def _step(prob, ctx, hp, mode="exact"):
    """Gate and expert FFN of one layer-step on h' [B][d]; returns y and the oracle's output for the gate's decisions."""
    cfg, B = prob.cfg, len(hp)
    x = torch.from_numpy(hp).cuda()
    idx = torch.empty((B, cfg.k), dtype=torch.int32, device="cuda")
    alpha = torch.empty((B, cfg.N), device="cuda")
    y = torch.full((B, cfg.d), 123.0, device="cuda")
    ctx.route_topk(0, x, B, idx, alpha)
    ctx.moe_ffn(0, mode, x, B, y)
    torch.cuda.synchronize()
    a, e = alpha.double().cpu().numpy(), idx.cpu().numpy()
    experts, shared = prob.oracle_experts(0), prob.oracle_shared(0)
    ref = np.stack([ao.moe_output(hp[b].astype(np.float64), e[b], a[b][e[b]] / a[b][e[b]].sum(), experts, shared) for b in range(B)])
    return y.double().cpu().numpy(), ref


def _rel(y, ref):
    return float(np.linalg.norm(y - ref) / np.linalg.norm(ref))


def test_an_overflowing_step_leaves_nothing_for_the_next():
    # two tokens, then four: the second step's routed pairs take rows of the scratch that held the first one's shared
    # expert (the wider of the two), whose intermediate overflows for this h' (finite, so the routing is ordinary)
    prob = _problem("bf16", d=512, N=2, k=2, I=72, I_shared=200, cfg_id=320)
    ctx = prob.make_ctx(max_batch=4)
    try:
        ctx.warm_all()
        rng = np.random.default_rng(320)
        hp = rng.standard_normal((4, 512)).astype(np.float32)
        hp = torch.from_numpy(hp).bfloat16().float().numpy()
        big, _ = _step(prob, ctx, hp[:2] * np.float32(2.0 ** 80))
        assert not np.isfinite(big).all()
        y, ref = _step(prob, ctx, hp)
        assert np.isfinite(y).all() and _rel(y, ref) <= 3e-5
    finally:
        ctx.destroy()
