"""Batched expert FFN (B > 1): which steps keep fp32 hidden states, and that no step leaves anything behind for the next."""
import numpy as np
import pytest
import torch

from oracle import apex_oracle as ao
from paper_2608_11688_b200 import binding, synth

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


@pytest.mark.parametrize("fmt", ["bf16", "fp8", "fp4"])
@pytest.mark.parametrize("I,I_shared,B", [(72, 0, 2), (192, 128, 5), (128, 200, 7), (320, 0, 40), (130, 72, 256)])
def test_batches_off_the_128_row_tiles_keep_fp32_hidden_states(fmt, I, I_shared, B):
    # h' with all 24 bits: rounding it to bf16 would show as about 2^-9.  The sums: a lane's chains of 16 products and 5 levels
    # of a tree per dot product, then at most I + I_shared fp32 additions into y, every one to half an ulp (2^-24) in
    # either direction; 2^-24 (16 + 5 + sqrt(I + I_shared)) of the terms' size is below 3e-6 for these shapes
    prob = _problem(fmt, d=512, N=8, k=2, I=I, I_shared=I_shared, cfg_id=321)
    ctx = prob.make_ctx(max_batch=B)
    try:
        ctx.warm_all()
        y, ref = _step(prob, ctx, np.random.default_rng(321 + B).standard_normal((B, 512)).astype(np.float32))
        rel = _rel(y, ref)
        print("fp32 h'", fmt, I, I_shared, B, rel)
        assert rel <= 3e-6
    finally:
        ctx.destroy()


@pytest.mark.parametrize("fmt", ["bf16", "fp8", "fp4"])
@pytest.mark.parametrize("N,k,I,I_shared,B", [(4, 2, 128, 256, 2), (5, 2, 256, 0, 31), (3, 1, 128, 384, 130), (2, 2, 1152, 128, 256),
                                              (6, 2, 768, 128, 40), (16, 3, 640, 256, 24)])
def test_grouped_gemm_tiles(fmt, N, k, I, I_shared, B):
    # the sizes the grouped GEMM takes: gate/up units of 32 rows (the first two, and on the e4m3 store the fifth) and of 128,
    # one and several chunks of K in the down projection, groups of 2 to 256 tokens: one part or several, and on the
    # quantised stores both accumulator layouts.  h' is bf16-representable; the intermediate is carried to 2^-17 (7.6e-6)
    prob = _problem(fmt, d=512, N=N, k=k, I=I, I_shared=I_shared, cfg_id=322)
    ctx = prob.make_ctx(max_batch=B)
    try:
        ctx.warm_all()
        hp = torch.from_numpy(np.random.default_rng(322 + B).standard_normal((B, 512)).astype(np.float32)).bfloat16().float().numpy()
        y, ref = _step(prob, ctx, hp)
        rel = _rel(y, ref)
        print("bf16 h'", fmt, I, I_shared, B, rel)
        assert rel <= 7.6e-6
    finally:
        ctx.destroy()


def _decode_inputs(cfg, B):
    hs = [synth.hidden_states(cfg, l, 1, B) for l in range(cfg.L)]
    return tuple(torch.from_numpy(np.stack([x[i][0] for x in hs])).cuda() for i in (0, 1))


@pytest.mark.parametrize("fmt", ["bf16", "fp8", "fp4"])
@pytest.mark.parametrize("d,N,k,I,I_shared,B", [(512, 16, 3, 512, 0, 24), (256, 4, 4, 1152, 0, 32), (256, 3, 2, 512, 1024, 9), (1024, 9, 3, 1024, 0, 4)])
def test_grouped_gemm_small_units(fmt, d, N, k, I, I_shared, B):
    """Gate/up units of 32 rows, two to a CTA, and down projections cut into more chunks of K than their length asks for (equal
    chunks or not).  Bounds as above."""
    if fmt != "bf16" and d == 256:
        d = 512
    prob = _problem(fmt, d=d, N=N, k=k, I=I, I_shared=I_shared, cfg_id=329)
    ctx = prob.make_ctx(max_batch=B)
    try:
        ctx.warm_all()
        hp = torch.from_numpy(np.random.default_rng(329 + B).standard_normal((B, d)).astype(np.float32)).bfloat16().float().numpy()
        y, ref = _step(prob, ctx, hp)
        assert _rel(y, ref) <= 7.6e-6
    finally:
        ctx.destroy()


@pytest.mark.parametrize("C", [6, 4])
def test_decode_goes_on_after_candidate_records_that_never_arrived(C):
    # C = N: the expert FFN of a layer is launched before its candidate records are waited for; C < N: after
    import harness
    B = 3
    cfg = synth.tiny_config(d=256, N=6, k=2, I=128, C=C, L=2, T=1, cfg_id=323)
    prob = harness.Problem(cfg)
    h, hp = _decode_inputs(cfg, B)
    out = []
    for what in (0, 3):
        ctx = prob.make_ctx(max_batch=B, wait_limit_ns=50_000_000)
        try:
            if C == cfg.N:
                ctx.warm_all()
            y = torch.zeros((cfg.L, B, cfg.d), device="cuda")
            if what:
                ctx.test_inject(what)
                with pytest.raises(binding.ApexError) as ei:
                    ctx.decode_token(h, hp, B, 0.9, "exact", y)
                assert ei.value.code == binding.APEX_ETIMEOUT and "candidate" in str(ei.value)
                torch.cuda.synchronize()
            ctx.decode_token(h, hp, B, 0.9, "exact", y)
            torch.cuda.synchronize()
            out.append(y.cpu().numpy())
        finally:
            ctx.destroy()
    np.testing.assert_allclose(out[1], out[0], rtol=0, atol=2e-6 * float(np.abs(out[0]).max()))  # (fp32 additions into y in another order)


def test_decode_right_behind_a_prediction_of_its_first_layer():
    # the prefetch stage of a batched step has no dependency wait of its own (the stand-in in front of it has): a prediction
    # still running on the same scratch must be complete before it
    import harness
    B, cfg = 64, synth.tiny_config(d=2048, N=64, k=4, I=128, C=64, L=1, T=2, cfg_id=324)
    prob = harness.Problem(cfg)
    ctx = prob.make_ctx(max_batch=B)
    try:
        ctx.warm_all()
        h, hp = _decode_inputs(cfg, B)
        other = torch.flip(h, dims=(1,)).contiguous()
        y = torch.zeros((1, B, cfg.d), device="cuda")
        ctx.decode_token(h, hp, B, 0.9, "exact", y)
        torch.cuda.synchronize()
        want, y_want = ctx.read_prediction(B), y.cpu().numpy()
        for _ in range(20):
            ctx.predict(0, other[0], B)
            ctx.decode_token(h, hp, B, 0.9, "exact", y)
            torch.cuda.synchronize()
            for a, b in zip(ctx.read_prediction(B), want):
                np.testing.assert_array_equal(a, b)
            np.testing.assert_allclose(y.cpu().numpy(), y_want, rtol=0, atol=2e-6 * float(np.abs(y_want).max()))
    finally:
        ctx.destroy()


@pytest.mark.parametrize("stage", ["prefetch", "gate"])
def test_batched_router_reports_a_wait_that_ran_out(stage):
    # one CTA of a batched router waits for bytes that nobody sends: its limit ends the wait, its cluster's tokens carry
    # no routing, the call (or the next one) reports it, and the context goes on
    import harness
    B, cfg = 40, synth.tiny_config(d=2048, N=24, k=3, I=128, C=24, L=1, T=1, cfg_id=325)
    prob = harness.Problem(cfg)
    ctx = prob.make_ctx(max_batch=B, wait_limit_ns=50_000_000)
    try:
        ctx.warm_all()
        h, hp = _decode_inputs(cfg, B)
        y = torch.zeros((1, B, cfg.d), device="cuda")
        ctx.decode_token(h, hp, B, 0.9, "exact", y)
        torch.cuda.synchronize()
        want = y.cpu().numpy()
        if stage == "prefetch":
            ctx.test_inject(4)
            with pytest.raises(binding.ApexError) as ei:
                ctx.decode_token(h, hp, B, 0.9, "exact", y)
            assert ei.value.code == binding.APEX_ETIMEOUT
        else:
            idx = torch.full((B, cfg.k), 7, dtype=torch.int32, device="cuda")
            alpha = torch.zeros((B, cfg.N), device="cuda")
            ctx.test_inject(4)
            ctx.route_topk(0, hp[0], B, idx, alpha)
            torch.cuda.synchronize()
            bad = (idx == -1).all(1)
            assert bad.any() and not bad.all() and ((idx >= 0).all(1) == ~bad).all()
            assert (torch.isnan(alpha).all(1) == bad).all() and torch.isfinite(alpha[~bad]).all()
            with pytest.raises(binding.ApexError) as ei:
                ctx.moe_ffn(0, "exact", hp[0], B, y[0])
            assert ei.value.code == binding.APEX_ETIMEOUT
        torch.cuda.synchronize()
        ctx.decode_token(h, hp, B, 0.9, "exact", y)
        torch.cuda.synchronize()
        np.testing.assert_allclose(y.cpu().numpy(), want, rtol=0, atol=2e-6 * float(np.abs(want).max()))
    finally:
        ctx.destroy()


@pytest.mark.parametrize("fmt", ["bf16", "fp4"])
def test_grouped_gemm_reads_this_steps_activations_every_time(fmt):
    # the rounded hidden states and the intermediate are written by some CTAs and read by the bulk loads of others; two
    # inputs in turn, so that a load that came too early would read the other one's
    import harness
    B, cfg = 160, synth.tiny_config(d=1024, N=16, k=4, I=256, C=16, L=2, T=2, I_shared=384, cfg_id=326)
    prob = harness.Problem(cfg, fp4=fmt == "fp4")
    ctx = prob.make_ctx(max_batch=B)
    try:
        ctx.warm_all()
        h, hp = _decode_inputs(cfg, B)
        inputs = [(h, hp), (torch.flip(h, dims=(2,)).contiguous(), torch.flip(hp, dims=(2,)).contiguous())]
        y = torch.zeros((cfg.L, B, cfg.d), device="cuda")
        want = []
        for n in range(60):
            ctx.decode_token(*inputs[n % 2], B, 0.9, "exact", y)
            torch.cuda.synchronize()
            if n < 2:
                want.append(y.clone())
            else:
                assert float((y - want[n % 2]).abs().max()) <= 2e-6 * float(want[n % 2].abs().max())
    finally:
        ctx.destroy()


@pytest.mark.parametrize("fmt", ["bf16", "fp8", "fp4"])
@pytest.mark.parametrize("I,I_shared", [(128, 0), (1024, 512)])
def test_grouped_gemm_stops_with_copies_in_flight_and_the_context_goes_on(fmt, I, I_shared):
    # one expert's slot-ready flag is withheld: the CTAs that wait for it run into the limit while others have weights,
    # activations and MMAs under way.  Units of 32 rows (the first shape) and of 128
    import harness
    B, cfg = 24, synth.tiny_config(d=1024, N=4, k=2, I=I, C=4, L=1, T=1, I_shared=I_shared, cfg_id=327)
    prob = harness.Problem(cfg, fp8=fmt == "fp8", fp4=fmt == "fp4")
    h, hp = _decode_inputs(cfg, B)
    y = torch.zeros((1, B, cfg.d), device="cuda")
    ref = prob.make_ctx(max_batch=B)
    try:
        ref.warm_all()
        ref.decode_token(h, hp, B, 0.9, "exact", y)
        torch.cuda.synchronize()
        want = y.cpu().numpy()
    finally:
        ref.destroy()
    for _ in range(3):
        ctx = prob.make_ctx(max_batch=B, wait_limit_ns=20_000_000)
        try:
            ctx.test_inject(2)
            late = 0
            for _ in range(3):
                try:
                    ctx.decode_token(h, hp, B, 1.0, "exact", y)
                except binding.ApexError as e:
                    assert e.code == binding.APEX_ETIMEOUT
                    late += 1
                torch.cuda.synchronize()
            assert late > 0 and ctx.get_stats()["timeouts"] > 0
            np.testing.assert_allclose(y.cpu().numpy(), want, rtol=0, atol=2e-6 * float(np.abs(want).max()))
        finally:
            ctx.destroy()


@pytest.mark.parametrize("mode,norm_topk", [("exact", 1), ("exact", 0), ("stall_free", 1)])
@pytest.mark.parametrize("B,C", [(2, 12), (33, 6), (256, 6)])
def test_pair_plan_in_lock_step(mode, norm_topk, B, C):
    # the plan of batches that stream pairs: one warp's worth of tokens, a second CTA with one token, all eight CTAs of the
    # cluster; demand waves (C < what the batch needs), substitution, and a gated shared expert
    import harness
    cfg = synth.tiny_config(d=512, N=12, k=3, I=72, C=C, L=2, T=2, I_shared=40, sigma_p=1.0, cfg_id=328)
    prob = harness.Problem(cfg, gated_shared=True)
    ctx = prob.make_ctx(C=C, max_batch=B, norm_topk=norm_topk)
    try:
        rep = harness.run_lockstep(prob, ctx, mode=mode, tau=0.8, T=2, B=B, C=C, norm_topk=bool(norm_topk), ffn_token_stride=max(1, B // 16))
        stats = ctx.get_stats()
        assert rep.near_ties == 0 and rep.worst_rel_l2 <= 3e-6
        assert stats["hits_R"] == rep.hits_R and stats["substitutions"] == rep.n_subst
        assert (stats["extra_waves"] > 0) == (mode == "exact" and rep.n_miss_steps > 0)
    finally:
        ctx.destroy()
