"""GPU parity: the CUDA library against the CPU oracle, element by element, through the C ABI."""
import numpy as np
import pytest
import torch

from paper_2608_11688_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _harness():
    import harness
    return harness


def _run(cfg, *, mode, tau, T, B=1, layers=None, C=None, norm_topk=1, cache_reuse=1, check_ffn_every=1,
         use_prefetch=True, prob=None, ffn_token_stride=1, flags=0, max_near_ties=0):
    hz = _harness()
    prob = prob or hz.Problem(cfg, layers=layers)
    apex = prob.make_ctx(C=C, max_batch=B, norm_topk=norm_topk, cache_reuse=cache_reuse, flags=flags)
    try:
        rep = hz.run_lockstep(prob, apex, mode=mode, tau=tau, T=T, B=B, C=C, norm_topk=bool(norm_topk),
                              cache_reuse=bool(cache_reuse), check_ffn_every=check_ffn_every,
                              use_prefetch=use_prefetch, ffn_token_stride=ffn_token_stride, max_near_ties=max_near_ties)
        stats = apex.get_stats()
    finally:
        apex.destroy()
    assert rep.near_ties <= max_near_ties
    if use_prefetch and rep.near_ties == 0:
        # S9: the device-side counters equal the oracle's metrics summed over the run (always, unless the caller
        # allowed near-tie steps and some occurred: the library's counters then include steps the oracle's sums skip)
        for key in ("sum_delta_hat", "sum_delta_star", "sum_ncand", "hits_P", "hits_R", "covered", "capped"):
            assert stats[key] == getattr(rep, key), (key, stats[key], getattr(rep, key))
        assert stats["prefetch_copies"] == rep.n_prefetch_copies and stats["demand_copies"] == rep.n_demand_copies
        assert stats["substitutions"] == rep.n_subst
    return rep, stats


# ------------------------------------------------------------------ tiny and ragged shapes
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
@pytest.mark.parametrize("d,N,k,I,C", [(256, 8, 2, 24, 4), (512, 12, 3, 40, 6), (768, 33, 5, 17, 9),
                                       (1024, 64, 8, 16, 16), (3072, 5, 1, 9, 2)])
def test_tiny_shapes_both_modes(d, N, k, I, C, mode):
    cfg = synth.tiny_config(d=d, N=N, k=k, I=I, C=C, T=12, sigma_p=1.0, cfg_id=200 + N)
    rep, stats = _run(cfg, mode=mode, tau=0.7, T=12)
    assert rep.layer_steps == 12 and rep.ffn_checked == 12 and rep.near_ties == 0
    assert stats["tokens"] == 12 and stats["routed"] == 12 * k
    if mode == "stall_free":
        assert rep.n_demand_copies == 0


@pytest.mark.parametrize("tau", [0.0, 0.3, 0.97, 1.0])
def test_tau_extremes_and_cap(tau):
    cfg = synth.tiny_config(d=256, N=16, k=4, I=32, C=8, T=10, sigma_p=0.8, cfg_id=210)
    rep, stats = _run(cfg, mode="exact", tau=tau, T=10)
    if tau == 0.0:
        assert stats["sum_delta_hat"] == 0
    if tau == 1.0:
        assert stats["sum_ncand"] == 10 * 8 and stats["capped"] == 10     # N-k = 12 capped to C-k = 4


def test_all_resident_cache_never_copies_twice():
    cfg = synth.tiny_config(d=256, N=8, k=2, I=32, C=8, T=30, cfg_id=211)
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=30)
    assert stats["prefetch_copies"] + stats["demand_copies"] <= 8


def test_minimal_cache_C_equals_k():
    cfg = synth.tiny_config(d=256, N=10, k=3, I=16, C=3, T=20, sigma_p=1.5, cfg_id=212)
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=20)
    assert rep.n_miss_steps > 0            # a noisy predictor with no spare slot misses
    if _harness().token_kernel_expected():     # (where launch calls may block the host corrects misses between launches)
        assert stats["extra_waves"] == 0       # B = 1: missing experts are waited for inside the one launch
    assert stats["demand_copies"] == rep.n_demand_copies > 0
    rep, stats = _run(cfg, mode="stall_free", tau=0.9, T=20)
    assert rep.n_subst > 0 and stats["substitutions"] == rep.n_subst


@pytest.mark.parametrize("how", ["flag", "environment"])
def test_exact_mode_with_host_side_miss_correction(how, monkeypatch):
    # B = 1, exact mode, no wait for the host inside the kernel: resident routed experts first, one further launch per
    # demand wave.  The setting for processes whose kernel launches block (it is chosen from the environment when the
    # context is created).  Same decisions, same table, same output as the oracle.
    if not _harness().token_kernel_expected():
        pytest.skip("launch calls already block in this process: every context corrects misses on the host, nothing to compare")
    cfg = synth.tiny_config(d=256, N=10, k=3, I=16, C=3, T=20, sigma_p=1.5, cfg_id=212)
    if how == "environment":
        monkeypatch.setenv("CUDA_LAUNCH_BLOCKING", "1")       # read by apex_create; the CUDA runtime of this process is already up
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=20, flags=binding.FLAG_HOST_WAVES if how == "flag" else 0)
    assert rep.n_miss_steps > 0 and rep.ffn_checked == 20
    assert stats["extra_waves"] == rep.n_miss_steps        # one more launch for every step that missed (C >= k: one wave)
    assert stats["demand_copies"] == rep.n_demand_copies > 0 and stats["timeouts"] == 0
    # through the pipelined whole-token call as well
    hz = _harness()
    cfg = synth.tiny_config(d=512, N=12, k=3, I=24, C=4, L=3, T=5, sigma_p=1.5, cfg_id=231)
    prob = hz.Problem(cfg)
    hs = [synth.hidden_states(cfg, l, cfg.T, 1) for l in range(cfg.L)]
    h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()
    hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
    outs = []
    for flags in (0, binding.FLAG_HOST_WAVES):
        if how == "environment" and flags == 0:
            monkeypatch.delenv("CUDA_LAUNCH_BLOCKING")
        elif how == "environment":
            monkeypatch.setenv("CUDA_LAUNCH_BLOCKING", "1")
        apex = prob.make_ctx(flags=flags if how == "flag" else 0)
        try:
            y = torch.zeros((cfg.T, cfg.L, 1, cfg.d), dtype=torch.float32, device="cuda")
            for t in range(cfg.T):
                apex.decode_token(h[t], hp[t], 1, 0.8, "exact", y[t])
            torch.cuda.synchronize()
            st = apex.get_stats()
            assert st["timeouts"] == 0 and (st["extra_waves"] > 0) == (flags != 0)
            outs.append((y.cpu().numpy(), st["demand_copies"], [apex.get_slot_table(l)[0].tolist() for l in range(cfg.L)]))
        finally:
            apex.destroy()
    assert outs[0][1] == outs[1][1] > 0 and outs[0][2] == outs[1][2]
    np.testing.assert_allclose(outs[1][0], outs[0][0], rtol=0, atol=2e-6 * float(np.abs(outs[0][0]).max()))


def test_load_use_evict_policy_and_unnormalised_gates():
    cfg = synth.tiny_config(d=512, N=12, k=3, I=24, C=7, T=12, sigma_p=1.0, cfg_id=213)
    rep, stats = _run(cfg, mode="stall_free", tau=0.8, T=12, cache_reuse=0)
    assert stats["prefetch_copies"] == stats["sum_ncand"]       # every candidate of every step is copied
    _run(cfg, mode="exact", tau=0.8, T=8, norm_topk=0)


def test_no_prefetch_baseline_demand_fetches_everything():
    cfg = synth.tiny_config(d=256, N=10, k=3, I=16, C=5, T=10, cfg_id=214)
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=10, use_prefetch=False)
    assert stats["prefetch_copies"] == 0 and stats["demand_copies"] == rep.n_demand_copies > 0


def test_shared_expert_and_multi_layer():
    cfg = synth.tiny_config(d=512, N=12, k=2, I=24, C=6, L=3, T=6, I_shared=40, cfg_id=215)
    rep, stats = _run(cfg, mode="exact", tau=0.8, T=6)
    assert rep.layer_steps == 18


@pytest.mark.parametrize("B", [2, 5, 16])
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_batched_tokens(B, mode):
    cfg = synth.tiny_config(d=512, N=20, k=3, I=24, C=8, T=5, I_shared=16, sigma_p=1.0, cfg_id=216)
    rep, stats = _run(cfg, mode=mode, tau=0.8, T=5, B=B)
    assert stats["tokens"] == 5 * B


@pytest.mark.parametrize("B", [16, 40, 97])
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_batched_tensor_core_path(B, mode):
    # shapes the tcgen05 grouped GEMM accepts (I, I_shared multiples of 128)
    cfg = synth.tiny_config(d=256, N=12, k=3, I=128, C=8, T=3, I_shared=256, sigma_p=1.0, cfg_id=230)
    rep, stats = _run(cfg, mode=mode, tau=0.8, T=3, B=B)
    assert stats["tokens"] == 3 * B and rep.ffn_checked >= 1 and rep.near_ties == 0
    print("tc", B, mode, rep)


def test_batched_exact_mode_runs_in_waves_when_cache_is_smaller_than_need():
    cfg = synth.tiny_config(d=256, N=16, k=4, I=16, C=5, T=4, cfg_id=217)
    rep, stats = _run(cfg, mode="exact", tau=0.5, T=4, B=8)
    assert stats["extra_waves"] >= 4 * 2          # at least two extra waves per step: need > 2 C


# ------------------------------------------------------------------ gated shared expert (no counterpart in the paper)
@pytest.mark.parametrize("B,fmt", [(1, "bf16"), (1, "fp8"), (1, "fp4"), (5, "bf16"), (24, "bf16"), (24, "fp8")])
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_gated_shared_expert(B, fmt, mode):
    # y = routed part + sigmoid(w_sg . h') * shared FFN: B = 1 the streaming kernel, B = 5 and 24 the grouped GEMM (the pairs of
    # other sizes, with the gate value from the plan kernel: test_gpu_batched_ffn.py)
    cfg = synth.tiny_config(d=512, N=12, k=3, I=128, C=8, L=2, T=3, I_shared=256, sigma_p=1.0, cfg_id=290)
    hz = _harness()
    prob = hz.Problem(cfg, fp8=(fmt == "fp8"), fp4=(fmt == "fp4"), gated_shared=True)
    rep, stats = _run(cfg, mode=mode, tau=0.8, T=3, B=B, prob=prob)
    assert rep.ffn_checked == 3 * 2 * B and rep.near_ties == 0
    # the gate matters: without it the same run must fail the output check
    prob.shared_gates = [None] * prob.L
    apex = prob.make_ctx(max_batch=B)
    try:
        for l in range(prob.L):
            apex.set_shared_gate(l, np.zeros(cfg.d, np.float32))      # weight 0.5 everywhere: differs from weight 1
        with pytest.raises(AssertionError, match="FFN output"):
            hz.run_lockstep(prob, apex, mode=mode, tau=0.8, T=1, B=B)
        for l in range(prob.L):
            apex.set_shared_gate(l, None)                             # back to weight 1: matches the ungated oracle
        hz.run_lockstep(prob, apex, mode=mode, tau=0.8, T=2, B=B)
    finally:
        apex.destroy()


# ------------------------------------------------------------------ e4m3 expert store (Sec. V-G)
def _run_fp8(cfg, *, mode, tau, T, B=1, layers=None, check_ffn_every=1, ffn_token_stride=1):
    hz = _harness()
    prob = hz.Problem(cfg, layers=layers, fp8=True)
    return _run(cfg, mode=mode, tau=tau, T=T, B=B, layers=layers, prob=prob, check_ffn_every=check_ffn_every,
                ffn_token_stride=ffn_token_stride)


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
@pytest.mark.parametrize("d,N,k,I,C,Ish", [(512, 12, 3, 40, 6, 0), (1024, 16, 4, 17, 8, 24), (2048, 8, 2, 9, 4, 0),
                                            (4096, 6, 2, 5, 3, 7)])
def test_fp8_store_tiny_shapes(d, N, k, I, C, Ish, mode):
    cfg = synth.tiny_config(d=d, N=N, k=k, I=I, C=C, T=8, I_shared=Ish, sigma_p=1.0, cfg_id=260 + N)
    rep, stats = _run_fp8(cfg, mode=mode, tau=0.7, T=8)
    assert rep.layer_steps == 8 and rep.ffn_checked == 8 and rep.near_ties == 0
    assert stats["bytes_copied"] == (rep.n_prefetch_copies + rep.n_demand_copies) * I * (3 * d + 16)
    print("fp8", d, mode, rep)


def test_fp8_store_small_batch_runs_streaming_kernel():
    # (these sizes run the grouped GEMM from two tokens on; batches that stream: test_gpu_batched_ffn.py)
    cfg = synth.tiny_config(d=512, N=12, k=3, I=128, C=8, T=3, I_shared=128, sigma_p=1.0, cfg_id=275)
    rep, stats = _run_fp8(cfg, mode="exact", tau=0.8, T=3, B=3)
    assert stats["tokens"] == 9


@pytest.mark.parametrize("B", [16, 40, 97])
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
@pytest.mark.parametrize("fmt", ["fp8", "fp4"])
def test_quantised_store_tensor_core_path(fmt, B, mode):
    # B >= 16 with d, I, I_shared the grouped GEMM accepts: converter warps expand the code tiles to bf16 operand tiles.
    # I = 256 gives two row blocks per expert and four K tiles in the down projection; I_shared = 384 a longer K there
    # (cut into chunks); d = 512 gives eight K tiles in gate / up, so the e2m1 scale bytes of a row cross no 16-byte group,
    # and the four column blocks of the down projection use all four scale offsets of one.
    cfg = synth.tiny_config(d=512, N=12, k=3, I=256, C=8, T=3, I_shared=384, sigma_p=1.0, cfg_id=276)
    rep, stats = (_run_fp8 if fmt == "fp8" else _run_fp4)(cfg, mode=mode, tau=0.8, T=3, B=B)
    assert stats["tokens"] == 3 * B and rep.ffn_checked == 3 * B and rep.near_ties == 0
    print("tc", fmt, B, mode, rep)


@pytest.mark.parametrize("B", [1, 24])
def test_fp8_store_of_subnormal_codes(B):
    # every code byte and-ed with 0x8F: exponent field 0 or 1 only, so half the weights are e4m3 subnormals and none is
    # large enough to hide them; B = 1 runs the streaming kernel, B = 24 the converters of the tensor-core path
    cfg = synth.tiny_config(d=512, N=12, k=3, I=128, C=8, T=2, I_shared=128, sigma_p=1.0, cfg_id=278)
    hz = _harness()
    prob = hz.Problem(cfg, fp8=True, fp8_code_mask=0x8F)
    codes = prob.stores[0][..., :3 * cfg.d].numpy()
    assert 0.3 < float(np.mean((codes >> 3) & 0xF == 0)) < 0.7 and int(((codes >> 3) & 0xF).max()) == 1
    rep, stats = _run(cfg, mode="exact", tau=0.8, T=2, B=B, prob=prob)
    assert rep.ffn_checked == 2 * B and rep.near_ties == 0


@pytest.mark.parametrize("fmt", ["bf16", "fp8", "fp4"])
@pytest.mark.parametrize("N,k,I,I_shared,B", [(4, 2, 72, 200, 2), (5, 2, 200, 0, 31), (3, 1, 130, 72, 130), (2, 2, 1100, 64, 256),
                                                  (6, 2, 700, 90, 40), (16, 3, 648, 200, 24)])
def test_grouped_gemm_tile_edges(fmt, N, k, I, I_shared, B):
    """Intermediate sizes off the grouped GEMM's 64- and 128-row tiles, which stream their pairs instead, for groups of 2 to 256
    tokens (the GEMM's own tile edges: test_grouped_gemm_tiles)."""
    cfg = synth.tiny_config(d=512, N=N, k=k, I=I, C=N, T=2, I_shared=I_shared, sigma_p=1.0, cfg_id=279)
    run = {"bf16": _run, "fp8": _run_fp8, "fp4": _run_fp4}[fmt]
    rep, stats = run(cfg, mode="exact", tau=0.8, T=2, B=B, ffn_token_stride=max(1, B // 16))
    assert stats["tokens"] == 2 * B and rep.near_ties == 0


def test_fp4_store_of_large_block_scales():
    # block scales above 2 (up) and tiny ones (down), which the converters apply in two multiplications: the factors cancel
    hz = _harness()
    cfg = synth.tiny_config(d=512, N=6, k=2, I=128, C=6, T=2, sigma_p=1.0, cfg_id=281)
    prob = hz.Problem(cfg, fp4=True)
    o = 3 * (cfg.d // 2)
    for st in prob.stores:
        up, down = st[..., o + cfg.d // 32:o + 2 * (cfg.d // 32)], st[..., o + 2 * (cfg.d // 32):o + 3 * (cfg.d // 32)]
        up[up > 0] += 14
        down[down > 0] -= 14
        assert int(up.max()) > 128
    rep, stats = _run(cfg, mode="exact", tau=0.8, T=2, B=24, prob=prob)
    assert rep.ffn_checked == 48 and rep.near_ties == 0


@pytest.mark.parametrize("fmt", ["fp8", "fp4"])
def test_quantised_store_tensor_core_path_wide(fmt):
    # d = 1024: sixteen K tiles, so the e2m1 scale bytes of a gate / up row span two 16-byte groups; 8 column blocks in
    # the down projection span two groups as well.  No shared expert.
    cfg = synth.tiny_config(d=1024, N=8, k=2, I=128, C=8, T=2, sigma_p=1.0, cfg_id=277)
    rep, stats = (_run_fp8 if fmt == "fp8" else _run_fp4)(cfg, mode="exact", tau=0.8, T=2, B=33)
    assert stats["tokens"] == 66 and rep.ffn_checked == 66 and rep.near_ties == 0


@pytest.mark.parametrize("fmt", ["fp8", "fp4"])
def test_quantised_store_config4_shape_tensor_core_batch(fmt):
    # config 4's shape (d = 2048, I = 768, 60 experts, 4 shared) at B = 32, one layer, FFN output of every 8th token
    cfg = synth.CONFIGS[4]
    rep, stats = (_run_fp8 if fmt == "fp8" else _run_fp4)(cfg, mode="exact", tau=0.9, T=1, layers=1, B=32, ffn_token_stride=8)
    assert stats["tokens"] == 32 and rep.ffn_checked >= 4 and rep.near_ties == 0
    print("config4-tc", fmt, rep, stats)


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_fp8_store_config1_shape_two_layers(mode):
    cfg = synth.CONFIGS[1]
    rep, stats = _run_fp8(cfg, mode=mode, tau=0.9, T=12, layers=2, check_ffn_every=3)
    assert rep.layer_steps == 24
    print("fp8 config1", mode, rep)


# ------------------------------------------------------------------ block-scaled e2m1 expert store
def _run_fp4(cfg, *, mode, tau, T, B=1, layers=None, check_ffn_every=1, ffn_token_stride=1):
    hz = _harness()
    prob = hz.Problem(cfg, layers=layers, fp4=True)
    return _run(cfg, mode=mode, tau=tau, T=T, B=B, layers=layers, prob=prob, check_ffn_every=check_ffn_every,
                ffn_token_stride=ffn_token_stride)


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
@pytest.mark.parametrize("d,N,k,I,C,Ish", [(512, 12, 3, 40, 6, 0), (1024, 16, 4, 17, 8, 24), (2048, 8, 2, 9, 4, 0),
                                            (4096, 6, 2, 5, 3, 7)])
def test_fp4_store_tiny_shapes(d, N, k, I, C, Ish, mode):
    cfg = synth.tiny_config(d=d, N=N, k=k, I=I, C=C, T=8, I_shared=Ish, sigma_p=1.0, cfg_id=300 + N)
    rep, stats = _run_fp4(cfg, mode=mode, tau=0.7, T=8)
    assert rep.layer_steps == 8 and rep.ffn_checked == 8 and rep.near_ties == 0
    assert stats["bytes_copied"] == (rep.n_prefetch_copies + rep.n_demand_copies) * I * synth.fp4_row_bytes(d)
    print("fp4", d, mode, rep)


def test_fp4_store_small_batch_runs_streaming_kernel():
    # (as above)
    cfg = synth.tiny_config(d=512, N=12, k=3, I=128, C=8, T=3, I_shared=128, sigma_p=1.0, cfg_id=315)
    rep, stats = _run_fp4(cfg, mode="exact", tau=0.8, T=3, B=5)
    assert stats["tokens"] == 15


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_fp4_store_config1_shape_two_layers(mode):
    cfg = synth.CONFIGS[1]
    rep, stats = _run_fp4(cfg, mode=mode, tau=0.9, T=12, layers=2, check_ffn_every=3)
    assert rep.layer_steps == 24
    print("fp4 config1", mode, rep)


# ------------------------------------------------------------------ speculative first fill of the expert FFN
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
@pytest.mark.parametrize("sigma_p", [0.0, 8.0])
def test_speculative_fill_with_good_and_useless_predictor(sigma_p, mode):
    # sigma_p = 0: most guesses are confirmed; sigma_p = 8: the prefetch ranking is almost unrelated to the
    # gate's, so nearly every speculative copy is dropped and its stage refilled
    cfg = synth.tiny_config(d=1024, N=24, k=6, I=96, C=12, T=10, I_shared=32, sigma_p=sigma_p, cfg_id=280)
    rep, stats = _run(cfg, mode=mode, tau=0.6, T=10, flags=binding.FLAG_SPECULATE)
    assert rep.layer_steps == 10 and rep.ffn_checked == 10 and rep.near_ties == 0
    if sigma_p == 8.0:
        assert stats["hits_P"] < 0.8 * stats["routed"]


def test_speculation_switch_changes_nothing_but_time():
    cfg = synth.tiny_config(d=1536, N=40, k=8, I=128, C=20, L=3, T=6, sigma_p=0.3, cfg_id=281)
    hz = _harness()
    prob = hz.Problem(cfg)
    hs = [synth.hidden_states(cfg, l, cfg.T, 1) for l in range(cfg.L)]
    h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()
    hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
    ys, stats = [], []
    for flags in (0, binding.FLAG_SPECULATE):
        apex = prob.make_ctx(flags=flags)
        try:
            y = torch.zeros((cfg.T, cfg.L, 1, cfg.d), dtype=torch.float32, device="cuda")
            for t in range(cfg.T):
                apex.decode_token(h[t], hp[t], 1, 0.8, "exact", y[t])
            torch.cuda.synchronize()
            ys.append(y.cpu().numpy())
            st = apex.get_stats()
            stats.append({k: st[k] for k in ("hits_P", "hits_R", "covered", "prefetch_copies", "demand_copies",
                                             "sum_delta_hat", "sum_delta_star", "substitutions", "timeouts")})
        finally:
            apex.destroy()
    assert stats[0] == stats[1] and stats[0]["timeouts"] == 0
    # same rows, same arithmetic per row; only the order of the fp32 atomic adds into y may differ
    np.testing.assert_allclose(ys[0], ys[1], rtol=0, atol=2e-6 * float(np.abs(ys[1]).max()))


# ------------------------------------------------------------------ throttled host link
def test_throttled_link_gives_the_same_results_later():
    import time
    cfg = synth.tiny_config(d=1024, N=16, k=4, I=256, C=8, T=8, sigma_p=1.0, cfg_id=320)     # 1.5 MiB experts
    hz = _harness()
    prob = hz.Problem(cfg)
    out = []
    for gbs in (0.0, 2.0):
        apex = prob.make_ctx(link_gbs=gbs)
        try:
            t0 = time.perf_counter()
            rep = hz.run_lockstep(prob, apex, mode="exact", tau=0.7, T=cfg.T)
            torch.cuda.synchronize()
            out.append((rep, apex.get_stats(), time.perf_counter() - t0))
        finally:
            apex.destroy()
    (r0, s0, _), (r1, s1, _) = out
    assert r0.n_prefetch_copies == r1.n_prefetch_copies and r0.n_demand_copies == r1.n_demand_copies
    assert s0["bytes_copied"] == s1["bytes_copied"] and s1["timeouts"] == 0
    # at 2 GB/s every copy of 1.5 MiB takes about 0.8 ms: the copy stream alone needs that long
    assert s1["bytes_copied"] / 2e9 > 0.02


def test_negative_link_bandwidth_is_refused():
    with pytest.raises(binding.ApexError):
        binding.Apex(d=256, N=8, k=2, I=8, C_slots=4, link_gbs=-1.0)


def test_expert_store_must_be_pinned_host_memory():
    a = binding.Apex(d=256, N=8, k=2, I=8, C_slots=4)
    try:
        dev_store = torch.zeros((8, 8, 3, 256), dtype=torch.bfloat16, device="cuda")
        with pytest.raises(binding.ApexError):
            a.register_experts(0, dev_store)
        pageable = torch.zeros((8, 8, 3, 256), dtype=torch.bfloat16)
        with pytest.raises(binding.ApexError):
            a.register_experts(0, pageable)
        a.register_experts(0, pageable.pin_memory())
    finally:
        a.destroy()


# ------------------------------------------------------------------ the paper-shaped configs
def test_config0_full():
    cfg = synth.CONFIGS[0]
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=cfg.T)
    assert rep.layer_steps == 128
    assert rep.worst_rel_l2 <= 2e-3 and rep.worst_max_abs <= 2e-2
    print("config0", rep, stats)


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_config1_shape_two_layers(mode):
    cfg = synth.CONFIGS[1]
    rep, stats = _run(cfg, mode=mode, tau=0.9, T=24, layers=2, check_ffn_every=3)
    assert rep.layer_steps == 48
    print("config1", mode, rep, stats)


@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_config2_shape_one_layer(mode):
    cfg = synth.CONFIGS[2]
    rep, stats = _run(cfg, mode=mode, tau=0.9, T=12, layers=1, check_ffn_every=3)
    print("config2", mode, rep, stats)


def test_config3_shape_one_layer():
    cfg = synth.CONFIGS[3]
    hz = _harness()
    prob = hz.Problem(cfg, layers=1)
    for mode in ("exact", "stall_free"):
        rep, stats = _run(cfg, mode=mode, tau=0.9, T=3, layers=1, prob=prob)
        print("config3", mode, rep, stats)


@pytest.mark.parametrize("B", [1, 8])
def test_config4_shape_one_layer(B):
    cfg = synth.CONFIGS[4]
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=2, layers=1, B=B)
    print("config4", B, rep, stats)


@pytest.mark.parametrize("B,stride", [(32, 8), (128, 32), (256, 64)])
def test_config4_shape_tensor_core_batches(B, stride):
    # the batched sweep of config 4 on the tcgen05 path; decisions checked for every token, FFN output for
    # every stride-th token (the oracle needs seconds per token at this size)
    cfg = synth.CONFIGS[4]
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=1, layers=1, B=B, ffn_token_stride=stride)
    assert stats["tokens"] == B and rep.ffn_checked >= B // stride
    print("config4-tc", B, rep, stats)


@pytest.mark.parametrize("d,N,k,C,B", [(768, 64, 8, 24, 200),    # clusters of 8: groups of 8 tokens, two passes, a ragged last group
                                        (512, 12, 3, 6, 250),     # clusters of 2: groups of 4 tokens, ragged
                                        (1024, 33, 4, 10, 131),   # clusters of 8, groups of 8, one ragged group
                                        (256, 5, 2, 3, 97)])      # one CTA per token
def test_batched_router_group_shapes(d, N, k, C, B):
    # the batched router / gate kernel walks groups of tokens per cluster: every token's ranking, budget, top-k and
    # gates against the oracle for group counts above and below the number of clusters the GPU holds
    cfg = synth.tiny_config(d=d, N=N, k=k, I=128, C=C, T=2, sigma_p=1.0, cfg_id=300 + N)
    for mode in ("exact", "stall_free"):
        rep, stats = _run(cfg, mode=mode, tau=0.8, T=2, B=B, ffn_token_stride=max(1, B // 8))
        assert stats["tokens"] == 2 * B and stats["routed"] == 2 * B * k


def test_tensor_core_path_more_units_than_one_descriptor_chunk():
    # gate/up GEMM: 64 experts x 112 row blocks = 7168 units, i.e. 49 per CTA on 148 SMs: the kernel describes its units 32
    # at a time, so this runs two chunks (the second one partial)
    cfg = synth.tiny_config(d=256, N=64, k=16, I=14336, C=64, T=1, sigma_p=1.0, cfg_id=377)
    rep, stats = _run(cfg, mode="exact", tau=0.9, T=1, B=256, ffn_token_stride=64)
    assert stats["tokens"] == 256 and rep.ffn_checked >= 4


# ------------------------------------------------------------------ API behaviour
@pytest.mark.parametrize("per_layer", [False, True])
def test_decode_token_matches_per_call_sequence_and_counts_launches(per_layer):
    cfg = synth.tiny_config(d=512, N=12, k=3, I=24, C=6, L=2, T=4, cfg_id=218)
    hz = _harness()
    prob = hz.Problem(cfg)
    a1, a2 = prob.make_ctx(flags=binding.FLAG_LAYER_LAUNCHES if per_layer else 0), prob.make_ctx()
    try:
        hs = [synth.hidden_states(cfg, l, cfg.T) for l in range(cfg.L)]
        h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()       # [T][L][1][d]
        hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
        y1 = torch.empty((cfg.L, 1, cfg.d), device="cuda"); y2 = torch.empty_like(y1)
        cand = torch.empty((1, cfg.C), dtype=torch.int32, device="cuda"); nc = torch.empty(1, dtype=torch.int32, device="cuda")
        idx = torch.empty((1, cfg.k), dtype=torch.int32, device="cuda"); al = torch.empty((1, cfg.N), device="cuda")
        for t in range(cfg.T):
            n0 = a1.launch_count()
            a1.decode_token(h[t], hp[t], 1, 0.9, "exact", y1)
            if per_layer:
                assert a1.launch_count() - n0 >= 4 * cfg.L      # fused predict+select, attention, gate, FFN
            else:
                assert a1.launch_count() - n0 == 1 or not hz.token_kernel_expected()   # one persistent kernel over all layers
            for l in range(cfg.L):
                a2.predict(l, h[t, l], 1); a2.select_candidates(l, 1, 0.9, cand, nc); a2.prefetch(l, 1)
                a2.attention_standin(l); a2.route_topk(l, hp[t, l], 1, idx, al)
                a2.moe_ffn(l, "exact", hp[t, l], 1, y2[l])
            torch.cuda.synchronize()
            torch.testing.assert_close(y1, y2, rtol=1e-4, atol=1e-5)
        # host-buffer variant
        hh = h[0].cpu().pin_memory(); hph = hp[0].cpu().pin_memory(); yh = torch.empty_like(hh).pin_memory()
        a3 = prob.make_ctx()
        a3.decode_token_host(hh, hph, 1, 0.9, "exact", yh)
        a4 = prob.make_ctx()
        a4.decode_token(h[0], hp[0], 1, 0.9, "exact", y1); torch.cuda.synchronize()
        torch.testing.assert_close(yh.cuda(), y1, rtol=1e-4, atol=1e-5)
        a3.destroy(); a4.destroy()
    finally:
        a1.destroy(); a2.destroy()


def test_ffn_in_two_halves_reset_stats_and_warm_all():
    # apex_moe_ffn_begin / apex_moe_ffn_end equal apex_moe_ffn; their ordering rules; apex_reset_stats; apex_warm_all
    cfg = synth.tiny_config(d=512, N=12, k=3, I=24, C=6, L=1, T=6, cfg_id=223)
    hz = _harness()
    prob = hz.Problem(cfg)
    a1, a2 = prob.make_ctx(), prob.make_ctx()
    full = prob.make_ctx(C=cfg.N)
    try:
        h, hp = synth.hidden_states(cfg, 0, cfg.T)
        hd, hpd = torch.from_numpy(h).cuda(), torch.from_numpy(hp).cuda()
        y1 = torch.empty((1, cfg.d), device="cuda"); y2 = torch.empty_like(y1)
        cand = torch.empty((1, cfg.C), dtype=torch.int32, device="cuda"); nc = torch.empty(1, dtype=torch.int32, device="cuda")
        idx = torch.empty((1, cfg.k), dtype=torch.int32, device="cuda"); al = torch.empty((1, cfg.N), device="cuda")
        with pytest.raises(binding.ApexError) as ei:
            a2.moe_ffn_end(0)                                   # nothing was begun
        assert ei.value.code == binding.APEX_ESTATE and "apex_moe_ffn_begin" in str(ei.value)
        for t in range(cfg.T):
            mode = "exact" if t % 2 == 0 else "stall_free"
            for a in (a1, a2):
                a.predict(0, hd[t], 1); a.select_candidates(0, 1, 0.9, cand, nc); a.prefetch(0, 1)
                a.attention_standin(0); a.route_topk(0, hpd[t], 1, idx, al)
            a1.moe_ffn(0, mode, hpd[t], 1, y1)
            a2.moe_ffn_begin(0, mode, hpd[t], 1, y2)
            if t == 0:
                with pytest.raises(binding.ApexError) as ei:    # the layer-step is not complete yet
                    a2.predict(0, hd[t], 1)
                assert ei.value.code == binding.APEX_ESTATE
            a2.moe_ffn_end(0)
            torch.cuda.synchronize()
            torch.testing.assert_close(y1, y2, rtol=1e-4, atol=1e-5)   # fp32 atomics: the order of the partial sums is free
            assert a1.get_last_copies(0) == a2.get_last_copies(0)
            t1, t2 = a1.get_slot_table(0), a2.get_slot_table(0)
            assert list(t1[0]) == list(t2[0]) and list(t1[1]) == list(t2[1])
        s = a1.get_stats()
        assert s["layer_steps"] == cfg.T and s["tokens"] == cfg.T and s["routed"] == cfg.T * cfg.k
        a1.reset_stats()
        assert all(v == 0 for v in a1.get_stats().values())
        # warm_all: only when every expert has a slot; afterwards nothing is ever copied
        with pytest.raises(binding.ApexError) as ei:
            a1.warm_all()
        assert ei.value.code in (binding.APEX_EINVAL, binding.APEX_ESTATE)
        full.warm_all()
        es, _, _ = full.get_slot_table(0)
        assert sorted(es) == list(range(cfg.N))
        full.reset_stats()
        for t in range(cfg.T):
            full.predict(0, hd[t], 1); full.select_candidates(0, 1, 0.9, cand, nc); full.prefetch(0, 1)
            full.route_topk(0, hpd[t], 1, idx, al); full.moe_ffn(0, "exact", hpd[t], 1, y1)
        torch.cuda.synchronize()
        s = full.get_stats()
        assert s["prefetch_copies"] == 0 and s["demand_copies"] == 0 and s["hits_R"] == s["routed"] == cfg.T * cfg.k
    finally:
        a1.destroy(); a2.destroy(); full.destroy()


def test_slot_table_checkpoint_and_resume():
    # snapshot the slot tables after a few tokens, restore them into a fresh context, continue: same outputs
    cfg = synth.tiny_config(d=512, N=12, k=3, I=24, C=6, L=2, T=8, cfg_id=222)
    hz = _harness()
    prob = hz.Problem(cfg)
    a1, a2 = prob.make_ctx(), prob.make_ctx()
    try:
        hs = [synth.hidden_states(cfg, l, cfg.T) for l in range(cfg.L)]
        h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()
        hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
        y1 = torch.empty((cfg.L, 1, cfg.d), device="cuda"); y2 = torch.empty_like(y1)
        for t in range(4):
            a1.decode_token(h[t], hp[t], 1, 0.8, "exact", y1)
        torch.cuda.synchronize()
        for l in range(cfg.L):
            es, st, clk = a1.get_slot_table(l)
            a2.set_slot_table(l, es, st, clk)
        for t in range(4, 8):
            a1.decode_token(h[t], hp[t], 1, 0.8, "exact", y1)
            a2.decode_token(h[t], hp[t], 1, 0.8, "exact", y2)
            torch.cuda.synchronize()
            torch.testing.assert_close(y1, y2, rtol=1e-4, atol=1e-5)
            for l in range(cfg.L):
                t1, t2 = a1.get_slot_table(l), a2.get_slot_table(l)
                assert list(t1[0]) == list(t2[0]) and list(t1[1]) == list(t2[1]) and t1[2] == t2[2]
    finally:
        a1.destroy(); a2.destroy()


def test_calls_out_of_order_and_bad_arguments():
    cfg = synth.tiny_config(d=256, N=8, k=2, I=16, C=4, cfg_id=219)
    hz = _harness()
    prob = hz.Problem(cfg)
    a = prob.make_ctx()
    try:
        y = torch.empty((1, cfg.d), device="cuda")
        with pytest.raises(binding.ApexError) as ei:
            a.moe_ffn(0, "exact", y, 1, y)
        assert ei.value.code == binding.APEX_ESTATE
        cand = torch.empty((1, cfg.C), dtype=torch.int32, device="cuda"); nc = torch.empty(1, dtype=torch.int32, device="cuda")
        with pytest.raises(binding.ApexError) as ei:
            a.select_candidates(0, 1, 0.9, cand, nc)
        assert ei.value.code == binding.APEX_ESTATE
        with pytest.raises(binding.ApexError) as ei:
            a.predict(3, y, 1)
        assert ei.value.code == binding.APEX_EINVAL
        with pytest.raises(binding.ApexError) as ei:
            a.set_cdf(0, np.zeros(cfg.N, np.float32), np.arange(cfg.N - cfg.k + 1, 0, -1).astype(np.float32))
        assert ei.value.code == binding.APEX_EINVAL
    finally:
        a.destroy()


def test_host_side_fault_hooks_copy_failure_and_withheld_flag():
    cfg = synth.tiny_config(d=256, N=8, k=2, I=16, C=4, T=4, cfg_id=220)
    hz = _harness()
    prob = hz.Problem(cfg)
    a = prob.make_ctx(wait_limit_ns=50_000_000)          # 50 ms bound on every wait
    try:
        h, hp = synth.hidden_states(cfg, 0, 4)
        hd, hpd = torch.from_numpy(h).cuda(), torch.from_numpy(hp).cuda()
        y = torch.empty((1, cfg.d), device="cuda")
        cand = torch.empty((1, cfg.C), dtype=torch.int32, device="cuda"); nc = torch.empty(1, dtype=torch.int32, device="cuda")
        idx = torch.empty((1, cfg.k), dtype=torch.int32, device="cuda"); al = torch.empty((1, cfg.N), device="cuda")
        # 1: the copy issue fails on the host
        a.predict(0, hd[0], 1); a.select_candidates(0, 1, 0.9, cand, nc)
        a.test_inject(1)
        with pytest.raises(binding.ApexError) as ei:
            a.prefetch(0, 1)
        assert ei.value.code == binding.APEX_ECUDA
        # the candidates whose copy was never issued must not count as resident: the same context goes on --
        # prefetch again, gate, exact-mode FFN -- and the output is the dense top-k mixture of the oracle
        from oracle import apex_oracle as ao
        es, _, _ = a.get_slot_table(0)
        cp, _ = a.get_last_copies(0)
        assert sorted(e for e, s in enumerate(es) if s >= 0) == sorted(e for e, _ in cp)    # only what was really copied
        a.prefetch(0, 1); a.attention_standin(0); a.route_topk(0, hpd[0], 1, idx, al)
        a.moe_ffn(0, "exact", hpd[0], 1, y)
        torch.cuda.synchronize()
        W_r, b_r, _, _ = prob.routers[0]
        _, K_r, alpha = ao.route_topk(W_r, b_r, hp[0, 0], cfg.k)
        ref = ao.moe_output(hp[0, 0], K_r, ao.gates(alpha, K_r), prob.oracle_experts(0))
        err = y[0].double().cpu().numpy() - ref
        assert np.linalg.norm(err) / np.linalg.norm(ref) <= hz.REL_L2_TOL and np.abs(err).max() <= hz.MAX_ABS_TOL
        assert sorted(idx[0].tolist()) == sorted(K_r)
        # and a failure of a demand copy: the expert FFN reports it, the table does not keep the expert, a second
        # attempt of the same layer-step's FFN completes
        a.predict(0, hd[1], 1); a.select_candidates(0, 1, 0.0, cand, nc); a.prefetch(0, 1)
        a.route_topk(0, hpd[1], 1, idx, al)
        pre_es, _, _ = a.get_slot_table(0)
        routed = idx[0].tolist()
        if any(pre_es[e] < 0 for e in routed):                    # (seeded inputs: this step does miss)
            a.test_inject(1)
            with pytest.raises(binding.ApexError) as ei:
                a.moe_ffn(0, "exact", hpd[1], 1, y)
            assert ei.value.code in (binding.APEX_ECUDA, binding.APEX_ETIMEOUT)
            torch.cuda.synchronize()
            try:
                a.moe_ffn(0, "exact", hpd[1], 1, y)
            except binding.ApexError as e:     # the first attempt's wait that ran out, reported late; this attempt's work is queued in full
                assert e.code == binding.APEX_ETIMEOUT
            torch.cuda.synchronize()
            _, K_r, alpha = ao.route_topk(W_r, b_r, hp[1, 0], cfg.k)
            ref = ao.moe_output(hp[1, 0], K_r, ao.gates(alpha, K_r), prob.oracle_experts(0))
            err = y[0].double().cpu().numpy() - ref
            assert np.linalg.norm(err) / np.linalg.norm(ref) <= hz.REL_L2_TOL and np.abs(err).max() <= hz.MAX_ABS_TOL
        # 2: a slot-ready flag is withheld: the device-side wait runs out and the call reports it;
        # the context stays usable afterwards
        a2 = prob.make_ctx(wait_limit_ns=50_000_000)
        a2.predict(0, hd[1], 1); a2.select_candidates(0, 1, 1.0, cand, nc)
        a2.test_inject(2)
        a2.prefetch(0, 1); a2.attention_standin(0); a2.route_topk(0, hpd[1], 1, idx, al)
        try:
            a2.moe_ffn(0, "stall_free", hpd[1], 1, y)
            torch.cuda.synchronize()
            # the status may arrive after the call returned: the next call reports it
            a2.predict(0, hd[2], 1); a2.select_candidates(0, 1, 1.0, cand, nc); a2.prefetch(0, 1)
            a2.route_topk(0, hpd[2], 1, idx, al); a2.moe_ffn(0, "stall_free", hpd[2], 1, y)
            torch.cuda.synchronize()
            raised = False
        except binding.ApexError as e:
            assert e.code == binding.APEX_ETIMEOUT
            raised = True
        assert raised or a2.get_stats()["timeouts"] > 0
        torch.cuda.synchronize()
        a2.predict(0, hd[3], 1); a2.select_candidates(0, 1, 0.9, cand, nc); a2.prefetch(0, 1)
        a2.route_topk(0, hpd[3], 1, idx, al)
        try:
            a2.moe_ffn(0, "exact", hpd[3], 1, y)
        except binding.ApexError as e:
            assert e.code == binding.APEX_ETIMEOUT          # a late report of the same timeout
        torch.cuda.synchronize()
        assert torch.isfinite(y).all()
        a2.destroy()
    finally:
        a.destroy()


def test_run_to_run_determinism_of_indices():
    cfg = synth.tiny_config(d=1024, N=32, k=8, I=32, C=16, T=6, cfg_id=221)
    hz = _harness()
    prob = hz.Problem(cfg)
    outs = []
    for rep in range(2):
        a = prob.make_ctx()
        h, hp = synth.hidden_states(cfg, 0, 6)
        cand = torch.empty((1, cfg.C), dtype=torch.int32, device="cuda"); nc = torch.empty(1, dtype=torch.int32, device="cuda")
        idx = torch.empty((1, cfg.k), dtype=torch.int32, device="cuda"); al = torch.empty((1, cfg.N), device="cuda")
        rec = []
        for t in range(6):
            a.predict(0, torch.from_numpy(h[t]).cuda(), 1); a.select_candidates(0, 1, 0.9, cand, nc)
            a.route_topk(0, torch.from_numpy(hp[t]).cuda(), 1, idx, al)
            torch.cuda.synchronize()
            rec.append((cand.cpu().numpy().copy(), idx.cpu().numpy().copy(), al.cpu().numpy().copy(), a.read_prediction(1)))
        outs.append(rec)
        a.destroy()
    for r0, r1 in zip(*outs):
        np.testing.assert_array_equal(r0[0], r1[0]); np.testing.assert_array_equal(r0[1], r1[1])
        np.testing.assert_array_equal(r0[2], r1[2])                      # bitwise: fixed reduction order
        for x, y2 in zip(r0[3], r1[3]):
            np.testing.assert_array_equal(x, y2)


# ------------------------------------------------------------------ the benchmark's launch configuration
@pytest.mark.parametrize("mode", ["exact", "stall_free"])
def test_config1_full_size_decode_token_sampled_layers(mode):
    """Config 1 at full size (32 layers, 20 slots, fitted confidence model) through apex_decode_token --
    the call bench.py times: fused prefetch router + budget, pipelined host work, in-kernel miss wait.
    Every token: slot tables of all layers before and after; sampled layers are replayed by the oracle
    from the pre-step table and compared (decisions bit-exact via the tables and copy lists, y by tolerance)."""
    from oracle import apex_oracle as ao
    hz = _harness()
    cfg = synth.CONFIGS[1]
    prob = hz.Problem(cfg, cdf="fitted")
    apex = prob.make_ctx()
    try:
        T = 3
        hs = [synth.hidden_states(cfg, l, T, 1) for l in range(cfg.L)]
        h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()      # [T][L][1][d]
        hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
        y = torch.empty((cfg.L, 1, cfg.d), device="cuda")
        worst = 0.0
        n_near = 0
        for t in range(T):
            pre = [apex.get_slot_table(l) for l in range(cfg.L)]
            apex.decode_token(h[t], hp[t], 1, 0.9, mode, y)
            torch.cuda.synchronize()
            g_y = y.cpu().numpy()
            for l in range((t * 5) % 7, cfg.L, 7):                           # five or so layers per token
                W_r, b_r, W_p, b_p = prob.routers[l]
                w, theta = prob.cdf[l]
                cache = ao.SlotCache(cfg.N, cfg.C)
                cache.set_state(*pre[l])
                out = ao.layer_step(cache, W_p=W_p, b_p=b_p, W_r=W_r, b_r=b_r, w=w, theta=theta, tau=0.9, k=cfg.k,
                                    h=hs[l][0][t], h_post=hs[l][1][t], mode=mode, expert_weights=prob.oracle_experts(l))
                tok = out["tokens"][0]
                near = bool(ao.near_tie_reasons(tok))
                post = apex.get_slot_table(l)
                cp, dm = apex.get_last_copies(l)
                same = (list(post[0]) == cache.expert_slot and list(post[1]) == cache.slot_stamp and post[2] == cache.clock
                        and cp == out["prefetch_copies"] and dm == out["demand_copies"])
                assert same or near, f"slot decisions differ t={t} l={l}"
                n_near += int(not same)
                if same:
                    err = g_y[l, 0].astype(np.float64) - tok["y"]
                    rel = float(np.linalg.norm(err) / np.linalg.norm(tok["y"]))
                    worst = max(worst, rel)
                    assert rel <= hz.REL_L2_TOL and float(np.abs(err).max()) <= hz.MAX_ABS_TOL, (t, l, rel)
        st = apex.get_stats()
        assert st["tokens"] == T * cfg.L and st["timeouts"] == 0
        assert n_near == 0, f"{n_near} sampled layer-steps excused as near-ties"
        print("config1 full", mode, "worst rel-L2", worst, "near-ties", n_near, st)
    finally:
        apex.destroy()


def test_config1_long_run_counts_near_ties():
    """1024 decode steps of one config-1 layer in lock-step: every decision of every step against the
    oracle (FFN output on every 64th step).  Reports how many steps had a near-tie (deciding logit gap
    below 1e-6) -- those are the only steps where an index may differ, and they are excused and counted."""
    cfg = synth.CONFIGS[1]
    hz = _harness()
    prob = hz.Problem(cfg, layers=1, cdf="fitted")
    apex = prob.make_ctx()
    try:
        rep = hz.run_lockstep(prob, apex, mode="exact", tau=0.9, T=cfg.T, check_ffn_every=64, max_near_ties=2)
    finally:
        apex.destroy()
    assert rep.layer_steps == 1024
    assert rep.near_ties <= 2, rep          # expected about 1e-3 per run for 40 logits of unit spread
    print("config1 long run:", rep)


def test_config1_long_run_stall_free_and_batched():
    """The same lock-step walk in stall-free mode (1024 steps), and with 8 tokens per step through the batched path
    (128 steps of a config-1 layer, execution sets of every token compared, FFN output on every 16th step)."""
    cfg = synth.CONFIGS[1]
    hz = _harness()
    prob = hz.Problem(cfg, layers=1, cdf="fitted")
    apex = prob.make_ctx()
    try:
        rep = hz.run_lockstep(prob, apex, mode="stall_free", tau=0.9, T=cfg.T, check_ffn_every=64, max_near_ties=2)
        st = apex.get_stats()
    finally:
        apex.destroy()
    assert rep.layer_steps == 1024 and rep.near_ties <= 2 and rep.n_demand_copies == 0
    assert st["substitutions"] >= rep.n_subst > 0 and (rep.near_ties > 0 or st["substitutions"] == rep.n_subst)
    apex = prob.make_ctx(max_batch=8)
    try:
        rep8 = hz.run_lockstep(prob, apex, mode="exact", tau=0.9, T=128, B=8, check_ffn_every=16, ffn_token_stride=3,
                               max_near_ties=2)
    finally:
        apex.destroy()
    assert rep8.layer_steps == 128 and rep8.near_ties <= 2
    print("config1 long run stall-free:", rep, "\nconfig1 long run B=8:", rep8)


def test_decode_token_output_does_not_depend_on_the_prefetch_policy():
    # exact mode: y is the router's top-k mixture whatever was prefetched -- with prefetching, without (tau < 0: the
    # attention stand-in then follows the previous layer's FFN and must wait for it), and with both alternating
    cfg = synth.tiny_config(d=1024, N=16, k=4, I=64, C=8, L=3, T=6, sigma_p=0.8, cfg_id=330)
    hz = _harness()
    prob = hz.Problem(cfg)
    hs = [synth.hidden_states(cfg, l, cfg.T, 1) for l in range(cfg.L)]
    h = torch.from_numpy(np.stack([x[0] for x in hs], 1)).cuda()
    hp = torch.from_numpy(np.stack([x[1] for x in hs], 1)).cuda()
    outs = []
    for taus in ([0.9] * cfg.T, [-1.0] * cfg.T, [0.9, -1.0] * (cfg.T // 2)):
        apex = prob.make_ctx()
        try:
            y = torch.zeros((cfg.T, cfg.L, 1, cfg.d), dtype=torch.float32, device="cuda")
            for t in range(cfg.T):
                apex.decode_token(h[t], hp[t], 1, taus[t], "exact", y[t])
            torch.cuda.synchronize()
            assert apex.get_stats()["timeouts"] == 0
            outs.append(y.cpu().numpy())
        finally:
            apex.destroy()
    scale = float(np.abs(outs[0]).max())
    for o in outs[1:]:
        np.testing.assert_allclose(o, outs[0], rtol=0, atol=2e-6 * scale)   # only the order of the fp32 atomics differs


def test_random_shapes_modes_and_options():
    """A fixed-seed walk over shapes and options that the hand-picked cases above do not combine: widths, expert counts
    up to 64, ragged I, shared experts, cache sizes from k to N, batch sizes on both sides of the tensor-core threshold,
    both modes, tau at and between the extremes, both cache policies, both gate normalisations, the quantised stores and
    the opt-in speculative fill.  Every decision and every output is compared with the oracle in lock-step."""
    import random
    rng = random.Random(20260811)
    hz = _harness()
    for it in range(36):
        d = rng.choice([256, 512, 768, 1024, 1536, 2048])
        N = rng.randint(2, 64)
        k = rng.randint(1, min(N, 16))
        C = rng.randint(k, N)
        I = rng.choice([8, 17, 40, 64, 128, 256])
        Ish = rng.choice([0, 0, 16, 128, 256])
        B = rng.choice([1, 1, 1, 2, 3, 5, 8, 16, 33])
        mode = rng.choice(["exact", "stall_free"])
        tau = rng.choice([0.0, 0.3, 0.7, 0.9, 0.99, 1.0])
        reuse, norm = rng.choice([1, 1, 0]), rng.choice([1, 1, 0])
        flags = rng.choice([0, 0, binding.FLAG_SPECULATE])
        fmt = rng.choice(["bf16", "bf16", "fp8", "fp4"]) if d in (512, 1024, 1536, 2048) else "bf16"
        L = rng.choice([1, 2])
        cfg = synth.tiny_config(d=d, N=N, k=k, I=I, C=C, L=L, T=4, I_shared=Ish, sigma_p=rng.choice([0.3, 1.0, 4.0]),
                                cfg_id=2000 + it)
        prob = hz.Problem(cfg, fp8=(fmt == "fp8"), fp4=(fmt == "fp4"))
        apex = prob.make_ctx(max_batch=B, norm_topk=norm, cache_reuse=reuse, flags=flags)
        try:
            rep = hz.run_lockstep(prob, apex, mode=mode, tau=tau, T=4, B=B, norm_topk=bool(norm), cache_reuse=bool(reuse))
            assert apex.get_stats()["timeouts"] == 0
            assert rep.layer_steps == 4 * L
        finally:
            apex.destroy()


def test_random_shapes_tensor_core_path_gated_shared_expert_and_token_kernel():
    """A second fixed-seed walk, over what the first one reaches rarely or not at all: batches of 16 to 40 tokens on shapes the
    grouped GEMMs accept (all three store formats), the gated shared expert, and B = 1 through apex_decode_token (the
    persistent token kernel, checked by replaying every layer against the oracle)."""
    import random
    rng = random.Random(20260812)
    hz = _harness()
    for it in range(24):
        tc = it % 2 == 0
        if tc:
            d, I, Ish, B = rng.choice([512, 1024]), rng.choice([128, 256]), rng.choice([0, 128, 384]), rng.choice([16, 24, 40])
        else:
            d, I, Ish, B = rng.choice([512, 1024, 1536, 2048]), rng.choice([8, 17, 64, 128]), rng.choice([0, 16, 128]), 1
        N = rng.randint(4, 64)
        k = rng.randint(1, min(N, 16))
        C = rng.choice([rng.randint(k, N), N])
        mode = rng.choice(["exact", "stall_free"])
        tau = rng.choice([0.0, 0.7, 0.9, 1.0])
        fmt = rng.choice(["bf16", "fp8", "fp4"])
        gated = Ish > 0 and rng.random() < 0.6
        L = rng.choice([1, 2, 3])
        cfg = synth.tiny_config(d=d, N=N, k=k, I=I, C=C, L=L, T=4, I_shared=Ish, sigma_p=rng.choice([0.3, 1.0, 4.0]), cfg_id=2100 + it)
        prob = hz.Problem(cfg, fp8=(fmt == "fp8"), fp4=(fmt == "fp4"), gated_shared=gated)
        apex = prob.make_ctx(max_batch=B)
        try:
            if tc:
                rep = hz.run_lockstep(prob, apex, mode=mode, tau=tau, T=3, B=B)
                assert rep.layer_steps == 3 * L
            else:
                n0 = apex.launch_count()
                rep = hz.run_decode_lockstep(prob, apex, mode=mode, tau=tau, T=4)
                assert apex.launch_count() - n0 == 4 or not hz.token_kernel_expected(), "the persistent token kernel did not run"
            assert apex.get_stats()["timeouts"] == 0 and rep.near_ties == 0
        finally:
            apex.destroy()

