"""GPU parity of apex_distill_router: the CUDA distillation of the prefetch router against the CPU one (oracle/distill.py)."""
import time

import numpy as np
import pytest
import torch

from paper_2608_11688_b200 import binding, build, synth

pytestmark = pytest.mark.gpu


def _teacher(cfg, T):
    """Calibration tokens of a config: h (before attention), and the router's distribution on h' (after)."""
    W_r, b_r, W_p, b_p = synth.router_weights(cfg, 0)
    h, hp = synth.hidden_states(cfg, 0, T, 1, calib=True)
    H, Hp = h[:, 0].astype(np.float64), hp[:, 0].astype(np.float64)
    Z = Hp @ W_r.astype(np.float64).T + b_r.astype(np.float64)
    Z -= Z.max(1, keepdims=True)
    Qr = np.exp(Z)
    Qr /= Qr.sum(1, keepdims=True)
    return H.astype(np.float32), Qr.astype(np.float32), W_r, b_r, W_p, b_p


@pytest.mark.parametrize("shape", ["tiny", "config1"])
def test_distillation_matches_cpu(shape):
    from oracle import distill
    build.build()
    if shape == "tiny":
        cfg, T, iters = synth.tiny_config(d=96, N=9, k=2, I=16, C=4, sigma_p=0.5, cfg_id=295), 501, 60
    else:
        cfg, T, iters = synth.CONFIGS[1], 2048, 40
    H, Qr, W_r, b_r, W_p, b_p = _teacher(cfg, T)
    t0 = time.perf_counter()
    W_ref, b_ref = distill.distill(H, Qr, W_p, b_p, iters=iters, lr=0.01)
    t_cpu = time.perf_counter() - t0
    Hd, Qd = torch.from_numpy(H).cuda(), torch.from_numpy(Qr).cuda()
    binding.distill_router(Hd, Qd, W_p, b_p, iters=iters, lr=0.01)       # warm-up
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    W, b = binding.distill_router(Hd, Qd, W_p, b_p, iters=iters, lr=0.01)
    t_gpu = time.perf_counter() - t0
    # same iterations in fp64 on both sides (sums in another order); outputs are fp32
    assert np.abs(W - W_ref).max() <= 2e-6 * max(1.0, float(np.abs(W_ref).max())), np.abs(W - W_ref).max()
    assert np.abs(b - b_ref).max() <= 2e-6 * max(1.0, float(np.abs(b_ref).max())), np.abs(b - b_ref).max()
    W2, b2 = binding.distill_router(Hd, Qd, W_p, b_p, iters=iters, lr=0.01)
    assert np.array_equal(W, W2) and np.array_equal(b, b2)             # bit-reproducible
    l0, l1 = distill.kl_loss(H, Qr, W_p, b_p), distill.kl_loss(H, Qr, W, b)
    assert l1 < l0
    print(f"distill {shape}: T={T} N={cfg.N} d={cfg.d} iters={iters}  gpu {t_gpu*1e3:.1f} ms  cpu {t_cpu*1e3:.1f} ms  "
          f"KL {l0:.4f} -> {l1:.4f}  max|dW| {np.abs(W - W_ref).max():.2e}")


@pytest.mark.parametrize("T,N,d", [(1, 1, 1), (63, 8, 64), (65, 9, 66), (257, 64, 130), (1190, 33, 68), (9601, 17, 36)])
def test_distillation_tile_edges(T, N, d):
    """Token tiles of one to eight warps and their remainders, expert tiles 1 to 8, columns off the 64-column tile and off
    16-byte rows, more tokens than one wave of CTAs."""
    from oracle import distill
    build.build()
    rng = np.random.default_rng(1000 * T + N)
    H = rng.standard_normal((T, d)).astype(np.float32)
    Z = rng.standard_normal((T, N))
    Qr = (np.exp(Z) / np.exp(Z).sum(1, keepdims=True)).astype(np.float32)
    W0 = (rng.standard_normal((N, d)) / np.sqrt(d)).astype(np.float32)
    b0 = rng.standard_normal(N).astype(np.float32)
    W_ref, b_ref = distill.distill(H, Qr, W0, b0, iters=4, lr=0.01)
    W, b = binding.distill_router(torch.from_numpy(H).cuda(), torch.from_numpy(Qr).cuda(), W0, b0, iters=4, lr=0.01)
    # a gradient that is exactly zero in one summation order and 1e-17 in another moves Adam by up to lr: not seen with
    # more than one expert; with one expert the softmax is 1 and every gradient is (1 - q_r) h
    assert np.abs(W - W_ref).max() <= 2e-6 * max(1.0, float(np.abs(W_ref).max()))
    assert np.abs(b - b_ref).max() <= 2e-6 * max(1.0, float(np.abs(b_ref).max()))


def test_distillation_rejects_bad_arguments():
    build.build()
    H = torch.zeros((8, 16), dtype=torch.float32, device="cuda")
    Q = torch.zeros((8, 70), dtype=torch.float32, device="cuda")
    with pytest.raises(binding.ApexError):
        binding.distill_router(H, Q, np.zeros((70, 16), np.float32), np.zeros(70, np.float32))      # N > 64


def test_distillation_reports_a_wait_that_ran_out():
    build.build()
    rng = np.random.default_rng(7)
    H = torch.from_numpy(rng.standard_normal((300, 128)).astype(np.float32)).cuda()
    Qr = torch.softmax(torch.from_numpy(rng.standard_normal((300, 9)).astype(np.float32)), 1).cuda()
    W0, b0 = rng.standard_normal((9, 128)).astype(np.float32), np.zeros(9, np.float32)
    want = binding.distill_router(H, Qr, W0, b0, iters=3)
    binding.load_library().apex_test_starve_distill()
    with pytest.raises(binding.ApexError) as ei:
        binding.distill_router(H, Qr, W0, b0, iters=3)
    assert ei.value.code == binding.APEX_ECUDA and "wait" in str(ei.value)
    got = binding.distill_router(H, Qr, W0, b0, iters=3)          # and the next call is not affected
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("T,N,d,iters", [
    (2369, 12, 128, 3),    # three warps of tokens per forward CTA; 19 segments of two stages, the last one of a token
    (4737, 20, 64, 3),     # five; one column tile, 25 segments of three stages
    (2368, 20, 64, 3),     # two; one column tile, 37 segments of one stage: the most there are
    (7104, 8, 256, 3),     # six; four column tiles, 37 segments of three stages
    (769, 40, 64, 3),      # thirteen segments of one stage: one more than the short sum of the step takes
    (768, 40, 64, 3),      # twelve
])
def test_distillation_splits(T, N, d, iters):
    """Warps per forward CTA and token segments of the backward pass, at the edges of their rules (fp64 on both sides, fp32
    outputs: half an ulp of values below 8, and sums in another order, are well inside 2e-6)."""
    from oracle import distill
    build.build()
    rng = np.random.default_rng(T)
    H = rng.standard_normal((T, d)).astype(np.float32)
    Z = rng.standard_normal((T, N))
    Qr = (np.exp(Z) / np.exp(Z).sum(1, keepdims=True)).astype(np.float32)
    W0 = (rng.standard_normal((N, d)) / np.sqrt(d)).astype(np.float32)
    b0 = rng.standard_normal(N).astype(np.float32)
    W_ref, b_ref = distill.distill(H, Qr, W0, b0, iters=iters, lr=0.01)
    W, b = binding.distill_router(torch.from_numpy(H).cuda(), torch.from_numpy(Qr).cuda(), W0, b0, iters=iters, lr=0.01)
    assert np.abs(W - W_ref).max() <= 2e-6 * max(1.0, float(np.abs(W_ref).max()))
    assert np.abs(b - b_ref).max() <= 2e-6 * max(1.0, float(np.abs(b_ref).max()))


def test_training_calls_from_two_threads_share_the_workspace_pool():
    """Two threads on two streams, different sizes in turn: what each gets is what it gets alone."""
    import threading
    build.build()
    g = torch.Generator(device="cuda").manual_seed(3)
    jobs = []
    for T, N, d in ((700, 9, 128), (3000, 40, 512)):
        H = torch.randn((T, d), generator=g, device="cuda")
        Qr = torch.softmax(torch.randn((T, N), generator=g, device="cuda"), 1).contiguous()
        jobs.append((H, Qr, np.zeros((N, d), np.float32), np.zeros(N, np.float32)))
    torch.cuda.synchronize()
    alone = [binding.distill_router(*j, iters=5) for j in jobs]
    got, errors = {}, []

    def work(i):
        try:
            s = torch.cuda.Stream()
            got[i] = [binding.distill_router(*jobs[(i + r) % 2], iters=5, stream=s) for r in range(6)]
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        for r in range(6):
            for a, b in zip(got[i][r], alone[(i + r) % 2]):
                np.testing.assert_array_equal(a, b)


def test_training_scratch_goes_back():
    """More than half a GB of scratch: at most 64 MB of it are kept when the call returns, and none after the trim."""
    build.build()
    H, Qr = torch.randn((1_000_000, 64), device="cuda"), torch.full((1_000_000, 64), 1.0 / 64, device="cuda")
    W0, b0 = np.zeros((64, 64), np.float32), np.zeros(64, np.float32)
    X, dstar = torch.softmax(torch.randn((500, 9), device="cuda", dtype=torch.float64), 1).sort(1, descending=True)[0].contiguous(), torch.zeros(500, dtype=torch.int32, device="cuda")
    binding.distill_router(H[:1000], Qr[:1000], W0, b0, iters=1)      # (modules and the pool itself are there from here on)
    binding.fit_cdf(X, dstar, 2, iters=2)
    torch.cuda.synchronize()
    binding.trim_scratch()
    free = torch.cuda.mem_get_info()[0]
    binding.distill_router(H, Qr, W0, b0, iters=1)
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    binding.fit_cdf(X, dstar, 2, iters=2)
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    binding.trim_scratch()
    assert torch.cuda.mem_get_info()[0] == free
