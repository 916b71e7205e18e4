"""Performance cases of the MoE decode library: what its users run, through the public entry points.

A case is a dict of plain values.  ``kind`` says which entry points it goes through:

* ``gate``     the context-free exact gate (``route_topk_static``): one small launch per call
* ``steps``    one layer-step after the other through the six separate calls of a caller that sequences the layers itself
* ``token``    all layers of a batch-1 decode token (``decode_token``, or ``decode_token_host`` with ``host``)
* ``batch``    all layers of a decode step of several tokens (``decode_token``)
* ``fit``      the confidence-model fit (``fit_cdf``)
* ``distill``  the distillation of the prefetch router (``distill_router``)

Decoding has one direction (forward) and no backward; the two training stages of the method are the last two kinds.
``C == N``: every expert is resident (what a 180 GB GPU affords for these models); ``C < N``: experts are copied from
pinned host memory while the step runs.  ``stores``: different host stores per context (layer l uses store l mod stores;
every layer has its own slots in HBM).  A context keeps several decode tokens and a pass takes the next one, as a
decode loop does, so that a limited cache keeps missing.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_11688_b200 import binding, synth

DEVICE = "cuda"
CTX_LEN = 1024          # the library's default context length (sizes the attention stand-in)
TOKENS = 8              # decode tokens a state holds
FMT_FLAGS = {"bf16": 0, "e4m3": binding.FLAG_FP8_EXPERTS, "e2m1": binding.FLAG_FP4_EXPERTS}


def _decode(name, kind, cfg_id, *, L, B, C=None, fmt="bf16", mode="exact", host=False, stores=1):
    """A decode case with the shape of one of the repository's configurations."""
    c = synth.CONFIGS[cfg_id]
    return {"name": name, "kind": kind, "cdf": cfg_id, "L": L, "d": c.d, "N": c.N, "k": c.k, "I": c.I, "I_shared": c.I_shared,
            "C": C or c.N, "B": B, "fmt": fmt, "mode": mode, "host": host, "tau": 0.9, "zipf_s": c.zipf_s,
            "sigma_p": c.sigma_p, "stores": stores}


def listed():
    return [
        # a serving process asks for the routed experts of one token: latency of one call
        {"name": "gate_b1", "kind": "gate", "N": 32, "d": 1024, "k": 8, "B": 1},
        # a caller that runs the layers itself, the single-layer configuration: launches and host work dominate
        _decode("steps_layer", "steps", 0, L=1, B=1),
        # the headline workload: batch-1 decode with half the experts in HBM, host buffers in and out
        _decode("token_slots_host", "token", 1, L=32, B=1, C=20, host=True, stores=4),
        # the same model with every expert resident: small experts, the per-layer chain dominates
        _decode("token_resident", "token", 1, L=32, B=1, mode="stall_free"),
        # one-byte expert weights, skewed expert popularity
        _decode("token_e4m3", "token", 2, L=16, B=1, fmt="e4m3"),
        # the largest experts: HBM streaming
        _decode("token_large", "token", 3, L=4, B=1),
        # a few concurrent requests, with the always-on shared expert
        _decode("batch_8", "batch", 4, L=4, B=8),
        # the largest decode step
        _decode("batch_256", "batch", 4, L=4, B=256),
        # an odd batch on half-byte expert weights
        _decode("batch_37_e2m1", "batch", 2, L=4, B=37, fmt="e2m1", mode="stall_free"),
        # a batched step with half the experts in HBM: prefetch and demand copies over the host link
        _decode("batch_32_slots", "batch", 4, L=2, B=32, C=30),
        # calibration, second stage: one layer's confidence model
        {"name": "fit_cdf", "kind": "fit", "T": 8192, "N": 40, "k": 8, "iters": 600},
        # calibration, first stage: one layer's prefetch router
        {"name": "distill", "kind": "distill", "T": 8192, "N": 40, "d": 1536, "iters": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_decode(rng, kind):
    fmt = rng.choice(("bf16", "bf16", "bf16", "e4m3", "e2m1"))
    d = rng.choice((512, 1024, 1536, 2048, 4096) if fmt != "bf16" else (256, 512, 768, 1024, 1536, 2048, 3072, 4096))
    N = _log_int(rng, 8, 64)
    k = rng.randint(1, min(8, N // 2))
    if kind == "batch":     # a multiple of 128, now and then one of 64
        unit = 64 if rng.random() < 0.25 else 128
        I = unit * _log_int(rng, 2, 4096 // unit)
        I_shared = 128 * _log_int(rng, 2, 44) if rng.random() < 0.4 else 0
        B = _log_int(rng, 2, 256)
    else:
        I = _log_int(rng, 128, 14336)
        I_shared = _log_int(rng, 128, 5632) if rng.random() < 0.25 else 0
        B = 1 if kind == "token" else _log_int(rng, 1, 8)
    slots = kind != "steps" and rng.random() < 0.25
    return {"kind": kind, "cdf": -1, "L": 1 if kind == "steps" else _log_int(rng, 1, 32), "d": d, "N": N, "k": k, "I": I,
            "I_shared": I_shared, "C": max(k, (N + 1) // 2) if slots else N, "B": B, "fmt": fmt,
            "mode": rng.choice(("exact", "stall_free")) if not slots else "exact", "host": rng.random() < 0.25 and kind != "steps",
            "tau": rng.choice((0.5, 0.75, 0.9)), "zipf_s": rng.choice((0.0, 1.1)), "sigma_p": rng.choice((0.3, 0.5)), "stores": 1}


def draw(rng):
    while True:
        kind = rng.choice(("gate", "steps", "token", "token", "token", "batch", "batch", "batch", "batch", "fit", "distill"))
        if kind == "gate":
            N = _log_int(rng, 8, 64)
            return {"kind": kind, "N": N, "d": rng.choice((256, 512, 768, 1024, 1536, 2048, 2880, 4096)),
                    "k": rng.randint(1, min(8, N)), "B": _log_int(rng, 1, 64)}
        if kind == "fit":
            N = rng.randint(8, 64)
            return {"kind": kind, "T": _log_int(rng, 256, 8192), "N": N, "k": rng.randint(1, min(8, N)), "iters": _log_int(rng, 100, 600)}
        if kind == "distill":
            c = {"kind": kind, "T": _log_int(rng, 256, 8192), "N": rng.randint(8, 64), "d": rng.choice((256, 768, 1024, 1536, 2048)),
                 "iters": _log_int(rng, 20, 100)}
            if c["T"] * c["N"] * c["d"] * c["iters"] <= 8192 * 40 * 1536 * 100:
                return c
            continue
        c = _draw_decode(rng, kind)
        expert = _row_bytes(c) * c["I"]
        copied = c["L"] * (c["N"] if c["B"] > 1 else c["C"]) * expert if c["C"] < c["N"] else 0
        # no larger than the listed ones: HBM for the slots, the host store, the bytes of a pass, the copies of a pass
        rows = c["B"] * c["k"] if c["I"] % 128 else _distinct(c)     # how often expert rows are read
        if c["L"] * c["C"] * expert <= 6e9 and c["N"] * expert <= 2.8e9 and work(c)["bytes"] <= 4e9 and copied <= 1e9 \
                and c["L"] * rows * expert <= 8e9:
            return c


def _row_bytes(case):
    """Bytes of one intermediate index of an expert: three vectors of d weights and their scales."""
    d = case["d"]
    return {"bf16": 6 * d, "e4m3": 3 * d + 16, "e2m1": synth.fp4_row_bytes(d)}[case["fmt"]]


def _store(case, gen, n, rows):
    """n experts of `rows` intermediate indices in the store layout and format, weights ~ N(0, 0.02^2), on the GPU."""
    d = case["d"]
    quantize = {"bf16": None, "e4m3": synth.quantize_store_fp8, "e2m1": synth.quantize_store_fp4}[case["fmt"]]
    parts = []
    step = max(1, int(3e8) // (3 * d * rows))
    for e in range(0, n, step):
        w = torch.empty((min(step, n - e), rows, 3, d), dtype=torch.bfloat16, device=DEVICE)
        w.normal_(0.0, 0.02, generator=gen)
        parts.append(w if quantize is None else quantize(w))
    return parts[0] if len(parts) == 1 else torch.cat(parts)


def _hidden(gen, shape):
    """h ~ N(0, 1) and h' = h + N(0, 0.25), bf16-representable values in fp32."""
    h = torch.randn(shape, generator=gen, device=DEVICE)
    hp = h + 0.5 * torch.randn(shape, generator=gen, device=DEVICE)
    return h.bfloat16().float(), hp.bfloat16().float()


def _prepare_decode(case, gen):
    L, d, N, k, I, B = (case[n] for n in ("L", "d", "N", "k", "I", "B"))
    a = binding.Apex(d=d, N=N, k=k, I=I, C_slots=case["C"], L=L, I_shared=case["I_shared"], max_batch=B, ctx_len=CTX_LEN,
                     flags=FMT_FLAGS[case["fmt"]])
    stores = []
    for _ in range(min(case["stores"], L)):
        w = _store(case, gen, N, I)
        s = torch.empty(w.shape, dtype=w.dtype, pin_memory=True)
        s.copy_(w)
        stores.append(s)
        del w
    for l in range(L):
        W_r = torch.randn((N, d), generator=gen, device=DEVICE) / math.sqrt(d)
        W_p = W_r + torch.randn((N, d), generator=gen, device=DEVICE) * (case["sigma_p"] / math.sqrt(d))
        b = np.zeros(N, np.float32)
        if case["zipf_s"] > 0:   # skewed popularity: 0.5 ln of Zipf frequencies over a random order of the experts
            perm = torch.randperm(N, generator=gen, device=DEVICE).cpu().numpy()
            f = (perm + 1.0) ** (-case["zipf_s"])
            b = (0.5 * np.log(f / f.sum())).astype(np.float32)
        a.set_router(l, W_r.cpu().numpy(), b)
        a.set_prefetch_router(l, W_p.cpu().numpy(), b)
        if case["cdf"] >= 0:
            a.set_cdf(l, *synth.cdf_params(synth.CONFIGS[case["cdf"]], l))
        else:
            a.set_cdf(l, *synth.handset_cdf_params(synth.tiny_config(d=d, N=N, k=k, I=I, C=case["C"])))
        a.register_experts(l, stores[l % len(stores)])
        if case["I_shared"] > 0:
            a.set_shared_expert(l, _store(case, gen, 1, case["I_shared"])[0])
    if case["C"] == N:
        a.warm_all()
    h, hp = _hidden(gen, (TOKENS, L, B, d))
    st = {"apex": a, "case": case, "t": 0}
    if case["host"]:
        st["h"], st["hp"] = h.cpu().pin_memory(), hp.cpu().pin_memory()
        st["y"] = torch.zeros((L, B, d), pin_memory=True)
    else:
        st["h"], st["hp"] = h, hp
        st["y"] = torch.zeros((L, B, d), device=DEVICE)
    if case["kind"] == "steps":
        i32 = dict(dtype=torch.int32, device=DEVICE)
        st["cand"], st["ncand"] = torch.zeros((L, B, case["C"]), **i32), torch.zeros((L, B), **i32)
        st["idx"], st["exec_idx"] = torch.zeros((L, B, k), **i32), torch.zeros((L, B, k), **i32)
        st["alpha"] = torch.zeros((L, B, N), device=DEVICE)
        st["exec_gate"] = torch.zeros((L, B, k), device=DEVICE)
    return st


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    kind = case["kind"]
    if kind == "gate":
        N, d, k, B = (case[n] for n in ("N", "d", "k", "B"))
        return {"case": case, "t": 0, "W": torch.randn((N, d), generator=gen, device=DEVICE) / math.sqrt(d),
                "b": torch.randn((N,), generator=gen, device=DEVICE) * 0.1, "hp": _hidden(gen, (TOKENS, B, d))[1],
                "idx": torch.zeros((B, k), dtype=torch.int32, device=DEVICE), "alpha": torch.zeros((B, N), device=DEVICE)}
    if kind in ("fit", "distill"):
        T, N = case["T"], case["N"]
        if kind == "fit":
            # prediction and routing of T tokens with a noisy predictor: x sorted descending, delta* = last rank needed - k
            k = case["k"]
            z = torch.randn((T, N), generator=gen, device=DEVICE, dtype=torch.float64)
            zr = z + 0.5 * torch.randn((T, N), generator=gen, device=DEVICE, dtype=torch.float64)
            X, order = torch.softmax(z, 1).sort(1, descending=True)
            rank = torch.empty_like(order).scatter_(1, order, torch.arange(N, device=DEVICE).expand(T, N))
            dstar = rank.gather(1, zr.topk(k, 1).indices).amax(1) + 1 - k
            return {"case": case, "X": X.contiguous(), "dstar": dstar.to(torch.int32).contiguous()}
        d = case["d"]
        H, Hp = _hidden(gen, (T, d))
        W_r = torch.randn((N, d), generator=gen, device=DEVICE) / math.sqrt(d)
        Qr = torch.softmax(Hp @ W_r.T, 1).contiguous()
        W0 = (W_r + torch.randn((N, d), generator=gen, device=DEVICE) * (0.3 / math.sqrt(d))).cpu().numpy()
        return {"case": case, "H": H, "Qr": Qr, "W0": W0, "b0": np.zeros(N, np.float32)}
    return _prepare_decode(case, gen)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fit":
        return binding.fit_cdf(state["X"], state["dstar"], case["k"], iters=case["iters"])
    if kind == "distill":
        return binding.distill_router(state["H"], state["Qr"], state["W0"], state["b0"], iters=case["iters"], lr=1e-4)
    t = state["t"]
    state["t"] = (t + 1) % TOKENS
    if kind == "gate":
        binding.route_topk_static(state["W"], state["b"], state["hp"][t], case["k"], state["idx"], state["alpha"])
        return {"idx": state["idx"], "alpha": state["alpha"]}
    a, h, hp, y, B, tau, mode = state["apex"], state["h"][t], state["hp"][t], state["y"], case["B"], case["tau"], case["mode"]
    if kind == "steps":
        for l in range(case["L"]):
            a.predict(l, h[l], B)
            a.select_candidates(l, B, tau, state["cand"][l], state["ncand"][l])
            a.prefetch(l, B)
            a.attention_standin(l)
            a.route_topk(l, hp[l], B, state["idx"][l], state["alpha"][l])
            a.moe_ffn(l, mode, hp[l], B, y[l], state["exec_idx"][l], state["exec_gate"][l])
        return {n: state[n] for n in ("y", "cand", "ncand", "idx", "alpha", "exec_idx", "exec_gate")}
    if case["host"]:
        a.decode_token_host(h, hp, B, tau, mode, y)
    else:
        a.decode_token(h, hp, B, tau, mode, y)
    if case["C"] == case["N"]:
        return y
    tables = [a.get_slot_table(l)[:2] for l in range(case["L"])]   # a limited cache is state that the step updates
    return {"y": y, "expert_slot": np.stack([s for s, _ in tables]), "slot_stamp": np.stack([s for _, s in tables])}


def _distinct(case):
    """Experts of a layer that a step executes: k for one token, the expected number of distinct ones for a batch."""
    N, k, B = case["N"], case["k"], case["B"]
    return N * (1.0 - (1.0 - k / N) ** B)


def work(case):
    kind = case["kind"]
    if kind == "fit":
        T, N, nth = case["T"], case["N"], case["N"] - case["k"] + 1
        return {"bytes": T * (8 * N + 4) + 4 * (N + nth), "flops": case["iters"] * T * (4 * N + 4 * nth)}
    if kind == "distill":
        T, N, d = case["T"], case["N"], case["d"]
        return {"bytes": 4 * T * (d + N) + 8 * N * (d + 1), "flops": 4 * case["iters"] * T * N * d}
    N, d, k, B = (case[n] for n in ("N", "d", "k", "B"))
    if kind == "gate":
        return {"bytes": 4 * (N * d + N + B * d + B * k + B * N), "flops": 2 * B * N * d}
    rows = _distinct(case) * case["I"] + case["I_shared"]
    layer = rows * _row_bytes(case) + 2 * 4 * N * d + 3 * 4 * B * d + 2 * (4 * d * d + 2 * CTX_LEN * d)
    return {"bytes": case["L"] * layer, "flops": case["L"] * B * (6 * d * (k * case["I"] + case["I_shared"]) + 4 * N * d)}


def tolerance(case):
    if case["kind"] in ("gate", "fit", "distill"):
        return {"rel": 1e-5}      # fp32 sums and softmax; fp64 fits rounded to fp32
    return {"rel": 3e-5}          # fp32 sums over exact weights; the batched path carries its intermediate to 2^-17
