"""The work whose speed this framework is judged by, through its public entry points.

Every case is one call (or, for training, one forward and its backward) as a user's program makes it.  The sizes
are those of the benchmark configurations and of the test suite, from the smallest call to a 32768-token prefill:
latency-bound single tiles, ordinary prefills and training shapes, ragged sequence lengths, odd GQA groups, partial
rotary widths, sliding window with ALiBi, block lists, 8-bit operands, and decoding against short and long caches.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_13612_b200 as af


def listed():
    return [
        # the smallest forward: one query tile of two heads; launch and host latency are all there is
        dict(name="fwd_tiny", op="fwd", B=1, Hq=2, Hkv=2, S=128, D=64, R=64, theta=1e4),
        # prefill of a 4096-token prompt in a grouped-query model of Llama-3-8B's geometry: the headline workload
        dict(name="fwd_llama3_8b", op="fwd", B=1, Hq=32, Hkv=8, S=4096, D=128, R=128, theta=5e5),
        # the same prefill as a server would run it: four prompts, keys rotated once (the recommended arm with GQA)
        dict(name="hybrid_batch4", op="hybrid", B=4, Hq=32, Hkv=8, S=2048, D=128, R=128, theta=5e5),
        # composed variant: RoPE, sliding window and ALiBi, no grouped queries
        dict(name="fwd_window_alibi", op="fwd", B=2, Hq=16, Hkv=16, S=8192, D=128, R=128, theta=1e4, window=1024, alibi=True),
        # prefill of a long document
        dict(name="fwd_long", op="fwd", B=1, Hq=32, Hkv=8, S=32768, D=128, R=128, theta=5e5, sigma=0.5),
        # prefill with 8-bit operands (rotation and quantisation done before the call)
        dict(name="fwd_fp8", op="fp8", B=1, Hq=32, Hkv=8, S=4096, D=128, R=0, theta=1e4),
        # training step of the Llama-3-8B geometry, and of GPT-2 small's (D = 64, no grouped queries)
        dict(name="train_llama3_8b", op="train", B=4, Hq=32, Hkv=8, S=2048, D=128, R=128, theta=5e5),
        dict(name="train_gpt2_small", op="train", B=4, Hq=12, Hkv=12, S=4096, D=64, R=64, theta=1e4),
        # a short ragged training step: odd length, odd group, partial rotary width, window and ALiBi
        dict(name="train_ragged", op="train", B=2, Hq=6, Hkv=2, S=777, D=128, R=64, theta=1e4, window=300, alibi=True),
        # training over block lists (a BigBird-like pattern in the same GPT-2 small geometry)
        dict(name="train_blocks", op="train", B=4, Hq=12, Hkv=12, S=4096, D=64, R=64, theta=1e4, causal=False, blocks=1),
        # decoding one token: a short cache (latency) and a large model's 32768-token cache (HBM)
        dict(name="decode_8b_4k", op="decode", B=1, Hq=32, Hkv=8, S=4096, D=128, R=0, theta=1e4),
        dict(name="decode_70b_32k", op="decode", B=1, Hq=64, Hkv=8, S=32768, D=128, R=0, theta=1e4),
    ]


def draw(rng):
    """One more case of the same kinds.  Lengths are spread over their logarithm, odd ones among them; batch sizes follow
    from a bound on the kept pairs, so that no drawn case costs more than the largest listed one."""
    op = rng.choice(["fwd", "fwd", "hybrid", "train", "train", "blocks", "decode", "decode", "fp8"])
    D = 128 if op == "fp8" else rng.choice([64, 128, 128])
    group = rng.choice([1, 2, 3, 4, 8])
    Hkv = rng.choice([1, 2, 4, 8, 12])
    while group * Hkv > 64:
        Hkv //= 2
    top = {"fwd": 16384, "hybrid": 16384, "train": 8192, "blocks": 8192, "decode": 65536, "fp8": 16384}[op]
    S = int(round(math.exp(rng.uniform(math.log(128 if op != "decode" else 256), math.log(top)))))
    if rng.random() < 0.3:   # whole tiles are as common as odd lengths
        S = max(128, S // 128 * 128)
    if op == "fp8":
        S = S // 16 * 16
    c = dict(op=op, B=1, Hq=group * Hkv, Hkv=Hkv, S=S, D=D, R=0, theta=rng.choice([1e4, 5e5]))
    if op not in ("decode", "fp8"):
        c["R"] = rng.choice([D, D, D, D // 2, 0 if op != "hybrid" else D])
    if op in ("fwd", "train", "decode") and rng.random() < 0.35:
        c["window"] = int(round(math.exp(rng.uniform(math.log(100), math.log(S + 100)))))
        c["alibi"] = rng.random() < 0.6
    if op == "fwd" and rng.random() < 0.15:
        c["causal"] = False
    if op == "blocks":
        c.update(op="train", causal=False, blocks=rng.randrange(2, 1000))
    # batch: up to a few thousand million kept pairs, and caches of at most 256 MB
    budget = 2e9 if op != "decode" else 1e9
    cost = float(c["Hq"]) * S * (S if op != "decode" else D)
    c["B"] = max(1, min(rng.choice([1, 2, 3, 4, 8, 16]), int(budget / cost)))
    return c


def _mask_blocks(case):
    """Active 128 x 128 blocks: diagonal, one global row and column of blocks, one random block per row."""
    nb = (case["S"] + 127) // 128
    rng = np.random.default_rng(case["blocks"])
    act = np.eye(nb, dtype=bool)
    act[:, 0] = True
    act[0, :] = True
    act[np.arange(nb), rng.integers(0, nb, size=nb)] = True
    return act


def _pairs(case):
    """Kept (query, key) pairs of one head."""
    S, w = case["S"], case.get("window", -1)
    if case["op"] == "decode":
        return S if w < 0 else min(S, w + 1)
    if case.get("blocks"):
        act = _mask_blocks(case)
        n = np.full(act.shape[0], 128.0)
        n[-1] = S - 128 * (act.shape[0] - 1)
        return float(n @ act @ n)
    if not case.get("causal", True):
        if w < 0:
            return float(S) * S
        w = min(w, S - 1)
        return float(S) * (2 * w + 1) - float(w) * (w + 1)
    w = S - 1 if w < 0 else min(w, S - 1)
    return float(S) * (w + 1) - w * (w + 1) / 2.0


def work(case):
    B, Hq, Hkv, S, D = (case[k] for k in ("B", "Hq", "Hkv", "S", "D"))
    fwd_flops = 4.0 * D * _pairs(case) * B * Hq
    if case["op"] == "decode":
        kept = _pairs(case)
        return {"bytes": 2.0 * B * Hkv * kept * D * 2 + 2.0 * B * Hq * D * 2 + 4.0 * B * Hq, "flops": fwd_flops}
    q, kv, lse = float(B) * Hq * S * D, float(B) * Hkv * S * D, 4.0 * B * Hq * S
    if case["op"] == "fp8":
        return {"bytes": q + 2 * kv + 2 * q + lse, "flops": fwd_flops}
    fwd_bytes = 2 * q + 4 * kv + 2 * q + lse
    if case["op"] != "train":
        return {"bytes": fwd_bytes, "flops": fwd_flops}
    # a training step: forward; then q, k, v, o, dO and L in, dQ (bf16), dK and dV (fp32) out
    return {"bytes": fwd_bytes + 2 * q + 4 * kv + 4 * q + lse + 2 * q + 8 * kv, "flops": 3.5 * fwd_flops}


def tolerance(case):
    # Against the same path in fp64 on the same inputs the bf16 path's outputs and gradients are off by 1.6e-3 to
    # 3.8e-3 (2-norm; the roundings of q', k', P, dS and the outputs, 2^-9 each) and by up to 0.075 of the root mean
    # square at one element; the 8-bit path by 2.1e-2 and 0.43 (P in E4M3).
    if case["op"] == "fp8":
        return {"rel": 0.03, "max": 0.6}
    return {"rel": 0.012, "max": 0.3}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    B, Hq, Hkv, S, D, op = (case[k] for k in ("B", "Hq", "Hkv", "S", "D", "op"))
    sigma = case.get("sigma", 1.0)

    def normal(*shape):
        return (torch.randn(*shape, generator=gen, device="cuda") * sigma).to(torch.bfloat16)

    st = {"op": op, "scale": 1.0 / math.sqrt(D)}
    slopes = None
    if case.get("alibi"):
        slopes = torch.tensor([2.0 ** (-8.0 * (h + 1) / Hq) for h in range(Hq)], dtype=torch.float32, device="cuda")
    st["mask"] = af.MaskSpec(causal=case.get("causal", True), window=case.get("window", -1), alibi_slopes=slopes)
    if op == "decode":
        st["q"] = normal(B, Hq, D)
        st["k"], st["v"] = normal(B, Hkv, S, D), normal(B, Hkv, S, D)
        st["workspace"] = af.decode_workspace(B, Hq, Hkv, S, D)
        return st
    q, k, v = normal(B, Hq, S, D), normal(B, Hkv, S, D), normal(B, Hkv, S, D)
    if op == "fp8":
        st["q"], st["k"] = q.to(torch.float8_e4m3fn), k.to(torch.float8_e4m3fn)
        st["v"] = v.transpose(2, 3).contiguous().to(torch.float8_e4m3fn)
        return st
    st["q"], st["k"], st["v"] = q, k, v
    st["rope"] = af.RopeSpec(theta=case["theta"], rotary_dim=case["R"])
    st["table"] = af.rope_table(st["rope"], S)
    st["blocks"] = af.BlockMask(_mask_blocks(case)) if case.get("blocks") else None
    if op == "hybrid":
        st["workspace"] = torch.empty(B * Hkv * S * D * 2, dtype=torch.uint8, device="cuda")
    if op == "train":
        st["do"] = normal(B, Hq, S, D)
        st["workspace"] = torch.empty(af.bwd_workspace_bytes(B, Hq, Hkv, S, D), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    op = st["op"]
    if op == "decode":
        return af.decode(st["q"], st["k"], st["v"], st["mask"], st["scale"], workspace=st["workspace"])
    if op == "fp8":
        return af.fwd_fp8(st["q"], st["k"], st["v"], st["mask"], st["scale"])
    args = (st["q"], st["k"], st["v"], st["rope"], st["table"], st["mask"], st["scale"])
    if op == "hybrid":
        return af.fwd_hybrid(*args, workspace=st["workspace"])
    if st["blocks"] is not None:
        o, lse = af.fwd_blocks(*args, st["blocks"])
    else:
        o, lse = af.fwd(*args)
    if op == "fwd":
        return o, lse
    dq, dk, dv = af.bwd(st["q"], st["k"], st["v"], o, lse, st["do"], st["rope"], st["table"], st["mask"], st["scale"],
                        workspace=st["workspace"], blocks=st["blocks"])
    return o, lse, dq, dk, dv
