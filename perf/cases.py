"""Workloads that performance is measured on, through the public entry points of the package.

Three kinds of call:
  step    bf16 Q, K, V on the device -> the quantizers and the attention forward -> O, LSE
  encode  the quantizers alone (operands that are quantized once and kept, K and V of a fixed context say)
  host    bf16 Q, K, V in pinned host memory -> fp4attn_attention_host -> O, LSE in pinned host memory

Sizes: head dimension 64 and 128, sequences of 128 to 32768 keys in whole 128-key tiles (any length below that as a
padded sequence), from one head up to about a million (head, token) rows.
"""
import math
import random

import torch

from paper_2609_04105_b200 import binding as fp4

# what one listed case at most costs: scores (batch x heads x N x N), rows (batch x heads x N) x head dimension, and the
# same for host buffers, whose preparation (pinning) is slow
MOST_SCORES = 16 * 32768 ** 2
MOST_ELEMENTS = 16 * 32768 * 128
MOST_HOST_ELEMENTS = 2 * 16 * 4096 * 128


def _case(kind, B, H, N, d, qk="mxfp4", kv_heads=0, p_map="ideal", p_rule="ceil", causal=False, ragged=False, pv="mxfp4",
          outliers=False, fixed_reference=False, schedule="one"):
    return {"kind": kind, "B": B, "H": H, "N": N, "d": d, "qk": qk, "kv_heads": kv_heads or H, "p_map": p_map, "p_rule": p_rule,
            "causal": causal, "ragged": ragged, "pv": pv, "outliers": outliers, "fixed_reference": fixed_reference,
            "schedule": schedule}


def listed():
    return [
        # the smallest call: a few query tiles, where the launches and the host's share of them are what a user waits for
        dict(_case("step", 1, 2, 256, 128), name="small"),
        # many short sequences in one batch: item boundaries, little reuse of K and V
        dict(_case("step", 32, 16, 1024, 128), name="batch_1k"),
        # one ordinary sequence of one layer with the paper's affine classifier
        dict(_case("step", 1, 16, 4096, 128, p_map="affine"), name="single_4k_affine"),
        # NVFP4 Q and K at head dimension 64
        dict(_case("step", 8, 16, 8192, 64, qk="nvfp4"), name="nvfp4_d64_8k"),
        # outlier channels in Q and K: large logits, a row reference that moves
        dict(_case("step", 1, 32, 16384, 128, outliers=True), name="outliers_16k"),
        # the longest sequence (video or long-context lengths): the headline workload
        dict(_case("step", 1, 16, 32768, 128), name="long_32k"),
        # the `fast` policy: affine classifier and constant row reference
        dict(_case("step", 4, 16, 8192, 128, p_map="affine", fixed_reference=True), name="fast_8k"),
        # the forward of a training step: causal, grouped K/V heads, one NVFP4 factor per head for the backward
        dict(_case("step", 2, 32, 4096, 128, qk="nvfp4_per_head", kv_heads=8, causal=True), name="causal_gqa_4k"),
        # a serving batch of sequences of unlike, odd lengths in padded buffers
        dict(_case("step", 6, 12, 2176, 64, p_rule="thr16", ragged=True), name="ragged_2k"),
        # FP8 probabilities and values (the training route)
        dict(_case("step", 2, 16, 8192, 128, pv="e4m3"), name="fp8_pv_8k"),
        # operands that live in host memory: copies in, the whole path, copies out
        dict(_case("host", 2, 16, 4096, 128, qk="nvfp4"), name="host_4k"),
        # quantization by itself, larger than the L2 cache
        dict(_case("encode", 4, 16, 8192, 128, qk="nvfp4"), name="encode_8k"),
    ]


def draw(rng):
    while True:
        kind = rng.choices(("step", "encode", "host"), (7, 2, 1))[0]
        d = rng.choice((64, 128))
        N = 128 * round(math.exp(rng.uniform(0.0, math.log(256))))
        H = rng.choice((1, 2, 3, 4, 5, 8, 12, 16, 24, 32, 40))
        B = round(math.exp(rng.uniform(0.0, math.log(64))))
        kw = {"qk": rng.choice(("mxfp4", "mxfp4", "nvfp4", "nvfp4_per_head"))}
        if kind == "host" and kw["qk"] == "nvfp4_per_head":
            kw["qk"] = "nvfp4"
        if kind == "step":
            kw["outliers"] = rng.random() < 0.15
            kw["kv_heads"] = rng.choice([h for h in (1, 2, 3, 4, 5, 8, 12, 16, 24, 32, 40) if H % h == 0]) if rng.random() < 0.3 else H
            per_head = kw["qk"] == "nvfp4_per_head"
            route = rng.choices(("plain", "fast", "fp8", "two", "hybrid", "mse"), (14, 2, 3, 1, 1, 1))[0]
            if route == "fast" and not per_head and not kw["outliers"]:
                kw.update(p_map="affine", fixed_reference=True)
            elif route == "fp8" and not per_head:
                kw.update(pv="e4m3")
            elif route == "two" and d == 64 and N % 256 == 0 and not per_head:
                kw.update(schedule="two", p_map=rng.choice(("ideal", "affine")))
            elif route == "hybrid" and not per_head:
                kw.update(p_map="hybrid8")
            elif route == "mse" and not per_head:
                kw.update(p_rule="mse")
            else:
                kw.update(p_map=rng.choice(("ideal", "ideal", "affine")), p_rule=rng.choices(("ceil", "thr16"), (5, 1))[0])
            if kw.get("schedule") != "two" and kw.get("p_map") != "hybrid8":
                kw["causal"] = rng.random() < 0.3
                kw["ragged"] = B <= 16 and rng.random() < 0.25
        elif kind == "encode" and kw["qk"] == "mxfp4":
            kw["pv"] = rng.choice(("mxfp4", "e4m3"))
        most = MOST_SCORES * (2 if kw.get("pv") != "e4m3" and kw.get("causal") else 1) // (2 if kw.get("pv") == "e4m3" else 1)
        if kind != "encode" and B * H * N * N > most:
            continue
        if B * H * N * d > (MOST_HOST_ELEMENTS if kind == "host" else MOST_ELEMENTS):
            continue
        return _case(kind, B, H, N, d, **kw)


def _lengths(case):
    """Token counts of a padded batch: one sequence fills its buffer, the others have any length from N / 8 on."""
    r = random.Random(case["B"] * 1000003 + case["N"])
    return [case["N"]] + [r.randint(max(1, case["N"] // 8), case["N"]) for _ in range(case["B"] - 1)]


def _tensor(case, heads, gen, outlier_channels=None):
    shape = (case["B"], heads, case["N"], case["d"])
    x = torch.randn(shape, generator=gen, dtype=torch.float32, device="cuda")
    if outlier_channels is not None:
        x[..., outlier_channels] *= 20.0                # 2 % of the channels, the same in Q and K
    if case["ragged"]:
        for b, n in enumerate(_lengths(case)):
            x[b, :, n:] = 0.0                           # what lies beyond a sequence is zero, as the quantizers ask for
    return x.to(torch.bfloat16)


_P_MAP = {"ideal": fp4.PMAP_IDEAL, "affine": fp4.PMAP_AFFINE, "hybrid8": fp4.PMAP_HYBRID}
_P_RULE = {"ceil": fp4.PSCALE_CEIL, "thr16": fp4.PSCALE_THR16, "mse": fp4.PSCALE_MSE}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    channels = None
    if case["outliers"]:
        channels = torch.randperm(case["d"], generator=gen, device="cuda")[: max(1, round(0.02 * case["d"]))]
    x = [_tensor(case, case["H"], gen, channels), _tensor(case, case["kv_heads"], gen, channels), _tensor(case, case["kv_heads"], gen)]
    s = {"kind": case["kind"], "qk": case["qk"], "pv": case["pv"]}
    if case["kind"] == "host":
        s["x"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in x]
        for h, t in zip(s["x"], x):
            h.copy_(t)
        s["fmt"] = fp4.FMT_MXFP4 if case["qk"] == "mxfp4" else fp4.FMT_NVFP4
        s["out"] = torch.empty(x[0].shape, dtype=torch.bfloat16, pin_memory=True)
        s["lse"] = torch.empty(x[0].shape[:3], dtype=torch.float32, pin_memory=True)
        n = fp4.fp4attn_attention_host_workspace_bytes(s["fmt"], case["B"], case["H"], case["N"], case["d"])
        s["workspace"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        return s
    s["x"] = x
    s["options"] = {"p_map": _P_MAP[case["p_map"]], "p_scale_rule": _P_RULE[case["p_rule"]], "causal": case["causal"]}
    if case["p_map"] == "hybrid8":
        s["options"]["exact_pairs"] = 0x5555
    if case["schedule"] == "two":
        s["options"]["schedule"] = fp4.SCHEDULE_TWO_QUERY
    if case["fixed_reference"]:
        s["options"]["fixed_reference"] = 0
    if case["ragged"]:
        s["lengths"] = _lengths(case)
        s["options"]["seq_len"] = torch.tensor(s["lengths"], dtype=torch.int32, device="cuda")
    return s


def _quantize_qk(x, role, qk):
    if qk == "nvfp4_per_head":
        return fp4.fp4attn_quantize_nvfp4_per_head(x, role)
    return fp4.fp4attn_quantize(x, fp4.FMT_NVFP4 if qk == "nvfp4" else fp4.FMT_MXFP4, role)


def run(state):
    if state["kind"] == "host":
        fp4.fp4attn_attention_host(*state["x"], state["fmt"], state["out"], state["lse"], state["workspace"])
        return state["out"], state["lse"]
    q, k, v = state["x"]
    q = _quantize_qk(q, fp4.ROLE_Q, state["qk"])
    k = _quantize_qk(k, fp4.ROLE_K, state["qk"])
    v = fp4.fp4attn_quantize_v_e4m3(v) if state["pv"] == "e4m3" else fp4.fp4attn_quantize(v, fp4.FMT_MXFP4, fp4.ROLE_V)
    if state["kind"] == "encode":
        return [(t.packed, t.scales, t.G) for t in (q, k, v)]
    out, lse = fp4.fp4attn_fwd(q, k, v, **state["options"])
    if "lengths" in state:          # the rows beyond a sequence's length have no meaning: each sequence's own rows
        return [(out[b, :, :n], lse[b, :, :n]) for b, n in enumerate(state["lengths"])]
    return out, lse


def work(case):
    B, H, N, d, rows = case["B"], case["H"], case["N"], case["d"], case["B"] * case["H"] * case["N"]
    kv_rows = B * case["kv_heads"] * N
    if case["kind"] == "encode":
        qk_out = 0.5 * d + d / (32 if case["qk"] == "mxfp4" else 16)
        v_out = d if case["pv"] == "e4m3" else 0.5 * d + d / 32
        return {"bytes": rows * (2.0 * d + qk_out) + kv_rows * (4.0 * d + qk_out + v_out), "flops": 0.0}
    lengths = _lengths(case) if case["ragged"] else [N] * B
    tokens, pairs = sum(lengths), sum(n * (n + 1) / 2 if case["causal"] else float(n) * n for n in lengths)
    return {"bytes": tokens * (H * (4.0 * d + 4.0) + case["kv_heads"] * 4.0 * d), "flops": 4.0 * H * d * pairs}


def tolerance(case):
    # Quantized operands are integers and one fp32 division: every correct implementation writes the same bits.
    # O is bf16 (half a spacing is 2^-9 of a value); a probability code within float32 rounding of a boundary may fall
    # either way, which moves single elements of short rows by more than that.
    return "exact" if case["kind"] == "encode" else {"rel": 5e-3, "max": 0.2}
