"""The work that a user has the library do, as cases to be timed: fused attention over the prefill and
encoder shapes of the benchmark definition and around them, the standalone row softmax in both output
forms, and the HiF8 conversions.  Every pass goes through the entry points of
``paper_2602_02071_b200.binding`` with torch tensors as device buffers, results allocated per call as
the binding does by default.

A case is a dict of plain values; ``kind`` names the path:
  attn       bf16 fused attention, the plain call
  attn_ex    the extended call: lambda, mode, B0 choice, statistics buffers
  attn_fp8   E4M3 Q / K with one power-of-two scale per 128-row tile
  attn_f32   float32 inputs, scores accumulated in double precision
  rows       row softmax, float output
  codes      row softmax, 8-bit output
  hif8       T to HiF8 codes, 8-bit exponent, codes back to values (Algorithm 2, step by step)
"""
import torch

from paper_2602_02071_b200 import binding, workloads

ATTN_KINDS = ("attn", "attn_ex", "attn_fp8", "attn_f32")


def _attn(name, kind, B, H, Hkv, S, D, causal, **more):
    case = {"name": name, "kind": kind, "B": B, "H": H, "Hkv": Hkv, "S": S, "D": D, "causal": causal}
    case.update(more)
    return case


def listed():
    return [
        # one head of 128 tokens in float32 with 64 x 64 tiles: the smallest call, all latency
        _attn("f32_single_head", "attn_f32", 1, 1, 1, 128, 64, False, block=64),
        # a short prompt on few heads: a handful of CTAs, launch cost counts
        _attn("short_prompt", "attn", 1, 4, 2, 512, 128, True),
        # odd number of query tiles, three query heads per kv head, D = 64
        _attn("odd_tiles_gqa3", "attn", 2, 6, 2, 640, 64, True),
        # image encoder: many short bidirectional sequences, per-token key bias
        _attn("vit_encoder", "attn", 32, 16, 16, 1024, 64, False, bias=0.5),
        # prompt prefill, one kv head per query head, outlier keys (frequent restarts)
        _attn("prefill_mha_outliers", "attn", 1, 32, 32, 4096, 128, True, outliers=0.01),
        # prompt prefill with grouped kv heads
        _attn("prefill_gqa", "attn", 2, 32, 8, 8192, 128, True),
        # long-context prefill, the largest call
        _attn("long_context", "attn", 1, 32, 8, 32768, 128, True),
        # prefill with quantised Q and K, statistics off
        _attn("prefill_fp8_qk", "attn_fp8", 1, 32, 8, 8192, 128, True),
        # non-fused path: score rows of a long context
        {"name": "rows_64k", "kind": "rows", "rows": 4096, "cols": 65536, "block_k": 128},
        # non-fused path: a row length that is no power of two
        {"name": "rows_odd_length", "kind": "rows", "rows": 20011, "cols": 3200, "block_k": 128},
        # rows that stay in 8 bits for a later product
        {"name": "codes_8k", "kind": "codes", "rows": 16384, "cols": 8192, "block_k": 128},
        # the conversions on a ragged array
        {"name": "hif8_ragged", "kind": "hif8", "n": 64 * 1024 * 1024 + 4099},
    ]


# No drawn case may cost more than the largest listed one.
MAX_ATTN_FLOPS = 2.0 * 32 * 32768.0 ** 2 * 128
MAX_ATTN_ELEMS = 32 * 32768 * 128
MAX_ELEMS = 1 << 28


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["attn", "attn", "attn", "attn_ex", "attn_fp8", "attn_f32", "rows", "rows", "codes", "hif8"])
    if kind == "hif8":
        return {"kind": kind, "n": _log_uniform(rng, 1000, MAX_ELEMS) | 1}
    if kind in ("rows", "codes"):
        cols = 128 * _log_uniform(rng, 1, 512)
        if rng.random() < 0.3:                       # the power-of-two lengths are common ones
            cols = 1 << rng.randint(10, 16)
        rows = max(1, _log_uniform(rng, cols, MAX_ELEMS) // cols)
        return {"kind": kind, "rows": rows, "cols": cols, "block_k": rng.choice([128, 128, 64])}
    if kind == "attn_f32":
        block = rng.choice([64, 128])
        hkv, group = rng.choice([(1, 1), (2, 1), (2, 2), (4, 1)])
        return {"kind": kind, "B": rng.randint(1, 2), "H": hkv * group, "Hkv": hkv,
                "S": block * _log_uniform(rng, 1, 1024 // block), "D": rng.choice([32, 64, 80, 128]),
                "causal": rng.random() < 0.5, "block": block}
    D = 128 if kind == "attn_fp8" else rng.choice([64, 128, 128])
    causal = rng.random() < 0.7
    while True:
        S = 128 * _log_uniform(rng, 1, 256)
        B = _log_uniform(rng, 1, 32)
        Hkv = rng.choice([1, 2, 4, 8, 16, 32])
        H = Hkv * rng.choice([1, 1, 3, 4, 8])
        flops = 4.0 * B * H * S * S * D / (2 if causal else 1)
        if H <= 64 and flops <= MAX_ATTN_FLOPS / 4 and B * H * S * D <= MAX_ATTN_ELEMS:
            break
    case = {"kind": kind, "B": B, "H": H, "Hkv": Hkv, "S": S, "D": D, "causal": causal}
    extra = rng.choice(["", "", "outliers", "bias"])
    if extra == "outliers":
        case["outliers"] = 0.01
    elif extra == "bias":
        case["bias"] = 0.5
    if kind == "attn_ex":
        mode = rng.choice([binding.MODE_E2E_HIF8, binding.MODE_E2E_HIF8, binding.MODE_EXP2_HIF8, binding.MODE_EXACT])
        case["mode"] = mode
        if mode == binding.MODE_E2E_HIF8:
            case["lam"] = rng.randint(0, 3)
            case["b0_last"] = rng.random() < 0.25
    return case


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _qkv(case, seed):
    """Unit-Gaussian Q, K, V; optionally a share of the key rows scaled by 8 (the same rows for all
    heads), or a per-token offset on the keys."""
    g = _gen(seed)
    B, H, Hkv, S, D = (case[n] for n in ("B", "H", "Hkv", "S", "D"))
    q = torch.randn(B, H, S, D, generator=g, device="cuda")
    k = torch.randn(B, Hkv, S, D, generator=g, device="cuda")
    v = torch.randn(B, Hkv, S, D, generator=g, device="cuda")
    if case.get("outliers"):
        n = max(1, int(round(case["outliers"] * S)))
        k[:, :, torch.randperm(S, generator=g, device="cuda")[:n], :] *= 8.0
    if case.get("bias"):
        k += torch.randn(B, Hkv, S, 1, generator=g, device="cuda") * case["bias"] ** 0.5
    return q, k, v


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind in ATTN_KINDS:
        q, k, v = _qkv(case, seed)
        if kind == "attn_fp8":
            state["q"], state["q_scale"], _ = workloads.quantize_e4m3_tiles(q)
            state["k"], state["k_scale"], _ = workloads.quantize_e4m3_tiles(k)
            state["v"] = v.bfloat16()
        else:
            dt = torch.float32 if kind == "attn_f32" else torch.bfloat16
            state["q"], state["k"], state["v"] = q.to(dt), k.to(dt), v.to(dt)
    elif kind in ("rows", "codes"):
        state["x"] = torch.randn(case["rows"], case["cols"], generator=_gen(seed), device="cuda").mul_(2.0)
    else:
        # T of score tiles: mostly below zero, a few above (rows whose maximum rose)
        state["x"] = torch.randn(case["n"], generator=_gen(seed), device="cuda").mul_(2.0).sub_(5.0)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "attn":
        return binding.baps_attention_fwd(state["q"], state["k"], state["v"], causal=case["causal"])
    if kind == "attn_f32":
        return binding.baps_attention_fwd_f32(state["q"], state["k"], state["v"], causal=case["causal"],
                                              block_q=case["block"], block_k=case["block"])
    if kind == "attn_ex":
        st = binding.baps_attention_fwd_ex(state["q"], state["k"], state["v"], causal=case["causal"], block_q=128,
                                           block_k=128, lam=case.get("lam", 1), mode=case["mode"],
                                           b0_last=case.get("b0_last", False))
        return [st.out, st.out_f32, st.row_m, st.row_d, st.restarts]
    if kind == "attn_fp8":
        return binding.baps_attention_fwd_fp8(state["q"], state["k"], state["v"], state["q_scale"], state["k_scale"],
                                              causal=case["causal"], want_stats=False).out
    if kind == "rows":
        return binding.baps_softmax_rows(state["x"], block_k=case["block_k"])
    if kind == "codes":
        return binding.baps_softmax_rows_codes(state["x"], block_k=case["block_k"])
    t = binding.baps_hif8_encode(state["x"])
    p = binding.baps_exp2_hif8(t)
    return t, p, binding.baps_hif8_decode(p)


def work(case):
    kind = case["kind"]
    if kind in ATTN_KINDS:
        B, H, Hkv, S, D = (case[n] for n in ("B", "H", "Hkv", "S", "D"))
        pairs = S * (S + 1) / 2 if case["causal"] else float(S) * S
        qk, v, out = {"attn_f32": (4, 4, 4), "attn_fp8": (1, 2, 2)}.get(kind, (2, 2, 2))
        nbytes = B * H * S * D * (qk + out) + B * Hkv * S * D * (qk + v)
        if kind == "attn_fp8":
            nbytes += 4 * (B * H + B * Hkv) * (S // 128)
        if kind == "attn_ex":                        # float32 output, two row statistics, restart counters
            nbytes += B * H * (S * D * 4 + S * 8 + S // 128 * 4)
        return {"bytes": nbytes, "flops": 4.0 * B * H * D * pairs}
    if kind in ("rows", "codes"):
        n = case["rows"] * case["cols"]
        if kind == "rows":
            return {"bytes": 8.0 * n, "flops": 0}
        return {"bytes": 5.0 * n + 4 * (n // case["block_k"]) + 4 * case["rows"], "flops": 0}
    return {"bytes": (4 + 1) * case["n"] + 2 * case["n"] + 5 * case["n"], "flops": 0}


def tolerance(case):
    """About four times what two correct computations of the same case were seen to differ by: the
    tensor-core path (fp32 scores, bf16 weights and output) against the same workflow with scores in
    double precision, rel 2.2e-3 and at most 0.04 on one value (a score next to a rounding boundary of
    the 8-bit format moves its weight by a whole step); the float32 path and the row softmax against
    the double-precision checker, rel 5.4e-5 and 1.4e-7.  Codes and exponents are whole numbers and
    come out the same; so do the conversions, their values included."""
    kind = case["kind"]
    if kind in ("attn", "attn_ex", "attn_fp8"):
        return {"rel": 8e-3, "max": 0.16}
    if kind == "attn_f32":
        return {"rel": 2e-4, "max": 0.04}
    return "exact" if kind == "hif8" else {"rel": 6e-7}
