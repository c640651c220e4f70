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


# ---- the same results in 64 bits, by plain torch ---------------------------------------------------

LOG2E = 1.4426950408889634074


def _hif8(x):
    """Nearest HiF8 value, ties to the larger magnitude: 3 / 2 / 1 mantissa bits for exponents up to 3 / 7 / 15
    in magnitude, powers of two from 2^-22 to 2^-16, nothing below 2^-23, infinity from 40960 on."""
    a = x.abs()
    e = torch.frexp(a.clamp(2.0 ** -22, 65536.0))[1] - 1
    ae = e.abs()
    bits = (ae <= 3).int() + (ae <= 7).int() + (ae <= 15).int()
    step = torch.ldexp(torch.ones_like(a), e - bits)
    r = torch.floor(a / step + 0.5) * step
    r = torch.where(a < 2.0 ** -23, 0.0, torch.where(a < 2.0 ** -22, 2.0 ** -22, r))
    r = torch.where(a >= 40960.0, float("inf"), r)
    return torch.copysign(r, x)


def _w8(t):
    return _hif8(torch.exp2(_hif8(t)))


def _update(s, m, lam, mode, first, whole_tile):
    """One block of Algorithm 1 (or of Eq. (2) in the other modes): base-2 scores s [..., rows, block] against
    the running max m [..., rows].  Returns the new max, the weights against it and the max the 8-bit
    arguments were taken against."""
    mx = s.amax(-1)
    if mode != binding.MODE_E2E_HIF8:
        new = torch.maximum(m, mx)
        t = s - new[..., None]
        return new, torch.exp2(t) if mode == binding.MODE_EXACT else _w8(t), new
    up = torch.maximum(m, torch.ceil(mx))
    if first:
        return up, torch.exp2(s - up[..., None]), up
    r8 = _hif8(mx - m)
    restart = r8 > lam
    if whole_tile:
        restart = restart.any(-1, keepdim=True)
    new = torch.where(restart, up, m + torch.ceil(r8).clamp_min(0.0))
    ref = torch.where(restart, up, m)
    return new, _w8(s - ref[..., None]) * torch.exp2(ref - new)[..., None], ref


def _exact_attention(q, k, v, causal, block, lam, mode, b0_last):
    """q [N,G,S,D], k, v [N,S,D] in 64 bits: N (batch, kv head) pairs of G query heads each.
    Returns out [N,G,S,D], row max and row sum [N,G,S], restart counts are left out."""
    N, G, S, D = q.shape
    n = S // block
    q = q.view(N, G, n, block, D) * (LOG2E / D ** 0.5)
    k, v = k.view(N, 1, n, block, D), v.view(N, 1, n, block, D)
    m = torch.full((N, G, n, block), -float("inf"), dtype=torch.float64, device=q.device)
    d, o = torch.zeros_like(m), torch.zeros_like(q)
    above = torch.ones(block, block, dtype=torch.bool, device=q.device).triu(1)

    def step(i0, kt, vt, diag, first):
        """Query tiles i0 .. against key tiles kt (one for all, or one each); diag: which of them are masked."""
        s = q[:, :, i0:] @ kt.transpose(-1, -2)
        if diag is not None:
            s[:, :, diag] = s[:, :, diag].masked_fill(above, -float("inf"))
        old = m[:, :, i0:]
        new, p, _ = _update(s, old, lam, mode, first, True)
        a = old - new
        a = torch.where(torch.isinf(old), 0.0, _w8(a) if mode == binding.MODE_EXP2_HIF8 else torch.exp2(a))
        d[:, :, i0:] = d[:, :, i0:] * a + p.sum(-1)
        o[:, :, i0:] = o[:, :, i0:] * a[..., None] + p @ vt
        m[:, :, i0:] = new

    if b0_last and mode == binding.MODE_E2E_HIF8:
        step(0, k[:, :, :1], v[:, :, :1], 0 if causal else None, True)
        if n > 1:
            last = slice(1, n) if causal else slice(n - 1, n)
            if causal:
                step(1, k[:, :, last], v[:, :, last], slice(0, n - 1), True)
            else:
                step(0, k[:, :, last], v[:, :, last], None, True)
        for j in range(1, n - 1):
            step(j + 1 if causal else 0, k[:, :, j:j + 1], v[:, :, j:j + 1], None, False)
    else:
        for j in range(n):
            step(j if causal else 0, k[:, :, j:j + 1], v[:, :, j:j + 1], 0 if causal else None, j == 0)
    return (o / d[..., None]).view(N, G, S, D), m.view(N, G, S), d.view(N, G, S)


def _exact_rows(x, block, codes):
    """Row softmax: probabilities, or (codes, exponents, row sums) with T rounded once to 32 bits."""
    rows, cols = x.shape
    xd = x.double() * (float(torch.tensor(LOG2E, dtype=torch.float32)) if codes else LOG2E)
    m = torch.full((rows, 1), -float("inf"), dtype=torch.float64, device=x.device)
    w, refs = torch.empty_like(xd), []
    for j in range(cols // block):
        at = slice(j * block, (j + 1) * block)
        s = xd[:, None, at]
        if codes and j:
            s = m[..., None] + (s - m[..., None]).float().double()
        new, p, ref = _update(s, m, 1, binding.MODE_E2E_HIF8, j == 0, False)
        if codes and j == 0:
            p = _w8((s - new[..., None]).float().double())
        w[:, at] = (p * torch.exp2(new - ref)[..., None])[:, 0]      # against ref
        refs.append(ref)
        m = new
    e = torch.cat(refs, 1) - m
    w = w.view(rows, -1, block)
    d = (w.sum(-1) * torch.exp2(e)).sum(-1)
    if codes:
        return _codes(w.view(rows, cols)), e.int(), d
    return w.mul_(torch.exp2(e)[..., None] / d[:, None, None]).view(rows, cols)


def _hif8_values():
    """The 256 values by code: sign, prefix-coded width of the exponent, sign-magnitude exponent, mantissa."""
    out = []
    for c in range(128):
        if c >> 5 == 3:
            width, mant, rest = 4, 1, c & 31
        elif c >> 5 == 2:
            width, mant, rest = 3, 2, c & 31
        elif c >> 5 == 1:
            width, mant, rest = 2, 3, c & 31
        elif c >> 4 == 1:
            width, mant, rest = 1, 3, c & 15
        elif c >> 3 == 1:
            width, mant, rest = 0, 3, c & 7
        else:
            out.append(2.0 ** (c - 23) if c else 0.0)
            continue
        exp = rest >> mant
        if width:
            mag = (1 << (width - 1)) | (exp & ((1 << (width - 1)) - 1))
            exp = -mag if exp >> (width - 1) else mag
        out.append((1 + (rest & ((1 << mant) - 1)) / (1 << mant)) * 2.0 ** exp)
    out[0x6F] = float("inf")
    neg = [-v for v in out]
    neg[0] = float("nan")
    return out + neg


def _codes(x):
    vals = torch.tensor(_hif8_values(), dtype=torch.float64, device=x.device)
    mags, order = vals[:128].sort()
    mids = (mags[:-1] + mags[1:]) / 2
    mids[-1] = 40960.0
    c = order[torch.searchsorted(mids, x.abs(), right=True)]
    return torch.where((x < 0) & (c > 0), c + 128, c).to(torch.uint8)


def exact(case, seed):
    kind = case["kind"]
    state = prepare(case, seed)
    if kind in ("rows", "codes"):
        return _exact_rows(state["x"], case["block_k"], kind == "codes")
    if kind == "hif8":
        vals = torch.tensor(_hif8_values(), dtype=torch.float64, device="cuda")
        t = _codes(state["x"].double())
        p = _codes(torch.exp2(vals))[t.long()]
        return t, p, vals[p.long()]
    B, H, Hkv, S, D = (case[n] for n in ("B", "H", "Hkv", "S", "D"))
    q, k, v = state["q"], state["k"], state["v"]
    if kind == "attn_fp8":
        q = (q.view(torch.float8_e4m3fn).float().view(B, H, -1, 128, D) * state["q_scale"][..., None, None]).view(B, H, S, D)
        k = (k.view(torch.float8_e4m3fn).float().view(B, Hkv, -1, 128, D) * state["k_scale"][..., None, None]).view(B, Hkv, S, D)
    block, G = case.get("block", 128), H // Hkv
    q, k, v = q.reshape(B * Hkv, G, S, D), k.reshape(B * Hkv, S, D), v.reshape(B * Hkv, S, D)
    part = max(1, (1 << 27) // (G * S * block))             # (batch, kv head) pairs at a time
    got = [_exact_attention(q[i:i + part].double(), k[i:i + part].double(), v[i:i + part].double(), case["causal"],
                            block, case.get("lam", 1), case.get("mode", binding.MODE_E2E_HIF8), case.get("b0_last", False))
           for i in range(0, B * Hkv, part)]
    out, m, d = (torch.cat([g[i] for g in got]).view(B, H, S, *([D] if i == 0 else [])) for i in range(3))
    return [out, out, m, d, None] if kind == "attn_ex" else out
