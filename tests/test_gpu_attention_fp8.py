"""GPU parity: attention with FP8 (E4M3) Q and K and per-tile power-of-two scales -- Q K^T on the
8-bit tensor-core path, the dequantisation folded into the score scale -- against the CPU checker fed
with the dequantised values (which are exact in float32, so both sides see the same numbers)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_02071_b200 import binding, workloads
from parity import EPS_REL, gate_attention
from tile_order import form

pytestmark = pytest.mark.gpu


def _np(t):
    return t.float().cpu().numpy()


def _check(w, tiles=None, mode=binding.MODE_E2E_HIF8, lam=1, what=""):
    q, k, v = workloads.make_qkv(w)
    q8, qs, qd = workloads.quantize_e4m3_tiles(q)
    k8, ks, kd = workloads.quantize_e4m3_tiles(k)
    st = binding.baps_attention_fwd_fp8(q8.cuda(), k8.cuda(), v.cuda(), qs.cuda(), ks.cuda(), causal=w.causal,
                                        lam=lam, mode=mode)
    binding.poll_async_error()
    if tiles is None:
        tiles = [tuple(x) for x in oracle.all_tiles(w.B, w.H, w.S, 128)]
    omode = {binding.MODE_E2E_HIF8: oracle.MODE_E2E_HIF8, binding.MODE_EXP2_HIF8: oracle.MODE_EXP2_HIF8}[mode]
    ref = oracle.attention(qd.numpy(), kd.numpy(), _np(v), causal=w.causal, block_q=128, block_k=128, lam=lam,
                           tiles=np.array(tiles, dtype=np.int32), mode=omode)
    out = st.out_f32.cpu().numpy()
    got = np.stack([out[b, h, i * 128:(i + 1) * 128] for b, h, i in tiles])
    gate_attention(got, ref, what=what or w.name)
    clear = ref.row_margin >= EPS_REL
    gm = np.stack([st.row_m.cpu().numpy()[b, h, i * 128:(i + 1) * 128] for b, h, i in tiles])
    if mode == binding.MODE_E2E_HIF8:
        assert np.array_equal(gm[clear], ref.row_m[clear])
        gr = np.array([st.restarts.cpu().numpy()[b, h, i] for b, h, i in tiles])
        assert np.array_equal(gr[clear.all(axis=1)], ref.restarts[clear.all(axis=1)])
    return st, (q, k, v)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("S", [128, 384, 1024])
def test_fp8_small_problems_all_tiles(causal, S):
    w = workloads.AttnWorkload("t", 2, 4, 2, S, 128, causal, 128, 128, outlier_frac=0.01, seed=90 + S + causal)
    _check(w, what=f"fp8 S={S} causal={causal}")


def test_fp8_exp2_setup_and_lambda():
    w = workloads.AttnWorkload("t", 1, 4, 2, 768, 128, True, 128, 128, seed=97)
    _check(w, mode=binding.MODE_EXP2_HIF8, what="fp8 exp2")
    _check(w, lam=0, what="fp8 lambda 0")


def test_fp8_full_size_sampled_and_close_to_the_bf16_path():
    """Configuration 2 at full size on sampled tiles, and the effect of the quantisation itself: against
    the bf16 path on the same inputs the 8-bit Q / K cost a few 1e-2 on average here (E4M3 keeps 3 mantissa
    bits of each factor, and this configuration's outlier keys, eight times larger than the rest, set the
    scale of their whole tile; the scores' errors average out over D = 128 products)."""
    w = workloads.WORKLOADS["c2_llm_prefill_mha"]
    st, (q, k, v) = _check(w, tiles=workloads.sample_tiles(w)[:8], what="c2 fp8")
    ref16 = binding.baps_attention_fwd_ex(q.cuda(), k.cuda(), v.cuda(), causal=True, block_q=128, block_k=128)
    diff = (st.out_f32 - ref16.out_f32).abs()
    assert float(diff.mean()) < 6e-2 and float(diff.max()) < 2.5


@pytest.mark.parametrize("S,causal,lam", [(640, True, 1), (768, True, 2), (256, False, 0)])
def test_fp8_two_query_tiles_per_cta_agree_with_one(S, causal, lam):
    """A few heads (one query tile per CTA) and the same heads repeated until the SMs are full several times over
    (two, an odd one left over at S = 640), outlier keys (restarts): the same decisions, and the same sums but for
    their order (2^-17, as for bf16 Q / K)."""
    n = 160
    assert form(128, 4, S // 128, causal) == "one tile" and form(128, 4 * n, S // 128, causal) == "two tiles"
    w = workloads.AttnWorkload("t", 1, 4, 2, S, 128, causal, 128, 128, outlier_frac=0.01, seed=400 + S + lam)
    few, (q, k, v) = _check(w, lam=lam, what=f"fp8 one tile S={S}")
    (q8, qs, _), (k8, ks, _) = (workloads.quantize_e4m3_tiles(t) for t in (q, k))
    many = binding.baps_attention_fwd_fp8(*(t.cuda().repeat(n, *[1] * (t.dim() - 1)) for t in (q8, k8, v, qs, ks)),
                                          causal=causal, lam=lam)
    assert torch.equal(few.row_m.expand_as(many.row_m), many.row_m)
    assert torch.equal(few.restarts.expand_as(many.restarts), many.restarts)
    assert torch.allclose(few.row_d.expand_as(many.row_d), many.row_d, rtol=2.0 ** -17, atol=0)
    # (a row's outputs are of the size of its largest, and what is left where they cancel is not)
    scale = few.out_f32.abs().amax(-1, keepdim=True)
    assert float(((few.out_f32 - many.out_f32).abs() / scale).max()) <= 2.0 ** -17
