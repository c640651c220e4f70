"""GPU parity of the fused attention where its number formats end, in every form of the kernel: a max that rounds to zero
from below, rows of NaN, weights near the largest factor, scores of -inf and +inf."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2602_02071_b200 import binding, workloads
from parity import EPS_REL, gate_attention
from tile_order import form

pytestmark = pytest.mark.gpu

# D, copies of two heads, the form of the kernel that this grid takes
FORMS = [(128, 1, "one tile"), (128, 80, "two tiles"), (64, 1, "one tile"), (64, 160, "two CTAs per SM")]


def _score_keys(scores, D):
    """Keys [2, S, D] whose base-2 score against every query with a 1 in column 0 is scores[key]."""
    k = torch.zeros(2, scores.numel(), D)
    k[..., 0] = scores * math.sqrt(D) / 1.4426950408889634
    return k.bfloat16()


def _run(q, k, v, n, want_form, causal, lam=1):
    """Two heads [2, S, D] repeated n times; the copies give the same bits.  -> statistics of one copy"""
    H, S, D = q.shape
    assert form(D, H * n, S // 128, causal) == want_form
    st = binding.baps_attention_fwd_ex(*(t[None].cuda().repeat(n, 1, 1, 1) for t in (q, k, v)), causal=causal,
                                       block_q=128, block_k=128, lam=lam)
    binding.poll_async_error()
    for t in (st.out, st.out_f32, st.row_m, st.row_d, st.restarts):
        assert torch.equal(t.nan_to_num(9e9), t[:1].nan_to_num(9e9).expand_as(t))
    return [t[0].float().cpu() for t in (st.out, st.out_f32, st.row_m, st.row_d, st.restarts)]


def _oracle(q, k, v, causal, lam=1):
    r = oracle.attention(*(t[None].float().numpy() for t in (q, k, v)), causal=causal, block_q=128, block_k=128, lam=lam)
    return r, tuple(x.reshape(q.shape[:2] + x.shape[2:]) for x in (r.out, r.row_m, r.row_d))


@pytest.mark.parametrize("first", [[-0.5], [-5.5, -0.5]])
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("D,n,want_form", FORMS)
def test_a_max_that_rounds_up_to_zero(D, n, want_form, causal, first):
    """The largest score so far lies in (-1, 0), in the first tile or after a restart, so that the max is zero; the scores
    of all later keys are zero exactly (padding): T = 0, weight 1."""
    S = 640
    g = torch.Generator().manual_seed(D)
    q = torch.randn(2, S, D, generator=g).bfloat16()
    q[..., 0] = 1.0
    scores = torch.zeros(S)
    scores[:128 * len(first)] = torch.tensor(first).repeat_interleave(128)
    k = _score_keys(scores, D)
    v = (torch.randn(2, S, D, generator=g) + (torch.arange(S) // 128)[:, None]).bfloat16()
    out, out_f32, row_m, row_d, restarts = _run(q, k, v, n, want_form, causal)
    ref, (want, want_m, want_d) = _oracle(q, k, v, causal)
    assert np.array_equal(row_m.numpy(), want_m) and np.array_equal(restarts.numpy().ravel(), ref.restarts)
    # all scores but the first tile's sit on table entries; those of the first tile have bf16 weights
    assert np.allclose(row_d.numpy(), want_d, rtol=2.0 ** -8, atol=0)
    assert np.abs(out_f32.numpy() - want).max() <= 1e-2


@pytest.mark.parametrize("D,n,want_form", FORMS)
def test_rows_without_a_score_keep_the_max_of_no_key(D, n, want_form):
    """A query row that holds a NaN has no scores: its output is NaN, its max that of no key (-inf), and no other row, max
    or restart count notices (the row is compared with one of zeros, which never votes for a restart either)."""
    S = 512
    g = torch.Generator().manual_seed(D + 1)
    q, k, v = (torch.randn(2, S, D, generator=g).bfloat16() for _ in range(3))
    k[:, 7::100] *= 8                                                   # restarts
    rows = [5, 200, S - 1]
    q[:, rows] = 0.0
    plain = _run(q, k, v, n, want_form, False)
    q[:, rows, 3] = float("nan")
    got = _run(q, k, v, n, want_form, False)
    others = [r for r in range(S) if r not in rows]
    for a, b in zip(plain[:4], got[:4]):
        assert torch.equal(a[:, others], b[:, others])
    assert torch.equal(plain[4], got[4]) and int(got[4].sum()) > 0
    for t in (got[0], got[1], got[3]):
        assert torch.isnan(t[:, rows]).all()
    assert (got[2][:, rows] == -float("inf")).all()


@pytest.mark.parametrize("D,n,want_form", FORMS)
def test_weights_stay_in_range_until_the_output_is_rebased(D, n, want_form):
    """The row maximum rises by three per tile up to 66, then stays: O~ and d are rebased before weights of 2^66 meet
    them.  V of 2^54 does not overflow (the sum over the keys of a tile adds 7 to the exponent, 2^64 times that is
    2^125), with 2^66 it would."""
    tiles = 30
    S = 128 * tiles
    g = torch.Generator().manual_seed(D + 2)
    q = torch.zeros(2, S, D).bfloat16()
    q[..., 0] = 1.0
    level = torch.tensor([0.0] + [3.0 * min(t, 22) - (0.3 if t <= 22 else 0.5) for t in range(1, tiles)])
    k = _score_keys(level.repeat_interleave(128), D)
    v = (torch.rand(2, S, D, generator=g) * 0.5 + 0.5).bfloat16()
    out, out_f32, row_m, row_d, restarts = _run(q, k, v * 2.0 ** 54, n, want_form, False, lam=3)
    ref, (want, want_m, want_d) = _oracle(q, k, v, False, lam=3)
    assert np.array_equal(row_m.numpy(), want_m) and (want_m == 66).all() and not restarts.any()
    assert np.allclose(row_d.numpy(), want_d, rtol=2.0 ** -8, atol=0)
    assert np.abs(out_f32.numpy() * 2.0 ** -54 - want).max() <= 1e-2


@pytest.mark.parametrize("D,n,want_form", FORMS)
def test_scores_of_minus_infinity_have_no_weight(D, n, want_form):
    """Keys whose scores overflow to -inf (masked by the caller), in the first tile, alone in a whole tile and scattered:
    weight 0, as the oracle has it for scores of -10^38."""
    S = 640
    g = torch.Generator().manual_seed(D + 3)
    q, k, v = (torch.randn(2, S, D, generator=g).bfloat16() for _ in range(3))
    q[..., 0] = 4.0
    k[..., 0] = 0.0
    masked = list(range(3, 60)) + list(range(256, 384)) + list(range(400, 640, 7))
    k[:, masked] = 0.0
    k[:, masked, 0] = -3e38                                             # 4 x -3e38: -inf in 32 bits
    out, out_f32, row_m, row_d, restarts = _run(q, k, v, n, want_form, False)
    ref, (want, want_m, want_d) = _oracle(q, k, v, False)
    gate_attention(out_f32.numpy(), ref, what=f"masked keys D={D} {want_form}")
    clear = (ref.row_margin >= EPS_REL).reshape(want_m.shape)
    assert np.array_equal(row_m.numpy()[clear], want_m[clear])


@pytest.mark.parametrize("D,n,want_form", FORMS)
def test_an_infinite_score_spoils_its_own_row_only(D, n, want_form):
    """A query row with an infinity has scores of +inf and -inf: its max is +inf from the first tile on, its output NaN; no
    other row, max or restart count notices."""
    S = 512
    g = torch.Generator().manual_seed(D + 4)
    q, k, v = (torch.randn(2, S, D, generator=g).bfloat16() for _ in range(3))
    k[:, 7::100] *= 8
    rows = [0, 133, S - 2]
    q[:, rows] = 0.0
    plain = _run(q, k, v, n, want_form, False)
    q[:, rows, 3] = float("inf")
    got = _run(q, k, v, n, want_form, False)
    others = [r for r in range(S) if r not in rows]
    for a, b in zip(plain[:4], got[:4]):
        assert torch.equal(a[:, others], b[:, others])
    assert torch.equal(plain[4], got[4]) and int(got[4].sum()) > 0
    assert torch.isnan(got[1][:, rows]).all() and (got[2][:, rows] == float("inf")).all()


@pytest.mark.parametrize("n,want_form", [(1, "one tile"), (80, "two tiles")])
def test_8_bit_rows_of_nan(n, want_form):
    """The same with E4M3 Q and K, whose score scale changes with the tile: a query row that holds the NaN code."""
    S, H = 512, 2
    assert form(128, H * n, S // 128, False) == want_form
    g = torch.Generator().manual_seed(5)
    q, k, v = (torch.randn(1, H, S, 128, generator=g) for _ in range(3))
    k[:, :, 7::100] *= 8
    q[:, :, 200] = 0.0
    (q8, qs, _), (k8, ks, _) = (workloads.quantize_e4m3_tiles(t) for t in (q, k))

    def run():
        st = binding.baps_attention_fwd_fp8(*(t.cuda().repeat(n, *[1] * (t.dim() - 1)) for t in (q8, k8, v.bfloat16(), qs, ks)),
                                            causal=False)
        binding.poll_async_error()
        return [t[n // 2].cpu() for t in (st.out_f32, st.row_d, st.row_m, st.restarts)]
    plain = run()
    q8[:, :, 200, 9] = 0x7F
    got = run()
    others = [r for r in range(S) if r != 200]
    for a, b in zip(plain[:3], got[:3]):
        assert torch.equal(a[:, others], b[:, others])
    assert torch.equal(plain[3], got[3]) and int(got[3].sum()) > 0
    assert torch.isnan(got[0][:, 200]).all() and (got[2][:, 200] == -float("inf")).all()
