"""The order in which the CTAs of the fused attention take query tiles and heads (``csrc/baps_tile_order.cuh``,
compiled here as plain C++): every tile once, chunks of kv heads even, and the SMs as evenly busy as without chunks."""
import heapq
import os
import random
import re

import pytest

from paper_2602_02071_b200 import build
from tile_order import SMS, form, one_tile_per_cta, tiles

RULES = open(os.path.join(build.CSRC, "baps_tile_order.cuh")).read()


def makespan(items, nq, pairs, slots):
    """CTAs handed out in order to whichever slot is free first (causal); costs as measured beside one_tile_per_cta, in
    tasks of a CTA with two query tiles: kTaskOne a task of a CTA with one, kFixed for either."""
    fixed, task_one = (float(re.search(n + r" = ([\d.]+)", RULES)[1]) for n in ("kFixed", "kTaskOne"))
    free = [0.0] * slots
    for tile, *_ in items:
        if pairs:
            lone = 2 * tile + 1 == nq
            cost = fixed + (2 * tile + 1) + (0 if lone else 2 * tile + 2)
        else:
            cost = fixed + task_one * (tile + 1)
        heapq.heapreplace(free, free[0] + cost)
    return max(free)


# B, H, Hkv, S, bytes of K and V per key (D = 128 bf16: 512, 8-bit keys: 384; D = 64: 256)
SHAPES = [(2, 32, 8, 8192, 384), (4, 32, 8, 4096, 384), (1, 36, 9, 8192, 512), (1, 16, 16, 16384, 512),
          (1, 9, 9, 16384, 256), (1, 176, 176, 2048, 512), (1, 176, 176, 2048, 256), (1, 176, 176, 1920, 512),
          (1, 40, 40, 8192, 512), (1, 96, 96, 4096, 512), (2, 32, 8, 8192, 512), (1, 32, 8, 32768, 512),
          (23, 7, 7, 1024, 256), (9, 15, 5, 2048, 512), (301, 2, 1, 1024, 512), (1, 1, 1, 128, 512), (3, 6, 2, 640, 256)]


def check(B, H, Hkv, S, key_bytes):
    nq = S // 128
    pairs = key_bytes != 256 and not one_tile_per_cta(B * H, nq, True)
    per_sm = 2 if key_bytes == 256 else 1
    n = (nq + 1) // 2 if pairs else nq
    for causal in (True, False):
        (size, wide), items = tiles(B, H, Hkv, n, S * key_bytes, causal, per_sm)
        assert sorted((b, h, t) for t, h, _, b in items) == [(b, h, t) for b in range(B) for h in range(H) for t in range(n)]
        assert all(hk == h // (H // Hkv) for _, h, hk, _ in items)
        assert 0 <= wide <= B * Hkv and (B * Hkv - wide * (size + 1)) % size == 0      # all of one size but for one head
    _, chunked = tiles(B, H, Hkv, n, S * key_bytes, True, per_sm)
    _, whole = tiles(B, H, Hkv, n, S * key_bytes, True, per_sm, whole=True)
    # 3 %: what reading K and V from L2 gives at these sizes; a ragged last chunk costs 5 to 35 % in this estimate
    assert makespan(chunked, nq, pairs, per_sm * SMS) <= 1.03 * makespan(whole, nq, pairs, per_sm * SMS)


@pytest.mark.parametrize("B,H,Hkv,S,key_bytes", SHAPES)
def test_every_tile_once_in_even_chunks_that_keep_the_sms_busy(B, H, Hkv, S, key_bytes):
    check(B, H, Hkv, S, key_bytes)


def test_random_shapes():
    rng = random.Random(5)
    for _ in range(60):
        Hkv, g, B = rng.randint(1, 48), rng.choice([1, 1, 2, 3, 4, 8]), rng.choice([1, 1, 2, 3, 5])
        nq, key_bytes = rng.choice([1, 3, 8, 16, 31, 64]), rng.choice([256, 384, 512])
        if B * Hkv * g * nq <= 30000:
            check(B, Hkv * g, Hkv, 128 * nq, key_bytes)


@pytest.mark.parametrize("D,causal,few,many", [
    (128, True, [(16, 512), (32, 1024), (16, 2048), (8, 4096), (3, 8192), (2, 16384), (1, 32768), (75, 384), (74, 256)],
     [(48, 640), (64, 512), (40, 1024), (20, 2048), (12, 4096), (6, 8192), (3, 16384), (2, 32768), (110, 256), (1, 128)]),
    (128, False, [(36, 512), (8, 2048), (2, 8192), (75, 384)], [(40, 512), (10, 2048), (3, 8192), (12, 4096)]),
    (64, True, [(36, 512), (24, 1024), (16, 2048), (8, 4096), (3, 8192), (2, 16384), (1, 32768), (74, 256), (74, 128)],
     [(48, 512), (40, 1024), (20, 2048), (10, 4096), (6, 8192), (3, 16384), (2, 32768), (110, 256), (200, 128)]),
    (64, False, [(36, 512), (8, 2048), (2, 8192), (74, 128)], [(40, 512), (10, 2048), (3, 8192), (200, 128)])])
def test_the_form_that_was_measured_to_be_faster(D, causal, few, many):
    """Sizes (heads, tokens) on both sides of the line, each at least 2 % faster in the form that is taken for it."""
    for heads, S in few:
        assert form(D, heads, S // 128, causal) == "one tile", (heads, S)
    for heads, S in many:
        assert form(D, heads, S // 128, causal) != "one tile", (heads, S)
