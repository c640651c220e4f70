"""The limit of the kernels' bounded waits does not count the time that the kernel ahead of them still takes.

In the wait-test build (every wait limited to 1 ms) a kernel that lets its dependents start at once keeps the stream
busy for 5 ms; every form of the fused attention and of the row softmax that waits for copies is launched right behind
it and has to give the result it gives alone, with no expired wait recorded.
"""
import ctypes

import pytest
import torch

from paper_2602_02071_b200 import binding, build
from tile_order import form

pytestmark = pytest.mark.gpu


@pytest.fixture
def wlib(monkeypatch):
    monkeypatch.setattr(binding, "LIB_PATH", build.build_wait_test())
    monkeypatch.setattr(binding, "_lib", None)
    lib = binding.load()
    lib.baps_test_keep_busy.argtypes = [ctypes.c_int, ctypes.c_void_p]
    return lib


def _attn(H, S, D, causal=True, want=None, **kw):
    assert want is None or form(D, H, S // 128, causal) == want
    q, k, v = (torch.randn(1, H, S, D, device="cuda").bfloat16() for _ in range(3))
    return lambda: binding.baps_attention_fwd_ex(q, k, v, causal=causal, block_q=128, block_k=128, **kw).out_f32


def _fp8(H, S, want):
    assert form(128, H, S // 128, True) == want
    q, k, v = (torch.randn(1, H, S, 128, device="cuda") for _ in range(3))
    q8, k8 = (t.to(torch.float8_e4m3fn) for t in (q, k))
    sc = torch.ones(1, H, S // 128, device="cuda")
    return lambda: binding.baps_attention_fwd_fp8(q8, k8, v.bfloat16(), sc, sc, causal=True).out_f32


def _rows(cols):
    x = torch.randn(64, cols, device="cuda")
    return lambda: binding.baps_softmax_rows(x)


@pytest.mark.parametrize("make", [
    lambda: _attn(2, 512, 128, want="one tile"),
    lambda: _attn(24, 2048, 128, want="two tiles"),
    lambda: _attn(2, 512, 128, mode=binding.MODE_EXACT),               # two query tiles per CTA, whatever the grid
    lambda: _attn(2, 512, 128, mode=binding.MODE_EXP2_HIF8),
    lambda: _attn(2, 512, 64, mode=binding.MODE_EXACT),
    lambda: _attn(2, 512, 64, want="one tile"),
    lambda: _attn(64, 1024, 64, causal=False, want="two CTAs per SM"),
    lambda: _fp8(24, 2048, "two tiles"), lambda: _fp8(2, 512, "one tile"), lambda: _rows(16384), lambda: _rows(65536)])
def test_waits_start_when_the_kernel_ahead_has_ended(wlib, make):
    call = make()
    want = call()
    binding.poll_async_error()
    for _ in range(3):
        assert wlib.baps_test_keep_busy(5000, binding._stream()) == 0
        got = call()
        binding.poll_async_error()                                     # raises after an expired wait
        assert torch.equal(got, want)
