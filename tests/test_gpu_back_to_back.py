"""Calls that follow one another on a stream without a wait between them, each reading what the one before wrote:
the kernels are launched before the kernel ahead has ended and wait for it themselves."""
import pytest
import torch

from paper_2602_02071_b200 import binding

pytestmark = pytest.mark.gpu


def _round(x, q, scales, wait):
    """Every kernel of the library once, all results feeding later calls; other kernels (torch's) in between."""
    y = binding.baps_hif8_decode(wait(binding.baps_exp2_hif8(wait(binding.baps_hif8_encode(x)))))
    codes, _, d = wait(binding.baps_softmax_rows_codes(wait(binding.baps_softmax_rows(wait(y)))))
    x = wait(binding.baps_hif8_decode(codes))
    x = wait(torch.where(torch.isfinite(x), x, torch.zeros_like(x)) * 3 - 1)
    a = wait(binding.baps_attention_fwd(q, q, q, causal=True))
    b = wait(binding.baps_attention_fwd(a, q, a, causal=False))
    f = wait(binding.baps_attention_fwd_f32(b.float(), a.float(), b.float(), causal=True))
    q8 = wait((f * 4).to(torch.float8_e4m3fn))
    e = wait(binding.baps_attention_fwd_fp8(q8, q8, b, scales, wait(scales * 0.5), causal=True, want_stats=False).out)
    q = wait(q + 0.5 * e)
    return x, wait(q / q.float().std().bfloat16()), d


@pytest.mark.parametrize("cols", [1024, 3200, 16384, 65536])
def test_dependent_calls_without_a_wait_between(cols):
    g = torch.Generator(device="cuda"); g.manual_seed(cols)
    x0 = torch.randn(9, cols, device="cuda", generator=g)
    q0 = torch.randn(1, 4, 512, 128, device="cuda", generator=g).bfloat16()
    scales = torch.full((1, 4, 4), 0.25, device="cuda")

    def chain(wait, n=12):
        x, q, out = x0, q0, []
        for _ in range(n):
            x, q, d = _round(x, q, scales, wait)
            out += [x, q, d]
        return out

    def synced(r):
        torch.cuda.synchronize()
        return r

    want = chain(synced)
    got = chain(lambda r: r)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = chain(lambda r: r, 3)
    graph.replay(); graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, captured))
