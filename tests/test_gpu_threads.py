"""Host threads that call the library at the same time, each with its own sizes and stream: the same kernel instances
at different row lengths and head sizes, which take different amounts of shared memory."""
import threading

import pytest
import torch

from paper_2602_02071_b200 import binding

pytestmark = pytest.mark.gpu


def _rows(cols, codes):
    x = torch.randn(1, cols, device="cuda")
    call = (lambda: binding.baps_softmax_rows_codes(x)[0]) if codes else (lambda: binding.baps_softmax_rows(x))
    return call, call()


def _f32(D, block):
    q = torch.randn(1, 1, block, D, device="cuda")
    call = lambda: binding.baps_attention_fwd_f32(q, q, q, causal=False, block_q=block, block_k=block)
    return call, call()


@pytest.mark.parametrize("small,large", [(lambda: _rows(8320, False), lambda: _rows(16256, False)),
                                         (lambda: _rows(8320, True), lambda: _rows(16256, True)),
                                         (lambda: _rows(16512, False), lambda: _rows(32640, False)),
                                         (lambda: _f32(64, 128), lambda: _f32(128, 128)),
                                         (lambda: _f32(64, 64), lambda: _f32(128, 64))])
def test_threads_with_different_sizes(small, large):
    jobs, failures = [small(), large(), small(), large()], []
    torch.cuda.synchronize()

    def work(call, want):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(1000):
                    got = call()
                torch.cuda.current_stream().synchronize()
                assert torch.equal(got, want)
        except Exception as e:                              # reported by the test's own thread
            failures.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
