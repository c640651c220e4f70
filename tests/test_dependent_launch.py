"""Rules of dependent launch that the sources have to keep: a kernel of the library may start before the kernel ahead
of it has ended, and the next one before it has ended itself.  Read from the sources: what breaks them is a wait that
never ends or stale data, which no test provokes on a GPU."""
import os
import re

import pytest

from paper_2602_02071_b200 import build

SRC = {n: open(os.path.join(build.CSRC, n)).read() for n in sorted(os.listdir(build.CSRC)) if n.endswith((".cu", ".cuh"))}
CODE = {n: re.sub(r"//[^\n]*", "", s) for n, s in SRC.items()}


def kernel_body(name):
    """Text of a __global__ function, from its name to the closing brace in the first column."""
    for code in CODE.values():
        m = re.search(r"__global__[^;{]*\b" + name + r"\(", code)
        if m:
            return code[m.start():code.index("\n}", m.start())]
    raise KeyError(name)


DEPENDENT = ["hif8_encode_kernel", "hif8_decode_kernel", "hif8_exp2_kernel", "softmax_rows_ring_kernel",
             "softmax_rows_quarters_kernel", "softmax_rows_group_kernel", "softmax_rows_warp_kernel",
             "attention_f32_kernel", "attention_tc_kernel", "attention_d64_kernel"]


@pytest.mark.parametrize("name", DEPENDENT)
def test_every_kernel_waits_for_the_kernel_ahead_and_lets_the_next_one_in(name):
    body = kernel_body(name)
    assert "await_previous_kernel(" in body and "allow_next_kernel()" in body


def test_tensor_memory_is_taken_between_the_kernel_ahead_and_the_next_one():
    """Two kernels on one SM that each hold tensor memory and wait for the other would wait for ever.  attention_d64_kernel
    leaves room beside it; attention_tc_kernel's CTA takes nearly all registers of an SM (640 threads x 96)."""
    body = kernel_body("attention_d64_kernel")
    alloc = body.index("tmem_alloc(")
    role = body.rindex("else if (warp == 9)", 0, alloc)
    assert body.index("await_previous_kernel()", role) < alloc < body.index("allow_next_kernel()")
    assert "__launch_bounds__(kTcThreads, 1)" in CODE["baps_attention_tc.cuh"]
    assert "kTcThreads = kTcSplit.threads;" in CODE["baps_attention_tc.cuh"]
    assert re.search(r"kTcSplit = \{640, ", CODE["baps_register_split.cuh"])


def test_no_load_asks_for_data_that_never_changes():
    """ld.global.nc (__ldg) may be served from data read before the kernel ahead wrote it."""
    for name, code in CODE.items():
        assert "__ldg(" not in code and "ld.global.nc" not in code, name


def test_the_paired_kernel_keeps_the_rules_too():
    """paired_attention_tc_kernel: the same calls, and a CTA as large as attention_tc_kernel's, so that nothing that uses
    tensor memory fits beside it."""
    body = kernel_body("paired_attention_tc_kernel")
    assert "await_previous_kernel(" in body and "allow_next_kernel()" in body
    # every role that touches caller memory, or starts a bounded wait, stands behind the wait for the kernel ahead: the
    # producer before its first load (ahead of the CTA-wide barrier that all other roles pass), the softmax warps at entry
    assert body.count("await_previous_kernel()") == 2
    producer, softmax = (m.start() for m in re.finditer(r"await_previous_kernel\(\)", body))
    assert producer < body.index("tma_load_2d(sbase + L::kQOff") < body.index("__syncthreads()")
    # (caller memory beside the tensor maps' is only touched by the softmax warps: the scales, outputs and statistics)
    touches = [m.start() for m in re.finditer(r"ldg_f32\(|p\.(?:q_scale|k_scale|out|out_f32|row_m|row_d|restarts)\b", body)]
    assert len(touches) >= 10 and body.index("setmaxnreg.inc") < softmax < min(touches)
    assert body.count("load_kv(l)") == 2 and producer < body.index("load_kv(l)")
    assert "__launch_bounds__(kTcThreads, 1)" in CODE["baps_attention_pair.cuh"]
