"""A kernel whose roles share out their registers waits for ever if it was compiled to fewer than they share: the rule
that the launch checks (``csrc/baps_register_split.cuh``, compiled here as plain C++), and the kernels as built."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2602_02071_b200 import build

SHIM = r"""
#include "baps_register_split.cuh"
using namespace baps;
extern "C" int fits(int threads, int few, int many_threads, int many, int regs)
{ return split_fits({threads, few, many_threads, many}, regs); }
extern "C" int tc_fits(int regs) { return split_fits(kTcSplit, regs); }
extern "C" int d64_fits(int regs) { return split_fits(kD64Split, regs); }
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(d / "shim.so"), str(d / "shim.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "shim.so"))


def test_the_shares_stay_within_the_pool(split):
    assert split.fits(384, 32, 256, 104, 80) and not split.fits(384, 32, 256, 104, 79)
    assert not split.fits(384, 32, 256, 112, 80) and not split.fits(384, 40, 256, 104, 80)
    assert split.tc_fits(96) and not split.tc_fits(88)
    assert split.d64_fits(80) and not split.d64_fits(72)


def test_the_kernels_take_their_shares_from_the_split_and_are_checked_before_the_launch():
    for name in ("baps_attention_tc.cuh", "baps_attention_d64.cuh"):
        code = open(os.path.join(build.CSRC, name)).read()
        assert re.findall(r'setmaxnreg\.\w+\.sync\.aligned\.u32 (\S+);" ::"n"\(k(?:Tc|D64)Split\.(few|many)\)', code) == [
            ("%0", "few"), ("%0", "many")]
        assert code.count("setmaxnreg.") == 2
    launch = open(os.path.join(build.CSRC, "baps_attention_launch.cuh")).read()
    assert launch.count("launch_kernel(") == 1
    assert launch.index("!has_registers_for<kernel>(split)") < launch.index("launch_kernel(")


def test_the_built_kernels_have_the_registers(split):
    """What ptxas reported when the library was built."""
    build.build()
    log = open(os.path.join(os.path.dirname(build.LIB), "build.log")).read()
    used = re.findall(r"Compiling entry function '\w*(attention_tc_kernel|attention_d64_kernel)\w*'.*?Used (\d+) registers", log, re.S)
    assert len(used) >= 15
    for name, regs in used:
        assert (split.tc_fits if name == "attention_tc_kernel" else split.d64_fits)(int(regs)), (name, regs)


def test_the_paired_kernel_takes_its_shares_from_the_split(split):
    code = open(os.path.join(build.CSRC, "baps_attention_pair.cuh")).read()
    assert re.findall(r'setmaxnreg\.\w+\.sync\.aligned\.u32 (\S+);" ::"n"\(kTcSplit\.(few|many)\)', code) == [
        ("%0", "few"), ("%0", "many")]
    assert code.count("setmaxnreg.") == 2 and "__launch_bounds__(kTcThreads, 1)" in code
    build.build()
    log = open(os.path.join(os.path.dirname(build.LIB), "build.log")).read()
    used = re.findall(r"Compiling entry function '\w*paired_attention_tc_kernel\w*'.*?Used (\d+) registers", log, re.S)
    assert len(used) == 2 and all(split.tc_fits(int(r)) for r in used)
