"""The choice of the fit kernel's variant (blocks per SM) on the CPU: a call
that one wave of blocks can hold gets one wave."""
import ctypes as C
import os
import shutil
import subprocess
import tempfile

import pytest

from tests.test_fit_host import CSRC


@pytest.fixture(scope="module")
def blocks_for():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    src = open(os.path.join(CSRC, "mkf_fit.cu")).read()
    a = src.index("constexpr int fit_blocks(int phys)")
    body = src[a:src.index("\n}\n", src.index("inline int fit_blocks_for")) + 3]
    d = tempfile.mkdtemp()
    with open(os.path.join(d, "b.cpp"), "w") as f:
        f.write("#include <cstdint>\n" + body + 'extern "C" int blocks_for(int phys, int backward, int blocks, int sms) '
                "{ return fit_blocks_for(phys, backward != 0, blocks, sms); }\n")
    so = os.path.join(d, "b.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-fPIC", "-shared", "-o", so, os.path.join(d, "b.cpp")], check=True)
    return C.CDLL(so).blocks_for


@pytest.mark.parametrize("sms", [152, 148, 1])
@pytest.mark.parametrize("backward", [0, 1])
def test_no_second_wave_where_one_is_enough(blocks_for, backward, sms):
    compiled = {0: (5, 6), 1: (4, 5, 6), 2: (3,)}
    for phys, ks in compiled.items():
        for blocks in list(range(1, 8 * sms)) + [100 * sms, 1 << 24]:
            k = blocks_for(phys, backward, blocks, sms)
            assert k in ks, (phys, blocks, k)
            if blocks <= max(ks) * sms:
                assert blocks <= k * sms, (phys, blocks, k)
            if blocks <= min(ks) * sms or blocks == 1 << 24 and phys == 0:
                assert k == min(ks), (phys, blocks, k)  # nothing spills
