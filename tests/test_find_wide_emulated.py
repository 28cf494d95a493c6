"""Seeds with wide windows on the CPU: find_kernel and find_wide_kernel compiled
for the host with the warp emulated (as in test_find_emulated.py).  Seeds are
left and found again with the same bits, and how many are left does not follow
from the grid of the hit bins."""
import json
import os
import re
import shutil
import subprocess
import sys
import tempfile

import numpy as np
import pytest

from tests.test_find_emulated import CSRC, HERE, ROOT

OUTPUTS = ("par", "cov", "chi2", "n_hits", "hits", "status", "counters")


@pytest.fixture(scope="module")
def wide_so():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    src = open(os.path.join(CSRC, "mkf_find.cu")).read()
    end = "}  // namespace"
    body = src[src.index("namespace {"):src.index(end, src.index("find_wide_kernel(const")) + len(end)]
    body = body.replace("extern __shared__ __align__(16) unsigned char smem[];", "unsigned char *smem = g_smem;")
    body = body.replace("__shared__ ", "static ")
    body = re.sub(r'asm volatile\("mov\.u64 %0, %%globaltimer;" : "=l"\(t\)\);', "t = 0;", body)
    body = body.replace('asm volatile("griddepcontrol.wait;" ::: "memory");', "")
    d = tempfile.mkdtemp()
    with open(os.path.join(d, "find_dev.inc"), "w") as f:
        f.write('#include "mkf_internal.h"\n' + body + "\n")
    so = os.path.join(d, "wide_emu.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-fPIC", "-shared", "-I" + os.path.join(HERE, "host"),
                    "-I" + d, "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", so,
                    os.path.join(HERE, "host", "wide_emu.cpp")], check=True)
    return so


def run(so, lines, n_best, tracks, noise, grid=None, config="dense45", events=(71,)):
    """One result per line (see wide_emu.cpp); the seeds left under "left"."""
    out = os.path.join(tempfile.mkdtemp(), "out.npz")
    cfg = dict(config=config, events=list(events), tracks=tracks, noise=noise, grid=grid, lines=lines, n_best=n_best)
    r = subprocess.run([sys.executable, os.path.join(HERE, "host", "run_wide_emu.py"), so, ROOT, out, json.dumps(cfg)],
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-2000:]
    z = np.load(out)
    res = [{k: z[f"{k}_{i}"] for k in OUTPUTS + ("fault", "left")} for i in range(len(lines))]
    for x in res:
        assert (x["fault"] == 0).all(), x["fault"]
    return res, int(z["n_seeds"])


@pytest.mark.parametrize("n_best,grid", [(1, (1024, 8)), (2, (1024, 8)), (1, (256, 32)), (2, (37, 5))])
def test_left_seeds_are_found_with_the_same_bits(wide_so, n_best, grid):
    """A line of less than a bin leaves every seed with a window of some phi bins."""
    lines = [-1.0, 1e-3, 0.5, 4.0]
    (ref, *others), n = run(wide_so, lines, n_best, 60, 20000, grid)
    assert int(ref["left"][0]) == 0
    left = [int(o["left"][0]) for o in others]
    assert n > left[0] >= left[1] >= left[2] > 0, (left, n)
    assert grid[0] < 1000 or left[0] > n // 2, (left, n)
    for o in others:
        for k in OUTPUTS:
            assert np.array_equal(o[k].view(np.uint32), ref[k].view(np.uint32)), k


def test_the_seeds_left_do_not_follow_the_grid(wide_so):
    """By the library's rule, against the 256 x 32 grid that it was measured on."""
    left = {}
    for grid in ((256, 32), (512, 32), (64, 8), (16, 4), (8, 64), (64, 1), (1, 1)):
        (out,), n = run(wide_so, [0.0], 3, 1500, 200000, grid)
        left[grid] = int(out["left"][0])
    want = left[256, 32]
    assert 4 <= want <= n // 20, (left, n)
    assert max(left.values()) <= 2 * want, (left, n)
