"""CPU check of duplicate removal where many tracks list one hit, with the kernel
of mkf_dedup.cu compiled for the host: the keep flags are the oracle's, and a
comparison of two tracks reads no more than it would read of the other track's
own list (the reads are counted)."""
import ctypes as C
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import oracle.dedup as D
from tests.test_dedup_host import CSRC, HERE, ROOT, _tracks

COUNTED = """
struct Counted {
    const int32_t *p;
    static long long &reads() { static long long n = 0; return n; }
    Counted(const int32_t *q) : p(q) {}
    const int32_t &operator[](int64_t i) const { ++reads(); return p[i]; }
};
extern "C" long long index_reads() { const long long n = Counted::reads(); Counted::reads() = 0; return n; }
"""


@pytest.fixture(scope="module")
def lib():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    src = open(os.path.join(CSRC, "mkf_dedup.cu")).read()
    a = src.index("namespace {")
    b = src.index("// Inverse index hit -> items of `lists`")
    body = src[a:b]
    k = body.index("tracks_decide_kernel(")
    body = body[:k] + body[k:].replace("const int32_t *items", "Counted items", 1) + "\n}  // namespace\n"
    body = body.replace("has = *L ==", "has = Counted(L)[0] ==")  # the look-up of a hit
    d = tempfile.mkdtemp()
    with open(os.path.join(d, "dedup_dev.inc"), "w") as f:
        f.write('#include "mkf_internal.h"\n' + COUNTED + body)
    so = os.path.join(d, "dedup_emu.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + os.path.join(HERE, "host"), "-I" + d,
                    "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", so,
                    os.path.join(HERE, "host", "dedup_emu.cpp")], check=True)
    lib = C.CDLL(so)
    lib.index_reads.restype = C.c_longlong
    return lib


def crowded(rows, n, per_hit, kind):
    """n tracks in groups of per_hit that share one hit (kind "one"), every hit ("same") or a part of them."""
    rng = np.random.default_rng(rows * 1000 + per_hit)
    group = np.arange(n) // per_hit * rows + np.arange(rows)[:, None]
    own = n * rows + np.arange(n) * rows + np.arange(rows)[:, None]
    if kind == "one":
        h = own.copy()
        h[rows // 2] = group[rows // 2]
    elif kind == "same":
        h = group
    else:
        h = np.where(rng.random((rows, n)) < 0.45, group, own)
        h[-1, ::5] = h[0, ::5]  # a hit listed twice
        h[1, ::9] = -1
    nh = rng.integers(rows - 1, rows + 1, n).astype(np.int32)
    return h.astype(np.int32), 2 * n * rows, nh, rng.integers(0, 50, n).astype(np.float32)


@pytest.mark.parametrize("kind", ["one", "same", "part"])
@pytest.mark.parametrize("rows,per_hit", [(6, 5), (6, 7), (6, 300), (12, 13), (23, 24), (23, 600)])
def test_flags_and_index_reads(lib, rows, per_hit, kind):
    n = 601
    h, n_hits, nh, c2 = crowded(rows, n, per_hit, kind)
    for f in (0.0, 0.5, 1.0):
        lib.index_reads()
        keep = _tracks(lib, h, n_hits, nh, c2, f)
        reads = lib.index_reads()
        assert (keep.astype(bool) == D.dedup_tracks(h, n_hits, nh, c2, f)).all(), f
        # each of a track's rows walks its hit's tracks (as often as they list it)
        # and compares with the better ones: at most rows^2 reads each
        lists = [np.unique(h[h[:, i] >= 0, i], return_counts=True) for i in range(n)]
        listed = np.zeros(n_hits, np.int64)
        for x, c in lists:
            listed[x] += c
        walked = sum(int((listed[x] * c).sum()) for x, c in lists)
        better = sum(int((np.maximum(listed[x] - 1, 0) * c).sum()) for x, c in lists)
        assert reads <= walked + better * rows * rows // 2 + better * rows, (f, reads, walked, better)
