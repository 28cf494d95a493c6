"""CPU check of the finder's processing order of a call on a list of seeds, with
the seed kernel and the order kernel compiled for the host: every place of the
order holds a seed of the list, also when the list names a seed more than once,
names seeds that do not exist or is short -- never what the buffer held before."""
import ctypes as C
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1811_04141_gb300 import _native as NN
from synth import make_batch
from tests.test_find_emulated import CSRC, HERE, ROOT, _device_part


@pytest.fixture(scope="module")
def lib():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    d = tempfile.mkdtemp()
    with open(os.path.join(CSRC, "mkf_find.cu")) as f:
        dev = _device_part(f.read())
    with open(os.path.join(d, "find_dev.inc"), "w") as f:
        f.write(dev)
    so = os.path.join(d, "order_emu.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-pthread", "-fPIC", "-shared", "-I" + os.path.join(HERE, "host"),
                    "-I" + d, "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", so,
                    os.path.join(HERE, "host", "order_emu.cpp")], check=True)
    return C.CDLL(so)


def _order(lib, n, n_events, lst, before):
    lay = make_batch("find20", [1], n_tracks=1).layers
    arr = (NN.MkfLayer * len(lay))()
    for i, d in enumerate(lay):
        arr[i] = NN.MkfLayer(int(d["kind"]), float(d["r_or_z"]), float(d["lo"]), float(d["hi"]), float(d["sigma_u"]),
                             float(d["sigma_v"]), int(d["n_phi"]), int(d["n_zr"]))
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    hits = np.full((3, n), -1, np.int32)  # recorded as a fault, each such seed keeps its place
    ev = (np.arange(n) % n_events).astype(np.int32)
    order = np.full(n, before, np.int32)
    fault = np.zeros(2, np.int32)
    l = None if lst is None else np.ascontiguousarray(lst, dtype=np.int32)
    padded = None if l is None else np.concatenate([l, np.full(max(0, n - l.size), 1 << 30, np.int32)])
    total = lib.emu_order(arr, len(lay), p(hits), p(ev), n, n_events, None if l is None else p(padded),
                          0 if l is None else int(l.size), p(order), p(fault))
    return total, order, ev


@pytest.mark.parametrize("n,n_events,lst", [
    (300, 3, None),
    (300, 3, np.arange(299, -1, -3)),
    (300, 3, np.repeat(np.arange(50), 6)),
    (300, 1, np.zeros(300, int)),
    (300, 3, np.concatenate([np.arange(100), np.arange(100)])),
    (300, 3, np.array([5, 5, -1, 400, 7, 5, 300, 7])),
    (300, 3, np.zeros(0, int))])
def test_every_place_holds_a_seed_of_the_list(lib, n, n_events, lst):
    for before in (-12345, 17, 1 << 29):
        total, order, ev = _order(lib, n, n_events, lst, before)
        want = np.arange(n) if lst is None else lst[(lst >= 0) & (lst < n)]
        assert total == want.size
        assert sorted(order[:total]) == sorted(want)  # each as often as it is listed
        assert (np.diff(ev[order[:total]]) >= 0).all()  # grouped by event
        assert (order[total:] == before).all()
