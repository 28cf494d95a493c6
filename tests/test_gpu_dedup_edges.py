"""Seed cleaning where the FP32 test of the eta difference cannot decide:
differences at the tolerance and within a few 1e-7 of it, angles next to 0 and
pi, and tolerances from 0 up; and tracks that list hits twice, with many rows."""
import numpy as np
import pytest
import torch

import oracle.dedup as D

pytestmark = pytest.mark.gpu


def _ctx():
    from paper_1811_04141_gb300 import Context, build
    build.build()
    return Context(0)


@pytest.mark.parametrize("tol", [0.0, 1e-7, 3e-4, 0.02, 1.0, 30.0])
def test_eta_differences_at_the_tolerance(tol):
    ctx = _ctx()
    rng = np.random.default_rng(int(tol * 1e4) + 1)
    n = 4001
    eta = rng.uniform(-4.0, 4.0, n)
    # pairs (2 k, 2 k + 1) share a hit; the second's eta is tol away, give or take
    eta[1::2] = eta[0:n - 1:2] + np.float32(tol) * rng.choice([-1.0, 1.0], n // 2) + rng.choice(
        [0.0, 1e-7, -1e-7, 1e-5, -1e-5, 1e-3, -1e-3], n // 2)
    th = (2.0 * np.arctan(np.exp(-eta))).astype(np.float32)
    th[5::97] = np.float32(1e-30)
    th[7::101] = np.float32(np.pi)
    th[11::103] = 0.0
    th[13::107] = np.nan
    par = np.zeros((6, n), np.float32)
    par[3] = 0.3
    par[4] = rng.choice([3.14159, -3.14159, 0.0], n)  # phi differences of 0, pi and 2 pi
    par[5] = th
    hits = np.arange(3 * n, dtype=np.int32).reshape(3, n)
    hits[1, 1::2] = hits[0, 0:n - 1:2]
    keep = ctx.seeds_clean(torch.as_tensor(hits, device="cuda"), 3 * n, torch.as_tensor(par, device="cuda"), 0.5, tol,
                           0.02).cpu().numpy()
    assert (keep.astype(bool) == D.clean_seeds(hits, 3 * n, par, 0.5, np.float32(tol), 0.02)).all()
    ctx.close()


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 16, 17, 72])
def test_tracks_with_repeated_hits_and_many_rows(rows):
    ctx = _ctx()
    rng = np.random.default_rng(rows)
    n, n_hits = 1500, 40 * rows
    hits = rng.integers(-2, n_hits + 2, size=(rows, n)).astype(np.int32)
    hits[rows // 2:, ::3] = hits[: rows - rows // 2, ::3]  # hits listed twice
    hits[:, 1::2] = np.where(rng.random((rows, n // 2)) < 0.6, hits[:, 0:n - 1:2], hits[:, 1::2])  # near twins
    nh = rng.integers(1, rows + 1, n).astype(np.int32)
    c2 = rng.integers(0, 3, n).astype(np.float32)
    for f in (0.0, 0.3, 0.5, 1.0):
        keep = ctx.tracks_dedup(torch.as_tensor(hits, device="cuda"), n_hits, torch.as_tensor(nh, device="cuda"),
                                torch.as_tensor(c2, device="cuda"), f).cpu().numpy()
        assert (keep.astype(bool) == D.dedup_tracks(hits, n_hits, nh, c2, f)).all(), f
    ctx.close()
