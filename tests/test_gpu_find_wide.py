"""Seeds with wide windows (find_wide_kernel) against the general path, bit for
bit: the finder with the MLP compiled in and nothing pruned (every logit is
above the threshold) searches every window with one lane per candidate."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import upload

pytestmark = pytest.mark.gpu


def _batch(grid=None):
    b = make_batch("dense45", [71, 72], n_tracks=1500, n_noise=200000, material=0.02, eloss=0.04)
    if grid:
        for d in b.layers:
            d["n_phi"], d["n_zr"] = grid
    return b


def _same(a, b):
    for k in a:
        x, y = a[k], b[k]
        if x.is_floating_point():
            x, y = x.view(torch.int32), y.view(torch.int32)
        assert torch.equal(x, y), k


def _ctx(b, field_alpha=None):
    from paper_1811_04141_gb300 import Context, build
    build.build()
    ctx = Context(0)
    ctx.geometry_load(b.layers, b.bz, field_alpha=field_alpha)
    return ctx


@pytest.mark.parametrize("n_best,cut,grid,alpha", [
    (1, 30.0, None, None), (2, 30.0, None, None), (5, 30.0, None, None), (10, 30.0, None, None), (16, 30.0, None, None),
    (10, 100.0, None, None), (10, 30.0, (37, 5), None), (3, 30.0, (1, 1), None), (10, 30.0, None, 1e-6),
    (1, 30.0, None, 1e-6)])
def test_wide_windows_match_the_general_path(n_best, cut, grid, alpha):
    b = _batch(grid)
    ctx = _ctx(b, alpha)
    d = upload(b)
    mlp = torch.zeros(897, dtype=torch.int16, device="cuda")
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    kw = dict(n_best=n_best, chi2_cut=cut)
    out = ctx.find(bins, d["seed_hits"], d["seed_event"], **kw)
    ref = ctx.find(bins, d["seed_hits"], d["seed_event"], mlp_bf16=mlp, mlp_tau=-1.0, **kw)
    ctx.sync()
    # some seeds test hundreds of hits where most test one a layer
    assert int(ref["counters"][1].max()) > 300
    _same(out, ref)
    # a subset in an order of its own, the other seeds' outputs untouched
    lst = torch.arange(d["seed_event"].shape[0] - 1, -1, -3, dtype=torch.int32, device="cuda")
    cnt = torch.tensor([lst.shape[0]], dtype=torch.int32, device="cuda")
    sub = {k: torch.full_like(v, -7) for k, v in ref.items()}
    ctx.find(bins, d["seed_hits"], d["seed_event"], out=sub, seed_list=lst, seed_count=cnt, **kw)
    ctx.sync()
    keep = torch.zeros(d["seed_event"].shape[0], dtype=torch.bool, device="cuda")
    keep[lst.long()] = True
    for k, v in ref.items():
        want = torch.where(keep, v, torch.full_like(v, -7))
        _same({k: sub[k]}, {k: want})
    ctx.close()


def test_wide_windows_with_the_gate_and_in_a_graph():
    from paper_1811_04141_gb300.runtime import CapturedStep
    b = _batch()
    ctx = _ctx(b)
    d = upload(b)
    mlp = torch.zeros(897, dtype=torch.int16, device="cuda")
    step = CapturedStep(ctx, d["xyz"], d["layer"], d["event_offsets"], d["seed_hits"], d["seed_event"], n_best=10)
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    ref = ctx.find(bins, d["seed_hits"], d["seed_event"], n_best=10, mlp_bf16=mlp, mlp_tau=-1.0)
    ref = {k: v.clone() for k, v in ref.items()}
    torch.cuda.synchronize()
    for _ in range(3):
        for v in step.out.values():
            v.fill_(-7)
        torch.cuda.synchronize()
        out = step.replay()
        torch.cuda.synchronize()
        _same(out, ref)
    # the gate flags the same seeds' best-hit tracks: every logit is 0 here
    for tau, flagged in ((-1.0, False), (1.0, True)):
        g = ctx.find(bins, d["seed_hits"], d["seed_event"], n_best=1, mlp_bf16=mlp, mlp_tau=tau, mlp_mode=1)
        p = ctx.find(bins, d["seed_hits"], d["seed_event"], n_best=1, mlp_bf16=mlp, mlp_tau=-1.0)
        ctx.sync()
        amb = (g["status"] & 64) != 0
        assert bool(amb.any()) == flagged
        g["status"] &= ~64
        _same(g, p)
    ctx.close()


@pytest.mark.parametrize("times,n_best,listed", [(1, 2, False), (14, 2, False), (40, 2, False), (1, 1, True), (30, 3, True)])
def test_the_line_over_the_number_of_seeds(times, n_best, listed):
    """The window size from which seeds are left grows with the call's seeds; the outputs do not change."""
    b = _batch()
    ctx = _ctx(b)
    d = upload(b)
    mlp = torch.zeros(897, dtype=torch.int16, device="cuda")
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    ref = ctx.find(bins, d["seed_hits"], d["seed_event"], n_best=n_best, mlp_bf16=mlp, mlp_tau=-1.0)
    n0 = d["seed_event"].shape[0]
    at = torch.arange(n0 * times, device="cuda") % n0
    kw = {}
    if listed:
        kw = dict(seed_list=torch.arange(n0 * times, dtype=torch.int32, device="cuda"),
                  seed_count=torch.tensor([n0 * times], dtype=torch.int32, device="cuda"))
    out = ctx.find(bins, d["seed_hits"][:, at].contiguous(), d["seed_event"][at].contiguous(), n_best=n_best, **kw)
    ctx.sync()
    _same(out, {k: v[..., at] for k, v in ref.items()})
    ctx.close()
