"""Hit lists with empty rows: the fit kernels read a track's rows one ahead, so
the same hits spread over more rows (-1 between them) must give the same bits,
whatever the number of rows; and an index out of range is reported wherever it
stands."""
import numpy as np
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import make_ctx, upload

pytestmark = pytest.mark.gpu


def _spread(hits, rows, seed):
    """The lists of `hits` [m, n] over `rows` rows, in order, -1 elsewhere; and the row of each hit."""
    m, n = hits.shape
    rng = np.random.default_rng(seed)
    at = np.sort(np.argsort(rng.random((rows, n)), axis=0)[:m], axis=0)
    out = np.full((rows, n), -1, np.int32)
    out[at, np.arange(n)[None, :]] = hits
    return out, at


def _bits(a, b):
    for k in a:
        x, y = a[k].cpu(), b[k].cpu()
        if x.is_floating_point():
            x, y = x.view(torch.int32), y.view(torch.int32)
        assert torch.equal(x, y), k


@pytest.mark.parametrize("cfg,kw", [("find20", {}), ("dense45", dict(material=0.02, eloss=0.04)),
                                    ("fit10", dict(field_alpha=1e-5))])
@pytest.mark.parametrize("m,rows", [(3, 3), (3, 4), (4, 5), (7, 9), (7, 64)])
def test_empty_rows_change_nothing(cfg, kw, m, rows):
    b = make_batch(cfg, [5], n_tracks=400, **kw)
    ctx = make_ctx(b)
    ctx.geometry_load(b.layers, b.bz, field_alpha=kw.get("field_alpha"))
    d = upload(b)
    hits = b.track_hits[:m]
    hits = np.ascontiguousarray(hits[:, (hits >= 0).all(0)][:, :333])  # not a multiple of the block
    wide, at = _spread(hits, rows, m * rows)
    t = lambda a: torch.as_tensor(a, device="cuda")
    f0 = ctx.fit(d["xyz"], d["layer"], t(hits))
    _bits(f0, ctx.fit(d["xyz"], d["layer"], t(wide)))
    _bits(ctx.fit_backward(d["xyz"], d["layer"], t(hits), f0["par"], f0["cov"], 10.0),
          ctx.fit_backward(d["xyz"], d["layer"], t(wide), f0["par"], f0["cov"], 10.0))
    s0 = ctx.fit_smooth(d["xyz"], d["layer"], t(hits), inflate=100.0)
    s1 = ctx.fit_smooth(d["xyz"], d["layer"], t(wide), inflate=100.0)
    n = hits.shape[1]
    full = {k: torch.full((rows,) + s0[k].shape[1:], float("nan"), device="cuda") for k in ("par", "cov")}
    for k in full:  # the rows of the hits, NaN elsewhere
        full[k].scatter_(0, t(at)[:, None, :].expand(m, s0[k].shape[1], n), s0[k])
        assert torch.equal(torch.isnan(full[k]), torch.isnan(s1[k])), k
        assert torch.equal(torch.nan_to_num(full[k]), torch.nan_to_num(s1[k])), k
    _bits({k: s0[k] for k in ("chi2", "ndf", "status")}, {k: s1[k] for k in ("chi2", "ndf", "status")})
    ctx.sync()
    ctx.close()


@pytest.mark.parametrize("row", [0, 2, 5, 8])
def test_invalid_index_is_reported_and_skipped(row):
    from paper_1811_04141_gb300._native import MkfError
    b = make_batch("fit10", [6], n_tracks=200)
    ctx = make_ctx(b)
    d = upload(b)
    bad = b.track_hits.copy()
    bad[row, 17] = b.n_hits
    hole = b.track_hits.copy()
    hole[row, 17] = -1
    few = np.full((3, 1), -1, np.int32)  # fewer than three hits: reported too
    few[2, 0] = b.n_hits + 5
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    for run in (lambda h: ctx.fit(d["xyz"], d["layer"], t(h)), lambda h: ctx.fit_smooth(d["xyz"], d["layer"], t(h))):
        ref = run(hole)
        ctx.sync()
        out = run(bad)
        with pytest.raises(MkfError):
            ctx.sync()
        ok = ~torch.isnan(ref["par"])
        assert torch.equal(ok, ~torch.isnan(out["par"])) and torch.equal(ref["par"][ok], out["par"][ok])
        assert torch.equal(ref["status"], out["status"])
        run(few)
        with pytest.raises(MkfError):
            ctx.sync()
    ctx.close()
