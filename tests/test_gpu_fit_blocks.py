"""Fits of as many tracks as make one variant of the fit kernel give way to the
next, against the same tracks in small calls."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import chi2_errors, make_ctx, par_errors, to_np, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("material", [False, True])
def test_variants_agree_around_the_lines(material):
    mat = dict(material=0.03, eloss=0.04) if material else {}
    b = make_batch("fit10", [5, 6], n_tracks=1000, **mat)
    ctx = make_ctx(b)
    d = upload(b)
    n0 = d["track_hits"].shape[1]
    ref = ctx.fit(d["xyz"], d["layer"], d["track_hits"])
    back = ctx.fit_backward(d["xyz"], d["layer"], d["track_hits"], ref["par"], ref["cov"], 100.0)
    ctx.sync()
    ref = {k: v.clone() for k, v in ref.items() if v is not None}
    back = {k: v.clone() for k, v in back.items() if v is not None}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for per_sm in (4, 5, 6, 8, 10, 12, 15, 18):
        for n in (128 * sms * per_sm, 128 * sms * per_sm + 1):
            at = torch.arange(n, device="cuda") % n0
            hits = d["track_hits"][:, at].contiguous()
            out = ctx.fit(d["xyz"], d["layer"], hits)
            rev = ctx.fit_backward(d["xyz"], d["layer"], hits, ref["par"][:, at].contiguous(),
                                   ref["cov"][:, at].contiguous(), 100.0)
            ctx.sync()
            for got, want in ((out, ref), (rev, back)):
                want = {k: v[..., at] for k, v in want.items()}
                assert torch.equal(got["status"], want["status"]) and torch.equal(got["ndf"], want["ndf"]), n
                g, w = to_np(got), to_np(want)
                assert par_errors(g["par"], w["par"]).max() <= 1.0, n
                assert chi2_errors(g["chi2"], w["chi2"], w["ndf"]).max() <= 1.0, n
    ctx.close()
