"""A launch that the CUDA runtime refuses is an error of its own call only."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import make_ctx, upload

pytestmark = pytest.mark.gpu


def test_calls_after_a_refused_launch():
    """The gradient of more than 65535 chunks of 256 samples asks for a grid that
    no device takes (the runtime refuses it before anything runs)."""
    from paper_1811_04141_gb300._native import MkfError
    from paper_1811_04141_gb300.api import mkf_mlp_forward, mkf_mlp_grad
    b = make_batch("fit10", [3], n_tracks=300)
    d = upload(b)
    ctx = make_ctx(b)
    want = ctx.fit(d["xyz"], d["layer"], d["track_hits"])
    ctx.sync()
    n = 65535 * 256 + 1
    feat = torch.zeros(n, 12, device="cuda")
    label = torch.zeros(n, device="cuda")
    w = torch.zeros(897, dtype=torch.int16, device="cuda")
    calls = (lambda: ctx.fit(d["xyz"], d["layer"], d["track_hits"]),
             lambda: ctx.fit_smooth(d["xyz"], d["layer"], d["track_hits"]),
             lambda: mkf_mlp_forward(ctx, w, feat[:100]))
    for call in calls:
        with pytest.raises(MkfError):
            mkf_mlp_grad(ctx, w, feat, label)
        call()
        ctx.sync()
    got = ctx.fit(d["xyz"], d["layer"], d["track_hits"])
    ctx.sync()
    for k in want:
        if want[k] is not None:
            assert torch.equal(got[k].view(torch.int32), want[k].view(torch.int32)), k
    ctx.close()
