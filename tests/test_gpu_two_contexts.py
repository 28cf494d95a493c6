"""Contexts on one device share its kernels: what one context's calls ask of
them (dynamic shared memory) and a launch that one call is refused leave the
other calls as they are."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import upload

pytestmark = pytest.mark.gpu


def test_second_context_keeps_the_first_ones_shared_memory():
    """N = 16 in blocks of 256 needs more shared memory than a block has by
    default; a context whose first call needs less comes in between."""
    from paper_1811_04141_gb300 import Context, build
    build.build()
    b = make_batch("dense45", [31], n_tracks=200, n_noise=2000)
    d = upload(b)

    def call(ctx, **kw):
        bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
        out = ctx.find(bins, d["seed_hits"], d["seed_event"], **kw)
        ctx.sync()
        return out

    big = dict(n_best=16, block_threads=256)
    a, c = Context(0), Context(0)
    for ctx in (a, c):
        ctx.geometry_load(b.layers, b.bz)
    want = call(a, **big)
    call(c, n_best=1, block_threads=32)
    got = call(a, **big)
    for k in want:
        assert torch.equal(got[k].view(torch.int32), want[k].view(torch.int32)), k
    # and the second context can ask for more later, the first one unharmed
    got = call(c, **big)
    for k in want:
        assert torch.equal(got[k].view(torch.int32), want[k].view(torch.int32)), k
    call(a, n_best=1)
    a.close()
    c.close()
