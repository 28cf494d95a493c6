"""The seeds' processing order around the line where a call's seeds all have a
warp at once (input order below it, grouped by event and |eta| above): the
outputs are those of the input order, bit for bit, eagerly and in a graph."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_best,threads,rows", [(10, 0, 3), (10, 256, 3), (16, 32, 2), (3, 64, 10), (1, 32, 32)])
def test_order_line(n_best, threads, rows):
    from paper_1811_04141_gb300 import Context, build
    build.build()
    b = make_batch("find20", [91, 92, 93], n_tracks=700)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = Context(0)
    ctx.geometry_load(b.layers, b.bz)
    d = upload(b)
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    n0 = d["seed_event"].shape[0]
    # `rows` seeds a warp, at most 16 warps of 128 registers on an SM: the line
    # lies at one of these multiples of a full row of warps, at its last seed
    for warps in (1, 4, 8, 12, 16):
        for n in (rows * warps * sms, rows * warps * sms + 1):
            at = torch.arange(n, device="cuda") % n0
            hits, ev = d["seed_hits"][:, at].contiguous(), d["seed_event"][at].contiguous()
            kw = dict(n_best=n_best, block_threads=threads)
            ref = ctx.find(bins, hits, ev, seed_order=1, **kw)
            out = ctx.find(bins, hits, ev, seed_order=0, **kw)
            ctx.sync()
            for k, v in ref.items():
                assert torch.equal(out[k].view(torch.int32), v.view(torch.int32)), (k, n)
    # the largest call in a graph (its scratch is already there)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    from paper_1811_04141_gb300.api import mkf_set_stream
    mkf_set_stream(ctx.handle, side)
    got = {k: torch.full_like(v, -7) for k, v in ref.items()}
    with torch.cuda.stream(side):
        ctx.find(bins, hits, ev, out=got, **kw)
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            ctx.find(bins, hits, ev, out=got, **kw)
        for v in got.values():
            v.fill_(-7)
        g.replay()
    side.synchronize()
    for k, v in ref.items():
        assert torch.equal(got[k].view(torch.int32), v.view(torch.int32)), k
    mkf_set_stream(ctx.handle, torch.cuda.current_stream())
    ctx.close()
