"""Finding with a list that names seeds more than once, in calls small enough
for the input order and large enough for the grouped one: the listed seeds'
outputs are those of a call on every seed, bit for bit, the others' stay."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("material,n_best", [(False, 10), (False, 1), (True, 4)])
@pytest.mark.parametrize("times", [1, 50])
def test_listed_more_than_once(material, n_best, times):
    from paper_1811_04141_gb300 import Context, build
    build.build()
    mat = dict(material=0.02, eloss=0.04) if material else {}
    b = make_batch("find20", [61, 62], n_tracks=1000, **mat)
    ctx = Context(0)
    ctx.geometry_load(b.layers, b.bz)
    d = upload(b)
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    n0 = d["seed_event"].shape[0]
    n = n0 * times
    at = torch.arange(n, device="cuda") % n0
    hits, ev = d["seed_hits"][:, at].contiguous(), d["seed_event"][at].contiguous()
    ref = ctx.find(bins, hits, ev, n_best=n_best)
    ref = {k: v.clone() for k, v in ref.items()}
    # every fifth seed, each four or five times in a row, and the first one often
    lst = torch.arange(n, device="cuda") // 5 * 5
    lst[::7] = 0
    lst = lst.to(torch.int32)
    cnt = torch.tensor([n], dtype=torch.int32, device="cuda")
    listed = torch.zeros(n, dtype=torch.bool, device="cuda")
    listed[lst.long()] = True
    for order in (0, 1):
        # a call on every seed leaves its own order in the scratch memory
        ctx.find(bins, hits, ev, n_best=n_best)
        got = {k: torch.full_like(v, -7) for k, v in ref.items()}
        ctx.find(bins, hits, ev, n_best=n_best, out=got, seed_list=lst, seed_count=cnt, seed_order=order)
        ctx.sync()
        for k, v in ref.items():
            want = torch.where(listed, v, torch.full_like(v, -7))
            assert torch.equal(got[k].view(torch.int32), want.view(torch.int32)), (k, order)
    ctx.close()
