"""Finding in the parameterised field around the line where the columns of a
move are no longer taken side by side: the outputs are the same bits."""
import pytest
import torch

from synth import make_batch
from tests.gpu_helpers import make_ctx, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_best,rows", [(1, 32), (4, 8), (10, 3), (16, 2)])
def test_columns_side_by_side_or_in_turn(n_best, rows):
    b = make_batch("find20", [96], n_tracks=300, field_alpha=1e-5)
    ctx = make_ctx(b)
    d = upload(b)
    bins = ctx.hits_bin(d["xyz"], d["layer"], d["event_offsets"])
    n0 = d["seed_event"].shape[0]
    ref = ctx.find(bins, d["seed_hits"], d["seed_event"], n_best=n_best)
    ctx.sync()
    ref = {k: v.clone() for k, v in ref.items()}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # `rows` seeds a warp, up to 16 warps on an SM; the line lies at half of them
    for warps in (2, 4, 6, 8, 16):
        for n in (rows * warps * sms, rows * warps * sms + 1):
            at = torch.arange(n, device="cuda") % n0
            out = ctx.find(bins, d["seed_hits"][:, at].contiguous(), d["seed_event"][at].contiguous(), n_best=n_best)
            ctx.sync()
            for k, v in ref.items():
                assert torch.equal(out[k].view(torch.int32), v[..., at].view(torch.int32)), (k, n)
    ctx.close()
