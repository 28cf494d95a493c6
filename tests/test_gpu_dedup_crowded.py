"""Duplicate removal where many tracks list one hit: the flags are the oracle's."""
import pytest
import torch

import oracle.dedup as D
from tests.test_dedup_crowded_host import crowded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n,per_hit,kind", [
    (1, 3000, 1500, "one"), (2, 900, 300, "same"), (8, 601, 9, "part"), (23, 601, 24, "part"), (23, 1203, 600, "part"),
    (23, 4000, 4000, "one"), (72, 300, 150, "part")])
def test_many_tracks_on_a_hit(rows, n, per_hit, kind):
    from paper_1811_04141_gb300 import Context, build
    build.build()
    ctx = Context(0)
    h, n_hits, nh, c2 = crowded(rows, n, per_hit, kind)
    for f in (0.0, 0.5, 1.0):
        keep = ctx.tracks_dedup(torch.as_tensor(h, device="cuda"), n_hits, torch.as_tensor(nh, device="cuda"),
                                torch.as_tensor(c2, device="cuda"), f).cpu().numpy()
        assert (keep.astype(bool) == D.dedup_tracks(h, n_hits, nh, c2, f)).all(), f
    ctx.close()
