"""gs_bin_sort into ranges on 4 bytes but not on 8 gives the lists it gives into
ranges of its own."""
import pytest
import torch

import paper_2405_19614_gb300 as gs
from gpu_util import make_rast, params_on_device, viewmats_on_device

import scenes

pytestmark = pytest.mark.gpu


def test_ranges_inside_another_array():
    c = scenes.config(1, scale=0.25)
    rast, vm = make_rast(c["scene"], c["cams"]), viewmats_on_device(c["cams"])
    rast.forward(params_on_device(c["scene"]), vm)
    want = {k: rast.bins[k].clone() for k in ("keys", "vals", "ranges")}
    arena = torch.full((2 * rast.n_tiles + 8,), -1, dtype=torch.int32, device="cuda")
    ranges = arena[1:2 * rast.n_tiles + 1].view(rast.n_tiles, 2)
    assert ranges.data_ptr() % 8 == 4
    bins = dict(rast.bins, ranges=ranges)
    for k in ("keys", "vals"):
        bins[k].fill_(-1)
    gs.gs_bin_sort(rast.proj, rast.n, rast.views, bins, rast.workspace)
    K = rast.n_pairs()
    assert K > 0 and torch.equal(ranges, want["ranges"])
    assert torch.equal(bins["keys"][:K], want["keys"][:K]) and torch.equal(bins["vals"][:K], want["vals"][:K])
    assert int(arena[0]) == -1 and bool((arena[2 * rast.n_tiles + 1:] == -1).all())
