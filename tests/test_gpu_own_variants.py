"""Images on each side of the pixel counts at which the library's own choice of
compositing variants changes, against the variants pinned for room-scale views:
the forward bit for bit, the gradients to the bar of the parity tests."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs
from gpu_util import GRAD_TOL, make_rast, params_on_device, rel_l2, t, viewmats_on_device

import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(64, 48), (322, 241), (361, 299), (640, 480)])
def test_own_choice_matches_pinned_variants(size):
    sc = scenes.cube_scene(2000, seed=size[0])
    cams = scenes.pinhole(*size, 0.9 * size[0])
    rast, p, vm = make_rast(sc, cams), params_on_device(sc), viewmats_on_device(cams)
    rng = np.random.default_rng(size[1])
    dC, dD = t(rng.normal(0, 1, (rast.n_pix, 3))), t(rng.normal(0, 1, rast.n_pix))
    saved = gs.gs_get_render_variants()[:2]
    out = []
    try:
        for fwd, bwd in ((-1, -1), (7, 9)):
            gs.gs_set_render_variants(fwd, bwd)
            rast.forward(p, vm)
            img = {k: v.clone() for k, v in rast.img.items()}
            rast.grad2d.zero_()
            gs.gs_render_bwd_splats(rast.proj, rast.n, rast.bins, rast.views, rast.img, dC, dD, None, rast.grad2d,
                                    rast.work_counter)
            torch.cuda.synchronize()
            out.append((img, rast.grad2d.cpu().numpy().reshape(-1, 12)[:, :10]))
    finally:
        gs.gs_set_render_variants(*saved)
    for k in out[0][0]:
        assert torch.equal(out[0][0][k], out[1][0][k]), k
    assert np.abs(out[1][1]).max() > 0
    assert rel_l2(out[0][1], out[1][1]) <= GRAD_TOL
