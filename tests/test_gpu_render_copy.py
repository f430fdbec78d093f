"""gs_render_fwd_copy writes the images it leaves in the image buffers, bit for
bit, on a launch of fewer bands than the GPU holds and on one of more, with
ragged edges."""
import pytest
import torch

import paper_2405_19614_gb300 as gs
import scenes
from gpu_util import params_on_device, viewmats_on_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(37, 23), (1283, 721)])
def test_copies_equal_the_images(size):
    from paper_2405_19614_gb300.build import build
    build()
    sc = scenes.cube_scene(3000, seed=3, sh_degree=1, log_scale=(-3.0, 0.5))
    cams = scenes.pinhole(size[0], size[1], 0.9 * size[0])
    rast = gs.Rasterizer(3000, 1, cams["intr"], cams["size"], pair_capacity=1 << 21)
    p, vm = params_on_device(sc), viewmats_on_device(cams)
    want = {k: v.clone() for k, v in rast.forward(p, vm).items()}
    copies = [torch.full_like(want[k], -1.0) for k in ("rgb", "depth", "alpha")]
    img = rast.forward(p, vm, copies=copies)
    assert rast.status() == 0
    for k in want:
        assert torch.equal(img[k], want[k]), k
    for k, c in zip(("rgb", "depth", "alpha"), copies):
        assert torch.equal(c, want[k]), k
    with pytest.raises(gs.GsError):
        rast.forward(p, vm, copies=[copies[0], copies[1], copies[0]])
