"""Depths around 2^126, beyond which the fast quotient of the projection's early
test gives zero: a Gaussian whose mean lies some pixels from a principal point
outside the image is drawn or not as the geometry contract says."""
import numpy as np
import pytest
import torch

import oracle
import paper_2405_19614_gb300 as gs
import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", ["left", "right", "above", "below"])
def test_depths_beyond_the_fast_quotient(side):
    z = np.array([8.4e37, 2.0 ** 126, 8.6e37, 8.6e37, 8.6e37, 1.2e38], np.float32)
    off = np.array([3.0e38, 3.2e38, 3.2e38, 3.3e38, -3.2e38, 3.2e38], np.float32)  # of the axis beside the image
    w, h = 64, 32
    intr = {"left": [1, 1, -3.9, 16], "right": [1, 1, 67.9, 16], "above": [1, 1, 32, -3.9], "below": [1, 1, 32, 35.9]}[side]
    sign = -1.0 if side in ("right", "below") else 1.0
    n = len(z)
    sc = scenes.cube_scene(n, seed=1, sh_degree=0, log_scale=(-3.0, 0.0), opacity=(3.0, 0.0))
    sc["means"][:] = 0.0
    sc["means"][:, 2] = z
    sc["means"][:, 0 if side in ("left", "right") else 1] = sign * off
    cams = scenes.cams_from([intr], [[w, h]], np.concatenate([np.eye(3), np.zeros((3, 1))], 1)[None])
    geom = oracle.project_geom(sc, cams)
    assert (geom["kept"][2:4] > 0).all() and geom["kept"][4] == 0
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    params = {k: dev(sc[k]) for k in ("means", "log_scales", "quats", "opacity_logit", "sh")}
    params["sh_degree"] = 0
    rast = gs.Rasterizer(n, 0, [intr], [[w, h]], pair_capacity=1 << 10)
    gs.gs_project(params, rast.views, dev(cams["viewmats"].reshape(-1, 12)), rast.proj, rast.near_z, rast.blur)
    np.testing.assert_array_equal(rast.proj["radii"].cpu().numpy(), geom["radius"])
    np.testing.assert_array_equal(rast.proj["tiles_touched"].cpu().numpy().view(np.uint32), geom["kept"])
