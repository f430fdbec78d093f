"""The projection's early test for Gaussians beside the image changes no
decision: radii and tile counts equal the oracle's geometry contract bit for bit
on Gaussians crowded around the image borders and the near plane, with scales
from far below a pixel to larger than the view, poses that are not orthonormal,
off-centre and extreme intrinsics, with and without the low-pass blur."""
import numpy as np
import pytest
import torch

import oracle
import paper_2405_19614_gb300 as gs
import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blur", [0.0, 0.3, 4.0])
@pytest.mark.parametrize("pose", ["rigid", "scaled", "skewed"])
def test_early_reject_equals_the_contract(pose, blur):
    from paper_2405_19614_gb300.build import build
    build()
    rng = np.random.default_rng(11)
    n = 20000
    size = [[64, 48], [321, 97], [33, 257]]
    intr = [[60.0, 60.0, 32.0, 24.0], [35.0, 700.0, -40.0, 200.0], [900.0, 20.0, 16.5, 128.5]]
    mats = []
    for k in range(3):
        E = scenes.look_at((0.1 * k, -0.2, 0.05), (0.2, 0.1 * k, 3.0)).astype(np.float64)
        if pose == "scaled":
            E[:, :3] *= (0.3, 2.5, 1.7)[k]
        if pose == "skewed":
            E[:, :3] = E[:, :3] @ np.array([[1.0, 0.8, 0.0], [0.0, 1.0, -0.6], [0.4, 0.0, 1.0]])
        mats.append(E.astype(np.float32))
    cams = scenes.cams_from(intr, size, mats)
    # camera points whose projection lies around the border, back to the world
    means = np.zeros((n, 3))
    for i, (k, side) in enumerate(zip(rng.integers(0, 3, n), rng.integers(0, 4, n))):
        fx, fy, cx, cy = intr[k]
        w, h = size[k]
        z = np.exp(rng.uniform(np.log(0.15), np.log(30.0)))
        u, v = rng.uniform(-0.5 * w, 1.5 * w), rng.uniform(-0.5 * h, 1.5 * h)
        off = np.exp(rng.uniform(np.log(0.01), np.log(3000.0)))
        if side == 0: u = -off
        if side == 1: u = w + off
        if side == 2: v = -off
        if side == 3: v = h + off
        pc = np.array([(u - cx) / fx * z, (v - cy) / fy * z, z])
        E = mats[k].astype(np.float64)
        means[i] = np.linalg.solve(E[:, :3], pc - E[:, 3])
    scene = scenes.cube_scene(n, seed=5, sh_degree=0)
    scene["means"] = means.astype(np.float32)
    scene["log_scales"] = rng.uniform(-7.0, 3.0, (n, 3)).astype(np.float32)
    geom = oracle.project_geom(scene, cams, blur=blur)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    params = {k: dev(scene[k]) for k in ("means", "log_scales", "quats", "opacity_logit", "sh")}
    params["sh_degree"] = 0
    rast = gs.Rasterizer(n, 0, intr, size, pair_capacity=1 << 16, blur=blur)
    gs.gs_project(params, rast.views, dev(cams["viewmats"].reshape(-1, 12)), rast.proj, rast.near_z, blur)
    radii = rast.proj["radii"].cpu().numpy()
    drawn = float((radii > 0).mean())
    assert 0.05 < drawn < 0.95
    np.testing.assert_array_equal(radii, geom["radius"])
    np.testing.assert_array_equal(rast.proj["tiles_touched"].cpu().numpy().view(np.uint32), geom["kept"])
