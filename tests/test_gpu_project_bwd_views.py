"""The projection backward over many views, where blocks leave early when no view
draws any of their Gaussians and warps walk only the views one of their lanes is
drawn in, against one call per view added up: 1 to 64 views around the sizes at
which the groups of views and the halves of the view mask change, every SH degree, a ragged last block, Gaussians drawn in no view,
gradients added and overwritten, pose only.

Both sides sum a Gaussian's terms over the views in the same order and differ by
one rounding of an addition per view, 64 x 2^-24 = 4e-6 of the terms' sizes, and
sums of opposite terms are some ten times smaller than those (1e-4 in the 2-norm,
where a missed view is 1e-2 and more); the twist's block sums arrive in any order, 1,000 terms a
view: 1e-4 of the largest twist."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs
import scenes

pytestmark = pytest.mark.gpu
KEYS = ("means", "log_scales", "quats", "opacity_logit", "sh")


@pytest.mark.parametrize("views,degree", [(1, 3), (7, 2), (8, 3), (9, 3), (16, 1), (17, 0), (33, 2), (64, 3)])
def test_views_together_equal_views_apart(views, degree):
    from paper_2405_19614_gb300.build import build
    build()
    rng = np.random.default_rng(views)
    n = 128 * 7 + 45
    scene = scenes.cube_scene(n, seed=views, sh_degree=degree)
    scene["means"][256:512, 0] += 1000.0  # two blocks that no view draws
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    params = {k: dev(scene[k]) for k in KEYS}
    params["sh_degree"] = degree
    intr, size = [[60.0, 60.0, 32.0, 24.0]] * views, [[64, 48]] * views
    at = [(rng.uniform(-1, 1), rng.uniform(-1, 1), rng.uniform(0.5, 6)) for _ in range(views)]
    mats = [scenes.look_at((0.3 * rng.uniform(-1, 1), 0.2, 0.1), a).astype(np.float32) for a in at]
    vm = dev(np.stack(mats).reshape(-1, 12))
    rast = gs.Rasterizer(n, degree, intr, size, pair_capacity=1 << 16)
    gs.gs_project(params, rast.views, vm, rast.proj)
    drawn = rast.proj["radii"].view(views, n) > 0
    assert 0 < int(drawn.sum()) and not bool(drawn[:, 256:512].any())
    g2 = dev(rng.normal(0, 1, (views, n, 12))) * drawn[:, :, None]
    zeros = lambda: {k: torch.zeros_like(params[k]) for k in KEYS}  # noqa: E731

    want, tw_want = zeros(), torch.zeros(views, 6, device="cuda")
    for v in range(views):
        one = gs.Rasterizer(n, degree, intr[v:v + 1], size[v:v + 1], pair_capacity=1 << 16)
        gs.gs_project(params, one.views, vm[v:v + 1].contiguous(), one.proj)
        assert torch.equal(one.proj["radii"], rast.proj["radii"].view(views, n)[v])
        gs.gs_project_bwd(params, one.views, vm[v:v + 1].contiguous(), one.proj, g2[v].clone(), want, tw_want[v:v + 1])
    for overwrite in (False, True):
        got, tw, g = zeros(), torch.zeros(views, 6, device="cuda"), g2.clone()
        if overwrite:
            got = {k: torch.full_like(t, 7.0) for k, t in got.items()}
        gs.gs_project_bwd(params, rast.views, vm, rast.proj, g, got, tw, overwrite_grads=overwrite)
        assert not bool(g.any())  # consumed
        for k in KEYS:
            assert float((got[k] - want[k]).norm()) <= 1e-4 * float(want[k].norm()), k
            assert not bool(got[k][256:512].any()), k
        assert float((tw - tw_want).abs().max()) <= 1e-4 * float(tw_want.abs().max())
    tw = torch.zeros(views, 6, device="cuda")
    gs.gs_project_bwd(params, rast.views, vm, rast.proj, g2.clone(), None, tw)
    assert float((tw - tw_want).abs().max()) <= 1e-4 * float(tw_want.abs().max())
