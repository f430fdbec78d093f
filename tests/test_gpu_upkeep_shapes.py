"""Map upkeep where its kernels change course: the spatial order of more means
than one round of blocks, compaction of rows that are not on 16 bytes or wider
than a block's share, densification at every SH degree with the capacity ending
inside a chunk of pixels, and rows that are not written left as they were."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs
import scenes
from gpu_util import t
from oracle import map_update as MU
from test_gpu_map_update import _morton_ranks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_19614_gb300.build import build
    build()


@pytest.mark.parametrize("n", [155_649, 400_003])  # 608 blocks of 256 and one mean; blocks of two or three rounds
def test_spatial_order_of_many_means(n):
    means = scenes.cube_scene(n, seed=n, sh_degree=0)["means"]
    new_index = torch.empty(n, dtype=torch.int32, device="cuda")
    ws = torch.empty(gs.gs_spatial_order_workspace_size(n), dtype=torch.uint8, device="cuda")
    gs.gs_spatial_order(t(means), new_index, ws)
    np.testing.assert_array_equal(new_index.cpu().numpy(), _morton_ranks(means))


def _rows(n, w, off):
    """[n, w] floats that start `off` floats behind a 16-byte boundary."""
    return torch.full((n * w + off,), -7.0, device="cuda")[off:].view(n, w)


@pytest.mark.parametrize("n,widths", [(5003, [4, 48, 3, 5, 12, 1]), (301, [2048, 2049, 2052, 8192, 8196, 8201])])
@pytest.mark.parametrize("src_off,dst_off", [(0, 0), (1, 0), (0, 1), (2, 3)])
def test_compaction_of_any_rows(n, widths, src_off, dst_off):
    rng = np.random.default_rng(n + src_off)
    keep = rng.random(n) < 0.6
    index = np.where(keep, np.cumsum(keep) - 1, -1).astype(np.int32)
    src, dst = [], []
    for w in widths:
        s = _rows(n, w, src_off)
        s.copy_(torch.from_numpy(rng.standard_normal((n, w)).astype(np.float32)))
        src.append(s)
        dst.append(_rows(n, w, dst_off))
    gs.gs_compact_rows(t(index, torch.int32), list(zip(src, dst)))
    m = int(keep.sum())
    for s, d in zip(src, dst):
        np.testing.assert_array_equal(d[:m].cpu().numpy(), s.cpu().numpy()[keep])
        assert bool((d[m:] == -7.0).all())


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("room", [1, 501, 3002, 10 ** 6])
def test_densification_at_every_degree(degree, room):
    rng = np.random.default_rng(degree)
    vms = np.stack([scenes.look_at((0.2 * k, -0.1, 0.0), (0.0, 0.2, 3.0)) for k in range(2)])
    cams = scenes.cams_from([[60, 60, 32, 24], [80, 75, 40.5, 30]], [[64, 48], [81, 61]], vms)
    P = 64 * 48 + 81 * 61
    alpha = rng.uniform(0, 1, P).astype(np.float32)
    depth = rng.uniform(0.5, 5.0, P).astype(np.float32)
    depth[rng.uniform(0, 1, P) < 0.1] = 0.0
    rgb = rng.uniform(0, 1, (P, 3)).astype(np.float32)
    idx, ref = MU.densify(alpha, rgb, depth, cams, 0.5, -1.0, degree)
    n_old, m = 37, min(room, len(idx))
    rows = n_old + m + 100  # a hundred rows beyond the capacity
    full = lambda *s: torch.full((rows, *s), 7.0, device="cuda")
    params = dict(means=full(3), log_scales=full(3), quats=full(4), opacity_logit=full(), sh=full((degree + 1) ** 2, 3),
                  sh_degree=degree)
    n_added = torch.zeros(1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(gs.gs_select_workspace_size(P), dtype=torch.uint8, device="cuda")
    gs.gs_densify(t(alpha), t(rgb), t(depth), gs.make_views(cams["intr"], cams["size"]),
                  t(cams["viewmats"].reshape(-1, 12)), 0.5, -1.0, params, n_old, n_old + m, n_added, ws, status)
    assert int(n_added) == m and (int(status) != 0) == (m < len(idx))
    for k in ("means", "log_scales", "quats", "opacity_logit", "sh"):
        got = params[k].cpu().numpy()
        np.testing.assert_allclose(got[n_old:n_old + m], ref[k][:m], rtol=2e-6, atol=2e-6, err_msg=k)
        assert (got[:n_old] == 7.0).all() and (got[n_old + m:] == 7.0).all(), k
