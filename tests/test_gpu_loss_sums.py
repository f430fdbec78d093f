"""The loss values' sums: gs_loss_l1 against numpy in 64 bits at the edges of
its launch shapes (one pixel, a block, a cluster of blocks, a whole GPU of
threads, several pixels a thread), and gs_loss_ssim's value equal in every run
and when added to a loss that is there already."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu


def _build():
    from paper_2405_19614_gb300.build import build
    build()


@pytest.mark.parametrize("gate", [False, True])
@pytest.mark.parametrize("P", [1, 255, 257, 2049, 2048 * 152 - 1, 2048 * 152 + 1, 777_777])
def test_l1_sum(P, gate):
    _build()
    rng = np.random.default_rng(P)
    f = lambda *s: rng.uniform(0.1, 1.0, s).astype(np.float32)  # noqa: E731
    rgb, t_rgb, z, t_z, alpha = f(P, 3), f(P, 3), f(P), f(P), f(P)
    c = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    d_rgb, d_z, loss = torch.empty(P, 3, device="cuda"), torch.empty(P, device="cuda"), torch.zeros(1, device="cuda")
    gs.gs_loss_l1(c(rgb), c(z), c(alpha), c(t_rgb), c(t_z), 0.5, 0.7, gate, 0.4, loss, d_rgb, d_z)
    D = np.float64
    l = 0.5 / (3 * P) * np.abs(rgb.astype(D) - t_rgb).sum(1) + 0.7 / P * np.abs(z.astype(D) - t_z)
    ref = float((l * (alpha > np.float32(0.4)) if gate else l).sum())
    # terms are positive, so the error is at most the roundings a term passes
    # through, 2^-24 each: 9 of its own, the thread's pixels (at most 1 + P / 77,824
    # on any GPU of 38 multiprocessors or more), two trees of 5, 8 blocks and at most
    # 152 additions to the running loss
    assert abs(float(loss) - ref) <= (9 + 1 + P / 77824 + 10 + 8 + 152) * 2.0 ** -24 * ref
    sign = np.sign(rgb - t_rgb) * ((alpha > np.float32(0.4))[:, None] if gate else 1.0)
    np.testing.assert_array_equal(np.sign(d_rgb.cpu().numpy()), sign)


@pytest.mark.parametrize("sizes", [[(64, 48)], [(641, 479)] * 4, [(320, 240), (33, 97)]])
def test_ssim_sum_is_one_addition(sizes):
    _build()
    rng = np.random.default_rng(7)
    P = sum(w * h for w, h in sizes)
    x = torch.from_numpy(rng.uniform(0, 1, (P, 3)).astype(np.float32)).cuda()
    y = (x + 0.1).clamp(0, 1)
    views = gs.make_views([[50, 50, 20, 20]] * len(sizes), sizes)
    ws = torch.full((gs.gs_ssim_workspace_size(P),), 255, dtype=torch.uint8, device="cuda")
    losses = []
    for start in (0.0, 0.0, 0.0, 0.25):
        loss, d_rgb = torch.full((1,), start, device="cuda"), torch.zeros(P, 3, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        gs.gs_loss_ssim(x, y, views, 0.3, loss, d_rgb, ws, status)
        assert gs.gs_get_device_status(status) == 0
        losses.append(np.float32(loss.item()))
    assert losses[0] == losses[1] == losses[2]
    assert losses[3] == np.float32(0.25) + losses[0]
