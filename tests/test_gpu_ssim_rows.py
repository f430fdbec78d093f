"""gs_loss_ssim with padded map rows (a workspace of gs_ssim_workspace_size)
against the pass without them (a workspace of 9 floats a pixel): the same sums
in the same order, so the gradients agree to a rounding of each operation
(1e-6 in the 2-norm); widths of every remainder modulo 4, at and around the
tile width, and views whose first pixel is not on 16 bytes."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(33, 40)], [(34, 59)], [(35, 47), (65, 49)], [(36, 33), (61, 97), (64, 48)],
                                   [(641, 35), (30, 130), (127, 48)], [(25, 25)], [(7, 90)]])
def test_padded_rows_equal_unpadded(sizes):
    from paper_2405_19614_gb300.build import build
    build()
    rng = np.random.default_rng(len(sizes))
    P = sum(w * h for w, h in sizes)
    x = rng.uniform(0, 1, (P, 3)).astype(np.float32)
    y = np.clip(x + rng.normal(0, 0.15, x.shape), 0, 1).astype(np.float32)
    views = gs.make_views([[50, 50, 20, 20]] * len(sizes), sizes)
    xt, yt = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    out = []
    for size in (gs.gs_ssim_workspace_size(P), 36 * P):
        # whatever the workspace held must not reach the sums
        ws = torch.full((size,), 255, dtype=torch.uint8, device="cuda")
        loss, d_rgb = torch.zeros(1, device="cuda"), torch.zeros(P, 3, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        gs.gs_loss_ssim(xt, yt, views, 0.3, loss, d_rgb, ws, status)
        assert gs.gs_get_device_status(status) == 0
        out.append((float(loss), d_rgb.cpu().numpy().astype(np.float64)))
    assert abs(out[0][0] - out[1][0]) <= 1e-6
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 1e-6 * np.linalg.norm(out[1][1])
