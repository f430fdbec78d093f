"""gs_pose_update against scipy's matrix exponential around the line between the
series and the closed form (0.1 rad), for several views in one call.  The update
is computed in FP64 and rounded once to FP32: half an ulp of entries below 8."""
import numpy as np
import pytest
import torch
from scipy.linalg import expm

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("angle", [0.0, 1e-7, 1e-3, 0.0999999, 0.1000001, 1.7, 3.1])
def test_exponential_of_the_twist(angle):
    from paper_2405_19614_gb300.build import build
    build()
    rng = np.random.default_rng(3)
    V = 5
    axis = rng.standard_normal((V, 3))
    axis /= np.linalg.norm(axis, axis=1, keepdims=True)
    xi = np.concatenate([rng.uniform(-1, 1, (V, 3)), angle * axis], 1).astype(np.float32)
    E = rng.uniform(-1, 1, (V, 12)).astype(np.float32)
    vm, tw = torch.from_numpy(E).cuda(), torch.from_numpy(xi).cuda()
    gs.gs_pose_update(vm, tw)
    got = vm.cpu().numpy().reshape(V, 3, 4).astype(np.float64)
    assert float(tw.abs().max()) == 0.0
    for v in range(V):
        r, p = xi[v, :3].astype(np.float64), xi[v, 3:].astype(np.float64)
        A = np.zeros((4, 4))
        A[:3, :3] = [[0, -p[2], p[1]], [p[2], 0, -p[0]], [-p[1], p[0], 0]]
        A[:3, 3] = r
        X = expm(A)
        M = E[v].reshape(3, 4).astype(np.float64)
        want = X[:3, :3] @ M
        want[:, 3] += X[:3, 3]
        assert np.abs(got[v] - want).max() <= 2.0 ** -22
