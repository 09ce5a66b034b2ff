"""The pose MLP's gradient over scenes around the 32 views that the update kernel stages at a time:
after one step from zero moments the first moment is 0.1 of the gradient, so every layer's gradient
(the sum over the views of dL/dz and the layer's input) is compared with the FP64 chain rule at the
device's own pose gradient.  FP32 forms it from two 128-term chains per layer and one term per view:
a few hundred roundings of terms no larger than the layer's largest entry, 1e-4 of it."""
import numpy as np
import pytest

import oracle.pose_mlp as pm
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

from paper_2607_00579_gb300 import _binding as B  # noqa: E402
from tests.test_gpu_selection import ring_pairs, tiny_scene  # noqa: E402


@pytest.mark.parametrize("n_views", [2, 31, 32, 33, 65, 160])
def test_gradient_of_every_layer(n_views):
    s = tiny_scene(n_views, ring_pairs(n_views, 2), seed=5, pose_param=B.EPO_POSE_MLP)
    theta = synth.pose_mlp_init(11)
    theta[-(12 * 128 + 12):] = np.random.default_rng(1).normal(0, 1e-3, 12 * 128 + 12).astype(np.float32)
    P0 = s.get_poses().reshape(-1, 12)
    s.set_poses(P0)
    B.epo_set_pose_mlp(s.handle, theta)
    T0, cache = pm.poses(theta.astype(np.float64), np.zeros((n_views, 3)), P0)
    assert np.abs(s.get_poses().reshape(-1, 12) - T0).max() < 1e-5
    _, G = s.loss_and_grad()
    gt, gd = pm.pose_backward(theta.astype(np.float64), cache, T0, G)
    s.step(1)
    m, v, dm, _ = B.epo_get_pose_mlp_moments(s.handle, 1, n_views)
    offs = np.cumsum([0] + [o * i + o for o, i in pm.DIMS])
    for l in range(6):
        g = gt[offs[l]:offs[l + 1]]
        assert np.abs(m[0][offs[l]:offs[l + 1]] / 0.1 - g).max() <= 1e-4 * np.abs(g).max(), l
    assert np.abs(dm / 0.1 - gd).max() <= 1e-4 * np.abs(gd).max()
