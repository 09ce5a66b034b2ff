"""The pose MLP's phi (Gram-Schmidt, FP64) with zero weights, on matrices far from rotations: its distance
from an extended-precision evaluation against that of numpy's correctly rounded FP64 operations.  Both
round as often; the order of a dot product and its fused operations leave 20 % between them (a
root and a division from refined approximations: 1.5 times)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

from paper_2607_00579_gb300 import _binding as B  # noqa: E402
from tests.test_gpu_selection import ring_pairs, tiny_scene  # noqa: E402


def phi(P):
    a1, a2 = P[:, :, 0], P[:, :, 1]
    b1 = a1 / np.sqrt((a1 * a1).sum(1))[:, None]
    u2 = a2 - (b1 * a2).sum(1)[:, None] * b1
    return np.stack([b1, u2 / np.sqrt((u2 * u2).sum(1))[:, None]], axis=2)


def test_columns_round_as_fp64_operations_do():
    n = 160
    s = tiny_scene(n, ring_pairs(n, 2), seed=5, pose_param=B.EPO_POSE_MLP)
    dev, host = [], []
    for seed in range(20):
        P = np.random.default_rng(seed).normal(0, 1, (n, 12))
        s.set_poses(P)
        want = phi(P.reshape(n, 3, 4).astype(np.longdouble))
        dev.append((s.get_poses().reshape(n, 3, 4)[:, :, :2] - want).astype(np.float64))
        host.append((phi(P.reshape(n, 3, 4)) - want).astype(np.float64))
    rms = lambda e: np.sqrt(np.mean(np.square(e), axis=(0, 1, 2)))
    assert np.all(rms(dev) <= 1.2 * rms(host)), (rms(dev), rms(host))
