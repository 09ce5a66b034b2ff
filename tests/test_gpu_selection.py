"""The block-wide selections of a step at the sizes where they change path or digit: the
sub-sampling's cut (one block per scene, 1,024 threads) against the oracle's subsets bit for bit,
and the schedule's 95th percentiles (rank counting up to 256 views, radix select above) against
the oracle's on the same poses.  The percentile's tolerance is the schedule test's: the angles come
from an arccosine near 1, whose argument carries ~1e-16, at angles of ~1e-3 rad or more."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import paper_2607_00579_gb300 as epo  # noqa: E402

B = epo._binding


def tiny_scene(n_views, pairs, seed=1, **opt):
    """Views of 16x12 pixels with a dozen records, cameras near the origin looking along z."""
    r = np.random.default_rng(seed)
    rec = np.zeros((12 * n_views, 4), np.float32)
    rec[:, 0], rec[:, 1] = r.integers(2, 14, len(rec)), r.integers(2, 10, len(rec))
    rec[:, 2] = r.uniform(2, 5, len(rec))
    y, x = np.mgrid[:12, :16]
    maps = [(np.abs(x - r.uniform(4, 12)) + 0.5 * np.abs(y - 6.0)).astype(np.float32) for _ in range(n_views)]
    T = np.tile(np.eye(3, 4).reshape(-1), (n_views, 1))
    T[:, [3, 7, 11]] = r.normal(0, 0.05, (n_views, 3))
    s = epo.Scene.single(np.full(n_views, 16), np.full(n_views, 12), np.tile([16.0, 16.0, 7.5, 5.5], (n_views, 1)),
                         12 * np.arange(n_views + 1), rec, maps, np.asarray(pairs, np.int32),
                         options=epo.default_options(**opt))
    s.set_poses(T)
    return s


def ring_pairs(n_views, k):
    return [(i, (i + 1 + j) % n_views) for i in range(n_views) for j in range(k)]


@pytest.mark.parametrize("n_pairs,budget", [(1, 1), (2, 1), (33, 32), (1023, 512), (1024, 1), (1025, 1024),
                                            (4100, 4099), (4100, 7)])
def test_subset_sizes(n_pairs, budget):
    n_views = 65
    pairs = [(p % n_views, (p * 7 + 1) % n_views) for p in range(n_pairs)]
    s = tiny_scene(n_views, pairs, pair_budget=budget, subsample_seed=77)
    for step in range(2):
        s.step(1)
        got = B.epo_get_pair_active(s.handle, n_pairs)
        assert np.array_equal(got, oracle.subsample(77, step, n_pairs, budget))


@pytest.mark.parametrize("n_views", [1, 2, 20, 21, 127, 255, 256, 257, 600])
def test_percentile_sizes(n_views):
    s = tiny_scene(n_views, ring_pairs(n_views, 2), schedule=1, lr_rot=2e-3, lr_trans=1e-2)
    for _ in range(3):
        T0 = s.get_poses()
        s.step(1)
        th = B.epo_get_schedule(s.handle, 1)[0][0]
        assert th == pytest.approx(oracle.theta95(T0, s.get_poses()), rel=1e-9, abs=1e-9)


def test_percentile_of_equal_changes():
    """Frozen views change by the same amount (zero): order statistics inside a run of equal values."""
    for n_views in (40, 300):
        s = epo.Scene.single(np.full(n_views, 16), np.full(n_views, 12), np.tile([16.0, 16.0, 7.5, 5.5], (n_views, 1)),
                             np.zeros(n_views + 1, np.int64), np.zeros((0, 4), np.float32),
                             [np.ones((12, 16), np.float32)] * n_views, np.asarray(ring_pairs(n_views, 1), np.int32),
                             fixed=np.ones(n_views, np.uint8), options=epo.default_options(schedule=1))
        T = np.tile(np.eye(3, 4).reshape(-1), (n_views, 1))
        T[:, 11] = 1.0
        s.set_poses(T)
        s.step(1)
        assert B.epo_get_schedule(s.handle, 1)[0][0] == oracle.theta95(T, s.get_poses())
