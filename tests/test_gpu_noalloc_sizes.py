"""The allocation-free call where its kernels change shape: records around the 256-record tiles,
more than 32 (pair, role) entries per view, views without pairs, and samples whose decisions lie on
their thresholds (identical poses and exact intrinsics put every sample exactly on a pixel, where the FP64 form decides).
Against the oracle within the parity tests' tolerances."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

from paper_2607_00579_gb300 import _binding as B  # noqa: E402
from tests.test_gpu_parity import check_against_oracle  # noqa: E402
from tests.test_zz_no_alloc import Problem  # noqa: E402


def scene(n, counts, pairs, W=70, H=50, spread=0.1, seed=3):
    r = np.random.default_rng([seed, n, len(pairs)])
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    rec = np.zeros((off[-1], 4), np.float32)
    rec[:, 0], rec[:, 1] = r.integers(0, W, len(rec)), r.integers(0, H, len(rec))
    rec[:, 2] = r.uniform(2, 5, len(rec))
    T = np.zeros((n, 3, 4))
    for v in range(n):
        T[v, :, :3] = synth._rotvec_to_matrix(r.normal(0, spread / 3, 3))
        T[v, :, 3] = r.normal(0, spread, 3)
    K = np.tile([1.1 * W, 1.05 * W, (W - 1) / 2 + 1.25, (H - 1) / 2 - 0.7], (n, 1))
    if spread == 0.0:  # identical poses, every operation exact: each sample returns to its own pixel
        K[:] = [64.0, 64.0, 34.5, 24.5]
        rec[:, 2] = r.choice([2.0, 4.0], len(rec))
    y, x = np.mgrid[:H, :W]
    maps = [(2.5 + 2 * np.sin(x / 6 + a) + 2 * np.cos(y / 5 + b) + 7 * (x > 50)).clip(0).astype(np.float32)
            for a, b in r.uniform(0, 6, (n, 2))]
    sc = synth.Scene(W=np.full(n, W, np.int32), H=np.full(n, H, np.int32), K=K, T_gt=T.reshape(n, 12),
                     T_init=T.reshape(n, 12), rec_off=off, rec=rec, edges=[], pairs=np.asarray(pairs, np.int32),
                     fixed=np.zeros(n, np.uint8), scale=1.0, depth_gt_at_rec=np.zeros(len(rec)))
    return sc, maps


def star(n):
    return [(0, v) for v in range(n)] + [(v, 0) for v in range(1, n)]


@pytest.mark.parametrize("n,counts,pairs,spread", [
    (2, [255, 257], [(0, 1), (1, 0)], 0.1),
    (3, [1, 0, 256], [(0, 1), (1, 0), (2, 1), (0, 2)], 0.1),
    (4, [513, 2, 300, 40], [(0, 0), (2, 3), (3, 2)], 0.1),
    (40, [60] * 40, star(40), 0.1),
    (6, [700] * 6, [(a, b) for a in range(6) for b in range(6) if a != b], 0.0),
    (70, [33] * 70, [(a, (a * 3 + b) % 70) for a in range(70) for b in range(20)], 0.3)])
@pytest.mark.parametrize("norm_mode", [B.EPO_NORM_VALID, B.EPO_NORM_ALL])
def test_sizes(n, counts, pairs, spread, norm_mode):
    sc, maps = scene(n, counts, pairs, spread=spread)
    got_loss, got_grad = Problem(sc, maps)(sc.T_init, norm_mode)
    o = oracle.scene_from_synth(sc, [m.astype(np.float64) for m in maps]).loss_grad(
        sc.T_init, lam=10.0, norm_mode=oracle.NORM_ALL if norm_mode == B.EPO_NORM_ALL else oracle.NORM_VALID)
    check_against_oracle(got_loss, got_grad, o, sc.pairs, sc.T_init)


def test_records_beyond_the_stated_maximum_are_left_out():
    """The tiles that max_records_per_view makes bound the work: of a view with more records only those
    of its first tiles (256 each) count."""
    sc, maps = scene(3, [600, 300, 256], [(0, 1), (1, 2), (2, 0)])
    run = Problem(sc, maps)
    run.prob.max_records_per_view = 250
    got_loss, got_grad = run(sc.T_init, B.EPO_NORM_VALID)
    keep = np.concatenate([np.arange(sc.rec_off[v], sc.rec_off[v] + 256) for v in range(3)])
    o = oracle.OracleScene(sc.W, sc.H, sc.K, np.arange(4, dtype=np.int64) * 256, sc.rec[keep],
                           [m.astype(np.float64) for m in maps], sc.pairs).loss_grad(sc.T_init, lam=10.0)
    check_against_oracle(got_loss, got_grad, o, sc.pairs, sc.T_init)


def test_views_of_different_sizes():
    """Each target's own width, height, intrinsics and map offset."""
    r = np.random.default_rng(8)
    W, H = np.array([70, 33, 128, 9, 61], np.int32), np.array([50, 90, 17, 12, 47], np.int32)
    n = len(W)
    off = np.concatenate([[0], np.cumsum([300, 513, 40, 256, 700])]).astype(np.int64)
    rec = np.zeros((off[-1], 4), np.float32)
    for v in range(n):
        part = rec[off[v]:off[v + 1]]
        part[:, 0], part[:, 1] = r.integers(0, W[v], len(part)), r.integers(0, H[v], len(part))
    rec[:, 2] = r.uniform(2, 5, len(rec))
    T = np.zeros((n, 3, 4))
    for v in range(n):
        T[v, :, :3] = synth._rotvec_to_matrix(r.normal(0, 0.03, 3))
        T[v, :, 3] = r.normal(0, 0.1, 3)
    K = np.stack([1.1 * W, 1.05 * H, W / 2 + 0.3, H / 2 - 0.7], axis=1)
    maps = [(2.5 + 2 * np.sin(np.arange(w) / 6 + v)[None, :] + 2 * np.cos(np.arange(h) / 5)[:, None]).clip(0).astype(np.float32)
            for v, (w, h) in enumerate(zip(W, H))]
    pairs = np.array([(a, b) for a in range(n) for b in range(n) if a != b], np.int32)
    sc = synth.Scene(W=W, H=H, K=K, T_gt=T.reshape(n, 12), T_init=T.reshape(n, 12), rec_off=off, rec=rec, edges=[],
                     pairs=pairs, fixed=np.zeros(n, np.uint8), scale=1.0, depth_gt_at_rec=np.zeros(len(rec)))
    got_loss, got_grad = Problem(sc, maps)(sc.T_init, B.EPO_NORM_VALID)
    o = oracle.scene_from_synth(sc, [m.astype(np.float64) for m in maps]).loss_grad(sc.T_init, lam=10.0)
    assert o["pair_stats"][:, 1].min() > 0
    check_against_oracle(got_loss, got_grad, o, sc.pairs, sc.T_init)
