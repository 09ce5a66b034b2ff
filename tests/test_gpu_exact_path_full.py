"""Work items with more samples on decision thresholds than a block's exact-path buffer holds: views of
one orientation, shifted by whole pixels, whose every operation is exact, so that each sample lies on a
pixel and takes its decisions in FP64 (cells, and the border for those on it).  The valid counts are the
oracle's integers whatever the schedule, and the results agree between schedules to the order of FP64
atomics (1e-12 leaves four digits for cancellation); values within the parity tests' tolerances."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import check_against_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import paper_2607_00579_gb300 as epo  # noqa: E402

B = epo._binding
W, H = 64, 48


def lattice(n_views, n_rec, k, lam, mixed=False, **opt):
    r = np.random.default_rng([n_views, n_rec, k])
    rec = np.zeros((n_rec * n_views, 4), np.float32)
    rec[:, 0], rec[:, 1] = r.integers(0, W, len(rec)), r.integers(0, H, len(rec))
    rec[:, 2] = r.choice([2.0, 4.0], len(rec))
    maps = [(r.uniform(0, 12, (H, W)).astype(np.float32).view(np.uint32) & 0xffff0000).view(np.float32) for _ in range(n_views)]
    pairs = np.array([(i, (i + j) % n_views) for i in range(n_views) for j in range(k)], np.int32)
    K = np.tile([64.0, 64.0, 31.5, 23.5], (n_views, 1))
    off = n_rec * np.arange(n_views + 1)
    T = np.tile(np.eye(3, 4).reshape(-1), (n_views, 1))
    T[:, 3] = np.arange(n_views) % 3 / 8.0  # 2 or 4 pixels each
    o = oracle.OracleScene([W] * n_views, [H] * n_views, K, off, rec, [m.astype(np.float64) for m in maps], pairs)
    kw, srec, smaps = {}, rec, maps
    if mixed:
        srec = np.zeros((len(rec), 4), np.uint16)
        srec[:, :2], srec[:, 2] = rec[:, :2], rec[:, 2].astype(np.float16).view(np.uint16)
        smaps = [(m.view(np.uint32) >> 16).astype(np.uint16) for m in maps]
        kw = dict(record_dtype=epo.EPO_F16, map_dtype=epo.EPO_BF16)
    s = epo.Scene.single([W] * n_views, [H] * n_views, K, off, srec, smaps, pairs,
                         options=epo.default_options(lambda0=lam, lambda1=lam, **opt), **kw)
    s.set_poses(T)
    return s, o, T, pairs


SCHEDULES = [dict(), dict(gather=epo.EPO_GATHER_TEX, block_threads=128, records_per_thread=4),
             dict(gather=epo.EPO_GATHER_TEX, block_threads=128, records_per_thread=4, tail_pairs=0),
             dict(gather=epo.EPO_GATHER_LDG, block_threads=256, records_per_thread=2, tail_pairs=0),
             dict(gather=epo.EPO_GATHER_TEX, block_threads=64, records_per_thread=8, grid_blocks=3),
             dict(gather=epo.EPO_GATHER_LDG, block_threads=512, records_per_thread=1, tail_pairs=-2),
             dict(gather=epo.EPO_GATHER_MIX, block_threads=96, records_per_thread=4, tail_pairs=3)]


@pytest.mark.parametrize("n_views,n_rec,k", [(1, 700, 1), (3, 3000, 3), (20, 1100, 7), (130, 2600, 9)])
@pytest.mark.parametrize("mixed", [False, True])
def test_pose_scenes(n_views, n_rec, k, mixed):
    ref = None
    for sched in SCHEDULES:
        s, o, T, pairs = lattice(n_views, n_rec, k, 10.0, mixed, **sched)
        loss, grad = s.loss_and_grad()
        st = s.pair_stats()
        queued, overflow = B.epo_fixup_stats(s.handle)
        xi = torch.zeros((n_views, 6), dtype=torch.float64, device="cuda")
        fl, fg = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(xi)
        B.epo_forward_dev(s.handle, xi, fl)
        B.epo_backward_dev(s.handle, xi, torch.ones_like(fl), fg)
        if ref is None:
            want = o.loss_grad(T, lam=10.0)
            check_against_oracle(loss[0], grad, want, pairs, T, stats=st)
            ref = loss, grad, st
        assert np.array_equal(st[:, 1], want["pair_stats"][:, 1])
        assert overflow == 0 and queued >= st[:, 1].sum()
        scale = max(np.abs(ref[1]).max(), 1e-3 * want["pair_abs"].max() / n_rec)
        for l, g in ((loss[0], grad), (fl.item(), fg.cpu().numpy())):
            assert abs(l - ref[0][0]) <= 1e-12 * ref[0][0]
            assert np.abs(g - ref[1]).max() <= 1e-12 * scale


@pytest.mark.parametrize("n_views,n_rec,k", [(1, 700, 1), (3, 3000, 3), (20, 1100, 7)])
def test_refinement_scenes(n_views, n_rec, k):
    ref = None
    for sched in (dict(), dict(gather=epo.EPO_GATHER_TEX, tail_pairs=0), dict(gather=epo.EPO_GATHER_LDG, block_threads=64),
                  dict(gather=epo.EPO_GATHER_TEX, block_threads=512, tail_pairs=-2, grid_blocks=5)):
        s, o, T, pairs = lattice(n_views, n_rec, k, 10.0, refine=1, **sched)
        out = B.epo_refine_loss_and_grad(s.handle, 1, n_views, n_rec * n_views)
        st = s.pair_stats()
        if ref is None:
            one, zero = np.ones(len(o.rec), np.float32), np.zeros(len(o.rec), np.float32)
            want = o.loss_grad(T, lam=10.0)
            full = o.loss_grad_full(T, np.zeros(n_views), one, zero, 10.0)
            ref = out
            check_against_oracle(out[0][0], out[1], want, pairs, T, stats=st)
            term = 2.0 * want["pair_maxterm"].max() / n_rec / len(pairs)  # one sample's share
            for got, w in zip(out[2:], (full["grad_gamma"], full["grad_alpha"], full["grad_beta"])):
                assert np.abs(got - w).max() <= 1e-4 * max(np.abs(w).max(), term)
        assert np.array_equal(st[:, 1], want["pair_stats"][:, 1])
        assert B.epo_fixup_stats(s.handle)[1] == 0
        for x, y in zip(out, ref):
            assert np.abs(x - y).max() <= 1e-12 * max(np.abs(y).max(), term * n_rec) + 1e-7 * term * (x.dtype == np.float32)
