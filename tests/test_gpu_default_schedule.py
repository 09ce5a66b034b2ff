"""The default schedule against plain loads in the 256-thread form, unsplit, on the same scene.  The sums of a work item are formed
in one order whatever the gather path and the split of its pairs, so the results agree to the order
of FP64 atomics (1e-12 leaves four digits for cancellation in the gradient)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import paper_2607_00579_gb300 as epo  # noqa: E402

B = epo._binding


def scene(W, H, n_views, n_rec, k, mixed, **opt):
    r = np.random.default_rng([W, H, n_views])
    rec = np.zeros((n_rec * n_views, 4), np.float32)
    rec[:, 0], rec[:, 1] = r.integers(0, W, len(rec)), r.integers(0, H, len(rec))
    rec[:, 2] = np.float16(r.uniform(2, 5, len(rec)))
    maps = [r.uniform(0, 12, (H, W)).astype(np.float32).view(np.uint32) & 0xffff0000 for _ in range(n_views)]
    maps = [m.astype(np.uint32).view(np.float32) for m in maps]
    T = np.tile(np.eye(3, 4).reshape(-1), (n_views, 1))
    T[:, [3, 7, 11]] = r.normal(0, 0.1, (n_views, 3))
    kw = {}
    if mixed:
        packed = np.zeros((len(rec), 4), np.uint16)
        packed[:, :2], packed[:, 2] = rec[:, :2], rec[:, 2].astype(np.float16).view(np.uint16)
        rec, maps = packed, [(m.view(np.uint32) >> 16).astype(np.uint16) for m in maps]
        kw = dict(record_dtype=epo.EPO_F16, map_dtype=epo.EPO_BF16)
    pairs = np.array([(i, (i + 1 + j) % n_views) for i in range(n_views) for j in range(k)], np.int32)
    s = epo.Scene.single(np.full(n_views, W), np.full(n_views, H), np.tile([W, W, (W - 1) / 2, (H - 1) / 2], (n_views, 1)),
                         n_rec * np.arange(n_views + 1), rec, maps, pairs, options=epo.default_options(**opt), **kw)
    s.set_poses(T)
    return s


def evaluate(s, refine):
    if refine:
        i = s.info()
        return B.epo_refine_loss_and_grad(s.handle, i.n_scenes, i.n_views, i.n_records)
    out = (*s.loss_and_grad(), s.pair_stats())
    xi = torch.full((s.n_views, 6), 1e-3, dtype=torch.float64, device="cuda")  # forward-only and adjoint-only
    loss, grad = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(xi)
    B.epo_forward_dev(s.handle, xi, loss)
    B.epo_backward_dev(s.handle, xi, torch.ones_like(loss), grad)
    return (*out, loss.cpu().numpy(), grad.cpu().numpy())


@pytest.mark.parametrize("W,H,n_views,n_rec,k", [(2, 2, 2, 9, 1), (3, 65, 3, 700, 2), (64, 48, 5, 513, 4),
                                                 (161, 123, 12, 1500, 11), (97, 80, 40, 5000, 8),
                                                 (80, 60, 130, 2600, 9)])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("refine", [0, 1])
def test_default_equals_plain_loads(W, H, n_views, n_rec, k, mixed, refine):
    a = scene(W, H, n_views, n_rec, k, mixed, refine=refine)
    if n_views == 130 and not refine:  # enough work for the 128-thread form of the default item
        assert (a.info().block_threads, a.info().records_per_thread) == (128, 4)
    b = scene(W, H, n_views, n_rec, k, mixed, refine=refine, gather=epo.EPO_GATHER_LDG, tail_pairs=0)
    assert (a.info().gather, b.info().gather) == (epo.EPO_GATHER_TEX, epo.EPO_GATHER_LDG)
    for x, y in zip(evaluate(a, refine), evaluate(b, refine)):
        assert np.abs(x - y).max() <= 1e-12 * max(np.abs(y).max(), 1e-300)


@pytest.mark.parametrize("W,H,n_views,n_rec,k", [(64, 48, 5, 513, 4), (97, 80, 40, 5000, 8), (80, 60, 130, 2600, 9),
                                                 (32, 24, 330, 4100, 18)])
@pytest.mark.parametrize("opt", [dict(), dict(pair_budget=37, subsample_seed=3), dict(refine=1)])
def test_split_items_equal_whole_ones(W, H, n_views, n_rec, k, opt):
    """The library's split of the items (also the last wave's alone, the largest scene here) against
    whole items, for the default schedule and for 128 threads with four records each."""
    for sched in (dict(), dict(gather=epo.EPO_GATHER_TEX, block_threads=128, records_per_thread=4)):
        if sched and "refine" in opt:
            continue
        a = scene(W, H, n_views, n_rec, k, False, **opt, **sched)
        whole = sched or dict(gather=epo.EPO_GATHER_TEX, block_threads=256, records_per_thread=2)
        if "refine" in opt:
            whole = dict(gather=epo.EPO_GATHER_TEX)
        b = scene(W, H, n_views, n_rec, k, False, tail_pairs=0, **opt, **whole)
        for x, y in zip(evaluate(a, "refine" in opt), evaluate(b, "refine" in opt)):
            assert np.abs(x - y).max() <= 1e-12 * max(np.abs(y).max(), 1e-300)
