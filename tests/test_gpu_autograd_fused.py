"""EdgeLoss's single pass (forward_grad, backward_from) against the forward-only and adjoint-only
kernels on the same inputs: the sums are the same, so gradients agree to FP64 rounding (1e-12 of the
largest leaves four digits for cancellation).  Twists on both sides of the series' limit of 0.05 rad."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import oracle  # noqa: E402
import paper_2607_00579_gb300 as epo  # noqa: E402
from tests.test_gpu_default_schedule import scene  # noqa: E402

B = epo._binding


def two_pass(s, x, w):
    loss, grad = torch.empty(s.n_scenes, dtype=torch.float64, device="cuda"), torch.empty_like(x)
    B.epo_forward_dev(s.handle, x, loss)
    B.epo_backward_dev(s.handle, x, w, grad)
    return loss, grad


@pytest.mark.parametrize("n_views,size", [(1, 0.01), (11, 0.0), (33, 0.02), (33, 0.2), (70, 0.04)])
@pytest.mark.parametrize("opt", [dict(), dict(refine=1), dict(pair_budget=9, subsample_seed=5), dict(norm_mode=1)])
def test_equals_two_passes(n_views, size, opt):
    s = scene(60, 44, n_views, 700, min(4, n_views), False, **opt)
    r = np.random.default_rng(n_views)
    xs = [torch.from_numpy(r.normal(0, size, (n_views, 6))).cuda().requires_grad_(True) for _ in range(2)]
    w = torch.tensor([1.7], dtype=torch.float64, device="cuda")
    if "refine" in opt:  # recomputes: the backward follows its forward
        outs = []
        for x in xs:
            L = epo.EdgeLoss.apply(x, s)
            outs.append((L, torch.autograd.grad((L * w).sum(), x)[0]))
    else:  # both forwards first, and an evaluation without a gradient between
        Ls = [epo.EdgeLoss.apply(x, s) for x in xs]
        with torch.no_grad():
            epo.EdgeLoss.apply(xs[1] + 0.1, s)
        outs = [(L, torch.autograd.grad((L * w).sum(), x)[0]) for L, x in zip(Ls, xs)]
    for x, (L, g) in zip(xs, outs):
        loss, grad = two_pass(s, x.detach(), w)
        assert torch.allclose(L, loss, rtol=1e-13, atol=0)
        scale = float(grad.abs().max())
        if n_views == 1:  # a view paired with itself: the two roles cancel exactly, the scale is their terms'
            st = s.pair_stats()[0]
            scale = 2.0 * w.item() * np.abs(st[2:]).max() / st[1]
        assert (g - grad).abs().max() <= 1e-12 * scale


def test_left_jacobian_and_twists_match_the_oracle():
    """backward_from alone on given gradients, and the poses through the loss's invariance: identity at 0."""
    s = scene(60, 44, 40, 50, 2, False)
    r = np.random.default_rng(2)
    x = r.normal(0, 1, (40, 6)) * np.geomspace(1e-9, 1.0, 40)[:, None]
    g = r.normal(0, 1, (40, 6))
    out = torch.empty((40, 6), dtype=torch.float64, device="cuda")
    B.epo_backward_from_dev(s.handle, torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda(),
                            torch.tensor([2.0], dtype=torch.float64, device="cuda"), out)
    want = np.stack([2.0 * oracle.se3_left_jacobian(x[v]).T @ g[v] for v in range(40)])
    # the closed form of the oracle loses digits to cancellation at small angles
    assert np.abs(out.cpu().numpy() - want).max() < 1e-9


def test_another_stream_keeps_no_buffer():
    """The kept gradient is torch's memory, so a pass on another stream than the scene's keeps none."""
    s = scene(60, 44, 20, 300, 4, False)
    x = torch.full((20, 6), 0.01, dtype=torch.float64, device="cuda", requires_grad=True)
    side = torch.cuda.Stream()
    out = []
    for st in (torch.cuda.current_stream(), side):
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            L = epo.EdgeLoss.apply(x, s)
            torch.cuda.synchronize()
            kept = len(L.grad_fn.saved_tensors)
            g = torch.autograd.grad(L.sum(), x)[0]
            torch.cuda.synchronize()
        out.append((kept, L.detach(), g))
    assert [k for k, _, _ in out] == [2, 1]
    assert torch.allclose(out[0][1], out[1][1], rtol=1e-13, atol=0)
    assert (out[0][2] - out[1][2]).abs().max() <= 1e-12 * out[0][2].abs().max()
