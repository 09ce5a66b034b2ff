"""Viewgraph estimation on the GPU (Section 3, Eq. 2; Algorithm 1 BuildViewgraph) against the
oracle: the round-trip fractions of every ordered pair are ratios of integer counts taken
with the same FP64 arithmetic in the same order, so they are compared exactly, as are the
kept pairs."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import paper_2607_00579_gb300 as epo  # noqa: E402


@pytest.mark.parametrize("preset,stride,which", [("RING8_128x96", 1, "T_gt"), ("RING8_128x96", 3, "T_init"),
                                                 ("RING32_518x392", 6, "T_init")])
def test_viewgraph_matches_oracle(preset, stride, which):
    sc = synth.make_scene(getattr(synth, preset), keep_depth=True)
    T = getattr(sc, which)
    frac, pairs = epo.build_viewgraph(sc.W, sc.H, sc.K, T, [torch.from_numpy(d).cuda() for d in sc.depth],
                                      stride=stride, tau=3.0, min_frac=0.125)
    want = oracle.viewgraph(sc.W, sc.H, sc.K, T, sc.depth, stride=stride, tau=3.0)
    assert np.array_equal(frac, want)
    assert np.array_equal(pairs, oracle.viewgraph_pairs(want, 0.125))
    assert 0 < len(pairs) <= sc.n_views * (sc.n_views - 1)


def test_viewgraph_argument_checks():
    d = torch.zeros(16, device="cuda")
    with pytest.raises(epo.EpoError):
        epo.build_viewgraph([4], [4], [[0.0, 1.0, 1.5, 1.5]], np.eye(4)[:3].reshape(1, 12), d)


@pytest.mark.parametrize("n,W,H,stride,tau,kind", [
    (2, 61, 47, 1, 3.0, "smooth"), (3, 40, 30, 2, 0.75, "identical"), (5, 97, 33, 3, 1.5, "half"),
    (9, 64, 48, 1, 3.0, "holes"), (4, 200, 150, 5, 10.0, "far"), (6, 80, 60, 2, 3.0, "sheared"),
    (40, 24, 20, 1, 2.0, "smooth"), (4, 50, 40, 1, 3.0, "tiny"), (1, 8, 8, 1, 3.0, "smooth")])
def test_viewgraph_counts_are_exact_where_decisions_are_close(n, W, H, stride, tau, kind):
    """Scenes that put decisions of the round trip on their thresholds: identical views (every pixel
    returns to itself, borders exactly on the border), shifts by half a pixel (every nearest-pixel
    choice a tie), missing depths, poses far from the origin, matrices that are no rotations, depths
    near the smallest floats."""
    r = np.random.default_rng([n, W, H])
    K = np.tile([1.1 * W, 1.1 * W, (W - 1) / 2, (H - 1) / 2], (n, 1))
    y, x = np.mgrid[:H, :W]
    depths = [(4 + np.sin(x / 9 + a) + 0.5 * np.cos(y / 7 + b)).astype(np.float32) for a, b in r.uniform(0, 6, (n, 2))]
    T = np.zeros((n, 3, 4))
    for v in range(n):
        w = r.normal(0, 0.03, 3)
        S = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
        T[v, :, :3] = np.linalg.inv(np.eye(3) - S / 2) @ (np.eye(3) + S / 2)
        T[v, :, 3] = r.normal(0, 0.2, 3)
    if kind in ("identical", "half", "tiny"):
        T[:] = np.eye(3, 4)
        depths = [np.full((H, W), 4.0, np.float32)] * n
    if kind == "half":
        T[:, 0, 3] = np.arange(n) * 0.5 * 4.0 / K[0, 0]
    if kind == "tiny":
        depths = [(d * np.float32(10.0) ** r.integers(-44, -36, (H, W)).astype(np.float32)) for d in depths]
    if kind == "holes":
        for d in depths:
            d[r.random((H, W)) < 0.3] = r.choice([0.0, -1.0, np.nan, np.inf])
    if kind == "far":
        T[:, :, 3] -= np.einsum("nij,j->ni", T[:, :, :3], [3e4, -2e4, 1e4])
        K[:, 2:] += r.uniform(-40, 40, (n, 2))
    if kind == "sheared":
        T[:, :, :3] = T[:, :, :3] @ (np.eye(3) + r.normal(0, 0.05, (n, 3, 3)))
    frac, pairs = epo.build_viewgraph(np.full(n, W), np.full(n, H), K, T.reshape(n, 12),
                                      [torch.from_numpy(d).cuda() for d in depths], stride=stride, tau=tau, min_frac=0.125)
    want = oracle.viewgraph(np.full(n, W), np.full(n, H), K, T.reshape(n, 12), depths, stride=stride, tau=tau)
    assert np.array_equal(frac, want)
    assert np.array_equal(pairs, oracle.viewgraph_pairs(want, 0.125))


def small_motion(r, n):
    T = np.zeros((n, 3, 4))
    for v in range(n):
        T[v, :, :3] = synth._rotvec_to_matrix(r.normal(0, 0.03, 3))
        T[v, :, 3] = r.normal(0, 0.2, 3)
    return T.reshape(n, 12)


@pytest.mark.parametrize("stride", [1, 3])
def test_views_of_different_sizes(stride):
    """Grids, borders and row pitches of each pair's own two views; 7 views, so that the pairs' grids
    are split over several blocks by the largest one."""
    r = np.random.default_rng(stride)
    W, H = np.array([61, 200, 17, 96, 33, 128, 5]), np.array([47, 31, 90, 96, 150, 12, 4])
    K = np.stack([1.1 * W, 1.2 * H, W / 2 - 0.3, H / 2 + 0.4], axis=1)
    T = small_motion(r, len(W))
    depths = [r.uniform(3, 5, (h, w)).astype(np.float32) for w, h in zip(W, H)]
    frac, _ = epo.build_viewgraph(W, H, K, T, [torch.from_numpy(d).cuda() for d in depths], stride=stride, tau=3.0)
    assert np.array_equal(frac, oracle.viewgraph(W, H, K, T, depths, stride=stride, tau=3.0))
    assert len(np.unique(frac)) > 20


def test_target_beyond_32_bit_pixel_indices():
    """A small view against one of 65536x40000 pixels, whose lower rows an int does not number.  Same
    pose, constant depth, powers of two throughout: pixel (x, y) of the one is (128 x, 128 y) of the
    other and every trip returns to its own pixel, except where the huge view's depth is cleared."""
    W, H = np.array([512, 65536]), np.array([313, 40000])
    K = np.array([[512, 256, 256, 160], [65536, 32768, 32768, 20480]], dtype=np.float64)
    depth = torch.full((512 * 313 + 65536 * 40000,), 4.0, device="cuda")
    depth[512 * 313:].view(40000, 65536)[36000:38000] = 0.0
    frac, _ = epo.build_viewgraph(W, H, K, np.tile(np.eye(3, 4).reshape(-1), (2, 1)), depth, stride=5, tau=0.75)
    del depth
    torch.cuda.empty_cache()
    cleared = lambda y: (y >= 36000) & (y < 38000)
    y = 128 * np.arange(0, 313, 5)
    assert frac[0, 1] == np.sum(~cleared(y)) / len(y)
    x, y = np.arange(0, 65536, 5), np.arange(0, 40000, 5)
    y = y[~cleared(y)]
    assert frac[1, 0] == int(np.sum(x <= 128 * 511)) * int(np.sum(y <= 128 * 312)) / (len(x) * len(y))


@pytest.mark.parametrize("far", [8e37, 9e37, 2e38, 3.4028234663852886e38])
@pytest.mark.parametrize("where", ["source", "both"])
def test_depths_near_the_largest_float(far, where):
    """Depths at which a reciprocal in FP32 is subnormal or zero (FLT_MAX marks the sky in some depth
    maps): every trip through them is decided in FP64."""
    r = np.random.default_rng(4)
    n, W, H = 4, 63, 47
    K = np.tile([70.0, 70.0, 30.3, 22.8], (n, 1))
    T = small_motion(r, n)
    T[1] = T[0]  # two views of one orientation, shifted
    T[1, 3] += 0.2
    depths = [r.uniform(3, 5, (H, W)).astype(np.float32) for _ in range(n)]
    for v, d in enumerate(depths):
        if where == "both" or v % 2 == 0:
            d[:30] = np.float32(far)
    frac, _ = epo.build_viewgraph(np.full(n, W), np.full(n, H), K, T, [torch.from_numpy(d).cuda() for d in depths],
                                  stride=1, tau=3.0)
    want = oracle.viewgraph(np.full(n, W), np.full(n, H), K, T, depths, stride=1, tau=3.0)
    assert np.array_equal(frac, want)
    assert where == "source" or want[0, 1] > 0.9


@pytest.mark.parametrize("W1,H1", [(49981, 42966), (50000, 50000)])  # 2^31 - 2 pixels, and beyond an int
def test_grids_at_and_beyond_32_bit_numbers(W1, H1):
    """Every pixel of a huge view against a small one: as above, with a few rows of valid depths."""
    W, H = np.array([W1, (W1 - 1) // 128 + 1]), np.array([H1, (H1 - 1) // 128 + 1])
    K = np.array([[65536, 65536, 32768, 32768], [512, 512, 256, 256]], dtype=np.float64)
    depth = torch.zeros(W1 * H1 + int(W[1]) * int(H[1]), device="cuda")
    depth[W1 * H1:] = 4.0
    rows = np.array([0, 1, 128, 128 * 200 - 1, 128 * 200, 128 * 300, H1 - 1])
    for y in rows:
        depth[W1 * y:W1 * (y + 1)] = 4.0
    frac, _ = epo.build_viewgraph(W, H, K, np.tile(np.eye(3, 4).reshape(-1), (2, 1)), depth, stride=1, tau=0.75)
    del depth
    torch.cuda.empty_cache()
    inside = int(np.sum(np.arange(W1) <= 128 * (W[1] - 1))) * int(np.sum(rows <= 128 * (H[1] - 1)))
    assert frac[0, 1] == inside / (W1 * len(rows))
    back = np.isin(128 * np.arange(H[1]), rows).sum()
    assert frac[1, 0] == int(back) / int(H[1])


def test_stride_beyond_the_image_and_too_many_grid_pixels():
    d = torch.full((2 * 40 * 30,), 4.0, device="cuda")
    K, T = np.tile([64.0, 64.0, 20.0, 15.0], (2, 1)), np.tile(np.eye(3, 4).reshape(-1), (2, 1))
    frac, _ = epo.build_viewgraph([40, 40], [30, 30], K, T, d, stride=2**31 - 1, tau=3.0)
    assert np.array_equal(frac, [[0, 1], [1, 0]])
    with pytest.raises(epo.EpoError):  # refused on the host, before the depths are touched
        epo.build_viewgraph([2**17, 40], [2**16, 30], K, T, d, stride=1, tau=3.0)
