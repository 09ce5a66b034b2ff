"""The distance transform at the sizes where its two passes change shape (32-pixel words, 16-word
loads, 1024-pixel segments; 4-column strips, the tallest image) and at every kind of mask, against
the oracle's exact transform.  Squared distances are integers below 2^24 and the root is correctly
rounded, so the two agree bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

import paper_2607_00579_gb300 as epo  # noqa: E402


def check(mask):
    got = epo.distance_field(torch.from_numpy(mask).cuda()).cpu().numpy()
    assert np.array_equal(got, oracle.edt(mask).astype(np.float32))


@pytest.mark.parametrize("W,H", [(1, 1), (1, 7), (2, 1), (3, 5), (31, 2), (32, 33), (33, 64), (511, 4), (512, 3),
                                 (513, 9), (1023, 5), (1024, 6), (1025, 7), (2049, 40), (3071, 3), (7, 1536)])
@pytest.mark.parametrize("density", [0.0, 0.002, 0.1, 1.0])
def test_sizes(W, H, density):
    r = np.random.default_rng([W, H])
    check(((r.random((H, W)) < density) * r.integers(1, 256, (H, W))).astype(np.uint8))


@pytest.mark.parametrize("W,H", [(2100, 70), (518, 392), (90, 300)])
def test_single_edges(W, H):
    for x, y in [(0, 0), (W - 1, H - 1), (W // 2, 0), (min(1023, W - 1), H // 2), (min(1024, W - 1), H // 3)]:
        m = np.zeros((H, W), np.uint8)
        m[y, x] = 255
        check(m)
