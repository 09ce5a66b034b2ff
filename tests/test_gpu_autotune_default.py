"""The autotuner's candidates include the schedule that the library picks by itself: where that splits
every item by pairs (small scenes with all pairs), which no other candidate does, tuning ends with it on
some of the scenes at least (by timing, so not on each)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA GPU required", allow_module_level=True)

from tests.test_gpu_default_schedule import scene  # noqa: E402


def schedule(s):
    i = s.info()
    return i.gather, i.block_threads, i.records_per_thread, i.tail_pairs


def test_default_schedule_is_a_candidate():
    kept = []
    for W, H, n in ((200, 150, 10), (200, 150, 14), (200, 150, 16), (200, 150, 20), (319, 241, 13), (319, 241, 14),
                    (319, 241, 16), (319, 241, 20), (96, 80, 16)):
        s = scene(W, H, n, W * H // 12, n - 1, False, autotune=1)
        own = schedule(s)
        assert own[3] < 0  # the default's, until the first evaluation tunes
        s.loss_and_grad()
        kept.append(schedule(s) == own)
    assert any(kept)
