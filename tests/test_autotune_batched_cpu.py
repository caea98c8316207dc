"""Host logic of the batched autotuner (no GPU): the height chosen on the
device from the images' sizes is among its candidates, and what it keeps for
one batch is not taken for batches of the same count and other sizes."""
import pytest
import torch

from paper_2312_00229_gb300 import api, autotune


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """The tuner with plans that only record their shape; `cost` gives times."""
    monkeypatch.setattr(autotune, "CACHE_PATH", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "_cache", None)
    monkeypatch.setattr(autotune, "_device_name", lambda device: "TestGPU")

    class Plan:
        def __init__(self, images, params=None, out_dtype=None, layout="chw", rows_per_tile=0,
                     outputs=None, tile_width=0):
            self.shape = (rows_per_tile, tile_width)

        def run(self):
            return self.shape

    cost = {}
    monkeypatch.setattr(api, "BatchedPlan", Plan)
    monkeypatch.setattr(autotune, "_time", lambda fn, reps: cost.get(fn(), 1.0))
    return cost


def _batch(sides, c=3):
    return [torch.zeros((c, h, w), dtype=torch.uint8) for h, w in sides]


SMALL, LARGE = _batch([(64, 80)] * 5), _batch([(1000, 900)] * 5)


def test_device_chosen_height_is_a_candidate_and_is_kept(tuner):
    tuner[(0, 118)] = 0.5
    times = autotune.tune_batched(SMALL)
    assert {w for r, w in times if r == 0} == set(autotune.BATCHED_TILE_WIDTHS)
    assert min(times, key=times.get) == (0, 118)
    assert autotune.lookup_batched(SMALL, None, "chw") == (0, 118)


def test_a_shape_is_kept_for_its_sizes_alone(tuner):
    tuner[(128, 247)] = 0.5
    autotune.tune_batched(LARGE)
    assert autotune.lookup_batched(LARGE, None, "chw") == (128, 247)
    assert autotune.lookup_batched(_batch([(1020, 880)] * 7), None, "chw") == (128, 247)
    for other in (SMALL, _batch([(1000, 900)] * 5, 1), _batch([(1000, 90)] * 5),
                  _batch([(1000, 900)] + [(40, 50)] * 4)):
        assert autotune.lookup_batched(other, None, "chw") == (0, 0)


def test_an_empty_batch_is_an_error(tuner):
    with pytest.raises(IndexError):
        autotune.lookup_batched([], None, "chw")
