"""Chains of zooms refuse what one zoom refuses, with the same errors, before
they allocate a level's output (a side of no samples has no 2n-1 grid)."""
import pytest
import torch

from paper_2312_00229_gb300 import api


@pytest.mark.parametrize("shape", [(1, 4, 0), (3, 0, 5), (1, 4, 6), (4, 0)])
def test_host_tensors_are_refused(shape):
    x = torch.zeros(shape)
    with pytest.raises(ValueError, match="must be a CUDA tensor"):
        api.zoom_to(x, 9, 9)
    with pytest.raises(ValueError, match="must be a CUDA tensor"):
        api.cascade_zoom(x, 2, api.Params(out_mode=1))


def test_no_level_is_no_zoom():
    x = torch.zeros((1, 4, 6))
    assert api.cascade_zoom(x, 0) is x


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1, 4, 0), (3, 0, 5), (4, 0)])
def test_empty_images_are_refused(shape):
    x = torch.zeros(shape, device="cuda")
    with pytest.raises(ValueError, match="empty input"):
        api.zoom_to(x, 9, 9)
    with pytest.raises(ValueError, match="empty input"):
        api.cascade_zoom(x, 2, api.Params(out_mode=1))
