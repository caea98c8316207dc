"""Chains of zooms whose intermediate type is left open (None) keep the input's
type between the levels, like a zoom whose output type is left open."""
import pytest
import torch

from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float16, torch.float32])
@pytest.mark.parametrize("n,m", [(9, 7), (16, 12)])
def test_open_intermediate_type(dtype, n, m):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand((2, n, m), generator=g, device="cuda")
    x = (x * 255).to(dtype) if dtype == torch.uint8 else x.to(dtype)
    for mode in (0, 1):
        p = api.Params(out_mode=mode)
        assert torch.equal(api.cascade_zoom(x, 3, p, out_dtype=torch.float32, inter_dtype=None),
                           api.cascade_zoom(x, 3, p, out_dtype=torch.float32, inter_dtype=dtype))
    assert torch.equal(api.zoom_to(x, 3 * n, 3 * m, inter_dtype=None),
                       api.zoom_to(x, 3 * n, 3 * m, inter_dtype=dtype))
