"""The adjoint's output-gradient loads: aligned column pairs, single columns of
misaligned or strided views and the odd last column of the 2n-1 grid take
different copies, and have to give the same gradient bit for bit."""
import pytest
import torch

from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu


def _view(g, kind):
    n, h, w = g.shape
    if kind == "offset":  # rows start on an odd element
        buf = torch.full((n, h, w + 3), float("nan"), device=g.device)
        v = buf[:, :, 1:1 + w]
    elif kind == "oddrows":  # an odd row stride: every other row is misaligned
        pad = 1 + w % 2
        buf = torch.full((n, h, w + pad), float("nan"), device=g.device)
        v = buf[:, :, :w]
    else:  # every second column of a wider buffer
        buf = torch.full((n, h, 2 * w), float("nan"), device=g.device)
        v = buf[:, :, ::2]
    v.copy_(g)
    return v


# sides around the sweeps' strips (115 and 179 columns of the extended grid,
# 108 and 172 of the image) and bands, and the smallest images
@pytest.mark.parametrize("n,m", [(1, 1), (2, 3), (9, 111), (17, 112), (40, 175), (33, 176),
                                 (21, 180), (64, 108), (50, 173)])
@pytest.mark.parametrize("mode", [0, 1])
def test_bwd_gradient_views(n, m, mode):
    gen = torch.Generator(device="cuda").manual_seed(1000 * n + m)
    p = api.Params(out_mode=mode)
    x = torch.rand((2, n, m), generator=gen, device="cuda")
    g = torch.randn((2, 2 * n - mode, 2 * m - mode), generator=gen, device="cuda")
    ref = api.zoom2x_bwd(x, g, p)
    for kind in ("offset", "oddrows", "strided"):
        assert torch.equal(api.zoom2x_bwd(x, _view(g, kind), p), ref), kind


def test_bwd_plane_equals_batch():
    """Each plane's gradient is that of the plane alone (workspace offsets)."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand((5, 70, 190), generator=gen, device="cuda")
    g = torch.randn((5, 140, 380), generator=gen, device="cuda")
    whole = api.zoom2x_bwd(x, g)
    for k in range(5):
        one = api.zoom2x_bwd(x[k:k + 1], g[k:k + 1])
        assert torch.allclose(one, whole[k:k + 1], rtol=0, atol=1e-6 * float(whole.abs().max()))
