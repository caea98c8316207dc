"""The gradient's bits do not depend on how the planes are batched: the launch
shape (strip width, band height) follows the plane count, and every shape sums a
sample's contributions in the same order."""
import pytest
import torch

from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [0.0, 1.0, 2.0, 3.0])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("c,n,m", [(5, 70, 190), (2, 40, 40), (8, 130, 250), (16, 64, 64),
                                   (7, 17, 500), (4, 500, 111), (40, 128, 128), (3, 33, 176)])
def test_bits_of_a_plane_alone_and_in_a_batch(c, n, m, mode, beta):
    gen = torch.Generator(device="cuda").manual_seed(n)
    p = api.Params(out_mode=mode, beta=beta)
    x = torch.rand((c, n, m), generator=gen, device="cuda")
    g = torch.randn((c, 2 * n - mode, 2 * m - mode), generator=gen, device="cuda")
    whole = api.zoom2x_bwd(x, g, p)
    for k in range(c):
        assert torch.equal(api.zoom2x_bwd(x[k:k + 1], g[k:k + 1], p), whole[k:k + 1])
