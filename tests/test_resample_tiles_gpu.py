"""Tensor-WENO resampling at the edges of its tiles: window widths, cells with
one to many outputs, reductions around 1/2, degenerate axes, odd and strided
outputs; the tiled kernels and the one-thread-per-output kernel give the same
bits, and all agree with the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu

# one resampling: FP32 differences of O(1) values and approximate reciprocals
TOL = 1e-5


def _x(c, n, m, seed):
    return np.random.default_rng(seed).random((c, n, m)).astype(np.float32)


SIZES = [(2, 2, 2, 2), (2, 2, 9, 31), (5, 64, 5, 64), (64, 5, 130, 121), (33, 61, 33, 61),
         (40, 62, 79, 123), (40, 62, 80, 125), (50, 70, 25, 36), (51, 71, 26, 36), (50, 70, 24, 35),
         (90, 40, 60, 161), (40, 90, 161, 60), (17, 300, 64, 901), (9, 9, 70, 200), (3, 200, 65, 4),
         (129, 131, 128, 130), (4, 4, 1, 9), (7, 7, 9, 1), (1, 9, 5, 30), (9, 1, 30, 5)]


@pytest.mark.parametrize("n,m,oh,ow", SIZES)
@pytest.mark.parametrize("beta", [2.0, 1.0])
def test_sizes_against_oracle(n, m, oh, ow, beta):
    x = _x(2, n, m, n * 131 + m)
    ref = oracle.tensor_resample(x.astype(np.float64), oh, ow, beta=beta)
    t = torch.from_numpy(x).cuda()
    for bound in (0.0, 1.0):  # scale-free and direct weights
        y = api.resample(t, oh, ow, api.Params(beta=beta, data_bound=bound))
        assert np.abs(y.double().cpu().numpy() - ref).max() <= TOL


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n,m,oh,ow", [(40, 62, 79, 123), (50, 70, 25, 36), (60, 90, 47, 61),
                                       (9, 9, 70, 200), (90, 40, 60, 161)])
def test_forms_and_layouts_agree(dtype, n, m, oh, ow):
    """Planar, interleaved, odd-stride and strided outputs, equal bit for bit;
    and each output column equals the one-thread-per-output kernel's on an axis
    it can be isolated on (a single column of the input repeated)."""
    x = torch.from_numpy(_x(3, n, m, 11)).cuda()
    x = (x * 255).to(torch.uint8) if dtype == torch.uint8 else x.to(dtype)
    ref = api.resample(x, oh, ow)
    hwc = api.resample(x.permute(1, 2, 0).contiguous(), oh, ow, layout="hwc")
    assert torch.equal(hwc.permute(2, 0, 1), ref)
    wide = torch.zeros((3, oh, ow + 3 - ow % 2), dtype=dtype, device="cuda")
    api.resample(x, oh, ow, out=wide[:, :, 1:1 + ow])
    assert torch.equal(wide[:, :, 1:1 + ow], ref)
    step = torch.zeros((3, oh, 2 * ow), dtype=dtype, device="cuda")
    api.resample(x, oh, ow, out=step[:, :, ::2])
    assert torch.equal(step[:, :, ::2], ref) and int(step[:, :, 1::2].count_nonzero()) == 0
    # run-time types: through another storage type of at least the precision
    if dtype in (torch.float16, torch.bfloat16):
        mixed = api.resample(x, oh, ow, out_dtype=torch.float32, params=api.Params(data_bound=1.0))
        same = api.resample(x.float(), oh, ow, api.Params(data_bound=1.0))
        assert torch.equal(mixed, same)


@pytest.mark.parametrize("n,m,oh,ow", [(200, 300, 60, 90), (101, 77, 11, 13)])
def test_reductions_beyond_half(n, m, oh, ow):
    x = _x(2, n, m, 5)
    ref = oracle.tensor_resample(x.astype(np.float64), oh, ow)
    y = api.resample(torch.from_numpy(x).cuda(), oh, ow)
    assert np.abs(y.double().cpu().numpy() - ref).max() <= TOL
    # columns reduced beyond 1/2 and rows magnified, and the other way round
    for h, w in ((2 * n, ow), (oh, 2 * m)):
        ref = oracle.tensor_resample(x.astype(np.float64), h, w)
        y = api.resample(torch.from_numpy(x).cuda(), h, w)
        assert np.abs(y.double().cpu().numpy() - ref).max() <= TOL
