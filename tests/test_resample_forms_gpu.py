"""The kernel forms of tensor-WENO resampling against the FP64 oracle, at the
edges of their tiles, and against each other bit for bit on data that isolates
one axis (an image of equal rows or equal columns keeps its values exactly
along that axis)."""
import numpy as np
import pytest
import torch

import oracle
import parity
from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu

TOL = 1e-5  # one resampling of O(1) values in FP32

# far magnified (by outputs), reduced columns with magnified rows, about the same
# spacing, single-sample axes and few rows (lines): tiles of 128 outputs, blocks
# of 32 and 256 columns and of 8 rows, and one more or less of each
SIZES = [(3, 3, 70, 400), (2, 2, 9, 1000), (9, 8, 64, 129), (20, 33, 161, 1100), (12, 40, 300, 640),
         (40, 300, 130, 160), (33, 257, 200, 129), (16, 131, 40, 128), (64, 130, 64, 131),
         (70, 200, 71, 190), (130, 135, 129, 134), (1, 40, 17, 257), (1, 9, 9, 31), (40, 1, 129, 33),
         (9, 1, 31, 1), (1, 1, 70, 300), (4, 300, 7, 513), (6, 6, 3, 300), (7, 40, 4, 20),
         (1, 300, 1, 100), (300, 1, 100, 5)]


@pytest.mark.parametrize("n,m,oh,ow", SIZES)
@pytest.mark.parametrize("beta", [2.0, 1.0, 0.0])
def test_forms_against_oracle(n, m, oh, ow, beta):
    x = np.random.default_rng(n * 977 + m).random((2, n, m)).astype(np.float32)
    ref = oracle.tensor_resample(x.astype(np.float64), oh, ow, beta=beta)
    t = torch.from_numpy(x).cuda()
    for bound in (0.0, 1.0):  # scale-free and direct weights
        y = api.resample(t, oh, ow, api.Params(beta=beta, data_bound=bound))
        assert np.abs(y.double().cpu().numpy() - ref).max() <= TOL


@pytest.mark.parametrize("dt", ["u8", "f16", "bf16"])
@pytest.mark.parametrize("n,m,oh,ow", [(3, 3, 70, 400), (40, 300, 130, 160), (70, 200, 71, 190),
                                       (1, 40, 17, 257), (40, 1, 129, 33), (4, 300, 7, 513),
                                       (40, 62, 79, 123), (60, 90, 47, 61), (50, 70, 24, 34)])
def test_storage_types_against_oracle(dt, n, m, oh, ow):
    x = parity.encode(np.random.default_rng(m).random((2, n, m)), dt)
    ref = oracle.tensor_resample(parity.decode(x), oh, ow)
    parity.compare(api.resample(x.cuda(), oh, ow), ref, dt)


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float16, torch.float32])
@pytest.mark.parametrize("n,m,oh,ow", [(3, 3, 70, 400), (40, 300, 130, 160), (70, 200, 71, 190),
                                       (1, 40, 17, 257), (40, 1, 129, 33), (4, 300, 7, 513)])
def test_layouts_and_strides_agree(dtype, n, m, oh, ow):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand((3, n, m), generator=g, device="cuda")
    x = (x * 255).to(dtype) if dtype == torch.uint8 else x.to(dtype)
    ref = api.resample(x, oh, ow)
    hwc = api.resample(x.permute(1, 2, 0).contiguous(), oh, ow, layout="hwc")
    assert torch.equal(hwc.permute(2, 0, 1), ref)
    wide = torch.zeros((3, oh + 2, ow + 3 - ow % 2), dtype=dtype, device="cuda")
    api.resample(x, oh, ow, out=wide[:, 1:1 + oh, 1:1 + ow])
    assert torch.equal(wide[:, 1:1 + oh, 1:1 + ow], ref)
    rest = wide.clone()
    rest[:, 1:1 + oh, 1:1 + ow] = 0
    assert int(rest.count_nonzero()) == 0  # nothing outside the view
    src = torch.full((3, n, 2 * m), 7, dtype=dtype, device="cuda")
    src[:, :, ::2] = x
    assert torch.equal(api.resample(src[:, :, ::2], oh, ow), ref)


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("beta", [2.0, 1.0])
@pytest.mark.parametrize("m,ow", [(40, 61), (40, 40), (40, 401), (40, 1000), (300, 290), (300, 200),
                                  (7, 500)])
def test_row_interpolants_are_the_forms_own(dtype, beta, m, ow):
    """Equal rows: the outputs of every form are the row interpolants."""
    g = torch.Generator(device="cuda").manual_seed(m + ow)
    line = torch.rand((2, 1, m), generator=g, device="cuda")
    line = (line * 255).to(dtype) if dtype == torch.uint8 else line
    p = api.Params(beta=beta)
    want = api.resample(line, 1, ow, p)  # lines
    assert torch.equal(api.resample(line, 9, ow, p), want.expand(2, 9, ow).contiguous())
    for n, oh in ((40, 40), (40, 70), (40, 25), (40, 9), (5, 7)):  # tiles, direct, lines
        y = api.resample(line.expand(2, n, m).contiguous(), oh, ow, p)
        assert torch.equal(y, want.expand(2, oh, ow)), (n, oh)


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("beta", [2.0, 1.0])
@pytest.mark.parametrize("n,oh", [(40, 61), (40, 40), (40, 401), (300, 290), (300, 160), (7, 500)])
def test_column_interpolants_are_the_forms_own(dtype, beta, n, oh):
    """Equal columns: the outputs of every form are the column interpolants."""
    g = torch.Generator(device="cuda").manual_seed(n + oh)
    line = torch.rand((2, n, 1), generator=g, device="cuda")
    line = (line * 255).to(dtype) if dtype == torch.uint8 else line
    p = api.Params(beta=beta)
    want = api.resample(line, oh, 1, p)  # lines
    assert torch.equal(api.resample(line, oh, 300, p), want.expand(2, oh, 300).contiguous())
    for m, ow in ((40, 40), (40, 100), (40, 1000), (40, 38), (40, 25), (40, 9)):  # tiles, direct
        y = api.resample(line.expand(2, n, m).contiguous(), oh, ow, p)
        assert torch.equal(y, want.expand(2, oh, ow)), (m, ow)


def test_infinite_sample_alone():
    """An axis of one sample is not interpolated along: infinity stays."""
    x = torch.full((1, 1, 1), float("inf"), device="cuda")
    for oh, ow in ((20, 30), (1, 300), (300, 1)):
        assert bool(torch.isposinf(api.resample(x, oh, ow)).all())
