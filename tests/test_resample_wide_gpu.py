"""Tensor-WENO resampling of images wider than 2^29 (FP32) and 2^30 (16-bit)
columns, where the byte offset of a column no longer fits 32 bits: reduced to
every second column, the right end has the bits of the same columns alone."""
import pytest
import torch

from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,cols", [(torch.float32, 2 ** 29 + 1001),
                                        (torch.float16, 2 ** 30 + 1001)])
def test_right_end_of_wide_images(dtype, cols):
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    gen = torch.Generator(device="cuda").manual_seed(7)
    keep = 2 * 900 + 1  # (odd: output column j is input column 2 j in both)
    end = torch.rand((4, keep), generator=gen, device="cuda").to(dtype)
    x = torch.zeros((1, 4, cols), dtype=dtype, device="cuda")
    x[0, :, -keep:] = end
    # 25 rows of 4: warps whose rows lie in the middle cell alone read rows
    # that need no clamping
    y = api.resample(x, 25, (cols + 1) // 2, out_dtype=torch.uint8)
    ref = api.resample(end[None].contiguous(), 25, (keep + 1) // 2, out_dtype=torch.uint8)
    n = 890  # (the columns whose neighbours are the same in both)
    assert torch.equal(y[0, :, -n:], ref[0, :, -n:])
    assert int(y[0, :, :1000].count_nonzero()) == 0
    del x, y
    torch.cuda.empty_cache()
