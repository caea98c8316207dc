"""The library's own choice of tile shapes: every plan gives the bits of one
fixed tile, from a single sample to several waves of CTAs, in the one-launch and
the batched form; and the kernels of a fixed storage pair give the bits of the
run-time-typed ones for beta != 2."""
import pytest
import torch

from paper_2312_00229_gb300 import api

pytestmark = pytest.mark.gpu


def _img(shape, seed, dtype=torch.uint8):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(0, 256, shape, generator=g, device="cuda", dtype=torch.uint8)
    return x if dtype == torch.uint8 else (x.float() * (1.0 / 255.0)).to(dtype)


@pytest.mark.parametrize("c,n,m", [(1, 1, 1), (3, 2, 7), (1, 3, 400), (3, 17, 118), (3, 48, 64),
                                   (1, 119, 119), (2, 200, 247), (3, 333, 500), (1, 1024, 130),
                                   (65, 40, 246), (3, 700, 900), (3, 512, 512), (1, 30, 182),
                                   (8, 64, 364), (24, 100, 183), (3, 300, 545)])
@pytest.mark.parametrize("mode", [0, 1])
def test_default_plan_bits(c, n, m, mode):
    x = _img((c, n, m), 7 * n + m)
    p = api.Params(out_mode=mode)
    ref = api.zoom2x_fwd(x, p, rows_per_tile=64, tile_width=247)
    assert torch.equal(api.zoom2x_fwd(x, p, rows_per_tile=0, tile_width=0), ref)
    for tw in (118, 119, 246, 247):  # band height chosen for a given width
        assert torch.equal(api.zoom2x_fwd(x, p, rows_per_tile=0, tile_width=tw), ref)
    for rows in (1, 2, 5, 33):  # width chosen for a given band height
        assert torch.equal(api.zoom2x_fwd(x, p, rows_per_tile=rows, tile_width=0), ref)


@pytest.mark.parametrize("sides", [[(1, 1)], [(5, 9)] * 3, [(64, 80), (1, 300), (300, 1)],
                                   [(100 + 7 * i, 90 + 11 * i) for i in range(33)],
                                   [(16 + i % 5, 20 + i % 3) for i in range(1100)],
                                   [(900, 700), (8, 8)]])
def test_batched_default_bits(sides):
    imgs = [_img((3, n, m), i) for i, (n, m) in enumerate(sides)]
    for rows, tw in ((0, 0), (0, 119), (0, 246), (24, 0)):
        outs = api.BatchedPlan(imgs, rows_per_tile=rows, tile_width=tw).run()
        step = max(1, len(imgs) // 40)
        for k in range(0, len(imgs), step):
            ref = api.zoom2x_fwd(imgs[k], rows_per_tile=64, tile_width=247)
            assert torch.equal(outs[k], ref), (rows, tw, k)


@pytest.mark.parametrize("beta", [0.1, 1.0, 1.5, 3.0])
@pytest.mark.parametrize("n,m,mode", [(37, 130, 0), (64, 246, 1), (5, 3, 0)])
def test_fixed_types_equal_run_time_types(beta, n, m, mode):
    p = api.Params(beta=beta, out_mode=mode)
    u8 = _img((2, n, m), 3)
    f32 = _img((2, n, m), 3, torch.float32)
    # uint8 -> FP32 runs the run-time-typed kernel, the same-type pairs do not
    ref = api.zoom2x_fwd(u8, p, out_dtype=torch.float32, rows_per_tile=16, tile_width=119)
    for tw in (118, 119, 246, 247):
        assert torch.equal(api.zoom2x_fwd(f32, p, tile_width=tw, rows_per_tile=0), ref)
        got = api.zoom2x_fwd(u8, p, tile_width=tw, rows_per_tile=0)
        assert torch.equal(got, api.zoom2x_fwd(f32, p, out_dtype=torch.uint8, tile_width=119,
                                               rows_per_tile=16))
    for dt in (torch.float16, torch.bfloat16):
        x = _img((2, n, m), 3, dt)
        ref16 = api.zoom2x_fwd(x.float(), p, rows_per_tile=0).to(dt)
        assert torch.equal(api.zoom2x_fwd(x, p, rows_per_tile=0), ref16)


@pytest.mark.parametrize("n,m", [(9, 7), (33, 61), (50, 50)])
def test_padded_inner_levels(n, m):
    """Inner levels with padded rows: the chain equals explicit contiguous levels."""
    x = _img((3, n, m), n)
    cur, bounds = x, api._level_bounds(x, api.Params(), 3)
    for lvl in range(3):
        cur = api.zoom2x_fwd(cur, api.Params(h=0.5 ** lvl, data_bound=bounds[lvl]),
                             out_dtype=torch.uint8 if lvl == 2 else torch.float32).contiguous()
    assert torch.equal(api.cascade_zoom(x, 3), cur)
    y = api.zoom_to(x, 3 * n, 3 * m)
    cur = x
    for lvl in range(2):
        cur = api.zoom2x_fwd(cur, api.Params(h=0.5 ** lvl, data_bound=bounds[lvl], out_mode=1),
                             out_dtype=torch.float32).contiguous()
    assert torch.equal(y, api.resample(cur, 3 * n, 3 * m, api.Params(h=0.25, data_bound=bounds[2]),
                                       out_dtype=torch.uint8))
