"""The 96-thread tile (182-column strips), which no caller can ask for: the sizes
below are ones for which the library's own plan takes it on 152 SMs (checked
on the CPU, the plan's header compiled for the host), so that the GPU tests run
it in every storage type and weight form, with bounds around its outputs."""
import os
import shutil
import subprocess

import pytest
import torch

from paper_2312_00229_gb300 import api

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2312_00229_gb300", "csrc")

# (planes, rows, columns): one strip, one of 180 and of 182 columns, two and three
# strips, bands that divide the rows and that do not
SIZES = [(96, 9, 182), (64, 20, 180), (30, 77, 182), (48, 130, 364), (3, 512, 512)]

SRC = r"""
#include <cstdio>
#include "wd_fwd_model.h"
int main() {
  int p, n, m;
  while (std::scanf("%d %d %d", &p, &n, &m) == 3) {
    const wdweno::FwdPlan q = wdweno::fwd_find_plan(n, m, p, 152, 0, 0, 0);
    std::printf("%d %d\n", q.threads, q.cols);
  }
}
"""


def test_the_plan_takes_it(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    text = "\n".join(" ".join(map(str, s)) for s in SIZES)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
    assert r.stdout.split("\n")[:-1] == ["96 2"] * len(SIZES)


@pytest.mark.gpu
@pytest.mark.parametrize("c,n,m", SIZES)
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("beta,bound", [(2.0, 0.0), (2.0, 1.0), (1.0, 0.0), (1.5, 0.0), (0.0, 0.0)])
def test_values_and_bounds(c, n, m, dtype, beta, bound):
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randint(0, 256, (c, n, m), generator=gen, device="cuda", dtype=torch.uint8)
    x = x if dtype == torch.uint8 else (x.float() * (1.0 / 255.0)).to(dtype)
    for mode in (0, 1):
        p = api.Params(beta=beta, out_mode=mode, data_bound=bound)
        ref = api.zoom2x_fwd(x, p, rows_per_tile=64, tile_width=247)
        oh, ow = ref.shape[1:]
        buf = torch.full((c, oh + 2, ow + 8), 77, dtype=dtype, device="cuda")
        got = buf[:, 1:1 + oh, 4:4 + ow]
        api.zoom2x_fwd(x, p, rows_per_tile=0, tile_width=0, out=got)
        assert torch.equal(got, ref)
        got.fill_(77)
        assert bool((buf == 77).all())  # nothing outside the view
