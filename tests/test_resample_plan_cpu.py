"""Every plan of a resampling call keeps the kernel's bounds (window columns,
input rows and cells of a warp, grid), and the form follows the measured rule:
by cells where a tile's cells have work for its lanes, by outputs where the
columns are magnified so far that they have not, lines for single-sample axes
and fewer rows than a tile has warps.  The plan's header, compiled for the
host."""
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2312_00229_gb300", "csrc")
SMS = 152
REDUCED, CELLS, OUTPUTS, DIRECT, LINES = range(5)

SRC = r"""
#include <cstdio>
#include "wd_resample_plan.h"
int main() {
  using namespace wdweno;
  std::printf("%d %d %d %d %d %d\n", RS_WC_DOWN, RS_WC_UP, RS_WC_OUT, RS_MAX_CELLS, RS_MAX_IN,
              RS_TC_MAX);
  long long p, n, m, no, mo;
  int bytes;
  while (std::scanf("%lld %lld %lld %lld %lld %d", &p, &n, &m, &no, &mo, &bytes) == 6) {
    const RsPlan r = rs_plan(RsShape{n, m, p, no, mo, bytes}, 152);
    std::printf("%d %d %d\n", r.form, r.cols, r.rows);
  }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")],
                   check=True)

    def run(shapes):
        text = "\n".join(" ".join(map(str, s)) for s in shapes)
        r = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True)
        lines = [tuple(map(int, x.split())) for x in r.stdout.splitlines()]
        assert len(lines) == len(shapes) + 1
        return lines[0], lines[1:]
    return run


def _cell(j, n, n_out):
    return 0 if n <= 1 or n_out <= 1 else min(j * (n - 1) // (n_out - 1), n - 2)


def _shapes():
    rng = random.Random(5)
    shapes = []
    for _ in range(6000):
        sides = []
        for _ in range(2):
            n = rng.choice([1, 2, 3, rng.randrange(1, 40), rng.randrange(1, 3000),
                            rng.randrange(1, 10 ** 6)])
            o = rng.choice([1, 2, n, max(1, int(n * rng.uniform(0.3, 1.1))),
                            int(n * rng.uniform(1, 3)) + 1, int(n * rng.uniform(1, 70)) + 1])
            sides.append((n, o))
        (n, no), (m, mo) = sides
        if no <= 524280:  # (the entry point's limit)
            shapes.append((rng.choice([1, 3, 64]), n, m, no, mo, rng.choice([1, 2, 4])))
    return shapes


def test_every_plan_keeps_the_kernels_bounds(plans):
    shapes = _shapes()
    (wc_down, wc_up, wc_out, max_cells, max_in, tc_max), got = plans(shapes)
    rng = random.Random(6)
    window = {REDUCED: wc_down, CELLS: wc_up, OUTPUTS: wc_out}
    seen = set()
    for (p, n, m, no, mo, _), (form, cols, rows) in zip(shapes, got):
        seen.add(form)
        if form == DIRECT:
            continue
        if form == LINES:
            assert cols in (1, 2, 4, 8, 16, 32, 64, 128, 256) and rows >= 1
            per_block = 256 // cols * (1 if m == 1 and n > 1 else rows)
            assert (no + per_block - 1) // per_block <= 65535
            continue
        assert n > 1 and m > 1 and cols >= 4 and cols % 4 == 0
        assert cols <= (tc_max if form == CELLS else 128)
        assert rows in (1, 2, 4, 8) and (rows < 8 or (no >= n and form != REDUCED))
        strips = (mo + cols - 1) // cols
        for s in {0, strips - 1, rng.randrange(strips)}:
            c0, c1 = s * cols, min(mo, (s + 1) * cols) - 1
            first, last = _cell(c0, m, mo), _cell(c1, m, mo)
            assert last - first + 4 <= window[form], (n, m, no, mo, form)
            if form == CELLS:  # every cell between has outputs
                assert mo >= m
        tile = 8 * rows
        tiles = (no + tile - 1) // tile
        assert tiles <= 65535
        for t in {0, tiles - 1, rng.randrange(tiles)}:
            r0, r1 = t * tile, min(no, (t + 1) * tile) - 1
            assert _cell(r1, n, no) - _cell(r0, n, no) + 4 <= max_in
            for q in range(r0, r1 + 1, rows):
                assert _cell(min(q + rows - 1, r1), n, no) - _cell(q, n, no) < max_cells
    assert seen == {REDUCED, CELLS, OUTPUTS, DIRECT, LINES}


@pytest.mark.parametrize("form,shapes", [
    (CELLS, [(3, 1080, 1920, 3240, 5760, 1), (3, 1080, 1920, 2160, 3840, 1),
             (3, 540, 960, 4320, 7680, 1), (3, 540, 960, 6480, 11520, 4),
             (3, 200, 300, 1200, 1800, 1)]),
    (OUTPUTS, [(3, 64, 64, 512, 512, 1), (3, 64, 64, 1024, 1024, 4), (3, 64, 64, 4096, 4096, 2),
               (3, 540, 960, 8640, 15360, 4), (1, 32, 32, 4096, 4096, 1), (1, 3, 3, 4000, 4000, 1),
               (3, 540, 960, 600, 1000, 1), (3, 540, 960, 4320, 500, 1),
               (3, 222, 987, 206, 914, 2)]),
    (REDUCED, [(3, 4317, 7677, 3240, 5760, 1), (3, 2160, 3840, 1270, 2258, 1)]),
    (LINES, [(1, 1, 1000, 1000, 3000, 1), (1, 400000, 1, 500000, 1, 1), (1, 1, 1, 1, 1, 4),
             (1, 6, 900, 7, 2000, 1)]),
    (DIRECT, [(3, 1080, 1920, 270, 480, 1), (3, 300, 300, 100, 900, 4)])])
def test_form_follows_the_rule(plans, form, shapes):
    assert [g[0] for g in plans(shapes)[1]] == [form] * len(shapes)
