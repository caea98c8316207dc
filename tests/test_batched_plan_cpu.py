"""The band height of a batch left open: the device's choice, its model compiled
for the host.  A few large images get heights whose tiles fill whole waves of
CTAs, small ones short bands, many large ones tall bands."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2312_00229_gb300", "csrc")
SMS = 152

SRC = r"""
#include <cstdio>
#include "wd_fwd_model.h"
using namespace wdweno;
int main() {
  int threads, cols, count;
  while (std::scanf("%d %d %d", &threads, &cols, &count) == 3) {
    FwdShape s = FWD_SHAPES[0];
    for (const FwdShape& q : FWD_SHAPES)
      if (q.threads == threads && q.cols == cols) s = q;
    BatchedCost c[BATCHED_CANDS] = {};
    for (int i = 0; i < count; ++i) {
      int p, n, m;
      if (std::scanf("%d %d %d", &p, &n, &m) != 3) return 1;
      for (int j = 0; j < BATCHED_CANDS; ++j)
        batched_add(c[j], n, float((m + fwd_strip(s) - 1) / fwd_strip(s) * p),
                    BATCHED_HEIGHTS.rows[j]);
    }
    int best = 0;
    for (int j = 1; j < BATCHED_CANDS; ++j)
      if (batched_us(s, 152, c[j]) < batched_us(s, 152, c[best])) best = j;
    std::printf("%d %.0f\n", BATCHED_HEIGHTS.rows[best], c[best].tiles);
  }
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("batched_plan")
    (d / "p.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")],
                   check=True)

    def run(images, shape=(64, 2)):
        text = " ".join(map(str, (*shape, len(images), *[v for im in images for v in im])))
        r = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True)
        rows, tiles = r.stdout.split()
        return int(rows), int(tiles)
    return run


@pytest.mark.parametrize("image,rows", [((3, 1080, 1920), {64}), ((3, 2000, 2000), {128}),
                                        ((1, 2000, 3000), {64}), ((3, 1000, 1000), {32}),
                                        ((3, 1500, 1500), {24, 32, 96}), ((3, 720, 1280), {32}),
                                        ((3, 2160, 3840), {64, 96, 128})])
def test_one_large_image_fills_whole_waves(choose, image, rows):
    """The measured best heights (us: 1080p 70 at 64 rows, 119 at 128; 2000x2000
    124 at 128, 137 at 64; the heights listed are within 5% of the best)."""
    got, tiles = choose([image])
    assert got in rows, (got, tiles)
    waves = tiles / (SMS * 6)
    assert waves - int(waves) == 0 or waves - int(waves) > 0.4, waves


def test_small_images_get_short_bands(choose):
    assert choose([(3, 61, 56), (3, 81, 77), (3, 48, 96), (3, 90, 50), (3, 70, 88)])[0] <= 4
    assert choose([(3, 512, 512)])[0] in (8, 12, 16)


def test_many_large_images_get_tall_bands(choose):
    assert choose([(3, 667 + i, 797 - i) for i in range(32)])[0] >= 96
    assert choose([(3, 3814, 3707)] * 3)[0] >= 96


@pytest.mark.parametrize("image,rows", [((3, 1080, 1920), {48}), ((3, 1000, 1000), {48}),
                                        ((3, 720, 1280), {24, 48}), ((1, 2000, 3000), {96}),
                                        ((3, 1500, 1500), {64, 128})])
def test_one_column_strips(choose, image, rows):
    """Strips of 119, beta = 1: within 3% of the measured best (1080p 115 us at 48
    rows, 129 at 64, 130 at 128)."""
    assert choose([image], (128, 1))[0] in rows
