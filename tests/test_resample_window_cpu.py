"""The tiled resampling kernel's window arithmetic at every width the entry
point accepts (below 2^31): the header the kernel includes is compiled for the
host and compared with exact integers."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2312_00229_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "wd_resample_window.h"
int main() {
  int kfirst, k0, m, first, rows_in, n, k, esz;
  while (std::scanf("%d %d %d %d %d %d %d %d", &kfirst, &k0, &m, &first, &rows_in, &n, &k, &esz) == 8)
    std::printf("%d %lld\n", (int)wdweno::window_inside(kfirst, k0, m, first, rows_in, n),
                (long long)wdweno::column_bytes(kfirst, k, esz));
}
"""


def _cases():
    top = 2 ** 31 - 1
    cases = []
    for m in (2, 63, 64, 65, 400, 2 ** 29 - 1, 2 ** 29 + 70, 2 ** 30 + 70, top - 64, top):
        for k0 in (0, 64, 256):
            edges = {-1, 0, 1, 2 ** 29 - 31, 2 ** 29, 2 ** 30 - 31, 2 ** 30}
            edges |= {m - d for d in (3, 2, 63, 64, 65, 64 + k0, 63 + k0, 65 + k0)}
            for kfirst in edges:
                if not -1 <= kfirst <= m - 2:  # cells 0 .. m - 2, one column before them
                    continue
                for first, rows_in, n in ((0, 11, 50), (1, 11, 11), (1, 11, 10), (40, 10, 49),
                                          (40, 10, 48), (top - 3, 4, top)):
                    for esz in (1, 2, 4):
                        cases.append((kfirst, k0, m, first, rows_in, n, k0 + 31, esz))
    return cases


# (traps on signed overflow, which the language leaves undefined)
@pytest.mark.parametrize("flags", [["-O2"], ["-O1", "-ftrapv"]])
def test_window_arithmetic_is_exact(tmp_path, flags):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", *flags, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    cases = _cases()
    text = "\n".join(" ".join(map(str, c)) for c in cases)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
    got = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    assert len(got) == len(cases)
    for (kfirst, k0, m, first, rows_in, n, k, esz), (inside, off) in zip(cases, got):
        want = (kfirst >= 0 and kfirst + k0 + 64 <= m and first >= 1
                and first - 1 + rows_in <= n)
        assert bool(inside) == want, (kfirst, k0, m, first, rows_in, n)
        assert off == (kfirst + k) * esz
