"""Where the fixed-point kernels read a link's entries (csrc/fixed.cuh), without a GPU: the address expression is
compiled for the host and compared with the FP64 storage layout, written out here, at sizes up to the library's
limit of 2^28 sites."""
import os
import subprocess

import pytest

from paper_2107_03747_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "fixed.cuh"
int main(int argc, char** argv) {
    const int Vp = atoi(argv[1]), s = atoi(argv[2]);
    for (int dir = 0; dir < 4; ++dir)
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j)
                for (int tr = 0; tr < 2; ++tr) printf("%lld\n", (long long)tgf::Su3Src::at(dir, s, i, j, tr != 0, Vp));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src, exe = d / "at.cu", d / "at"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), *build.ARCH,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    return str(exe)


def layout(dir, s, e, Vp):
    """Doubles from the field's start: planes of entries (0,1), (2,3), (4,5), (6,7), four doubles a site, then
    entry 8, two doubles a site."""
    base = dir * 18 * Vp
    return base + 16 * Vp + 2 * s if e == 8 else base + (e // 2) * 4 * Vp + 4 * s + 2 * (e % 2)


@pytest.mark.parametrize("Vp", [32, 2304, 178956960, 178956992, 192432384, 1 << 28])
def test_links_are_read_where_the_layout_puts_them(program, Vp):
    for s in (0, 1, Vp // 2 + 1, Vp - 1):
        got = [int(x) for x in subprocess.run([program, str(Vp), str(s)], check=True, capture_output=True).stdout.split()]
        want = [layout(dir, s, 3 * j + i if tr else 3 * i + j, Vp)
                for dir in range(4) for i in range(3) for j in range(3) for tr in range(2)]
        assert got == want
