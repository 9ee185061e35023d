"""Where the fixed-point kernels read a link's entries (csrc/fixed.cuh), without a GPU: the planes' offsets are
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
    for (int e = 0; e < 8; ++e) {
        const auto p = tgf::Su3Src::plane(e, atoi(argv[1]));  // a pointer offset, of the type that the kernels add
        printf("%lld\n", (long long)(size_t)p);
    }
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


@pytest.mark.parametrize("Vp", [32, 2304, 178956960, 178956992, 192432384, 1 << 28])
def test_links_are_read_where_the_layout_puts_them(program, Vp):
    """Planes of entries (0,1), (2,3), (4,5), (6,7), four doubles a site."""
    got = [int(x) for x in subprocess.run([program, str(Vp)], check=True, capture_output=True).stdout.split()]
    assert got == [(e // 2) * 4 * Vp + 2 * (e % 2) for e in range(8)]
