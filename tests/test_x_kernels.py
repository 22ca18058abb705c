"""Which x kernel runs a grid (csrc/kernels.cuh), from the library without a GPU."""
import os

import pytest

from device_code import program_output


@pytest.fixture(scope="module")
def library():
    from conftest import build_flusi
    libdir = os.path.dirname(build_flusi().LIB_PATH)
    return ["-L", libdir, "-lflusi", "-Xlinker", f"-rpath={libdir}"]


def test_x_kernel_of_every_length(library, tmp_path):
    """0 the shared-memory kernel, 1 a line kernel of its own, 2 the general line
    kernels: in FP32 also at 256, 128 and 64 points without the fused sponge."""
    out = program_output(r"""
#include <cstdio>
#include "kernels.cuh"
using namespace flusi;
int main()
{
    for (int fp64 = 0; fp64 < 2; ++fp64)
        for (int sponge = 0; sponge < 2; ++sponge)
            for (int nx : {8, 12, 16, 48, 64, 96, 128, 192, 256, 384, 512, 1024})
                for (int generic = 0; generic < 2; ++generic) {
                    Geom g{};
                    g.nx = nx;
                    g.xgeneric = generic;
                    printf("%d %d %d %d %d\n", fp64, sponge, nx, generic, xpass_kernel(fp64, g, sponge));
                }
    return 0;
}
""", tmp_path, *library)
    lines = [tuple(map(int, l.split())) for l in out.splitlines()]
    assert len(lines) == 96
    for fp64, sponge, nx, generic, kernel in lines:
        own = nx in (96, 512, 1024) or (nx in (64, 128, 256) and (fp64 or sponge))
        want = 0 if generic else 1 if own else 2 if not fp64 and nx >= 16 else 0
        assert kernel == want, (fp64, sponge, nx, generic)
