"""The autotuner's rules (csrc/tuning.cuh), from the library without a GPU."""
import os

import pytest

from device_code import program_output

HEAD = r"""
#include <cstdio>
#include <string>
#include "kernels.cuh"
#include "tuning.cuh"
using namespace flusi;
"""


@pytest.fixture(scope="module")
def library():
    from conftest import build_flusi
    libdir = os.path.dirname(build_flusi().LIB_PATH)
    return ["-L", libdir, "-lflusi", "-Xlinker", f"-rpath={libdir}"]


def test_plans_are_scored_by_every_kernel_they_change(library, tmp_path):
    """In FP32 the z plan decides between the staged and the two-pass kernels of
    both z passes, so both are timed for it, as both y passes are for theirs."""
    out = program_output(HEAD + r"""
int main()
{
    for (const TuneKnob& k : tune_knobs) {
        const char* name = k.field == &flusi_tuning::y_plan ? "y_plan" : k.field == &flusi_tuning::zf_plan ? "zf_plan" : "-";
        for (const char* s : k.kernels) printf("%s %s\n", name, s ? s : "-");
    }
    return 0;
}
""", tmp_path, *library)
    timed = {}
    for line in out.splitlines():
        name, kernel = line.split()
        timed.setdefault(name, set()).add(kernel)
    assert timed["y_plan"] == {"yinv", "yfwd"}
    assert timed["zf_plan"] == {"zinv_curl", "zfwd"}
