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


SIGNATURES = HEAD + r"""
int main()
{
    const double L[3] = {1.0, 1.0, 1.0};
    const int n[][3] = {%s};
    for (auto& m : n) {
        flusi_t h = nullptr;
        if (flusi_create(m[0], m[1], m[2], L, 0.01, 1e-2, %s, &h) != FLUSI_OK) return 1;
        for (int y = 0; y < 3; ++y)
            for (int z = 0; z < 3; ++z)
                for (int x = 0; x < 2; ++x) {
                    flusi_tuning t{};
                    t.y_plan = y, t.zf_plan = z, t.x_kernel = x;
                    if (flusi_set_tuning(h, &t) != FLUSI_OK) return 2;
                    printf("%%d %%d %%d %%d %%d %%d %%s\n", m[0], m[1], m[2], y, z, x, tuning_signature(h).c_str());
                }
        flusi_destroy(h);
    }
    return 0;
}
"""


def _signatures(library, tmp_path, grids, prec):
    text = SIGNATURES % (", ".join("{%d, %d, %d}" % g for g in grids), prec)
    out = {}
    for line in program_output(text, tmp_path, *library).splitlines():
        *k, sig = line.split()
        k = tuple(map(int, k))
        out[k[:3], k[3:]] = sig
    return out


def test_two_pass_and_staged_kernels_are_told_apart(library, tmp_path):
    """At 64, 192, 384 and 512 rows plans 0 and 1 have the same radices; in FP32
    plan 1 runs the two-pass kernels and plan 0 the staged ones."""
    grids = [(96, n, n) for n in (64, 192, 384, 512)]
    sig = _signatures(library, tmp_path, grids, "FLUSI_FP32")
    for g in grids:
        assert sig[g, (0, 1, 0)] != sig[g, (1, 1, 0)] and sig[g, (1, 0, 0)] != sig[g, (1, 1, 0)], g
        assert sig[g, (1, 1, 0)] != sig[g, (1, 1, 1)], g
        # the staged kernels with the same radices stay one setting
        if sig[g, (0, 0, 0)].split(",")[:2] == sig[g, (2, 2, 0)].split(",")[:2] and g[1] in (64, 512):
            assert sig[g, (0, 0, 0)] == sig[g, (2, 2, 0)], g
    # without two-pass kernels (FP64; 48 and 729 rows), equal radices are one setting
    sig = _signatures(library, tmp_path, [(96, 512, 64)], "FLUSI_FP64")
    assert sig[(96, 512, 64), (0, 0, 0)] == sig[(96, 512, 64), (1, 1, 0)] == sig[(96, 512, 64), (2, 2, 0)]
    sig = _signatures(library, tmp_path, [(96, 48, 729)], "FLUSI_FP32")
    assert sig[(96, 48, 729), (1, 0, 0)] == sig[(96, 48, 729), (1, 1, 0)]


def test_cache_lines_belong_to_one_build(library, tmp_path):
    """Which setting is best depends on the kernels, so a line of another build
    does not apply: the key ends in the library's source hash."""
    out = program_output(HEAD + r"""
int main()
{
    const double L[3] = {1.0, 1.0, 1.0};
    flusi_t h = nullptr;
    if (flusi_create(96, 64, 512, L, 0.01, 1e-2, FLUSI_FP32, &h) != FLUSI_OK) return 1;
    printf("%s\n", tuning_key(h).c_str());
    return flusi_destroy(h);
}
""", tmp_path, *library)
    from conftest import build_flusi
    build_flusi()
    from paper_1506_06513_gb300 import _build
    key = out.strip()
    assert "96x64x512|fp32|ab2|nowake" in key and " " not in key
    assert key.split("|")[-1] == _build.source_hash()
