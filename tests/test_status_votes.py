"""A kernel whose threads share tables or barriers leaves a failed step as a whole
block (block_leaves in csrc/common.cuh): the status word can be written while its
blocks start, and threads that leave on their own reading of it would strand the
rest.  Read from the sources; the GPU side is test_gpu_failed_state.py and
test_gpu_failed_sponge.py.
"""
import glob
import os
import re

from device_code import CSRC


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = f.read()
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\([^;{]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield os.path.basename(path), m.group(1), text[m.end():end]


def test_kernels_leave_whole():
    seen = []
    for where, name, body in _kernels():
        seen.append(name)
        alone = re.search(r"status\s*!=\s*0\s*\)\s*return", body)
        shares = re.search(r"__shared__|__syncthreads|\bsmem_raw\b|bar\.sync", body)
        assert not (alone and shares), f"{where}: {name} leaves thread by thread"
    assert {"k_xpass", "k_xpass_sq", "k_xline_phys", "k_ypass", "k_ycol", "k_zinv", "k_zcol_inv", "k_zupdate"} <= set(seen)
