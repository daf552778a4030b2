"""Registers and spills of the kernels whose speed hangs on them, as the compiler reports them (no GPU needed)."""
import os
import re
import subprocess

import pytest

from __graft_entry__ import CSRC, NVCC_FLAGS

# kernel -> registers a thread may have for the CTAs per SM that were measured to be best; none of them spills
LIMITS = {
    "lightkv_fd": {
        "fd_stream_kernel<__nv_bfloat16, 1, 6, 2>": 64,        # sixteen CTAs of two warps
        "fd_stream_kernel<__nv_bfloat16, 2, 3, 2>": 72,        # fourteen
        "fd_stream_kernel<float, 2, 4, 2>": 96,                # ten
    },
    "lightkv_kernels": {
        "kv_compact_kernel<__nv_bfloat16, 256, 2, false>": 48,        # five CTAs of 256 threads
        "kv_compact_kernel<__nv_bfloat16, 512, 4, false>": 64,        # two of 512
        "kv_compact_kernel<float, 256, 2, false>": 64,                # four of 256
    },
}


@pytest.mark.parametrize("name", sorted(LIMITS))
def test_registers_and_spills(name, tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    log = subprocess.run([nvcc] + NVCC_FLAGS + ["-Xptxas", "-v", "-cubin", "-o", str(tmp_path / "out.cubin"),
                                                os.path.join(CSRC, name + ".cu")],
                         check=True, stdout=subprocess.PIPE, stderr=subprocess.STDOUT).stdout.decode()
    log = subprocess.run(["c++filt"], input=log.replace("'_Z", "' _Z"), check=True, capture_output=True, text=True).stdout
    found = {}
    for kernel, report in re.findall(r"Compiling entry function '\s*(.*?)' for(.*?Used \d+ registers)", log, re.S):
        found[kernel] = (int(re.search(r"Used (\d+) registers", report).group(1)),
                         int(re.search(r"(\d+) bytes spill loads", report).group(1)))
    for kernel, limit in LIMITS[name].items():
        (registers, spilled), = [v for k, v in found.items() if "lkv::" + kernel + "(" in k]
        assert registers <= limit and spilled == 0, (kernel, registers, spilled)
