"""Which output buffers the kernels store to directly: plain memory of the current device.
Another device's memory, managed and host memory are written by copies.  Host code of
csrc/emb_internal.cuh, run without a GPU."""
from __future__ import annotations

import os
import subprocess

import pytest

from paper_2512_01251_gb300 import build as B

MAIN = r"""
#include <stdio.h>
#include "emb_internal.cuh"
int main()
{
    const cudaMemoryType type[] = {cudaMemoryTypeDevice, cudaMemoryTypeManaged, cudaMemoryTypeHost, cudaMemoryTypeUnregistered};
    for (int t = 0; t < 4; ++t)
        for (int dev = 0; dev < 3; ++dev)
            for (int here = 0; here < 3; ++here) {
                cudaPointerAttributes a = {};
                a.type = type[t];
                a.device = dev;
                printf("%d %d %d %d\n", t, dev, here, (int)emb_plain_device(a, here));
            }
}
"""


def test_only_memory_of_the_current_device_is_stored_to(tmp_path):
    if not os.path.exists(B.NVCC):
        pytest.skip("nvcc not available")
    src = tmp_path / "view.cu"
    src.write_text(MAIN)
    exe = str(tmp_path / "view")
    subprocess.check_call([B.NVCC, *B.ARCH, "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.HERE, "..", "include"),
                           "-diag-suppress", "177", "-o", exe, str(src)])
    rows = [[int(x) for x in r.split()] for r in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 36
    for t, dev, here, direct in rows:
        assert direct == (t == 0 and dev == here)
