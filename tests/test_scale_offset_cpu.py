"""The offset at which the tensor-core quantiser stores a row's scales, computed on the host by the kernels' own function."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_20586_b200", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "quant_math.cuh"
int main() {
    for (uint32_t tile : {0u, 1u, (1u << 23) - 1u, 1u << 23, (1u << 24) - 1u, (1u << 29) - 1u})
        for (uint32_t row : {0u, 7u, 31u, 32u, 127u})
            printf("%u %u %llu %lld\n", tile, row, (unsigned long long)mx::sf_row_offset(tile, row / 32u, row % 32u),
                   (long long)mx::sf_native_offset(row, 4ll * tile, 1ll << 29));
}
"""


def test_scale_rows_beyond_four_gigabytes(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "offsets.cu", tmp_path / "offsets"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(lines) == 30
    for line in lines:
        tile, row, got, native = map(int, line.split())
        assert got == native == tile * 512 + row % 32 * 16 + row // 32 * 4, (tile, row)
