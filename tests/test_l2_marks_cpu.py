"""Which launches of the tensor-core quantiser mark their input as the first to leave L2, by the library's own function."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_20586_b200", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "kernels.h"
static int marked(int n, long long rows, long long cols, bool layer, bool values = false) {
    mx::QuantArgs a[4] = {};
    float y;
    for (int v = 0; v < n; ++v) { a[v].rows = rows; a[v].cols = cols; a[v].layer = layer; a[v].y_out = values ? &y : nullptr; }
    return mx::quant_input_leaves_l2(a, n);
}
int main() {
    printf("%d %d %d ", marked(4, 4096, 3032, true), marked(4, 4096, 3040, true), marked(4, 65536, 65536, true));      // a layer: 125.7, 126.1 MB and more
    printf("%d %d ", marked(2, 4096, 8192, true), marked(2, 1024, 8192, true));                                        // dY's two views: 169.9, 42.5 MB
    printf("%d %d %d %d ", marked(1, 8192, 6056, false), marked(1, 8192, 6144, false), marked(1, 8192, 8192, false), marked(1, 8192, 8704, false));   // one view: 125.6, 127.4, 169.9, 180.5 MB
    printf("%d %d\n", marked(1, 8192, 6144, false, true), marked(2, 4096, 8192, false));                               // its values written; two views of no layer
}
"""


def test_input_marks(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "marks.cu", tmp_path / "marks"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["0", "1", "1", "1", "0", "0", "1", "1", "0", "0", "0"]
