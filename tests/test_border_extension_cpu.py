"""The border extension of one axis: the form without a division against the general one and numpy's padding, at every
distance within three lengths of the axis (compiled for the host from the kernels' own header)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
INC = os.path.join(HERE, "..", "paper_2201_06174_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SRC = r"""
#include <cstdio>
#include "sal_internal.cuh"
int main() {
    for (int n = 1; n <= 19; ++n)
        for (int mode = 0; mode < 3; ++mode)
            for (int i = -3 * n; i < 4 * n; ++i)
                std::printf("%d %d %d %d %d\n", n, mode, i, sal::ext_index(i, n, mode), sal::ext_index_any(i, n, mode));
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_extension_without_a_division_is_the_general_one(tmp_path):
    src, exe = tmp_path / "ext.cu", tmp_path / "ext"
    src.write_text(SRC)
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-I", INC, "-I", os.path.join(HERE, "..", "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True, timeout=300)
    rows = np.loadtxt(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n"), dtype=int)
    assert np.array_equal(rows[:, 3], rows[:, 4])
    for n in (1, 2, 7, 19):
        for mode, pad in ((0, "symmetric"), (1, "wrap")):
            sel = rows[(rows[:, 0] == n) & (rows[:, 1] == mode)]
            assert np.array_equal(sel[:, 3], np.pad(np.arange(n), 3 * n, mode=pad))
        z = rows[(rows[:, 0] == n) & (rows[:, 1] == 2)]
        assert np.array_equal(z[:, 3], np.where((z[:, 2] >= 0) & (z[:, 2] < n), z[:, 2], -1))
