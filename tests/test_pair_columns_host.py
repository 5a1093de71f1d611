"""The complex back-substitution of the interpolation (csrc/qdt.cu) gives a right-hand column to a pair of lanes; the pairs
left over in a warp read a column too, and it must be one that their own warp writes (another warp may be writing
its columns at that moment). No GPU needed: the column choice is compiled for the host and every warp of every
count of right-hand sides is walked through."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def column(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("cols") / "pair_column_check.so")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o",
                    so, os.path.join(HERE, "cuda", "pair_column_check.cu")], check=True, capture_output=True)
    return ctypes.CDLL(so).pair_column


@pytest.mark.parametrize("threads", [256, 512])
def test_left_over_pairs_read_their_own_warps_columns(column, threads):
    for n_rhs in range(1, threads + 3):
        for q0 in range(0, n_rhs, threads // 2):
            for warp in range(threads // 32):
                first = q0 + 16 * warp
                if first >= n_rhs:
                    continue   # the whole warp leaves
                own = set(range(first, min(first + 16, n_rhs)))
                read = [column(q, n_rhs) for q in range(first, first + 16)]
                assert set(read) == own
                assert read[:len(own)] == sorted(own)
