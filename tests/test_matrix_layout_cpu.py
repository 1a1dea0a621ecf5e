"""The sliced layout of matrices whose rows are strips, not lines (detector
response, wide bins): ``tests/host/ray_packs_check.cpp`` builds it with the
library's own host code and unpacks it again."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.sparse as sp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_13344_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


def strips(n, angles, bins, spacing, width):
    """CSR of parallel strips `width` pixels wide, `spacing` apart."""
    r, c = np.divmod(np.arange(n * n), n)
    x, y = c + 0.5 - n / 2, r + 0.5 - n / 2
    rows, cols = [], []
    for a in range(angles):
        th = np.pi * (a + 0.3) / angles
        pos = -x * np.sin(th) + y * np.cos(th)
        for b in range(bins):
            at = np.nonzero(np.abs(pos - (b - (bins - 1) / 2) * spacing) <= width / 2)[0]
            rows.append(np.full(len(at), a * bins + b))
            cols.append(at)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    val = (0.1 + (rows * 7 + cols * 3) % 11 / 16.0).astype(np.float32)
    return sp.csr_matrix((val, (rows, cols)), shape=(angles * bins, n * n))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    out = str(tmp_path_factory.mktemp("host") / "ray_packs_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", CUDA_INC, os.path.join(ROOT, "tests", "host", "ray_packs_check.cpp"),
                    os.path.join(CSRC, "csr_host.cpp"), "-o", out], check=True)
    return out


def check(exe, tmp_path, A, n, angles):
    with open(tmp_path / "in.bin", "wb") as f:
        np.array([n, angles, A.shape[0], A.nnz], np.int32).tofile(f)
        A.indptr.astype(np.int32).tofile(f)
        A.indices.astype(np.int32).tofile(f)
        A.data.astype(np.float32).tofile(f)
    out = subprocess.run([exe, str(tmp_path / "in.bin")], check=True, capture_output=True,
                         text=True).stdout
    assert out.split("\n")[:4] == [f"{lanes} 1 0" for lanes in (1, 2, 4, 8)]


@pytest.mark.parametrize("n", [256, 512])
@pytest.mark.parametrize("width", [8, 16, 24, 31, 32, 33, 48])
def test_wide_rows_fit_the_sliced_layout(exe, tmp_path, n, width):
    # one shallow and one steep angle among four; some rows empty or ragged
    A = strips(n, 4, 9, n / 7, width)
    A.sort_indices()
    check(exe, tmp_path, A, n, 4)


def test_unsorted_and_empty_rows(exe, tmp_path):
    A = strips(60, 6, 21, 5.0, 2)
    A.sort_indices()
    rng = np.random.default_rng(3)
    for i in range(0, A.shape[0], 2):
        s, e = A.indptr[i], A.indptr[i + 1]
        turn = rng.permutation(e - s)
        A.indices[s:e] = A.indices[s:e][turn]
        A.data[s:e] = A.data[s:e][turn]
    check(exe, tmp_path, A, 60, 6)
