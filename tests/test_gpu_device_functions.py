"""Device functions of the library alone, through tests/device_checks.cu (built here with the
library's own flags), where the entry points cannot reach the cases that matter."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1904_04825_gb300 import _build as B
    out = str(tmp_path_factory.mktemp("dev") / "device_checks.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_checks.cu")
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", src, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


def _inverse(dev, M):
    out = np.empty_like(M)
    D = ctypes.POINTER(ctypes.c_double)
    assert dev.fp64_inverse(len(M), np.ascontiguousarray(M).ctypes.data_as(D), out.ctypes.data_as(D)) == 0
    return out


def _exact_inverse(M):
    """Gauss-Jordan in extended precision, pivots by scaled rows."""
    n, A = len(M), np.concatenate([M, np.eye(len(M))], 1).astype(np.longdouble)
    for c in range(n):
        q = c + int(np.argmax(np.abs(A[c:, c]) / np.abs(A[c:, :n]).max(1)))
        A[[c, q]] = A[[q, c]]
        A[c] /= A[c, c]
        f = A[:, c].copy()
        f[c] = 0
        A -= f[:, None] * A[c]
    return A[:, n:]


@pytest.mark.parametrize("n", [36, 40, 64, 100, 135, 144])
def test_fp64_block_inverse_at_every_width(dev, n):
    """Widths whose rows, two threads each up to 100, end inside a warp and whose last panel is 4, 7, 8
    or 16 columns wide.  M = 4 I + G, G of entries N(0, 1/n): cond below 10, so n u cond = 144 * 1.1e-16
    * 10 = 1.6e-13 per entry, relative to the largest."""
    M = 4.0 * np.eye(n) + np.random.default_rng(n).standard_normal((n, n)) / np.sqrt(n)
    want = _exact_inverse(M)
    assert np.abs(_inverse(dev, M) - want).max() < 1.6e-13 * np.abs(want).max()


@pytest.mark.parametrize("nblk", [1, 2, 19, 32])
def test_grid_barrier_over_the_wrap_of_its_counter(dev, nblk):
    """The counter of a long solve wraps: rounds that begin at zero, below 2^32 and below 2^31 (where
    the difference of signed values would turn) all separate the notes before from those behind, and
    carry the done bit."""
    for start in (0, 2**32 - 40 * nblk, 2**31 - 40 * nblk):
        assert dev.check_barrier(nblk, ctypes.c_uint(start), 60) == 0
