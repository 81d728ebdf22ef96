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


@pytest.mark.parametrize("nblk", [1, 2, 19, 32])
def test_grid_barrier_over_the_wrap_of_its_counter(dev, nblk):
    """The counter of a long solve wraps: rounds that begin at zero, below 2^32 and below 2^31 (where
    the difference of signed values would turn) all separate the notes before from those behind, and
    carry the done bit."""
    for start in (0, 2**32 - 40 * nblk, 2**31 - 40 * nblk):
        assert dev.check_barrier(nblk, ctypes.c_uint(start), 60) == 0
