"""A wait of the FP32 tensor-core correlation that runs out leaves no score unwritten: the entry point
without a handle returns before the kernel has run, so what it could not finish must show in
the result.  The kernel is built with a limit of 0.2 ms; 128 signals of 32768 entries with an infinity
each keep the accumulating warps of a block on a tile's chains for several milliseconds, and
the blocks that have a second tile (20480 atoms are 160 tiles, 152 or fewer blocks) give up on it.
Unlike a wait, the chains end by themselves, and so does every block."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1302_5010_gb300 import build as libbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
DERR_TIMEOUT = 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("tf32") / "libtf32_wait.so")
    subprocess.run([libbuild.nvcc(), *libbuild.ARCH, *libbuild.NVCC_FLAGS, "-I", libbuild.INCLUDE, "-shared", "-o", out,
                    os.path.join(HERE, "tf32_wait_limit.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _run(lib, A, R, C):
    import torch
    err = ctypes.c_int(-1)
    torch.cuda.synchronize()
    rc = lib.run_tf32(ctypes.c_void_p(A.data_ptr()), A.shape[1], A.shape[0], ctypes.c_void_p(R.data_ptr()), R.shape[0],
                      ctypes.c_void_p(C.data_ptr()), ctypes.byref(err))
    assert rc == 0
    return err.value


def test_unfinished_tiles_are_nan(lib):
    import torch
    n, m, p = 32768, 20480, 128
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(m, n, device="cuda", generator=g)
    R = torch.randn(p, n, device="cuda", generator=g)
    C = torch.full((p, m), 7.0e7, device="cuda")
    # the limit is no obstacle to finite inputs
    assert _run(lib, A, R, C) == 0
    ref = R[:4].double() @ A[:64].double().T
    assert (C[:4, :64].double() - ref).abs().max().item() < 1e-2
    assert int((C == 7.0e7).sum()) == 0
    C.fill_(7.0e7)
    R[:, 100] = float("inf")
    A[:, 100] = A[:, 100].abs() + 1.0
    assert _run(lib, A, R, C) == DERR_TIMEOUT
    assert int((C == 7.0e7).sum()) == 0, "scores that were never written"
    # a score is the infinity it should be, or NaN; the first tile of every block was finished
    assert bool((torch.isposinf(C) | torch.isnan(C)).all())
    assert bool(torch.isposinf(C).any()) and bool(torch.isnan(C).any())
    np.testing.assert_array_equal(torch.isnan(C).any(dim=0).cpu().numpy(), torch.isnan(C).all(dim=0).cpu().numpy())
