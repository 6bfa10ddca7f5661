"""Active sets above the host's bound on |S|, which picks the kernels of the master problems and sizes
the grid of the Gram growth: reported (MPL_ERR_CUDA in a solve), not passed over.  Sets within the
bound are worked on beside them.  Bounds at every variant: 24 and 32 (a warp per signal), 64, 96 and
128 (registers), 200 (shared memory) and 300 (streamed)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1302_5010_gb300 import build as libbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
DERR_SHAPE = 3


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("bound") / "libbound.so")
    objs = [os.path.join(libbuild.BUILD, os.path.basename(s)[:-3] + ".o") for s in libbuild._sources()]
    subprocess.run([libbuild.nvcc(), *libbuild.ARCH, *libbuild.NVCC_FLAGS, "-I", libbuild.INCLUDE, "-shared", "-o", out,
                    os.path.join(HERE, "active_set_bound.cu"), *objs], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _run(lib, what, s0, s1, bound, smax):
    x, g = np.zeros((2, smax), dtype=np.float32), np.zeros((2, smax, smax), dtype=np.float32)
    err = lib.run_bound(what, s0, s1, bound, smax, x.ctypes.data_as(ctypes.c_void_p), g.ctypes.data_as(ctypes.c_void_p))
    return err, x, g


@pytest.mark.parametrize("bound", [24, 32, 64, 96, 128, 200, 300])
def test_master_problems(lib, bound):
    smax = 400
    want = np.maximum(np.arange(1, smax + 1) - 0.5, 0.0)  # identity block: the soft-thresholded h
    for s1 in (bound, smax):
        err, x, _ = _run(lib, 0, 5, s1, bound, smax)
        assert err == (0 if s1 <= bound else DERR_SHAPE)
        np.testing.assert_allclose(x[0, :5], want[:5], rtol=1e-4)
        if s1 <= bound:
            np.testing.assert_allclose(x[1, :s1], want[:s1], rtol=1e-4)
        else:
            assert not np.any(x[1])


@pytest.mark.parametrize("bound", [24, 64, 100])
def test_gram_growth(lib, bound):
    smax = 400
    for s1 in (bound, smax):
        err, _, g = _run(lib, 1, 5, s1, bound, smax)
        assert err == (0 if s1 <= bound else DERR_SHAPE)
        np.testing.assert_array_equal(g[0, :5, :5], np.eye(5))
        if s1 <= bound:
            np.testing.assert_array_equal(g[1, :s1, :s1], np.eye(s1))
