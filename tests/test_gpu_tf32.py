"""The FP32 correlation on the tensor cores (operands split into two TF32 parts): every score
within the error bound that the selection's band uses, on ragged sizes around its tiles (128
atoms, 16 to 256 signals, 32 columns of n, rows that are and are not 16-byte multiples), no
less accurate than an FP32 chain over n, and infinite or NaN where the FP32 product is."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import mpl

pytestmark = pytest.mark.gpu


def _noalloc(At, R):
    import torch
    m, n = At.shape
    p = R.shape[0]
    C = torch.full((p, m), float("nan"), device="cuda")
    rc = mpl.mpl_correlate_noalloc(torch.from_numpy(At).cuda(), n, m, torch.from_numpy(R).cuda(), p, C)
    assert rc == mpl.MPL_OK
    torch.cuda.synchronize()
    return C.cpu().numpy()


def _data(n, m, p, seed):
    rng = np.random.default_rng(seed)
    At = rng.standard_normal((m, n)).astype(np.float32)
    At /= np.linalg.norm(At, axis=1, keepdims=True)
    return At, (rng.standard_normal((p, n)) * 0.3).astype(np.float32)


# (n just below the kernel's first size takes the chain)
SHAPES = [(127, 300, 20), (128, 1, 9), (128, 128, 16), (129, 127, 17), (130, 129, 255), (160, 257, 256),
          (161, 1000, 257), (255, 513, 272), (256, 128, 1000), (777, 6001, 99), (1000, 2050, 130), (2044, 32771, 33),
          (4096, 640, 513), (8193, 150, 40)]


@pytest.mark.parametrize("n,m,p", SHAPES)
def test_within_bound_of_fp64(n, m, p):
    At, R = _data(n, m, p, 3 * n + m + p)
    C = _noalloc(At, R).astype(np.float64)
    exact = R.astype(np.float64) @ At.astype(np.float64).T
    absdot = np.abs(R.astype(np.float64)) @ np.abs(At.astype(np.float64)).T
    tf = 98.0 * 2.0 ** -22 + (n / 32.0 + 2.0) * 2.0 ** -24
    assert np.all(np.abs(C - exact) <= tf * absdot)
    # and far below it on average: a stale tile or a lost low part would be off by 2^-11
    assert np.linalg.norm(C - exact) <= 2.0 ** -19 * np.linalg.norm(exact)


@pytest.mark.parametrize("n", [128, 200, 512, 1024, 4096])
def test_no_less_accurate_than_an_fp32_chain(n):
    """2-norm of the error against FP64, beside that of one FP32 accumulation chain per score."""
    At, R = _data(n, 512, 48, n)
    C = _noalloc(At, R).astype(np.float64)
    exact = R.astype(np.float64) @ At.astype(np.float64).T
    acc = np.zeros((48, 512), dtype=np.float64)
    for k in range(n):  # fused multiply-add: one rounding per term
        acc = (acc + R[:, k].astype(np.float64)[:, None] * At[:, k].astype(np.float64)[None, :])
        acc = acc.astype(np.float32).astype(np.float64)
    assert np.linalg.norm(C - exact) <= np.linalg.norm(acc - exact)


@pytest.mark.parametrize("n,m,p", [(256, 300, 40), (333, 130, 300)])
def test_non_finite_values(n, m, p):
    At, R = _data(n, m, p, n)
    R[3, 5] = np.inf
    R[7, n - 1] = -np.inf
    R[8, 0] = np.nan
    At[10, 2] = np.inf
    At[11, 1] = np.nan
    At[12, 7] = 0.0
    R[9, 7] = np.inf           # 0 * inf at atom 12
    At[13, 4], R[17, 4] = 2.0 ** -100, 3.4e38  # finite, but rounding it to TF32 is not
    with np.errstate(invalid="ignore", over="ignore"):
        exact = (R.astype(np.float64)[:, None, :] * At.astype(np.float64)[None, :, :]).sum(axis=2)
    C = _noalloc(At, R)
    fin = np.isfinite(exact) & (np.abs(exact) < 1e38)
    np.testing.assert_array_equal(np.isnan(C), np.isnan(exact))
    np.testing.assert_array_equal(C[np.isinf(exact)], exact[np.isinf(exact)].astype(np.float32))
    assert np.all(np.isfinite(C[fin]))
    np.testing.assert_allclose(C[fin], exact[fin], rtol=2e-5, atol=2e-5)
    # rows and columns without such values are untouched by them
    At2, R2 = _data(n, m, p, n)
    clean = np.ix_([i for i in range(p) if i not in (3, 7, 8, 9, 17)], [j for j in range(m) if j not in (10, 11, 12, 13)])
    np.testing.assert_array_equal(C[clean], _noalloc(At2, R2)[clean])


@pytest.mark.parametrize("n,m,p", [(130, 20000, 128), (192, 20001, 65), (225, 39000, 16), (256, 20100, 129),
                                   (161, 20000, 257), (300, 19999, 512)])
def test_several_tiles_per_block(n, m, p):
    """Up to 128 signals, and more where their tiles run side by side, take three stages: slices that are
    2, 0 and 2 modulo 3, so that consecutive
    tiles of a block start in different stages; the others take the wide kernel's two.  Bound as above."""
    At, R = _data(n, m, p, n + m + p)
    C = _noalloc(At, R).astype(np.float64)
    exact = R.astype(np.float64) @ At.astype(np.float64).T
    absdot = np.abs(R.astype(np.float64)) @ np.abs(At.astype(np.float64)).T
    tf = 98.0 * 2.0 ** -22 + (n / 32.0 + 2.0) * 2.0 ** -24
    assert np.all(np.abs(C - exact) <= tf * absdot)
    assert np.linalg.norm(C - exact) <= 2.0 ** -19 * np.linalg.norm(exact)
