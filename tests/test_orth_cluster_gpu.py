"""lp_orth where the block's rows change how they are dealt to the CTAs of a
cluster (thresholds of d per padded k, fewer rows than slices, rows beyond shared
memory) and where the FP32 Cholesky hands over to the FP64 one.

Tolerances: the second CholQR pass starts from a basis whose Gram is within
d u32 of the identity, so Z^T Z - I is a few d-term FP32 sums of entries of size
1/d off, well below k 2^-20 (3e-5 at k = 32); Z itself differs from the FP64
factorisation by the FP32 triangular solve's backward error, a few k u32 times the
condition number of the columns scaled to norm one (below 4 here)."""
import numpy as np
import pytest

import oracle as O
from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = 32 * 2.0 ** -20


def _orth(Y, fp64):
    ctx = B.lp_create(0)
    try:
        return B.lp_orth(ctx, Y, kxk_fp64=fp64)
    finally:
        B.lp_destroy(ctx)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("d", [33, 128, 129, 256, 257, 513, 1024, 2049])
def test_orth_over_cluster_sizes(gpu_lib, d, k, fp64):
    rng = np.random.default_rng(1000 * d + k)
    Y = rng.standard_normal((3, d, k)) @ (np.eye(k) + 0.1 * rng.standard_normal((k, k)) / np.sqrt(k))
    Z = _orth(Y, fp64)
    for b in range(3):
        assert np.abs(Z[b].T @ Z[b] - np.eye(k)).max() < TOL
        assert np.abs(Z[b] - O.orth(Y[b])).max() < TOL


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("d,k", [(8, 8), (5, 1), (32, 32), (9000, 32), (20011, 16)])
def test_orth_few_rows_and_rows_beyond_shared_memory(gpu_lib, d, k, fp64):
    rng = np.random.default_rng(d + k)
    Y = np.linalg.qr(rng.standard_normal((d, k)))[0] @ np.triu(np.ones((k, k)) * 0.1 + np.eye(k))
    Z = _orth(Y[None], fp64)[0]
    assert np.abs(Z.T @ Z - np.eye(k)).max() < TOL
    assert np.abs(Z - O.orth(Y)).max() < TOL


@pytest.mark.parametrize("d,k", [(100, 5), (1024, 16), (700, 32)])
def test_orth_small_pivot_takes_the_fp64_factor(gpu_lib, d, k):
    """The last column 1,500 times shorter: its pivot, 4.4e-7 of the largest
    diagonal entry, is below the FP32 factorisation's floor of 1e-6."""
    rng = np.random.default_rng(d)
    U = O.orth(rng.standard_normal((d, k)))
    scale = np.ones(k)
    scale[-1] = 1.0 / 1500.0
    Z = _orth((U * scale)[None], False)[0]
    assert np.abs(Z.T @ Z - np.eye(k)).max() < TOL
    assert np.abs(Z - U).max() < TOL
