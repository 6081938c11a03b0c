"""Sign-fixing where the inner products that decide it are far below the rounding
of an FP32 sum: the signs must be those of the exact products (sgn(0) = +1), at
row counts around the slices a block's threads take."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 5, 16, 31])
@pytest.mark.parametrize("d", [64, 257, 1024])
def test_sign_of_nearly_orthogonal_columns(gpu_lib, d, k):
    rng = np.random.default_rng(d + k)
    m = 5
    Z = rng.standard_normal((m, d, k)).astype(np.float32).astype(np.float64)
    h = d // 2
    Z[0, h:2 * h] = Z[0, :h]
    Z[0, 0] = Z[0, h] = 1.0
    for i in range(1, m):
        for j in range(k):
            # the products cancel in pairs but for 2^-24 of either sign; or they are all zero
            Z[i, h:2 * h, j] = -Z[i, :h, j]
            Z[i, 2 * h:, j] = 0.0
            Z[i, 0, j], Z[i, h, j] = [(0.0, 0.0), (1.0, -1.0 + 2.0 ** -24), (1.0 - 2.0 ** -24, -1.0)][(i + j) % 3]
            if (i + j) % 3 == 0:
                Z[i, :, j] = 0.0
    Z32 = Z.astype(np.float32).astype(np.float64)
    dots = np.array([[float(np.sum([np.longdouble(a) * np.longdouble(b) for a, b in zip(Z32[i, :, j], Z32[0, :, j])]))
                      for j in range(k)] for i in range(m)])
    ctx = B.lp_create(0)
    try:
        _, D = B.lp_align_aggregate(ctx, "sign", 0, np.ones(m) / m, Z, Z)
    finally:
        B.lp_destroy(ctx)
    for i in range(1, m):
        assert np.array_equal(np.diag(D[i]), np.where(dots[i] < 0, -1.0, 1.0))
