"""Sign-fixing where the products of the columns' entries lie at or below FP32's
smallest numbers: the signs must be those of the exact inner products (sgn(0) = +1),
also where an FP32 sum has lost the terms that decide."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _columns(rng, d, kind):
    """x, y of d entries (FP32 values): kinds 0-2 are unit columns but for tiny terms, 3 random tiny products."""
    x, y = np.zeros(d), np.zeros(d)
    if kind == 3:
        x, y = rng.standard_normal((2, d)) * 2.0 ** -74.5
        x, y = x.astype(np.float32), y.astype(np.float32)
    else:
        x[0] = y[1] = 1.0
        few, one = [(0.4, -0.6), (-0.45, 0.7), (0.49, -1.6)][kind]
        e, f = np.sqrt(abs(few)) * 2.0 ** -74.5, np.sqrt(abs(one)) * 2.0 ** -74.5
        n = max(3, (d - 3) // 2)
        x[2:2 + n], y[2:2 + n] = e, np.sign(few) * e
        x[-1], y[-1] = f, np.sign(one) * f
    p = rng.permutation(d)
    return x[p].astype(np.float32).astype(np.float64), y[p].astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("k", [1, 4, 8, 12, 32])
@pytest.mark.parametrize("d", [6, 40, 257, 1024])
def test_sign_of_products_below_the_normal_range(gpu_lib, d, k):
    if k > d:
        pytest.skip("k exceeds d")
    rng = np.random.default_rng(d + k)
    m = 5
    Z = np.zeros((m, d, k))
    want = np.ones((m, k))
    for j in range(k):
        x, y = _columns(rng, d, (j + d) % 4)
        Z[0, :, j] = x
        for i in range(1, m):
            Z[i, :, j] = y * (1.0 if i % 2 else -1.0)
            dot = sum(Fraction(a) * Fraction(b) for a, b in zip(Z[i, :, j], Z[0, :, j]))
            want[i, j] = -1.0 if dot < 0 else 1.0
    ctx = B.lp_create(0)
    try:
        _, G = B.lp_align_aggregate(ctx, "sign", 0, np.ones(m) / m, Z, Z)
    finally:
        B.lp_destroy(ctx)
    for i in range(1, m):
        assert np.array_equal(np.diag(G[i]), want[i])
