"""A solve's Procrustes alignments take no longer than the launch on its own would lead one
to expect: started while the reduction before it still holds SMs, a launch of some more
CTAs than SMs is packed on the free ones, and FP64 ones then share a pipe.

182 partitions of 24 columns, k = 17: two aligning rounds cost the difference between the
solve with Procrustes and the one without; packed it was 4.2 times the solve without,
spread 2.2 times.  The limit, 3.2, lies between."""
import time

import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


def test_fp64_procrustes_in_a_solve_is_spread_over_the_chip(gpu_lib):
    import torch
    n, d, k, m = 11_418, 24, 17, 182
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn(n, d, device="cuda", generator=g)
    parts = [p.contiguous() for p in A.split([n // m + (j < n % m) for j in range(m)])]
    y0 = np.random.default_rng(3).standard_normal((d, k))
    torch.cuda.synchronize()
    best = {}
    for agg in ("identity", "opt"):
        with B.LocalPower(parts) as lp:
            ts = []
            for _ in range(20):
                t = time.perf_counter()
                B.lp_solve(lp.ctx, k, [4, 4], agg, y0, 0, B.LP_FLAG_KXK_FP64)
                B.lp_result(lp.ctx, d, k)
                ts.append(time.perf_counter() - t)
            best[agg] = min(ts)
    assert best["opt"] - best["identity"] < 3.2 * best["identity"], best
