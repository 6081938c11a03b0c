"""lp_orth where many blocks take one CTA each (FP64 k x k work, and FP32 at k <= 8) or
larger clusters than few blocks would: the sums keep their order, so every block has the
bits that it has in a small batch (rows around whole rounds of the 85 or 25 FP64 slices
and the rows widened at a time, limits of the choice in blocks and rows, rows that fill
shared memory).

Tolerances against the FP64 factorisation as for the clusters, k 2^-20, on blocks with
four times as many rows as columns (square Gaussian blocks are not well-conditioned)."""
import numpy as np
import pytest

import oracle as O
from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = 32 * 2.0 ** -20


@pytest.mark.parametrize("k,d,batch", [
    (8, 8, 81), (1, 33, 183), (5, 84, 300), (8, 85, 153), (7, 86, 101), (5, 255, 92), (8, 257, 200), (3, 384, 92),
    (5, 385, 122), (8, 512, 152), (5, 1_408, 201), (5, 1_025, 149), (8, 2_600, 122), (6, 3_800, 152), (6, 4_200, 152),
    (16, 16, 183), (9, 24, 200), (16, 25, 190), (12, 26, 183), (13, 126, 183), (16, 384, 183), (10, 448, 251),
    (16, 768, 151), (11, 1_000, 152), (16, 2_250, 129), (16, 2_400, 151),
    (32, 4_300, 24), (20, 4_000, 24), (16, 6_000, 40), (7, 12_000, 40)])
def test_many_fp64_blocks_have_the_bits_of_few(gpu_lib, k, d, batch):
    _many_and_few(k, d, batch, True)


@pytest.mark.parametrize("k,d,batch", [
    (8, 8, 600), (5, 1_024, 153), (5, 1_025, 77), (3, 3_072, 153), (8, 3_073, 153), (8, 5_120, 77), (5, 5_121, 100),
    (5, 4_272, 250), (5, 4_000, 170), (16, 2_500, 153), (12, 4_200, 100), (32, 1_500, 153), (20, 2_300, 80)])
def test_many_fp32_blocks_have_the_bits_of_few(gpu_lib, k, d, batch):
    _many_and_few(k, d, batch, False)


def _many_and_few(k, d, batch, fp64):
    import torch
    g = torch.Generator(device="cuda").manual_seed(d + k)
    mix = torch.eye(k, dtype=torch.float64, device="cuda") + 0.1 / k
    Y = torch.randn(batch, d, k, dtype=torch.float64, device="cuda", generator=g) @ mix
    torch.cuda.synchronize()
    ctx = B.lp_create(0)
    try:
        Z = B.lp_orth(ctx, Y, kxk_fp64=fp64)
        few = torch.cat([B.lp_orth(ctx, y.contiguous(), kxk_fp64=fp64) for y in Y.split(20)])
    finally:
        B.lp_destroy(ctx)
    assert torch.equal(Z, few)
    for b in (0, batch - 1) if d >= 4 * k else ():
        z, y = Z[b].cpu().numpy(), Y[b].cpu().numpy()
        assert np.abs(z.T @ z - np.eye(k)).max() < TOL
        assert np.abs(z - O.orth(y)).max() < TOL
