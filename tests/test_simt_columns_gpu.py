"""The FP32 step's second pass with four threads to four columns of A: widths around its
groups of four and of 512 columns, ranks in each padded size, rows around the 8- and 16-row
tiles, several partitions and segments a block, and rows with a pitch above d."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 33, 130, 511, 513, 766, 1021, 1024])
@pytest.mark.parametrize("k", [1, 8, 11, 16, 17, 32])
@pytest.mark.parametrize("sizes", [[32], [47, 33], [5_003, 100, 64]])
def test_step_against_fp64(gpu_lib, d, k, sizes):
    import torch
    g = torch.Generator(device="cuda").manual_seed(d * 37 + k)
    A = torch.randn(sum(sizes), d, device="cuda", generator=g)
    z = np.linalg.qr(np.random.default_rng(k).standard_normal((len(sizes), d, k)))[0]
    torch.cuda.synchronize()
    with B.LocalPower(list(A.split(sizes)), dtype="f32") as lp:
        got = torch.from_numpy(lp.power_step(k, z, shared=False)).cuda()
    for i, a in enumerate(A.double().split(sizes)):
        zi = torch.from_numpy(z[i]).cuda()
        # FP32 sums of d products, then of the rows: each within (terms) 2^-24 of the absolute sums,
        # and Z's own rounding
        bound = (d + sizes[i] + 4) * 2.0 ** -24 * (a.abs().T @ (a.abs() @ zi.abs())) / sizes[i]
        assert bool(((got[i] - a.T @ (a @ zi) / sizes[i]).abs() <= bound).all())
