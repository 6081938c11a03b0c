"""The pass-split step with ring slots of half a unit (64 columns): where they are chosen
(a short ring, or many units a tile) against the ring of whole units that a set ring size
asks for.  Both add the same products in the same order, so the results are equal bit for
bit: one partition and several a cluster, tiles of one row, widths whose last unit has one
64-column chunk or part of one, fewer tiles than clusters and several segments a cluster."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,k,dtype", [(1024, 32, "bf16"), (724, 20, "bf16"), (961, 17, "bf16"), (1024, 4, "bf16"),
                                       (362, 16, "f32_bf16x2"), (448, 3, "f32_bf16x2"), (1000, 12, "f32_bf16x2")])
@pytest.mark.parametrize("sizes", [[32], [129], [2049, 33, 1000], [40] * 90, [12_000, 9_001]])
def test_half_unit_slots(gpu_lib, d, k, dtype, sizes):
    import torch
    g = torch.Generator(device="cuda").manual_seed(d + k)
    A = torch.randn(sum(sizes), d, device="cuda", generator=g)
    if dtype == "bf16":
        A = A.to(torch.bfloat16)
    parts = list(A.split(sizes))
    z = np.linalg.qr(np.random.default_rng(d).standard_normal((len(sizes), d, k)))[0]
    out = []
    torch.cuda.synchronize()
    for ring in (0, 8):  # 8: as many whole units as fit
        with B.LocalPower(parts, dtype=dtype) as lp:
            B.lp_set_tuning(lp.ctx, ring_units=ring, kernel="pair")
            out.append(lp.power_step(k, z, shared=False))
    assert np.array_equal(out[0], out[1])
    A64 = A.double()
    for i, a in enumerate(A64.split(sizes)):
        zi = torch.from_numpy(z[i]).cuda()
        bound = 2e-4 * (a.abs().T @ (a.abs() @ zi.abs())) / sizes[i]  # 2^-16 of |a| in W, FP32 sums
        assert bool(((torch.from_numpy(out[0][i]).cuda() - a.T @ (a @ zi) / sizes[i]).abs() <= bound).all())
