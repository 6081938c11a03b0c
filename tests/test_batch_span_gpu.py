"""A batch's short steps take several row ranges a cluster, so that several groups share
the chip.  Only the grid changes: every instance, each a group of its own, equals the solve
on a context of its own bit for bit, for row ranges that do not divide by the span, fewer
tiles than clusters, two planes and padded rows, and groups of one and of several units."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

# (partition sizes, d, k, dtype): 1, 2, 5, 73 and all ranges of the grid, and steps too long to share
SHAPES = [([100], 64, 4, "bf16"), ([129, 100], 90, 16, "bf16"), ([70] * 9, 256, 8, "f32_bf16x2"),
          ([4_000, 5_301], 128, 32, "bf16"), ([9_000, 12_345, 64], 181, 12, "bf16"), ([30_001], 1024, 5, "bf16")]


@pytest.mark.parametrize("count", [2, 3, 6])
def test_batch_steps_equal_the_lone_solve(gpu_lib, count):
    import torch
    data = []
    for i, (sizes, d, k, dtype) in enumerate(SHAPES[:count] if count > 2 else SHAPES[3:5]):
        g = torch.Generator(device="cuda").manual_seed(i)
        A = torch.randn(sum(sizes), d, device="cuda", generator=g) * (0.9 ** torch.arange(d, device="cuda"))
        parts = [p.contiguous() for p in (A if dtype != "bf16" else A.to(torch.bfloat16)).split(sizes)]
        data.append((parts, k, np.random.default_rng(i).standard_normal((d, k)), dtype))
    torch.cuda.synchronize()
    with B.Batch() as bt:
        for parts, k, y0, dtype in data:
            bt.add(parts, k, [4, 2, 1], "sign", y0, dtype=dtype, flags=0)
        for _ in range(2):
            bt.solve()
            got = [bt.result(i)[0] for i in range(len(data))]
            for z, (parts, k, y0, dtype) in zip(got, data):
                with B.LocalPower(parts, dtype=dtype) as lp:
                    assert np.array_equal(z, lp.solve(k, [4, 2, 1], "sign", y0, ritz=False)[0])
