"""One solve launched in every form gives the same bits: dependent launches that overlap
(captured and one by one), separated launches (timed), and through the server, directly and,
with a schedule of more launches than a stream takes, as a graph; on every step kernel,
including shapes whose clusters own several pieces of several partitions."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

CASES = [("f32", 100, 5, [900, 1_100]), ("f32", 1024, 16, [700, 333, 90]), ("f32", 300, 24, [5_000]),
         ("bf16", 362, 8, [40] * 50 + [20_011]), ("bf16", 2048, 32, [1_500, 129]),
         ("f32_bf16x2", 1024, 16, [5_003, 200]), ("e4m3", 700, 12, [3_001, 64])]


@pytest.mark.parametrize("dtype,d,k,sizes", CASES)
@pytest.mark.parametrize("agg", ["sign", "opt"])
def test_forms_of_one_solve(gpu_lib, dtype, d, k, sizes, agg):
    import torch
    g = torch.Generator(device="cuda").manual_seed(d)
    A = torch.randn(sum(sizes), d, device="cuda", generator=g) * (0.95 ** torch.arange(d, device="cuda"))
    scales = None
    if dtype == "bf16":
        A = A.to(torch.bfloat16)
    elif dtype == "e4m3":
        s = A.abs().amax(1) / 448
        A, scales = (A / s[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), list(s.split(sizes))
    parts = [p.contiguous() for p in A.split(sizes)]
    y0 = np.random.default_rng(k).standard_normal((d, k))
    torch.cuda.synchronize()
    for schedule in ([3, 2, 1, 1], [1] * 300 if d == 100 else [2]):
        out = []
        for flags in (0, B.LP_FLAG_NO_GRAPH, B.LP_FLAG_TIMING, B.LP_FLAG_TIMING | B.LP_FLAG_NO_GRAPH):
            with B.LocalPower(parts, dtype=dtype, row_scales=scales) as lp:
                B.lp_solve(lp.ctx, k, schedule, agg, y0, 1, flags)
                out.append(B.lp_result(lp.ctx, d, k)[0])
        with B.Server() as srv:
            ids = [srv.submit(parts, k, schedule, agg, y0, dtype=dtype, row_scales=scales, refine_rounds=1, flags=0)
                   for _ in range(3)]
            done = set()
            while len(done) < 3:
                done.update(srv.progress())
            out += [srv.result(i)[0] for i in ids]
        assert all(np.array_equal(out[0], o) for o in out[1:])
