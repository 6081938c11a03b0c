"""A server that can run one request at a time gives each the whole chip: requests
that wait behind it (by the active limit or by the memory budget) do not make its
steps leave SMs to them.

One step of 9,728 x 1,024 BF16 is eight units a cluster on 76 clusters, 32 on a
quarter of them, so its kernel takes about twice as long when it makes room; the
factor allowed, 1.3, is far from both."""
import time

import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

N, D, K, M = 9_728, 1_024, 16, 4
FLAGS = B.LP_FLAG_TIMING


def _step_ms(srv, parts, y0, at_once):
    """Mean step-kernel time of each request, `at_once` submitted before the first is admitted."""
    out = []
    while len(out) < 5:
        ids = [srv.submit(parts, K, [4] * 8, "sign", y0, dtype="bf16", flags=FLAGS) for _ in range(at_once)]
        done, t0 = set(), time.time()
        while len(done) < len(ids):
            done.update(srv.progress())
            assert time.time() - t0 < 60
        for i in ids:
            st = srv.result(i)[2]
            out.append(st["ms_step_kernels"] / st["step_launches"])
    return out


@pytest.mark.parametrize("limit", ["max_active", "budget"])
def test_waiting_requests_do_not_narrow_the_running_one(gpu_lib, limit):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn(N, D, device="cuda", generator=g) * (0.97 ** torch.arange(D, device="cuda"))
    parts = [p.contiguous() for p in A.to(torch.bfloat16).split(N // M)]
    y0 = np.random.default_rng(4).standard_normal((D, K))
    torch.cuda.synchronize()
    with B.Server(max_active=1) as srv:
        _step_ms(srv, parts, y0, 1)
        alone = min(_step_ms(srv, parts, y0, 1))
        need = srv.query()["hbm_peak"]
    args = dict(max_active=1) if limit == "max_active" else dict(max_active=8, hbm_budget_bytes=need + need // 2)
    with B.Server(**args) as srv:
        waited = _step_ms(srv, parts, y0, 5)
    # the median: the last of the five has nothing behind it
    assert sorted(waited)[2] < 1.3 * alone, (waited, alone)
