"""Loading FP32 rows as hi/lo planes: aligned and unaligned rows, widths that are
not a multiple of the eight columns a thread converts, more partitions than one
launch takes, a source pitch wider than d, and partitions shorter than a thread
block's share, from host and from device memory."""
import numpy as np
import pytest

from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [8, 61, 64, 90, 257, 1024])
@pytest.mark.parametrize("m,rows", [(1, 1000), (3, 7), (130, 40), (257, 9)])
def test_planes_from_device_and_host_rows(gpu_lib, d, m, rows):
    import torch
    k = 4
    rng = np.random.default_rng(d + m)
    sizes = [rows + i % 3 for i in range(m)]
    A = rng.standard_normal((sum(sizes), d)).astype(np.float32)
    z = np.linalg.qr(rng.standard_normal((d, k)))[0]
    offs = np.concatenate([[0], np.cumsum(sizes)])
    host = [A[offs[i]:offs[i + 1]] for i in range(m)]
    dev = torch.from_numpy(A).cuda()
    torch.cuda.synchronize()
    out = []
    for parts in (host, [dev[offs[i]:offs[i + 1]] for i in range(m)]):
        with B.LocalPower(parts, dtype="f32_bf16x2") as lp:
            out.append(lp.power_step(k, z))
    assert np.array_equal(out[0], out[1])
    for i in range(m):
        a = host[i].astype(np.float64)
        # stored values within 2^-17 of a in either product, and the step's own rounding
        bound = 2e-5 * (np.abs(a).T @ (np.abs(a) @ np.abs(z))) / sizes[i]
        assert np.all(np.abs(out[1][i] - a.T @ (a @ z) / sizes[i]) <= bound)


def test_planes_from_pitched_device_rows(gpu_lib):
    import torch
    rng = np.random.default_rng(5)
    d, k, y0 = 100, 3, np.random.default_rng(6).standard_normal((100, 3))
    wide = rng.standard_normal((4000, 133)).astype(np.float32)
    dev = torch.from_numpy(wide).cuda()
    torch.cuda.synchronize()
    sizes = [1500, 2500]
    with B.Server() as srv:
        rid = srv.submit([dev[:1500], dev[1500:]], k, [2, 1], "sign", y0, dtype="f32_bf16x2", row_pitch=133, d=d)
        while rid not in srv.progress():
            pass
        Z, _, _ = srv.result(rid)
    parts = [np.ascontiguousarray(wide[:1500, :d]), np.ascontiguousarray(wide[1500:, :d])]
    assert [p.shape[0] for p in parts] == sizes
    with B.LocalPower(parts, dtype="f32_bf16x2") as lp:
        Zh, _, _ = lp.solve(k, [2, 1], "sign", y0, ritz=True)
    assert np.array_equal(Z, Zh)
