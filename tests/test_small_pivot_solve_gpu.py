"""A start block whose FP32 Gram has a last pivot that is not positive in FP32 but
positive in FP64 (nearly dependent columns): the FP64 factor takes over and the
padded columns of the basis (k < K) have to stay zero, since the aggregation with
Procrustes aligners multiplies whole rows of K.

The blocks are chosen on the CPU by the same sums: rows fall into slices r mod S,
each summed row by row with fused FP32 multiply-adds, the slices added in a fixed
order.  Tolerance: the FP32 bar of a whole solve, 1e-6; the start's own error is
gone after 18 local steps across the spectrum's gap (at most 0.25 a step)."""
import numpy as np
import pytest

import oracle as O
import synth
from paper_2002_08014_gb300 import binding as B

pytestmark = pytest.mark.gpu

F32 = np.float32
D = 160


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F32)


def _gram(Y, K):
    P = np.zeros((len(Y), K), F32)
    P[:, :Y.shape[1]] = Y
    S = 256 // (K // 4) ** 2
    acc = np.zeros((S, K, K), F32)
    for r, row in enumerate(P):
        acc[r % S] = _fma(row[:, None], row[None, :], acc[r % S])
    s = np.zeros((4, K, K), F32)
    for q in range(S):
        s[q % 4] = s[q % 4] + acc[q]
    return (s[0] + s[1]) + (s[2] + s[3])


def _last_pivot(G, k, dtype):
    """Pivot k - 1 of the right-looking factorisation, or an earlier one that is not positive."""
    A = G[:k, :k].astype(dtype)
    for j in range(k - 1):
        if not A[j, j] > 0:
            return A[j, j]
        my = (A[j] * (dtype(1) / np.sqrt(A[j, j]))).astype(dtype)
        if dtype is F32:
            A[j + 1:, j + 1:] = _fma(-my[j + 1:, None], my[None, j + 1:], A[j + 1:, j + 1:])
        else:
            A[j + 1:, j + 1:] -= np.outer(my[j + 1:], my[j + 1:])
    return A[k - 1, k - 1]


def _block(k, seed):
    rng = np.random.default_rng(seed)
    Y = rng.standard_normal((D, k))
    Y[:, -1] = Y[:, :-1] @ rng.standard_normal(k - 1) / np.sqrt(k - 1) + 2e-4 * rng.standard_normal(D)
    return Y.astype(F32)


@pytest.mark.parametrize("agg", ["opt", "sign"])
@pytest.mark.parametrize("k,K,seeds", [(5, 8, (9, 16, 24)), (12, 16, (1, 2, 5)), (24, 32, (5, 19, 20))])
def test_solve_from_a_start_with_a_negative_fp32_pivot(gpu_lib, k, K, seeds, agg):
    sizes = [1_900, 2_100, 1_500]
    lam = np.concatenate([0.9 ** np.arange(k), 0.2 * 0.9 ** np.arange(k, D)])
    parts = synth.split_rows(synth.spiked_rows(sum(sizes), D, lam, 0.0, 7 + k, threads=4), sizes)
    for seed in seeds:
        Y0 = _block(k, seed)
        G = _gram(Y0, K)
        assert _last_pivot(G, k, F32) <= 0 and _last_pivot(G, k, np.float64) > 1e-9 * G.max()
        with B.LocalPower(parts, dtype="f32") as lp:
            B.lp_solve(lp.ctx, k, [3] * 6, agg, Y0.astype(np.float64), 0, 0)
            Z = B.lp_result(lp.ctx, D, k)[0]
        assert np.isfinite(Z).all()
        ref = O.localpower([p.astype(np.float64) for p in parts], k, [3] * 6, agg, Y0.astype(np.float64))["Z"]
        assert O.subspace_dist(Z, ref) < 1e-6
