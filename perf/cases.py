"""Performance cases of the LocalPower library: what a user has it do, through
the public entry points of ``paper_2002_08014_gb300.binding``.

Kinds of case
  step     ``lp_power_step``: one fused local power step over every loaded
           partition (the hot operation of every solve), device tensors in and out
  orth     ``lp_orth``: the orthonormalisation of a batch of blocks
  solve    a whole solve on loaded partitions and its result
  refresh  new rows of the same shapes loaded into a context, then a solve (a
           loop that refreshes its data)
  batch    ``Batch``: many independent instances solved by one launch
  serve    ``Server``: a burst of requests admitted, solved and fetched

The rows are spiked Gaussian, a = U diag(sqrt(lam)) g + sigma e, with the
spectra of the workloads in ``synth.configs`` and of the benchmark's batching
and serving workloads, drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2002_08014_gb300 import binding as B

DEV = "cuda"
L2_BYTES = 129e6
ELEM = {"f32": 4, "f32_bf16x2": 4, "bf16": 2, "e4m3": 1}
# pool widths of the batching and serving workloads
WIDTHS = [64, 90, 128, 181, 256, 362, 512, 724, 1024]
# the serving workload's decaying schedule (with 3 refinement rounds)
SERVING = "4x10,2x10,1x60"


# --------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest call: the plain workload's step (the paper's smallest datasets), all latency
        dict(name="step_plain", kind="step", dtype="f32", n=4_000, d=100, k=5, m=4, shared=True),
        # the plain workload's whole solve: sign-fixing, p = 4, 20 rounds, Ritz vectors and singular values
        dict(name="solve_plain", kind="solve", dtype="f32", n=4_000, d=100, k=5, m=4, schedule="4x20", refine=0,
             agg="sign", ritz=True, kxk_fp64=False),
        # plain FP32 storage at the rounds workload's shape, every partition with its own basis (j > 1 of a round)
        dict(name="step_fp32", kind="step", dtype="f32", n=250_000, d=1024, k=16, m=64, shared=False),
        # plain FP32 storage, Procrustes alignment, ragged partitions and an iteration rank above the target rank
        dict(name="solve_fp32_opt", kind="solve", dtype="f32", n=60_007, d=362, k=24, m=20,
             schedule="4x4,2x3,1x3", refine=0, agg="opt", ritz=False, kxk_fp64=False),
        # the headline workload's step: FP32 rows held as hi/lo BF16 planes, full size
        dict(name="step_planes", kind="step", dtype="f32_bf16x2", n=1_000_000, d=1024, k=16, m=64, shared=False),
        # the headline data path with new rows each pass: load (split into planes on the device), solve, read back
        dict(name="refresh_planes", kind="refresh", dtype="f32_bf16x2", n=131_072, d=1024, k=16, m=64,
             schedule="4x2,2x2,1x2", refine=0, agg="sign", ritz=False, kxk_fp64=False),
        # BF16 storage at a middle width of the batching workload (padded rows), small k
        dict(name="step_bf16", kind="step", dtype="bf16", n=150_001, d=362, k=8, m=24, shared=False),
        # the precision workload's step, BF16 storage, a quarter of its rows
        dict(name="step_bf16_wide", kind="step", dtype="bf16", n=1_000_000, d=2048, k=32, m=128, shared=False),
        # the precision workload's step, FP8 codes with row scales, a quarter of its rows
        dict(name="step_e4m3_wide", kind="step", dtype="e4m3", n=1_000_000, d=2048, k=32, m=128, shared=False),
        # the precision workload's local orthonormalisation: FP64 Gram and Cholesky, one block per partition
        dict(name="orth_fp64", kind="orth", d=2048, k=32, batch=128, kxk_fp64=True),
        # batching: instances of mixed shapes, BF16 rows, p = 4 with a few closing p = 1 rounds
        dict(name="batch", kind="batch", dtype="bf16", count=24, n_lo=8_000, n_hi=100_000, mix=1,
             schedule="4x6,1x4", refine=0, agg="sign", ritz=False, kxk_fp64=False),
        # serving: a burst of requests through the server, the serving workload's schedule
        dict(name="serve", kind="serve", dtype="bf16", count=8, n_lo=8_000, n_hi=100_000, mix=2,
             schedule=SERVING, refine=3, agg="sign", ritz=True, kxk_fp64=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "solve", "solve", "refresh", "orth", "batch", "serve"])
    fp64 = rng.random() < 0.3
    if kind == "orth":
        d, k = _log(rng, 64, 2048), rng.randint(1, 32)
        return dict(kind=kind, d=d, k=min(k, d), batch=_log(rng, 1, 128), kxk_fp64=fp64)
    if kind in ("batch", "serve"):
        batch = kind == "batch"
        return dict(kind=kind, dtype="bf16", count=rng.randint(4, 24 if batch else 8), n_lo=8_000,
                    n_hi=_log(rng, 16_000, 100_000), mix=rng.randint(3, 1 << 20),
                    schedule="4x6,1x4" if batch else SERVING, refine=0 if batch else 3, agg="sign",
                    ritz=not batch, kxk_fp64=False)
    dtype = "f32_bf16x2" if kind == "refresh" else rng.choice(["f32", "f32_bf16x2", "bf16", "e4m3"])
    d = _log(rng, 64, 1024 if dtype in ("f32", "f32_bf16x2") else 2048)
    k = rng.choice([1, 3, 4, 5, 8, 12, 16, 24, 32])
    if kind != "step" and dtype == "f32" and d <= 128:
        k = min(k, 8)  # the plain workload's spectrum: further columns lie in its noise
    # rows: in whole solves enough per partition that the local bases stay near the shared one,
    # at most about the listed cases' elements
    m = _log(rng, 1, 128 if kind == "step" else 32)
    most = {"step": 3e8 if dtype == "f32" else 1e9, "solve": 2.2e7, "refresh": 1.3e8}[kind]
    lo = max(2_000, m * (2048 if kind != "step" else 64))
    n = _log(rng, lo, max(lo + 1, min(1_000_000, int(most / d))))
    case = dict(kind=kind, dtype=dtype, n=n, d=d, k=k, m=m)
    if kind == "step":
        return dict(case, shared=rng.random() < 0.3)
    return dict(case, schedule=rng.choice(["4x4,2x3,1x3", "4x2,2x2,1x2", "8x1,4x2,2x2,1x4"]),
                refine=rng.choice([0, 2]), agg=rng.choice(["sign", "opt", "sign", "identity"]), ritz=False,
                kxk_fp64=fp64)


# --------------------------------------------------------------------------- data

def _schedule(text):
    out = []
    for part in text.split(","):
        p, times = part.split("x")
        out += [int(p)] * int(times)
    return out


def _sizes(n, m):
    q, r = divmod(n, m)
    return [q + (1 if i < r else 0) for i in range(m)]


def _spectrum(dtype, d, k):
    """(lam, noise sigma) of the workload whose storage this is."""
    if dtype in ("f32_bf16x2",) or (dtype == "f32" and d > 128):
        q = min(d, max(32, k + 8))
        return 10.0 * 0.9 ** np.arange(1, q + 1), math.sqrt(0.1)
    if dtype == "f32":
        return 0.8 ** np.arange(1, d + 1), 0.1
    if d >= 1536:
        j1, j2 = np.arange(1, k + 1), np.arange(k + 1, 4 * k + 1)
        return np.concatenate([j1 ** -1.5, 0.5 * j2 ** -1.5]), math.sqrt(1e-3)
    # 0.85^j; what lies beyond 96 spikes (1e-7 of the first) is below the stored rows' rounding
    return 0.85 ** np.arange(1, min(d, 96) + 1), 0.0


def _rows(n, d, lam, sigma, seed):
    """n x d FP32 spiked-Gaussian rows on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    q = len(lam)
    U = torch.linalg.qr(_gauss((d, q), seed + 5).float())[0]
    basis = (U.to(DEV) * torch.tensor(lam, device=DEV, dtype=torch.float32).sqrt()).T.contiguous()
    out = torch.empty(n, d, device=DEV)
    for r in range(0, n, 131_072):
        e = min(n, r + 131_072)
        blk = torch.randn(e - r, q, device=DEV, generator=g) @ basis
        if sigma:
            blk += sigma * torch.randn(e - r, d, device=DEV, generator=g)
        out[r:e] = blk
    return out


def _encode(rows, dtype):
    """(stored tensor, row scales or None) of FP32 rows."""
    if dtype in ("f32", "f32_bf16x2"):
        return rows, None
    if dtype == "bf16":
        return rows.to(torch.bfloat16), None
    codes = torch.empty(rows.shape, device=DEV, dtype=torch.uint8)
    scales = torch.empty(rows.shape[0], device=DEV)
    for r in range(0, rows.shape[0], 131_072):
        blk = rows[r:r + 131_072]
        sc = blk.abs().amax(dim=1) / 448.0
        sc[sc == 0] = 1.0
        scales[r:r + 131_072] = sc
        q = (blk / sc[:, None]).clamp(-448.0, 448.0).to(torch.float8_e4m3fn)
        codes[r:r + 131_072] = q.view(torch.uint8)
    return codes, scales


def _data(case, seed):
    """(list of stored partitions, list of row scales or None) on the GPU."""
    lam, sigma = _spectrum(case["dtype"], case["d"], case["k"])
    stored, scales = _encode(_rows(case["n"], case["d"], lam, sigma, seed), case["dtype"])
    sizes = _sizes(case["n"], case["m"])
    torch.cuda.synchronize()  # the library reads the rows on a stream of its own
    return list(stored.split(sizes)), None if scales is None else list(scales.split(sizes))


def _gauss(shape, seed):
    g = torch.Generator().manual_seed(int(seed) + 77)
    return torch.randn(shape, dtype=torch.float64, generator=g)


def _bases(case, seed):
    """The FP64 blocks a step multiplies: one shared orthonormal basis or one per partition."""
    c = 1 if case["shared"] else case["m"]
    z = torch.linalg.qr(_gauss((c, case["d"], case["k"]), seed))[0].contiguous().to(DEV)
    return z[0] if case["shared"] else z


def _instances(case, seed):
    """Shapes of a mix of instances: n log-uniform, d among the pool widths, m and k as the batching workload.
    The shapes belong to the case, the rows to the seed."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        out.append(dict(n=n, d=int(rng.choice(WIDTHS)), m=int(round(math.exp(rng.uniform(math.log(4), math.log(16))))),
                        k=int(rng.choice([4, 8, 16, 32])), seed=int(seed) * 1000 + i))
    return [dict(o, dtype=case["dtype"]) for o in out]


def _iterates(case, seed):
    """Blocks as M Z leaves them: columns of falling norm (the precision workload's spectrum), somewhat mixed."""
    k = case["k"]
    lam = torch.tensor(np.arange(1, k + 1) ** -1.5)
    mix = torch.eye(k, dtype=torch.float64) + 0.3 * _gauss((k, k), seed + 1) / math.sqrt(k)
    y = _gauss((case["batch"], case["d"], k), seed).to(DEV)
    return (y @ (lam[:, None] * mix).to(DEV)).contiguous()


def _flags(case):
    return (B.LP_FLAG_RITZ if case["ritz"] else 0) | (B.LP_FLAG_KXK_FP64 if case["kxk_fp64"] else 0)


# --------------------------------------------------------------------------- the protocol

def prepare(case, seed):
    state = _prepare(case, seed)
    torch.cuda.synchronize()  # what was drawn on torch's stream is there for the library's
    return state


def _prepare(case, seed):
    kind = case["kind"]
    if kind == "orth":
        return dict(case=case, ctx=B.lp_create(), y=_iterates(case, seed))
    if kind == "batch":
        batch = B.Batch()
        for inst in _instances(case, seed):
            parts, _ = _data(inst, inst["seed"])
            batch.add(parts, inst["k"], _schedule(case["schedule"]), case["agg"],
                      _gauss((inst["d"], inst["k"]), inst["seed"]).numpy(), dtype=case["dtype"],
                      refine_rounds=case["refine"], flags=_flags(case))
        return dict(case=case, batch=batch)
    if kind == "serve":
        reqs = []
        for inst in _instances(case, seed):
            parts, _ = _data(inst, inst["seed"])
            reqs.append((parts, inst["k"], _gauss((inst["d"], inst["k"]), inst["seed"]).numpy()))
        return dict(case=case, server=B.Server(max_active=64), reqs=reqs, schedule=_schedule(case["schedule"]))
    parts, scales = _data(case, seed)
    lp = B.LocalPower(parts, dtype=case["dtype"], row_scales=scales)
    state = dict(case=case, lp=lp)
    if kind == "step":
        state["z"] = _bases(case, seed)
        state["out"] = torch.empty((case["m"], case["d"], case["k"]), dtype=torch.float64, device=DEV)
        return state
    state["y0"] = _gauss((case["d"], case["k"]), seed).numpy()
    state["schedule"] = _schedule(case["schedule"])
    if kind == "refresh":
        state["parts"] = parts
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        lp = state["lp"]
        return B.lp_power_step(lp.ctx, case["k"], state["z"], case["shared"], case["m"], case["d"], out=state["out"])
    if kind == "orth":
        return B.lp_orth(state["ctx"], state["y"], kxk_fp64=case["kxk_fp64"])
    if kind == "batch":
        batch = state["batch"]
        batch.solve()
        return [batch.result(i)[0] for i in range(case["count"])]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(parts, k, state["schedule"], case["agg"], y0, dtype=case["dtype"],
                          refine_rounds=case["refine"], flags=_flags(case)) for parts, k, y0 in state["reqs"]]
        done = {}
        while len(done) < len(ids):
            for rid in srv.progress():
                done[rid] = srv.result(rid)
        return [list(done[rid][:2]) for rid in ids]
    lp = state["lp"]
    if kind == "refresh":
        B.lp_load_partitions(lp.ctx, state["parts"], case["dtype"])
    Z, sigma, _ = lp.solve(case["k"], state["schedule"], case["agg"], state["y0"], refine_rounds=case["refine"],
                           ritz=case["ritz"], kxk_fp64=case["kxk_fp64"])
    return [Z, sigma] if case["ritz"] else Z


# --------------------------------------------------------------------------- least work

def _solve_work(n, d, k, m, dtype, schedule, refine, ritz, load):
    steps = sum(_schedule(schedule)) + refine + (1 if ritz else 0)
    a = float(n) * d * ELEM[dtype] + (4.0 * n if dtype == "e4m3" else 0.0)
    # each local step depends on the one before: A is read once for each step, or once in all where it fits L2
    reads = steps if a > L2_BYTES else 1
    return dict(bytes=a * (reads + (1 if load else 0)) + 16.0 * d * k, flops=4.0 * n * d * k * steps)


def work(case):
    kind = case["kind"]
    if kind == "orth":
        b, d, k = case["batch"], case["d"], case["k"]
        return dict(bytes=16.0 * b * d * k, flops=2.0 * b * d * k * k)
    if kind == "step":
        n, d, k, m = case["n"], case["d"], case["k"], case["m"]
        a = float(n) * d * ELEM[case["dtype"]] + (4.0 * n if case["dtype"] == "e4m3" else 0.0)
        return dict(bytes=a + 8.0 * d * k * ((1 if case["shared"] else m) + m), flops=4.0 * n * d * k)
    if kind in ("batch", "serve"):
        ws = [_solve_work(i["n"], i["d"], i["k"], i["m"], case["dtype"], case["schedule"], case["refine"], case["ritz"],
                          kind == "serve") for i in _instances(case, 0)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    return _solve_work(case["n"], case["d"], case["k"], case["m"], case["dtype"], case["schedule"], case["refine"],
                       case["ritz"], kind == "refresh")


# --------------------------------------------------------------------------- FP64 values

def _f64(part, scale, dtype):
    if dtype == "e4m3":
        return part.view(torch.float8_e4m3fn).to(torch.float64) * scale.to(torch.float64)[:, None]
    return part.to(torch.float64)


def _orth64(Y):
    """Orthonormal basis with positive diagonal of R, blocks d x k: two passes of Gram and Cholesky in FP64
    (the second removes what the conditioning of the first leaves), equal to a Householder QR with that sign."""
    for _ in range(2):
        L = torch.linalg.cholesky((Y.mT @ Y).cpu())
        Y = Y @ torch.linalg.inv(L).mT.to(DEV)
    return Y


class _Local64:
    """M_i Z_i = A_i^T (A_i Z_i) / s_i in FP64, partitions padded with zero rows to one stacked tensor."""

    def __init__(self, parts, scales, dtype):
        self.s = torch.tensor([float(p.shape[0]) for p in parts], dtype=torch.float64, device=DEV)
        smax, d = max(p.shape[0] for p in parts), parts[0].shape[1]
        self.A = torch.zeros(len(parts), smax, d, dtype=torch.float64, device=DEV)
        for i, p in enumerate(parts):
            self.A[i, :p.shape[0]] = _f64(p, None if scales is None else scales[i], dtype)

    def step(self, Z):
        return self.A.mT @ (self.A @ Z) / self.s[:, None, None]


def _solve64(parts, scales, dtype, k, schedule, refine, agg, y0, ritz):
    op = _Local64(parts, scales, dtype)
    m, n = len(parts), float(op.s.sum())
    w = (op.s / n)[:, None, None]
    base = int(torch.argmax(op.s))
    Z = _orth64(torch.as_tensor(y0, device=DEV))
    for p in list(schedule) + [1] * refine:
        Zi = Z.expand(m, -1, -1)
        for j in range(p):
            if j:
                Zi = _orth64(Yi)
            Yi = op.step(Zi)
        if p > 1 and agg == "sign":
            dots = (Zi * Zi[base]).sum(dim=1)
            Yi = Yi * torch.where(dots < 0, -1.0, 1.0).to(torch.float64)[:, None, :]
        elif p > 1 and agg == "opt":
            W1, _, W2 = torch.linalg.svd((Zi.mT @ Zi[base]).cpu())
            D = W1 @ W2
            D[base] = torch.eye(k, dtype=torch.float64)
            Yi = Yi @ D.to(DEV)
        Z = _orth64((w * Yi).sum(dim=0))
    if not ritz:
        return Z.cpu().numpy(), None
    H = Z.T @ (w * op.step(Z.expand(m, -1, -1))).sum(dim=0)
    lam, V = torch.linalg.eigh(((H + H.T) / 2).cpu())
    lam, V = lam.flip(0).to(DEV), V.flip(1).to(DEV)
    # a Ritz vector's sign: along the column of Z_T that it has most of
    V = V * torch.sign(V.gather(0, V.abs().argmax(dim=0, keepdim=True)))
    return (Z @ V).cpu().numpy(), (n * lam.clamp(min=0)).sqrt().cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "orth":
        return _orth64(_iterates(case, seed))
    if kind in ("batch", "serve"):
        out = []
        for inst in _instances(case, seed):
            parts, scales = _data(inst, inst["seed"])
            Z, sigma = _solve64(parts, scales, case["dtype"], inst["k"], _schedule(case["schedule"]), case["refine"],
                                case["agg"], _gauss((inst["d"], inst["k"]), inst["seed"]).numpy(), case["ritz"])
            out.append([Z, sigma] if case["ritz"] else Z)
        return out
    parts, scales = _data(case, seed)
    if kind == "step":
        z = _bases(case, seed)
        out = torch.empty((case["m"], case["d"], case["k"]), dtype=torch.float64, device=DEV)
        for i, p in enumerate(parts):
            a = _f64(p, None if scales is None else scales[i], case["dtype"])
            out[i] = a.T @ (a @ (z if case["shared"] else z[i])) / p.shape[0]
        return out
    Z, sigma = _solve64(parts, scales, case["dtype"], case["k"], _schedule(case["schedule"]), case["refine"],
                        case["agg"], _gauss((case["d"], case["k"]), seed).numpy(), case["ritz"])
    return [Z, sigma] if case["ritz"] else Z
