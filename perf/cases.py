"""The work a program has this solver do, as measurable cases.

Every case is one call (or the short sequence of calls that belongs together)
through the package's public entry points, on inputs drawn on the GPU from a
seed.  The systems are Kalman-smoother normal equations (the generator of
paper_2509_03015_gb300/inputs.py with every step's blocks distinct), since
those are what the solver is used for:
  A_kk = Q^-1 + G_{k+1}^T Q^-1 G_{k+1} + H_k^T R^-1 H_k,  A_{k+1,k} = -Q^-1 G_{k+1},
with Q = 0.1 I, R = 0.5 I, G_k = rho (orthogonal) + a small step-dependent
part, H_k Gaussian with m = n / 2 rows.

  kind        call
  solve       Solver.factor_solve                 (factor and solve one system)
  resolve     Solver.solve                        (new right-hand sides, stored factors)
  likelihood  Solver.factor_solve + logdet        (one evaluation of a Gaussian likelihood)
  grad        block_tri_solve + autograd.grad     (forward and backward)
  batch       BatchSolver.run                     (uneven systems in one launch)
  assemble    kalman_assemble                     (normal equations from a per-step model)
"""
import math

import torch

from paper_2509_03015_gb300 import BatchSolver, Solver, block_tri_solve, kalman_assemble

DEV = "cuda"


def listed():
    return [
        # a short smoother: the smallest call, where latency is everything
        dict(name="short-smoother", kind="solve", precision="fp64", N=64, n=8, d=1, rho=0.95),
        # a model whose sizes are multiples of nothing
        dict(name="odd-sizes", kind="solve", precision="fp64", N=777, n=37, d=3, rho=0.95),
        # a long smoother in FP64: the benchmark's headline workload
        dict(name="long-fp64", kind="solve", precision="fp64", N=16384, n=64, d=4, rho=0.95),
        # the same system in mixed precision (FP32 factors, FP64 refinement)
        dict(name="long-fp32", kind="solve", precision="fp32_ir", N=16384, n=64, d=4, rho=0.95),
        # a wide state in FP64: the paper's N = 1024, n = 256 shape
        dict(name="wide-fp64", kind="solve", precision="fp64", N=1024, n=256, d=1, rho=0.95),
        # a short wide system, as long as the paper's neuroscience instance, in FP32
        dict(name="wide-short-fp32", kind="solve", precision="fp32_ir", N=100, n=256, d=1, rho=0.95),
        # the benchmark's ill-conditioned wide workload in TF32: the largest one
        dict(name="wide-tf32", kind="solve", precision="tf32_ir", N=4096, n=256, d=16, rho=0.99),
        # a smoother that is factored once and solved for many measurement sets
        dict(name="resolve", kind="resolve", precision="fp64", N=4096, n=64, d=16, rho=0.95),
        # a likelihood evaluation inside a hyperparameter search
        dict(name="likelihood", kind="likelihood", precision="fp64", N=2000, n=24, d=1, rho=0.95),
        # differentiable smoother layer
        dict(name="grad", kind="grad", N=2048, n=32, d=8, rho=0.95),
        # condensed model-predictive-control problems of uneven horizons
        dict(name="mpc-batch", kind="batch", K=512, N_lo=32, N_hi=2048, d=1, rho=0.95),
        # building the normal equations on the device
        dict(name="assemble", kind="assemble", N=16384, n=64, m=32, diag=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "resolve", "likelihood", "grad", "batch", "assemble"])
    rho = rng.choice([0.9, 0.95, 0.99])
    if kind == "batch":
        K = _log_int(rng, 32, 512)
        return dict(kind="batch", K=K, N_lo=_log_int(rng, 8, 64), N_hi=_log_int(rng, 256, 2048), d=1, rho=rho)
    if kind == "assemble":
        n = _log_int(rng, 8, 256)
        m = max(1, int(n * rng.choice([0.5, 1.0, 2.0])))
        N = _log_int(rng, 32, max(64, min(16384, 2 ** 32 // (n * n * (n + m)))))
        return dict(kind="assemble", N=N, n=n, m=m, diag=rng.random() < 0.5)
    if kind == "grad":
        n = _log_int(rng, 4, 64)
        N = _log_int(rng, 32, max(64, min(8192, 2 ** 29 // n ** 3)))
        return dict(kind="grad", N=N, n=n, d=rng.choice([1, 2, 8]), rho=rho)
    if kind in ("resolve", "likelihood"):
        n = _log_int(rng, 4, 128)
        N = _log_int(rng, 32, max(64, min(16384, 2 ** 31 // n ** 3)))
        return dict(kind=kind, precision="fp64", N=N, n=n, d=1 if kind == "likelihood" else rng.choice([1, 4, 16]),
                    rho=rho)
    precision = rng.choice(["fp64", "fp64", "fp32_ir", "tf32_ir"])
    n = _log_int(rng, 8, 256) if precision == "fp64" else _log_int(rng, 32, 256)
    N = _log_int(rng, 32, max(64, min(16384, 2 ** 33 // n ** 3)))
    return dict(kind="solve", precision=precision, N=N, n=n, d=rng.choice([1, 2, 4, 16]), rho=rho)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _system(g, N, n, d, rho):
    """A_diag, A_sub, B of one smoother with distinct blocks."""
    m = max(1, n // 2)
    U = torch.linalg.qr(_randn(g, n, n))[0]
    G = rho * U + 0.02 * _randn(g, max(N - 1, 0), n, n) / math.sqrt(n)
    H = _randn(g, N, m, n) / math.sqrt(n)
    A = 2.0 * torch.bmm(H.transpose(1, 2), H)
    A.diagonal(dim1=1, dim2=2).add_(10.0)
    if N > 1:
        A[:-1] += 10.0 * torch.bmm(G.transpose(1, 2), G)
    return A.contiguous(), (-10.0 * G).contiguous(), _randn(g, N, n, d)


def _batch_shapes(case, seed):
    r = torch.Generator().manual_seed(7)  # the shapes are the case's, the numbers the seed's
    u = torch.rand(case["K"], 2, generator=r, dtype=torch.float64)
    lo, hi = math.log(case["N_lo"]), math.log(case["N_hi"])
    return [(max(1, int(math.exp(lo + (hi - lo) * float(a)))), (12, 24, 48)[min(2, int(3 * float(b)))]) for a, b in u]


def _batch_systems(g, case, seed):
    shapes = _batch_shapes(case, seed)
    d, out = case["d"], [None] * case["K"]
    for n in (12, 24, 48):  # one long draw per block size, cut into the instances
        ks = [k for k, s in enumerate(shapes) if s[1] == n]
        if not ks:
            continue
        A, S, B = _system(g, sum(shapes[k][0] for k in ks), n, d, case["rho"])
        at = 0
        for k in ks:
            N = shapes[k][0]
            out[k] = (A[at:at + N], S[at:at + N - 1], B[at:at + N])
            at += N
    return out


def _model(g, case):
    N, n, m = case["N"], case["n"], case["m"]
    G = 0.5 * _randn(g, N, n, n) / math.sqrt(n)
    H = _randn(g, N, m, n) / math.sqrt(n)
    Mq = _randn(g, N, n, n)
    Qinv = torch.bmm(Mq, Mq.transpose(1, 2)) / n
    Qinv.diagonal(dim1=1, dim2=2).add_(1.0)
    if case["diag"]:
        Rinv = 1.0 + _randn(g, N, m).abs()
    else:
        Mr = _randn(g, N, m, m)
        Rinv = torch.bmm(Mr, Mr.transpose(1, 2)) / m
        Rinv.diagonal(dim1=1, dim2=2).add_(1.0)
    return dict(G=G, H=H, Qinv=Qinv, Rinv=Rinv, z=_randn(g, N, m), zeta=_randn(g, N, n))


def _inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    if case["kind"] == "batch":
        return _batch_systems(g, case, seed)
    if case["kind"] == "assemble":
        return _model(g, case)
    out = _system(g, case["N"], case["n"], case["d"], case["rho"])
    return out + (_randn(g, case["N"], case["n"], case["d"]),) if case["kind"] == "grad" else out


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "assemble":
        st.update(x)
    elif kind == "batch":
        # solutions in one buffer, instance after instance (16-byte aligned)
        sizes = [B.numel() for _, _, B in x]
        starts = [0]
        for s in sizes:
            starts.append(starts[-1] + (s + 1) // 2 * 2)
        flat = torch.zeros(starts[-1], dtype=torch.float64, device=DEV)
        views = [flat[a:a + s].view(B.shape) for a, s, (_, _, B) in zip(starts, sizes, x)]
        st.update(flat=flat, batch=BatchSolver(x, X=views))
    elif kind == "grad":
        A, S, B, W = x
        st.update(A=A.requires_grad_(), S=S.requires_grad_(), B=B.requires_grad_(), W=W)
    else:
        A, S, B = x
        solver = Solver(case["N"], case["n"], d_max=case["d"], precision=case["precision"])
        st.update(A=A, S=S, B=B, solver=solver)
        if kind == "resolve":
            solver.factor(A, S)
    return st


def run(st):
    kind = st["kind"]
    if kind == "solve":
        return st["solver"].factor_solve(st["A"], st["S"], st["B"])
    if kind == "resolve":
        return st["solver"].solve(st["B"])
    if kind == "likelihood":
        X = st["solver"].factor_solve(st["A"], st["S"], st["B"])
        return X, st["solver"].logdet()
    if kind == "grad":
        X = block_tri_solve(st["A"], st["S"], st["B"])
        return (X.detach(),) + torch.autograd.grad(X, (st["A"], st["S"], st["B"]), st["W"])
    if kind == "batch":
        st["batch"].run(graph=True)
        return st["flat"]
    return kalman_assemble(st["G"], st["H"], st["Qinv"], st["Rinv"], st["z"], st["zeta"])


def _work_system(N, n, d, solve_only=False):
    """Block Cholesky along the chain: per block n^3/3 + n^3 (coupling solve) +
    n^2 (n + 1) (symmetric update), 2 n^2 d and 4 n^2 d per block and coupling."""
    nn = 8.0 * n * n
    flops = N * 2.0 * n * n * d + (N - 1) * 4.0 * n * n * d
    if solve_only:  # the stored factor (lower triangles) and couplings, b and x
        return (N * 0.5 + (N - 1)) * nn + 16.0 * N * n * d, flops
    return (2 * N - 1) * nn + 16.0 * N * n * d, flops + N * n ** 3 / 3 + (N - 1) * (2.0 * n ** 3 + n * n)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = [_work_system(N, n, case["d"]) for N, n in _batch_shapes(case, 0)]
        return dict(bytes=sum(b for b, _ in ws), flops=sum(f for _, f in ws))
    N, n = case["N"], case["n"]
    if kind == "assemble":
        m = case["m"]
        rr = m if case["diag"] else m * m
        by = 8.0 * N * (2 * n * n + m * n + rr + m + n) + 8.0 * N * (2 * n * n + n)
        fl = N * (2.0 * n ** 3 + n * n * (n + 1) + n * n * (m + 1) + 4.0 * n * n + 2.0 * m * n)
        return dict(bytes=by, flops=fl + N * (m * n if case["diag"] else 2.0 * m * m * n + 2.0 * m * m))
    d = case["d"]
    by, fl = _work_system(N, n, d, kind == "resolve")
    if kind == "grad":
        # the adjoint solve, the gradients' outer products; W in, gradients out
        by += 8.0 * (2 * N - 1) * n * n + 16.0 * N * n * d
        fl += _work_system(N, n, d, True)[1] + (2 * N - 1) * 4.0 * n * n * d
    return dict(bytes=by, flops=fl)


# ---- the same results in plain torch, 64 bits -------------------------------

def _sym(A):
    return 0.5 * (A + A.transpose(-1, -2))


def _reduce(A, S, B):
    """A X = B and log det A by eliminating every other block at once, level by
    level (batched torch.linalg in FP64).  A symmetric."""
    N = A.shape[0]
    if N == 1:
        L = torch.linalg.cholesky(A)
        return torch.cholesky_solve(B, L), 2.0 * L.diagonal(dim1=1, dim2=2).log().sum()
    Lo = torch.linalg.cholesky(A[1::2])
    k = (N - 1) // 2  # eliminated blocks with a right neighbour
    WL = torch.linalg.solve_triangular(Lo, S[0::2], upper=False)
    WR = torch.linalg.solve_triangular(Lo[:k], S[1::2].transpose(1, 2), upper=False)
    y = torch.linalg.solve_triangular(Lo, B[1::2], upper=False)
    Ae, Be = A[0::2].clone(), B[0::2].clone()
    e = WL.shape[0]
    Ae[:e] -= WL.transpose(1, 2) @ WL
    Be[:e] -= WL.transpose(1, 2) @ y
    Ae[1:1 + k] -= WR.transpose(1, 2) @ WR
    Be[1:1 + k] -= WR.transpose(1, 2) @ y[:k]
    Xe, ld = _reduce(_sym(Ae), -(WR.transpose(1, 2) @ WL[:k]), Be)
    t = y - WL @ Xe[:e]
    t[:k] -= WR @ Xe[1:1 + k]
    X = torch.empty_like(B)
    X[0::2] = Xe
    X[1::2] = torch.linalg.solve_triangular(Lo.transpose(1, 2), t, upper=True)
    return X, ld + 2.0 * Lo.diagonal(dim1=1, dim2=2).log().sum()


def _apply(A, S, X):
    R = A @ X
    if S.shape[0]:
        R[1:] += S @ X[:-1]
        R[:-1] += S.transpose(1, 2) @ X[1:]
    return R


def _solve(A, S, B):
    A = _sym(A)
    X, ld = _reduce(A, S, B)
    X = X + _reduce(A, S, B - _apply(A, S, X))[0]  # one step of refinement
    return X, ld


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "assemble":
        G, H, Q, z, zeta = x["G"], x["H"], x["Qinv"], x["z"][..., None], x["zeta"][..., None]
        Rz = x["Rinv"][..., None] * z if case["diag"] else x["Rinv"] @ z
        RH = x["Rinv"][..., None] * H if case["diag"] else x["Rinv"] @ H
        QG = Q[1:] @ G[1:]
        A = Q + H.transpose(1, 2) @ RH
        A[:-1] += G[1:].transpose(1, 2) @ QG
        b = H.transpose(1, 2) @ Rz + Q @ zeta
        b[:-1] -= G[1:].transpose(1, 2) @ (Q[1:] @ zeta[1:])
        return A, -QG, b
    if kind == "batch":
        flat = []
        shapes = _batch_shapes(case, seed)
        X = [None] * case["K"]
        for n in (12, 24, 48):  # the instances of one block size in one chain, uncoupled from each other
            ks = [k for k, s in enumerate(shapes) if s[1] == n]
            if not ks:
                continue
            zero = torch.zeros(1, n, n, dtype=torch.float64, device=DEV)
            S = torch.cat([t for k in ks for t in (x[k][1], zero)])[:-1]
            Y, _ = _solve(torch.cat([x[k][0] for k in ks]), S, torch.cat([x[k][2] for k in ks]))
            for k, part in zip(ks, torch.split(Y, [shapes[k][0] for k in ks])):
                X[k] = part.reshape(-1)
        for part in X:
            flat.append(part)
            if part.numel() % 2:
                flat.append(torch.zeros(1, dtype=torch.float64, device=DEV))
        return torch.cat(flat)
    X, ld = _solve(*x[:3])
    if kind == "likelihood":
        return X, float(ld)
    if kind == "grad":
        Lam, _ = _solve(x[0], x[1], x[3])
        LX = Lam @ X.transpose(1, 2)
        dS = -(Lam[1:] @ X[:-1].transpose(1, 2) + X[1:] @ Lam[:-1].transpose(1, 2))
        return X, -_sym(LX), dS, Lam
    return X
