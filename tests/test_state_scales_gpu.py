"""GPU: systems whose state components have different units.  With the state
scaled by powers of two, A -> D A D and b -> D b, every operation of the
elimination commutes with the scaling, so that X / D^-1 has to be as accurate
as the solution of the unscaled system, component by component: a normwise
measure would see the largest rows and the smallest-scaled unknowns only."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _scales(N, n, decades, seed):
    """Powers of two over `decades` powers of ten, in another order in every block."""
    rng = np.random.default_rng(seed)
    e = np.round(np.linspace(-0.5, 0.5, n) * decades / np.log10(2.0))
    return 2.0 ** np.stack([rng.permutation(e) for _ in range(N)])


def _scaled(s, D):
    return dict(A_diag=s["A_diag"] * D[:, :, None] * D[:, None, :], A_sub=s["A_sub"] * D[1:, :, None] * D[:-1, None, :],
                B=s["B"] * D[:, :, None])


# the unscaled system has kappa(A) below 1e3 and is solved to a few units of
# 1e-16 kappa; 1e-13 is the bar for both
DECADES = (3, 8, 12)


@pytest.mark.parametrize("N,n,d", [(9, 32, 1), (9, 48, 3), (12, 37, 16), (33, 64, 16)])
@pytest.mark.parametrize("decades", DECADES)
def test_blocks_up_to_64(oracle_mod, N, n, d, decades):
    """Factor + solve and the solve with stored factors (its many-column form
    from d = 9 on)."""
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    D = _scales(N, n, decades, seed=n)
    t = _scaled(s, D)
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    sol = Solver(N, n, d_max=d)
    sol.set_option("schur_emu", 1)
    X = sol.factor_solve(_dev(t["A_diag"]), _dev(t["A_sub"]), _dev(t["B"])).cpu().numpy()
    X2 = sol.solve(_dev(t["B"])).cpu().numpy()
    sol.close()
    for x in (X, X2):
        assert oracle_mod.forward_error(x * D[:, :, None], Xo) <= 1e-13


@pytest.mark.parametrize("N,n,d", [(1, 100, 1), (9, 96, 2), (5, 130, 17), (6, 256, 16)])
@pytest.mark.parametrize("decades", DECADES)
def test_blocks_above_64(oracle_mod, N, n, d, decades):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    D = _scales(N, n, decades, seed=n)
    t = _scaled(s, D)
    As = t["A_sub"] if N > 1 else np.zeros((1, n, n))
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    sol = Solver(N, n, d_max=d)
    X = sol.factor_solve(_dev(t["A_diag"]), _dev(As), _dev(t["B"])).cpu().numpy()
    X2 = sol.solve(_dev(t["B"])).cpu().numpy()
    sol.close()
    for x in (X, X2):
        assert oracle_mod.forward_error(x * D[:, :, None], Xo) <= 1e-13


# a target that the FP32 solution meets at once: what the FP32 factors give,
# unrefined; kappa(A) u_32 is below 1e-4, and 1e-4 is the bar
@pytest.mark.parametrize("N,n,d,precision", [(40, 24, 1, "fp32_ir"), (40, 64, 4, "fp32_ir"), (9, 96, 2, "fp32_ir"),
                                             (6, 256, 16, "tf32_ir")])
@pytest.mark.parametrize("decades", (3, 8))
def test_unrefined_fp32_factors(oracle_mod, N, n, d, precision, decades):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    D = _scales(N, n, decades, seed=n)
    t = _scaled(s, D)
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    sol = Solver(N, n, d_max=d, precision=precision)
    sol.set_option("target_berr_e18", 10 ** 18)
    X = sol.factor_solve(_dev(t["A_diag"]), _dev(t["A_sub"]), _dev(t["B"])).cpu().numpy()
    assert sol.last_info.iters == 0
    X2 = sol.solve(_dev(t["B"])).cpu().numpy()
    sol.close()
    for x in (X, X2):
        assert oracle_mod.forward_error(x * D[:, :, None], Xo) <= 1e-4


@pytest.mark.parametrize("N,n,precision", [(257, 20, "fp32_ir"), (257, 24, "fp32_ir"), (130, 31, "tf32_ir"),
                                           (257, 33, "fp32_ir"), (65, 32, "fp64"), (65, 47, "fp64"), (9, 65, "fp64"),
                                           (9, 100, "fp32_ir")])
def test_workspace_guards_hold(N, n, precision):
    """The exponents' buffers among the others: 64 to a block whatever its size."""
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, 1, seed=n)
    sol = Solver(N, n, d_max=1, precision=precision)
    if precision == "fp64":
        sol.set_option("schur_emu", 1)
    sol.set_option("debug_guards", 1)
    sol.factor_solve(_dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"]))
    sol.close()


@pytest.mark.parametrize("N,n,m,diag", [(3, 2, 3, False), (4, 24, 12, False), (5, 33, 65, False), (4, 64, 32, True),
                                        (3, 100, 70, False), (3, 256, 130, True)])
@pytest.mark.parametrize("decades", DECADES)
def test_kalman_assembly(N, n, m, diag, decades):
    """x = S x', z = T z': G -> S_k+1 G S_k^-1, H -> T H S^-1, Qinv -> S^-1 Qinv
    S^-1, Rinv -> T^-1 Rinv T^-1.  Every entry against the sums of magnitudes it
    is formed from, as a chain of FP64 multiply-adds would give it."""
    from paper_2509_03015_gb300 import kalman_assemble
    mod = inputs.kalman_model(N, n, m, seed=N + n + m)
    S, T = _scales(N, n, decades, seed=n), _scales(N, m, decades, seed=m + 1)
    G, H, Q, R = mod["G"].copy(), mod["H"], mod["Qinv"], mod["Rinv"]
    G[1:] *= S[1:, :, None] / S[:-1, None, :]
    H = H * T[:, :, None] / S[:, None, :]
    Q = Q / (S[:, :, None] * S[:, None, :])
    R = R / (T[:, :, None] * T[:, None, :])
    if diag:
        R = np.stack([np.diag(np.diag(r)) for r in R])
    Rin = np.ascontiguousarray(np.einsum("kii->ki", R)) if diag else R
    A, E, _ = kalman_assemble(_dev(G), _dev(H), _dev(Q), _dev(Rin))
    A, E = A.cpu().numpy(), E.cpu().numpy()
    ld = np.longdouble
    aG, aH, aQ, aR = np.abs(G), np.abs(H), np.abs(Q), np.abs(R)
    for k in range(N):
        want = Q[k].astype(ld) + H[k].T.astype(ld) @ (R[k].astype(ld) @ H[k].astype(ld))
        mag = aQ[k] + aH[k].T @ (aR[k] @ aH[k])
        if k + 1 < N:
            QG = Q[k + 1].astype(ld) @ G[k + 1].astype(ld)
            want = want + G[k + 1].T.astype(ld) @ QG
            mag = mag + aG[k + 1].T @ (aQ[k + 1] @ aG[k + 1])
            # n products each within eps of its own size
            assert (np.abs(E[k] + QG) <= (n + 4) * 2.0 ** -52 * (aQ[k + 1] @ aG[k + 1])).all()
        assert (np.abs(A[k] - want) <= 2 * (n + m + 4) * 2.0 ** -52 * mag).all()


@pytest.mark.parametrize("n", [5, 48, 80])
def test_kalman_assembly_with_uneven_diagonal_precisions(n):
    """Process precisions over eight decades beside a G of O(1): A_{k+1,k} entry by
    entry.  An entry is one product; G's entries are of one magnitude, and a column
    is cut 62 bits below its own largest."""
    from paper_2509_03015_gb300 import kalman_assemble
    N = 3
    mod = inputs.kalman_model(N, n, 4, seed=n)
    rng = np.random.default_rng(n)
    G = rng.uniform(0.25, 1.0, (N, n, n)) * rng.choice([-1.0, 1.0], (N, n, n)) / np.sqrt(n)
    q = np.logspace(-4, 4, n)
    Q = np.stack([np.diag(np.random.default_rng(k).permutation(q)) for k in range(N)])
    Q[1, 0, 0] = 0.0  # no information at all on one component
    A, E, _ = kalman_assemble(_dev(G), _dev(mod["H"]), _dev(Q), _dev(mod["Rinv"]))
    want = -np.matmul(Q[1:], G[1:])
    assert (np.abs(E.cpu().numpy() - want) <= 8 * 2.0 ** -52 * np.abs(want)).all()
    Ad = Q + np.matmul(mod["H"].transpose(0, 2, 1), np.matmul(mod["Rinv"], mod["H"]))
    Ad[:-1] += np.matmul(G[1:].transpose(0, 2, 1), np.matmul(Q[1:], G[1:]))
    s = np.sqrt(np.einsum("kii->ki", Ad))
    assert (np.abs(A.cpu().numpy() - Ad) <= 4 * (n + 4) * 2.0 ** -52 * s[:, :, None] * s[:, None, :]).all()
