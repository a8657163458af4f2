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
