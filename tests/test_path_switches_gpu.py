"""GPU: options that choose between factorisation paths, switched between the
factorisations and solves of one handle.  Every result is checked against the
CPU oracle, on systems drawn apart from each other, so that factors left from
an earlier one cannot pass."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _put(s):
    return _dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"])


# random_btd has kappa(A) below 1e3: 1e-12 forward in FP64, 1e-11 where the call
# refines to a backward error of 1e-14


@pytest.mark.parametrize("N,n,precision", [(40, 32, "fp32_ir"), (40, 32, "tf32_ir"), (9, 128, "fp32_ir"),
                                           (9, 128, "tf32_ir"), (5, 256, "fp32_ir"), (5, 256, "tf32_ir")])
@pytest.mark.parametrize("persistent", [1, 0])
def test_schur_emu_off_changes_nothing_in_mixed_precision(oracle_mod, N, n, precision, persistent):
    """The option is an FP64 one; on the other handles 0 is accepted and leaves
    the path, and its results, as they are."""
    from paper_2509_03015_gb300 import Solver
    s1, s2 = inputs.random_btd(N, n, 2, seed=1), inputs.random_btd(N, n, 2, seed=2)
    L, C = oracle_mod.factor(s2["A_diag"], s2["A_sub"])
    Xo = oracle_mod.solve(L, C, s2["B"])
    sol = Solver(N, n, d_max=2, precision=precision, persistent=bool(persistent))
    sol.factor(*_put(s1)[:2])
    launches = sol.launch_stats()[0]
    sol.set_option("schur_emu", 0)
    Ad, As, B = _put(s2)
    sol.factor(Ad, As)
    assert sol.launch_stats()[0] == launches
    ld = sol.logdet()
    X = sol.solve(B).cpu().numpy()
    sol.close()
    # each of the N n pivots' logarithms is within a few FP32 roundings
    assert abs(ld - oracle_mod.logdet(L)) <= N * n * 2.0 ** -20
    assert oracle_mod.forward_error(X, Xo) <= 1e-11
    assert oracle_mod.backward_error(s2["A_diag"], s2["A_sub"], X, s2["B"]) <= 1e-14


@pytest.mark.parametrize("d", [1, 12])
def test_factors_of_another_path_are_not_taken_for_the_tensor_core_ones(oracle_mod, d):
    """Tensor-core factors of one system, then the one-cluster path's factors of
    another, then a solve with the tensor-core option on again."""
    from paper_2509_03015_gb300 import Solver
    N, n = 40, 32
    s1, s2 = inputs.random_btd(N, n, d, seed=3), inputs.random_btd(N, n, d, seed=4)
    sol = Solver(N, n, d_max=d)
    sol.set_option("schur_emu", 1)
    sol.factor(*_put(s1)[:2])
    sol.set_option("schur_emu", 0)
    sol.set_option("small_cluster", 1)
    Ad, As, B = _put(s2)
    sol.factor(Ad, As)
    sol.set_option("schur_emu", 1)
    X = sol.solve(B).cpu().numpy()
    sol.close()
    assert oracle_mod.forward_error(X, oracle_mod.solve_system(s2["A_diag"], s2["A_sub"], s2["B"])) <= 1e-12


@pytest.mark.parametrize("N,n,nstar", [(100, 32, 2), (100, 48, 7), (37, 64, 2), (9, 40, 64), (130, 33, 3)])
@pytest.mark.parametrize("d", [1, 16])
def test_stored_factors_with_a_serial_top(oracle_mod, N, n, nstar, d):
    """Tensor-core factors below a serial sweep of up to nstar top blocks: the
    separators of the last level are that sweep's, not eliminated blocks."""
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n + nstar)
    sol = Solver(N, n, d_max=d)
    sol.set_option("schur_emu", 1)
    sol.set_option("nstar", nstar)
    Ad, As, B = _put(s)
    X = sol.factor_solve(Ad, As, B).cpu().numpy()
    X2 = sol.solve(B).cpu().numpy()
    sol.close()
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    for x in (X, X2):
        assert oracle_mod.forward_error(x, Xo) <= 1e-12
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1e-14


# the choice between the solve passes over tensor-core factors, both sides of its
# lines (one launch: the persistent kernel, over the other path's factors)
@pytest.mark.parametrize("N,n,d,one", [(130, 52, 3, False), (130, 51, 4, True), (65, 60, 1, False), (65, 59, 2, True),
                                       (65, 64, 5, True), (65, 64, 6, True), (65, 56, 7, False), (65, 55, 8, True),
                                       (65, 32, 9, False), (65, 32, 8, True), (2049, 60, 1, True)])
def test_choice_of_the_solve_pass(oracle_mod, N, n, d, one):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    sol = Solver(N, n, d_max=d)
    sol.set_option("schur_emu", 1)
    Ad, As, B = _put(s)
    sol.factor(Ad, As)
    X = sol.solve(B).cpu().numpy()
    launches = sol.launch_stats()[0]
    sol.close()
    assert (launches == 1) == one
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    assert oracle_mod.forward_error(X, Xo) <= 1e-12
    assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], X, s["B"]) <= 1e-14


@pytest.mark.parametrize("N,n,d,one", [(40, 20, 4, False), (40, 31, 5, True), (40, 32, 64, False), (40, 33, 23, False),
                                       (40, 39, 24, True), (40, 40, 24, False)])
def test_choice_of_the_solve_pass_in_mixed_precision(oracle_mod, N, n, d, one):
    """With a target that the unrefined solution meets: the pass and one residual."""
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    sol = Solver(N, n, d_max=d, precision="fp32_ir")
    Ad, As, B = _put(s)
    sol.factor(Ad, As)
    X = sol.solve(B).cpu().numpy()
    sol.set_option("target_berr_e18", 10 ** 18)
    sol.solve(B)
    launches = sol.launch_stats()[0]
    sol.close()
    assert (launches == 2) == one
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    assert oracle_mod.forward_error(X, Xo) <= 1e-11


# five to eight right-hand sides: the factorisation's line (launches of the call)
@pytest.mark.parametrize("N,n,d,tc", [(1600, 43, 5, False), (1600, 43, 8, False), (1600, 44, 5, True), (1600, 43, 9, True),
                                      (1600, 43, 4, True), (8192, 40, 5, True)])
def test_choice_of_the_factorisation_for_several_columns(oracle_mod, N, n, d, tc):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    sol = Solver(N, n, d_max=d)
    X = sol.factor_solve(*_put(s)).cpu().numpy()
    launches = sol.launch_stats()[0]
    sol.close()
    assert (launches > 1) == tc
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    assert oracle_mod.forward_error(X, Xo) <= 1e-12
    assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], X, s["B"]) <= 1e-14
