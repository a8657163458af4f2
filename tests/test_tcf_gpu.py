"""GPU: factorisation of n <= 64 blocks with the coupling solves and Schur
products on the tensor cores (digit products), against the CPU oracle and the
FP64-ALU path, at the edges of its tiles: 32 and 64 rows, odd n, one or both
couplings, right-hand sides across the 16-column rounds."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _solve(s, tc, host=False):
    from paper_2509_03015_gb300 import Solver
    N, n, _ = s["A_diag"].shape
    sol = Solver(N, n, d_max=s["B"].shape[-1])
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()) if host else _dev
    try:
        sol.set_option("schur_emu", int(tc))
        sol.set_option("debug_guards", 1)
        Ad, As, B = put(s["A_diag"]), put(s["A_sub"]), put(s["B"])
        X = sol.factor_solve(Ad, As, B).cpu().numpy()
        ld = sol.logdet()
        X2 = sol.solve(B).cpu().numpy()
        return X, X2, ld
    finally:
        sol.close()


# random_btd blocks are diagonally dominant with kappa(A) below 1e3, so a
# backward-stable solve is within kappa u times a small factor of the oracle:
# 1e-12 forward, 1e-14 backward (the repository's bar), log det relative 1e-12
@pytest.mark.parametrize("N,n,d", [(2, 32, 1), (3, 34, 2), (4, 32, 16), (5, 33, 17), (6, 47, 3), (7, 63, 1),
                                   (8, 64, 33), (9, 64, 1), (33, 40, 4), (130, 36, 5), (257, 64, 2)])
def test_matches_oracle(oracle_mod, N, n, d):
    s = inputs.random_btd(N, n, d, seed=900 + N + n)
    X, X2, ld = _solve(s, True)
    L, C = oracle_mod.factor(s["A_diag"], s["A_sub"])
    Xo = oracle_mod.solve(L, C, s["B"])
    ldo = oracle_mod.logdet(L)
    for x in (X, X2):
        assert oracle_mod.forward_error(x, Xo) <= 1e-12
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1e-14
    assert abs(ld - ldo) <= 1e-12 * max(1.0, abs(ldo))


def test_repeats_and_host_inputs_give_the_same_bits():
    s = inputs.random_btd(70, 52, 3, seed=5)
    X, X2, ld = _solve(s, True)
    Y, Y2, ld2 = _solve(s, True, host=True)
    assert np.array_equal(X, Y) and np.array_equal(X2, Y2) and ld == ld2


@pytest.mark.parametrize("n", [32, 64])
def test_wide_row_scales(oracle_mod, n):
    """Rows and columns over sixteen binades each way: every operand row is cut
    below its own maximum."""
    s = inputs.random_btd(9, n, 2, seed=12)
    sc = np.logspace(-5, 5, n)
    s["A_diag"] = s["A_diag"] * sc[None, :, None] * sc[None, None, :]
    s["A_sub"] = s["A_sub"] * sc[None, :, None] * sc[None, None, :]
    s["B"] = s["B"] * sc[None, :, None]
    X, _, _ = _solve(s, True)
    assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], X, s["B"]) <= 1e-14


@pytest.mark.parametrize("what", ["not_spd", "nan_coupling"])
def test_bad_pivot_is_reported(what):
    from paper_2509_03015_gb300 import BDSSError
    s = inputs.random_btd(12, 40, 1, seed=3)
    if what == "not_spd":
        s["A_diag"][6] -= 1e4 * np.eye(40)
    else:
        s["A_sub"][5, 3, 4] = np.nan
    with pytest.raises(BDSSError) as e:
        _solve(s, True)
    assert e.value.status == 2
    if what == "not_spd":
        assert e.value.info.block == 6 and e.value.info.level == 1


# mixed precision takes the path by size; the call refines to a backward error
# of 1e-14, and kappa(A) below 1e3 then bounds the forward error by 1e-11
@pytest.mark.parametrize("N,n,d,precision", [(2048, 40, 1, "fp32_ir"), (2049, 63, 3, "tf32_ir"),
                                             (2100, 64, 17, "fp32_ir")])
def test_mixed_precision_matches_oracle(oracle_mod, N, n, d, precision):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    sol = Solver(N, n, d_max=d, precision=precision)
    X = sol.factor_solve(_dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"])).cpu().numpy()
    X2 = sol.solve(_dev(s["B"])).cpu().numpy()
    sol.close()
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    for x in (X, X2):
        assert oracle_mod.forward_error(x, Xo) <= 1e-11
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1.1e-14


# the line of the choice by size, both sides of it (launches of the call: one
# for the persistent kernel), with the tolerances above
@pytest.mark.parametrize("N,n,d,tc", [(127, 48, 1, False), (128, 48, 1, True), (128, 47, 1, False), (128, 48, 2, False),
                                      (1536, 40, 2, True), (1535, 40, 2, False)])
def test_choice_by_size(oracle_mod, N, n, d, tc):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, d, seed=N + n)
    sol = Solver(N, n, d_max=d)
    X = sol.factor_solve(_dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"])).cpu().numpy()
    launches = sol.launch_stats()[0]
    sol.close()
    assert (launches > 1) == tc
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    assert oracle_mod.forward_error(X, Xo) <= 1e-12
    assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], X, s["B"]) <= 1e-14
