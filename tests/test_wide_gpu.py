"""GPU: factorisation of 64 < n <= 256 blocks with its products on the tensor
cores, against the CPU oracle, at the edges of its panels (one column past a
panel, odd n, unequal last panels), of its levels (one to nine blocks) and of
its right-hand-side tiles."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _solve(s, host=False, precision="fp64"):
    from paper_2509_03015_gb300 import Solver
    N, n, _ = s["A_diag"].shape
    sol = Solver(N, n, d_max=s["B"].shape[-1], precision=precision)
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()) if host else _dev
    try:
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
@pytest.mark.parametrize("N,n,d", [(1, 65, 1), (2, 66, 2), (3, 96, 17), (4, 127, 3), (5, 128, 16), (6, 129, 1),
                                   (7, 192, 33), (3, 193, 4), (9, 200, 5), (5, 255, 1), (4, 256, 64), (33, 72, 1)])
def test_matches_oracle(oracle_mod, N, n, d):
    s = inputs.random_btd(N, n, d, seed=700 + N + n)
    X, X2, ld = _solve(s)
    L, C = oracle_mod.factor(s["A_diag"], s["A_sub"])
    Xo = oracle_mod.solve(L, C, s["B"])
    ldo = oracle_mod.logdet(L)
    for x in (X, X2):
        assert oracle_mod.forward_error(x, Xo) <= 1e-12
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1e-14
    assert abs(ld - ldo) <= 1e-12 * max(1.0, abs(ldo))


def test_repeats_and_host_inputs_give_the_same_bits():
    s = inputs.random_btd(9, 100, 3, seed=5)
    X, X2, ld = _solve(s)
    Y, Y2, ld2 = _solve(s, host=True)
    assert np.array_equal(X, Y) and np.array_equal(X2, Y2) and ld == ld2


@pytest.mark.parametrize("n", [72, 160])
def test_wide_row_scales(oracle_mod, n):
    """Rows and columns over sixteen binades each way: every operand row is cut
    below its own maximum."""
    s = inputs.random_btd(5, n, 2, seed=12)
    sc = np.logspace(-5, 5, n)
    s["A_diag"] = s["A_diag"] * sc[None, :, None] * sc[None, None, :]
    s["A_sub"] = s["A_sub"] * sc[None, :, None] * sc[None, None, :]
    s["B"] = s["B"] * sc[None, :, None]
    X, _, _ = _solve(s)
    assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], X, s["B"]) <= 1e-14


@pytest.mark.parametrize("what", ["not_spd", "nan_coupling"])
def test_bad_pivot_is_reported(what):
    from paper_2509_03015_gb300 import BDSSError
    s = inputs.random_btd(12, 80, 1, seed=3)
    if what == "not_spd":
        s["A_diag"][6] -= 1e4 * np.eye(80)
    else:
        s["A_sub"][5, 3, 4] = np.nan
    with pytest.raises(BDSSError) as e:
        _solve(s)
    assert e.value.status == 2
    if what == "not_spd":
        assert e.value.info.block == 6 and e.value.info.level == 1


# FP32 factors refined to a backward error of 1e-14 (the call fails otherwise);
# kappa(A) below 1e3 then bounds the forward error by 1e-11.  Shapes whose
# inverse is streamed and shapes (n % 4, d > 16) whose is not; N = 1: the FP64
# top block alone.
@pytest.mark.parametrize("N,n,d", [(1, 100, 2), (2, 65, 1), (3, 66, 3), (5, 128, 16), (6, 132, 17), (9, 193, 2),
                                   (4, 256, 1), (17, 256, 16)])
def test_mixed_precision_matches_oracle(oracle_mod, N, n, d):
    s = inputs.random_btd(N, n, d, seed=800 + N + n)
    X, X2, ld = _solve(s, precision="fp32_ir")
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    for x in (X, X2):
        assert oracle_mod.forward_error(x, Xo) <= 1e-11
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1e-14
    L, _ = oracle_mod.factor(s["A_diag"], s["A_sub"])
    # each of the N n pivots' logarithms is within a few FP32 roundings
    assert abs(ld - oracle_mod.logdet(L)) <= N * n * 2.0 ** -20
