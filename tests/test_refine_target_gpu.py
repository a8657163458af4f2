"""GPU: the refinement stops at the first iterate whose backward error meets
the target, however narrowly."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.mark.parametrize("N,n,precision", [(40, 24, "fp32_ir"), (9, 96, "tf32_ir")])
@pytest.mark.parametrize("krylov", [0, 1, 2])
def test_a_target_just_above_the_attained_error_is_met(N, n, precision, krylov):
    from paper_2509_03015_gb300 import Solver
    s = inputs.random_btd(N, n, 2, seed=N + n)
    Ad, As, B = _dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"])
    sol = Solver(N, n, d_max=2, precision=precision)
    sol.set_option("target_berr_e18", 10 ** 18)
    X0 = sol.factor_solve(Ad, As, B)
    first = sol.last_info.backward_err  # the unrefined solution's, the same in every call
    sol.set_option("refine_krylov", krylov)
    for margin in (1.001, 1.02, 1.04):
        sol.set_option("target_berr_e18", int(first * 1e18 * margin) + 1)
        X = sol.factor_solve(Ad, As, B)
        assert sol.last_info.backward_err <= first * margin * (1 + 1e-9)
        assert sol.last_info.iters == 0 and torch.equal(X, X0)
    sol.close()
