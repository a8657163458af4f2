"""GPU: diagonal blocks of condition 1e8 and more, coupled as strongly as an SPD
system allows.  The tensor-core paths multiply with the inverse of a block's
triangular factor where a substitution would do; the solution has to be as
backward stable."""
import numpy as np
import pytest

from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _system(N, n, d, kappa, seed):
    """A_ii = U diag(1 .. 1/kappa) U^T, A_{i+1,i} = 0.45 A_{i+1,i+1}^1/2 (orthogonal)
    A_ii^1/2: kappa(A) is about 10 kappa."""
    rng = np.random.default_rng(seed)
    lam = np.logspace(0.0, -np.log10(kappa), n)
    A, H = np.empty((N, n, n)), np.empty((N, n, n))
    for i in range(N):
        U = inputs.haar_orthogonal(rng, n)
        A[i], H[i] = (U * lam) @ U.T, (U * np.sqrt(lam)) @ U.T
        A[i] = 0.5 * (A[i] + A[i].T)
    S = np.stack([0.45 * H[i + 1] @ inputs.haar_orthogonal(rng, n) @ H[i] for i in range(N - 1)])
    return dict(A_diag=A, A_sub=S, B=rng.standard_normal((N, n, d)))


# a CPU model of the elimination gives 2e-17 with substitutions and 5e-17 with the
# inverses at any kappa; 1e-15 leaves room, and two solutions that stable differ by
# kappa(A) times a few u
@pytest.mark.parametrize("N,n,d", [(9, 40, 1), (33, 64, 16), (9, 96, 2), (5, 256, 1)])
@pytest.mark.parametrize("kappa", [1e8, 1e11])
def test_fp64_is_backward_stable(oracle_mod, N, n, d, kappa):
    from paper_2509_03015_gb300 import Solver
    s = _system(N, n, d, kappa, seed=n)
    sol = Solver(N, n, d_max=d)
    sol.set_option("schur_emu", 1)
    X = sol.factor_solve(_dev(s["A_diag"]), _dev(s["A_sub"]), _dev(s["B"])).cpu().numpy()
    X2 = sol.solve(_dev(s["B"])).cpu().numpy()
    sol.close()
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    for x in (X, X2):
        assert oracle_mod.backward_error(s["A_diag"], s["A_sub"], x, s["B"]) <= 1e-15
        assert oracle_mod.forward_error(x, Xo) <= 10 * kappa * 2.2e-16 * 50
