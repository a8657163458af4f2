"""GPU: assembly of the Kalman-smoother normal equations on both sides of the line
between the FP64-ALU tiles (few or small steps) and the digit products."""
import numpy as np
import pytest

import oracle
from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# sums of at most n + m <= 97 products of O(1) terms round to within 97 eps of the
# largest magnitude; 1e-13 leaves room
RTOL = 1e-13


@pytest.mark.parametrize("N,n,m", [(1, 48, 48), (1, 48, 49), (1, 90, 6), (20, 24, 24), (20, 24, 25), (33, 40, 8), (33, 1, 48),
                                   (128, 10, 10), (128, 10, 11), (2000, 5, 5), (2000, 5, 6), (2000, 1, 9), (2000, 1, 12),
                                   (1301, 2, 17), (1300, 7, 4), (700, 9, 3)])
@pytest.mark.parametrize("diag", [False, True])
def test_matches_oracle(N, n, m, diag):
    from paper_2509_03015_gb300 import kalman_assemble
    mod = inputs.kalman_model(N, n, m, seed=N + 3 * n + m)
    if diag:
        mod["Rinv"] = np.ascontiguousarray(np.einsum("kii->ki", mod["Rinv"]))
    d = {k: torch.from_numpy(v).cuda() for k, v in mod.items()}
    got = kalman_assemble(d["G"], d["H"], d["Qinv"], d["Rinv"], d["z"], d["zeta"])
    full = np.stack([np.diag(r) for r in mod["Rinv"]]) if diag else mod["Rinv"]
    want = oracle.kalman_assemble(mod["G"], mod["H"], mod["Qinv"], full, mod["z"], mod["zeta"])
    for g, w in zip(got, want):
        if w.size:
            scale = max(1.0, float(np.abs(w).max()))
            np.testing.assert_allclose(g.cpu().numpy(), w, rtol=0, atol=RTOL * scale)
