"""GPU: assembly of the Kalman-smoother normal equations at the edges of its
tiles: odd numbers of steps (two steps share a tile up to n = 64), 32 and 64
columns, one column more, several K chunks, diagonal precisions."""
import numpy as np
import pytest

import oracle
from paper_2509_03015_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the oracle's sums of at most n + m <= 556 products of O(1) terms round to
# within 556 eps of the largest magnitude; 1e-12 leaves room
RTOL = 1e-12


@pytest.mark.parametrize("N,n,m,diag", [(1, 1, 1, False), (3, 31, 64, False), (2, 32, 65, True), (5, 33, 1, False),
                                        (4, 63, 129, True), (3, 64, 63, False), (2, 65, 64, False), (3, 128, 130, True),
                                        (2, 129, 33, False), (2, 256, 300, False)])
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
