"""GPU: the device memory a handle takes."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bytes(*args, **kw):
    from paper_2509_03015_gb300 import Solver
    Solver(*args, **kw).close()  # context, modules
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    sol = Solver(*args, **kw)
    free1, _ = torch.cuda.mem_get_info()
    sol.close()
    return free0 - free1


def test_mixed_precision_above_64():
    """In FP32: L and L^{-1} of every block, L^{-T} of half of them, the couplings of
    all levels (2 N slots), and three vectors of N n d_max (d_max beyond the sliced
    residual's): 4.5 N n^2 + 3 N n d values, 4.7 N n^2 here; a second set of
    coupling slots would make it 6.7."""
    N, n = 1024, 256
    assert _bytes(N, n, d_max=17, precision="fp32_ir") <= 5 * 4 * N * n * n


@pytest.mark.parametrize("precision,d,before", [("fp32_ir", 1, 8), ("fp64", 1, 6)])
def test_a_handle_without_the_tensor_core_buffers_still_works(oracle_mod, precision, d, before):
    """Where size alone chose the tensor-core path, a handle whose buffers for it do
    not fit runs the persistent kernel, as all of its size once did.  `before`
    allocations come first (fewer of them: the call fails)."""
    import numpy as np
    from paper_2509_03015_gb300 import BDSSError, Solver, _lib, inputs
    N, n = 200, 48
    s = inputs.random_btd(N, n, d, seed=5)
    dev = [torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("A_diag", "A_sub", "B")]
    Xo = oracle_mod.solve_system(s["A_diag"], s["A_sub"], s["B"])
    lib = _lib.load()
    try:
        for k in range(before, before + 6):
            assert lib.bdss_debug_fail_alloc(k) == 0
            if k == before:
                with pytest.raises(BDSSError) as e:
                    Solver(N, n, d_max=d, precision=precision)
                assert e.value.status == 4
                continue
            sol = Solver(N, n, d_max=d, precision=precision)
            lib.bdss_debug_fail_alloc(0)
            sol.set_option("debug_guards", 1)
            X = sol.factor_solve(*dev).cpu().numpy()
            sol.factor(*dev[:2])
            launches = sol.launch_stats()[0]
            X2 = sol.solve(dev[2]).cpu().numpy()
            sol.close()
            assert (launches == 1) == (k <= before + 4)  # the fifth is beyond the path's four buffers
            for x in (X, X2):
                assert oracle_mod.forward_error(x, Xo) <= 1e-11
    finally:
        lib.bdss_debug_fail_alloc(0)
