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
