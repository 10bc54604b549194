"""Boxes of few dofs in large numbers: the persistent, tensor-core and warp-per-box forms of their correction."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_large_levels import sweep_of_sampled_boxes  # noqa: E402
from tests.test_gpu_parity import TOL32, TOL64  # noqa: E402


# both sides of every line: one-cell boxes with 5, 33 and 85 dofs, 2 x 2 boxes with 16, on levels of 1,024, 4,096 and
# 16,384 boxes; IB boxes beside IB-free ones
@pytest.mark.parametrize("dtype,tol", [(torch.float32, TOL32), (torch.float64, TOL64)], ids=["f32", "f64"])
@pytest.mark.parametrize("b,o,N", [(1, 0, 32), (1, 0, 64), (1, 0, 128), (1, 1, 32), (1, 1, 64), (1, 1, 128), (1, 2, 64),
                                   (1, 2, 128), (2, 0, 64), (2, 0, 128)])
def test_small_boxes(b, o, N, dtype, tol):
    sweep_of_sampled_boxes(I.thin_ellipse_re(N, kappa=1e2), b, o, dtype, tol, (1, 0) if dtype == torch.float32 else (1,))


# 65,536 boxes of five dofs in FP64 take about as long as 16,384 of sixteen: both are a pass over the level
def test_time_of_one_cell_boxes():
    N, times = 256, {}
    for b in (1, 2):
        S = sib.solver_for(I.no_structure(N, rho=1.0, seed=4), smoother=sib.SMOOTHER_RAS, box=b, box_overlap=0)
        x, r = torch.zeros(3 * N * N, device="cuda", dtype=torch.float64), torch.ones(3 * N * N, device="cuda",
                                                                                   dtype=torch.float64)
        S.smooth(S.num_levels - 1, x, r, 5)
        best = float("inf")
        for _ in range(5):
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            S.smooth(S.num_levels - 1, x, r, 20)
            e.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(e))
        times[b] = best
        S.close()
    assert times[1] < 2 * times[2], times
