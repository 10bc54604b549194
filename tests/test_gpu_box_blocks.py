"""The FP64 correction of 16 x 16 IB boxes, a block each: blocks do not share an SM while others are idle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402


def test_time_follows_the_largest_box():
    """16 boxes at 64^2 and 64 at 128^2, of about the same size, all at once: the same time but for the shared part."""
    times = {}
    for N in (64, 128):
        S = sib.solver_for(I.paper_problem("circle", N, 50.0), smoother=sib.SMOOTHER_RAS, box=16, box_overlap=4)
        x = torch.zeros(3 * N * N, device="cuda", dtype=torch.float64)
        b = torch.ones_like(x)
        S.smooth(S.num_levels - 1, x, b, 2)
        best = float("inf")
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            S.smooth(S.num_levels - 1, x, b, 4)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times[N] = best
        S.close()
    assert times[128] < 1.3 * times[64], times
