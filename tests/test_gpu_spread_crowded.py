"""Spreading where cells hold many markers, against the oracle, and its time beside an even distribution's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ib  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import cu  # noqa: E402

EPS = 2.0 ** -53


def solver(N, X):
    S = sib.Solver(N, n_min=4)
    S.set_options(restart=1, max_it=1)
    S.set_structure(cu(X), torch.tensor([[0, len(X) - 1]], dtype=torch.int32, device="cuda"), cu(np.array([1.0])))
    S.setup()
    return S


# the largest cell at, and one above, what the thread-per-column form takes (24 + M / 6000, where the other markers lie
# one a cell); grids of one tile and smaller; a cell at the seam; a line of crowded cells; cells the counting sort
# leaves to the network
@pytest.mark.parametrize("N,where,per", [(128, "cell", 24), (128, "cell", 25), (4, "cell", 40), (16, "cell", 300),
                                         (32, "seam", 70), (64, "seam", 25), (256, "line", 30), (128, "line", 80)])
def test_crowded_cells(N, where, per):
    rng = np.random.default_rng(1000 * N + per)
    if where == "line":
        X = np.stack([rng.uniform(0.0, 1.0, N * per), (N // 2 + 0.3 + rng.uniform(0.0, 0.4, N * per)) / N], 1)
    else:
        cell = np.array([N - 1, N - 1] if where == "seam" else [N // 2, 1])
        X = (cell + 0.55 + 0.4 * rng.uniform(0.0, 1.0, (per, 2))) / N   # one bin of both components
        i = np.arange(0, N, 2)   # other cells: one marker each
        rest = (np.stack(np.meshgrid(i, i), -1).reshape(-1, 2) + 0.25) / N
        X = np.concatenate([X, rest[np.abs(rest * N - cell).max(1) > 1.5]])
    M = len(X)
    F = rng.standard_normal((M, 2))
    S = solver(N, X)
    f = S.spread(cu(F)).cpu().numpy()
    ref = ib.spread_force(N, X, F)
    # at most five roundings a term beside those of the weights (a few ulp of 1), at most M terms a face
    mag = np.concatenate([abs(ib.spread_matrix(N, X, c)) @ np.abs(F[:, c]) for c in (0, 1)])
    tol = (2 * M + 8) * EPS * mag + 64 * EPS * N * N * np.abs(F).max()
    assert (np.abs(f - ref) <= tol).all(), np.abs(f - ref).max()
    assert torch.equal(S.spread(cu(F)), S.spread(cu(F)))
    S.close()


# 20,000 markers in one cell: every one of 16 faces sums them all, which a warp does in some 0.1 ms (a single thread
# takes 6 ms); evenly over 128^2 the same markers take about 25 us
def test_time_of_a_crowded_cell():
    rng = np.random.default_rng(0)
    U = rng.uniform(0.0, 1.0, (20000, 2))
    times = []
    for X in (U, (5.0 + U) / 128):
        S = solver(128, X)
        F = cu(rng.standard_normal(X.shape))
        for _ in range(3):
            S.spread(F)
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(10):
                S.spread(F)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 10)
        times.append(best)
        S.close()
    assert times[1] < 40 * times[0], times


# the call without allocations, whose tiles choose their form on the device: crowded tiles beside ordinary ones, the
# largest cell on both sides of the line, a grid below a tile
@pytest.mark.parametrize("N,per", [(64, 24), (64, 25), (64, 2000), (32, 100), (256, 40), (16, 100)])
def test_crowded_cells_without_allocations(N, per):
    import ctypes

    rng = np.random.default_rng(2000 * N + per)
    X = np.concatenate([(np.array([1, N // 2]) + 0.55 + 0.4 * rng.uniform(0.0, 1.0, (per, 2))) / N,
                        rng.uniform(0.0, 1.0, (500, 2))])
    M = len(X)
    F = rng.standard_normal((M, 2))
    Xd, Fd, f = cu(X), cu(F), torch.full((2 * N * N,), 7.0, dtype=torch.float64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = sib.load().sib_spread_noalloc(N, M, p(Xd), p(Fd), p(f),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == sib.SIB_OK
    ref = ib.spread_force(N, X, F)
    mag = np.concatenate([abs(ib.spread_matrix(N, X, c)) @ np.abs(F[:, c]) for c in (0, 1)])
    tol = (2 * M + 8) * EPS * mag + 64 * EPS * N * N * np.abs(F).max()
    assert (np.abs(f.cpu().numpy() - ref) <= tol).all()
