"""Kernels at the sizes where their tiling can go wrong, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ib, multigrid, system  # noqa: E402
from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import TOL32, TOL64, cu, host, rand, rel  # noqa: E402

EPS = 2.0 ** -53


# grids below, at and above one 32 x 8 tile; single markers; a cell that holds every marker, with as many as
# the counting sort orders itself and one more; markers outside the unit square (they wrap); more chunks of
# bins than a scan block has threads
@pytest.mark.parametrize("N,M,where", [(4, 1, "any"), (8, 3, "any"), (16, 200, "any"), (32, 1, "seam"), (32, 700, "cell"),
                                       (64, 999, "any"), (64, 64, "seam"), (128, 5001, "any"), (256, 37, "outside"),
                                       (32, 64, "cell"), (32, 65, "cell"), (1024, 20000, "any")])
def test_spread_tiles(N, M, where):
    rng = np.random.default_rng(100 * N + M)
    X = rng.uniform(0.0, 1.0, (M, 2))
    if where == "cell":
        X = (5.0 + rng.uniform(0.0, 1.0, (M, 2))) / N
    elif where == "seam":
        X[:, 0] = rng.uniform(-1.0, 1.0, M) / N
    elif where == "outside":
        X = X * 3.0 - 1.0
    F = rng.standard_normal((M, 2))
    edges = np.array([[0, M - 1]], dtype=np.int32)
    S = sib.Solver(N, n_min=4)
    S.set_structure(cu(X), torch.as_tensor(edges, device="cuda"), cu(np.array([1.0])))
    S.setup()
    f = S.spread(cu(F)).cpu().numpy()
    ref = ib.spread_force(N, X, F)
    # every term carries at most five roundings beside those of the weights (phi to a few ulp of its
    # terms' magnitude, 1), and a face sums at most M of them; magnitudes from |S| |F|
    mag = np.concatenate([abs(ib.spread_matrix(N, X, c)) @ np.abs(F[:, c]) for c in (0, 1)])
    tol = (2 * M + 8) * EPS * mag + 64 * EPS * N * N * np.abs(F).max()
    assert (np.abs(f - ref) <= tol).all(), np.abs(f - ref).max()
    assert torch.equal(S.spread(cu(F)), S.spread(cu(F)))
    S.close()


# Box set-up by block elimination: one cell, one face row more than the box, ragged row tiles (12, 48 and
# 192 owned rows in tiles of 32), the widest subdomain it takes (14 cells) and subdomains whose faces wrap
# around a small level.  One FP64 sweep per level to the repository's FP64 bar.
@pytest.mark.parametrize("b,o,N,kappa", [(1, 0, 32, 1e2), (1, 2, 32, 1e2), (2, 6, 32, 1e2), (4, 5, 32, 1e4), (8, 3, 32, 1e2),
                                         (4, 1, 16, 1e4)])
def test_box_inverses(b, o, N, kappa):
    prob = I.thin_ellipse_stokes(N, kappa=kappa)
    H = multigrid.Hierarchy(prob, smoother="ras", box=b, overlap=o)
    S = sib.solver_for(prob, smoother=sib.SMOOTHER_RAS, box=b, box_overlap=o)
    for l in range(1, len(H.levels)):
        n3 = 3 * H.levels[l].n
        x, rhs = rand(n3, 7000 + l), rand(n3, 7100 + l, 10.0)
        y = cu(x.copy())
        S.smooth(l, y, cu(rhs), 1)
        ref = H.smooth(l, x, rhs, 1)
        assert rel(host(y), ref) < TOL64, (l, rel(host(y), ref))
    S.close()


# The tensor-core tiles of narrow boxes on a level above 128^2 (levels up to 128^2 take the split form), 64
# and 128 boxes a row; one FP32 sweep to the repository's FP32 bar, with the CUDA-core form beside it.
@pytest.mark.parametrize("make,b,o", [(lambda: I.thin_ellipse_re(256, kappa=1e4), 4, 1),
                                      (lambda: I.no_structure(256, rho=1.0, seed=4), 2, 1)], ids=["4x4", "2x2"])
def test_narrow_boxes_on_tensor_cores(make, b, o):
    prob = make()
    H = multigrid.Hierarchy(prob, smoother="ras", box=b, overlap=o)
    S = sib.solver_for(prob, smoother=sib.SMOOTHER_RAS, box=b, box_overlap=o)
    l = len(H.levels) - 1
    x = rand(3 * H.levels[l].n, 7200 + b).astype(np.float32).astype(np.float64)
    rhs = rand(3 * H.levels[l].n, 7300 + b, 10.0).astype(np.float32).astype(np.float64)
    ref = H.smooth(l, x, rhs, 1)
    for tc in (1, 0):
        S.set_options(ras_tc=tc)
        y = cu(x, torch.float32)
        S.smooth(l, y, cu(rhs, torch.float32), 1)
        assert rel(host(y), ref) < TOL32, (tc, rel(host(y), ref))
    y = cu(x)
    S.smooth(l, y, cu(rhs), 1)
    assert rel(host(y), ref) < TOL64, rel(host(y), ref)
    S.close()


# Galerkin windows of every level, down to 4 x 4 cells, where window offsets alias, and the coarsest
# pseudo-inverse by block elimination (4 and 8 cells) and by Gauss-Jordan (16), with and without a density
@pytest.mark.parametrize("n_min", [4, 8, 16])
@pytest.mark.parametrize("make", [lambda: I.disk_stokes(32, kappa=1e4, seed=1), lambda: I.thin_ellipse_re(64, kappa=1e4)],
                         ids=["stokes", "re"])
def test_coarse_levels(make, n_min):
    prob = make()
    H = multigrid.Hierarchy(prob, n_min=n_min)
    st = prob.structure
    S = sib.Solver(prob.N, n_min=n_min)
    S.set_fluid(prob.rho, prob.mu, prob.dt)
    S.set_structure(cu(st.X), torch.as_tensor(st.edges, device="cuda"), cu(st.kappa))
    S.setup()
    for l, lev in enumerate(H.levels):
        u = rand(2 * lev.n, 7400 + l)
        assert rel(host(S.apply_ib(l, cu(u))), lev.B @ u) < TOL64, l
    b = rand(3 * n_min * n_min, 7500)
    assert rel(host(S.coarse_solve(cu(b))), H.coarse_pinv @ b) < TOL64
    S.close()


# 16 x 16 boxes in FP32 on levels with a whole and with a partial group of eight IB boxes, and with boxes
# that have none: the correction of a residual that FP32 holds exactly (a sweep from zero) against the FP64
# level's, to the repository's FP32 bar
@pytest.mark.parametrize("kind,N,gamma,o", [("circle", 64, 50.0, 4), ("circle", 128, 500.0, 4), ("annulus", 128, 5.0, 4),
                                            ("circle", 128, 50.0, 2)])
def test_wide_boxes_in_pairs_of_floats(kind, N, gamma, o):
    S = sib.solver_for(I.paper_problem(kind, N, gamma), smoother=sib.SMOOTHER_RAS, box=16, box_overlap=o)
    for l in range(1, S.num_levels):
        n3 = 3 * (8 << l) ** 2
        b = rand(n3, 7700 + l).astype(np.float32)
        y32, y64 = cu(np.zeros(n3), torch.float32), cu(np.zeros(n3))
        S.smooth(l, y32, cu(b, torch.float32), 1)
        S.smooth(l, y64, cu(b.astype(np.float64)), 1)
        assert rel(host(y32), host(y64)) < TOL32, l
    S.close()


# The cluster kernel's levels: one, two and three of them, strips of one, two and four rows, as the whole
# V-cycle or below a 64^2 level, with and without IB windows; to the repository's bar for an FP32 V-cycle
@pytest.mark.parametrize("n_min,N", [(4, 8), (4, 16), (4, 32), (8, 16), (8, 32), (8, 64), (4, 64)])
@pytest.mark.parametrize("make", [lambda N: I.disk_stokes(N, kappa=1e2, seed=1), lambda N: I.no_structure(N, rho=1.0, seed=4)],
                         ids=["disk", "fluid"])
def test_cluster_levels(make, n_min, N):
    prob = make(N)
    H = multigrid.Hierarchy(prob, n_min=n_min)
    st = prob.structure
    S = sib.Solver(N, n_min=n_min)
    S.set_fluid(prob.rho, prob.mu, prob.dt)
    if st.M > 0:
        S.set_structure(cu(st.X), torch.as_tensor(st.edges, device="cuda"), cu(st.kappa))
    S.setup()
    b = rand(3 * N * N, 7600 + N).astype(np.float32).astype(np.float64)
    b[2 * N * N:] -= b[2 * N * N:].mean()
    z = S.vcycle(cu(b, torch.float32))
    assert rel(host(z), H.vcycle(b)) < 1e-4
    assert torch.equal(S.vcycle(cu(b, torch.float32)), z)
    S.close()


# Arnoldi steps of one, two and three groups of eight vectors, on vectors shorter than a slice and longer; the
# true residual, formed after the solve, is the stopping test's to rounding
@pytest.mark.parametrize("N,n_min", [(8, 4), (32, 8), (128, 8)])
@pytest.mark.parametrize("restart", [7, 8, 9, 17, 100])
def test_arnoldi_lengths(N, n_min, restart):
    prob = I.disk_stokes(N, kappa=1e2, seed=1)
    st, its = prob.structure, []
    for graphs in (1, 0):
        S = sib.Solver(N, n_min=n_min)
        S.set_fluid(prob.rho, prob.mu, prob.dt)
        S.set_options(rtol=1e-10, restart=restart, max_it=200, use_graphs=graphs)
        S.set_structure(cu(st.X), torch.as_tensor(st.edges, device="cuda"), cu(st.kappa))
        S.setup()
        S.solve(cu(prob.g))
        assert S.stats.converged and S.stats.rel_residual < 2e-10, (graphs, S.stats.rel_residual)
        its.append(S.stats.iterations)
        S.close()
    assert abs(its[0] - its[1]) <= 1, its


# The V-cycle on the caller's arrays (grids from 2048^2 on) and on the level's (an array that is not aligned, an
# output that is the input) are the same kernels on the same values
@pytest.mark.parametrize("dtype,smoother", [(torch.float32, 0), (torch.float64, 0), (torch.float32, sib.SMOOTHER_RAS)])
def test_vcycle_on_the_callers_arrays(dtype, smoother):
    N = 2048
    S = sib.solver_for(I.thin_ellipse_re(N, kappa=1e2), smoother=smoother, restart=1, max_it=1)
    b = torch.randn(3 * N * N + 1, device="cuda", dtype=dtype)
    z = S.vcycle(b[:-1])
    off = b[:-1].new_empty(3 * N * N + 1)
    off[1:] = b[:-1]
    assert torch.equal(S.vcycle(off[1:]), z)
    same = b[:-1].clone()
    assert S.vcycle(same, same) is same and torch.equal(same, z)
    S.close()


# Orthogonalisation steps in a cluster: levels of up to 128^2 (the largest it takes) and 256^2 (above), stages of one
# to five steps, both precisions; the V-cycle to the repository's bars
@pytest.mark.parametrize("N,nu1,nu2", [(16, 1, 1), (32, 2, 3), (128, 2, 2), (128, 5, 1), (256, 1, 2)])
def test_wrapped_steps_in_a_cluster(N, nu1, nu2):
    prob = I.disk_stokes(N, kappa=1e2, seed=1)
    H = multigrid.Hierarchy(prob, smoother="vanka", krylov=True, nu1=nu1, nu2=nu2)
    S = sib.solver_for(prob, smooth_krylov=1, nu1=nu1, nu2=nu2)
    b = system.rhs(prob).astype(np.float32).astype(np.float64)
    ref = H.vcycle(b)
    assert rel(host(S.vcycle(cu(b))), ref) < TOL64
    assert rel(host(S.vcycle(cu(b, torch.float32))), ref) < 1e-4
    S.close()
