"""Kernels that only large levels take: the staged residual restriction (FP32 from 2048^2), the persistent FP64 box
correction (narrow boxes from 512^2), the tiled FP32 one of wide boxes, the V-cycle launched on the caller's arrays;
and, at the other end, that the smallest levels are one launch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import system  # noqa: E402
from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import TOL32, TOL64, cu, host, rand  # noqa: E402


# aligned arrays take TMA copies inside and single loads at the periodic seam, arrays one value off single loads
# throughout; with and without IB-active tiles; against the FP64 kernel, which stages nothing, each component to its
# own largest value
@pytest.mark.parametrize("make", [lambda: I.thin_ellipse_re(2048, kappa=1e4), lambda: I.no_structure(2048, rho=1.0, seed=4)],
                         ids=["ellipse", "fluid"])
def test_staged_residual_restriction(make):
    prob = make()
    N = prob.N
    S = sib.solver_for(prob, restart=1, max_it=1)
    l, n3 = S.num_levels - 1, 3 * N * N
    gen = torch.Generator(device="cuda").manual_seed(5)
    x, b = (torch.randn(n3, generator=gen, device="cuda") for _ in range(2))
    b = b * 1e4   # of the size of L x on the velocities
    ref = S.residual_restrict(l, x.double(), b.double()).reshape(3, -1)
    shifted = []
    for t in (x, b):
        s = torch.empty(n3 + 1, device="cuda")
        s[1:] = t
        shifted.append(s[1:])
    for args in ((x, b), shifted):
        got = S.residual_restrict(l, *args).double().reshape(3, -1)
        err = (got - ref).abs().amax(1) / ref.abs().amax(1)
        assert (err < TOL32).all(), err
    S.close()


def box(N, b, o, k):
    """dofs of box k's subdomain and which of them the box owns"""
    nb, e = N // b, b + 2 * o
    i0, j0 = (k % nb) * b - o, (k // nb) * b - o
    dofs, own = [], []
    for comp, (wi, wj) in enumerate(((e + 1, e), (e, e + 1), (e, e))):
        jj, ii = np.meshgrid(np.arange(wj), np.arange(wi), indexing="ij")
        dofs.append((comp * N * N + (j0 + jj) % N * N + (i0 + ii) % N).ravel())
        own.append(((ii >= o) & (ii < o + b) & (jj >= o) & (jj < o + b)).ravel())
    return np.concatenate(dofs), np.concatenate(own)


def sweep_of_sampled_boxes(prob, b, o, dtype, tol, tcs):
    """One sweep of the finest level against the local solves of boxes at the corners, of IB boxes and of others"""
    N, nb = prob.N, prob.N // b
    S = sib.solver_for(prob, smoother=sib.SMOOTHER_RAS, box=b, box_overlap=o)
    L = system.operator_of(prob).tocsr()
    rim = (prob.structure.X[:: max(1, prob.structure.M // 12)] * nb).astype(int) % nb
    picks = [0, nb - 1, nb * (nb - 1), nb * nb - 1, nb * (nb // 2) + nb // 2] + [int(j * nb + i) for i, j in rim]
    round_ = (lambda v: v) if dtype == torch.float64 else (lambda v: v.astype(np.float32).astype(np.float64))
    x, rhs = round_(rand(3 * N * N, 8500 + b)), round_(rand(3 * N * N, 8600 + b, 10.0))
    r = rhs - L @ x
    for tc in tcs:
        S.set_options(ras_tc=tc)
        y = cu(x, dtype)
        S.smooth(S.num_levels - 1, y, cu(rhs, dtype), 1)
        y = host(y)
        scale = np.abs(y).max()
        for k in picks:
            d, own = box(N, b, o, k)
            want = x[d[own]] + np.linalg.solve(L[d][:, d].toarray(), r[d])[own]
            assert np.abs(y[d[own]] - want).max() < tol * scale, (tc, k)
    S.close()


# FP64 narrow boxes in the persistent kernel, 48 owned rows of its 64 lanes
def test_persistent_fp64_boxes():
    sweep_of_sampled_boxes(I.thin_ellipse_re(512, kappa=1e4), 4, 1, torch.float64, TOL64, (1,))


# FP32 boxes in tiles: three, 12 and 48 owned rows (one and two rows a lane) of subdomains above six cells, on the CUDA
# cores and on the tensor cores
@pytest.mark.parametrize("b,o", [(1, 3), (2, 3), (4, 2)])
def test_tiled_fp32_boxes(b, o):
    sweep_of_sampled_boxes(I.thin_ellipse_re(256, kappa=1e4), b, o, torch.float32, TOL32, (1, 0))


# the Schur-complement smoother on the caller's arrays and (an array off 16 bytes) on the level's
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_schur_complement_vcycle_on_the_callers_arrays(dtype):
    N = 2048
    S = sib.solver_for(I.thin_ellipse_re(N, kappa=1e2), smoother=sib.SMOOTHER_SC, restart=1, max_it=1)
    b = torch.randn(3 * N * N, device="cuda", dtype=dtype)
    kept = b.clone()
    z = S.vcycle(b)
    off = b.new_empty(3 * N * N + 1)
    off[1:] = b
    assert torch.equal(S.vcycle(off[1:]), z) and torch.equal(b, kept)
    S.close()


# FP32 Vanka levels up to 32^2 are one launch together, in the V-cycle of a 32^2 grid the only one; FP64 and the
# other smoothers keep more
def test_smallest_levels_are_one_launch():
    counts = {}
    for key, dtype, opts in (("cluster", torch.float32, {}), ("separate", torch.float32, dict(fuse_small=0)),
                             ("fp64", torch.float64, {}), ("sc", torch.float32, dict(smoother=sib.SMOOTHER_SC))):
        S = sib.solver_for(I.thin_ellipse_stokes(32, kappa=1e2), **opts)
        b = cu(rand(3 * 32 * 32, 8700), dtype)
        S.vcycle(b)
        before = S.launch_count
        S.vcycle(b)
        counts[key] = S.launch_count - before
        S.close()
    assert counts["cluster"] == 1 and min(counts["separate"], counts["fp64"], counts["sc"]) > 4, counts


# a V-cycle from 2048^2 on copies nothing; one on an array off 16 bytes, or below that size, copies its input and its output
@pytest.mark.parametrize("N,shift,copies", [(2048, 0, 0), (2048, 1, 2), (1024, 0, 2)])
def test_copies_of_a_vcycle(N, shift, copies):
    from torch.profiler import ProfilerActivity, profile

    S = sib.solver_for(I.thin_ellipse_re(N, kappa=1e2), restart=1, max_it=1)
    b = torch.randn(3 * N * N + 1, device="cuda")[shift: 3 * N * N + shift]
    z = torch.empty_like(b)
    S.vcycle(b, z)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        S.vcycle(b, z)
        torch.cuda.synchronize()
    assert sum(e.count for e in p.key_averages() if "Memcpy DtoD" in e.key) == copies
    S.close()
