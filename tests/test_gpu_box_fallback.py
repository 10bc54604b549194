"""Box inverses whose velocity blocks lose their definiteness to rounding: the set-up inverts with pivoting instead."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import smoothers, system  # noqa: E402
from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import TOL64, cu, host, rand  # noqa: E402

N = 32


def set_up(prob, b, o):
    st = prob.structure
    S = sib.Solver(N)
    S.set_fluid(prob.rho, prob.mu, prob.dt)
    S.set_options(smoother=sib.SMOOTHER_RAS, box=b, box_overlap=o)
    S.set_structure(cu(st.X), torch.as_tensor(st.edges, device="cuda"), cu(st.kappa))
    before = S.launch_count
    S.setup()
    return S, S.launch_count - before


# twelve springs whose stiffness swallows the stencil (1e22: the rounding errors of a block's entries are 100 times the
# stencil's), a narrow and a wide box: one more launch a level, and the boxes away from these springs as the oracle has them
@pytest.mark.parametrize("b,o", [(4, 1), (8, 2)])
def test_indefinite_blocks(b, o):
    prob = I.thin_ellipse_stokes(N, kappa=1e2)
    st = prob.structure
    S, usual = set_up(prob, b, o)
    S.close()
    near = np.abs(st.X[:, 0] - 0.8) + np.abs(st.X[:, 1] - 0.5) < 0.1
    stiff = near[st.edges[:, 0]] & near[st.edges[:, 1]]
    assert stiff.sum() == 12
    st.kappa[stiff] = 1e22
    S, launches = set_up(prob, b, o)
    levels = [l for l in range(1, S.num_levels) if not smoothers.ras_wraps(S.level_size(l), b, o)]
    assert launches - usual == len(levels)
    l = S.num_levels - 1
    L = system.operator_of(prob).tocsr()
    rhs = rand(3 * N * N, 8300 + b, 10.0)
    y = cu(np.zeros(3 * N * N))
    S.smooth(l, y, cu(rhs), 1)
    y, omega, checked = host(y), S.opts.omega if S.opts.omega > 0 else 1.0, 0
    assert np.isfinite(y).all()
    for d, own in smoothers.ras_boxes(N, b, o):
        A = L[d][:, d].toarray()
        if np.abs(A).max() > 1e10:
            continue
        want = omega * np.linalg.solve(A, rhs[d])[own]
        assert np.abs(y[d[own]] - want).max() < TOL64 * np.abs(want).max()
        checked += 1
    assert checked >= 12
    S.close()


# stiffnesses whose products overflow: no inverse by either elimination, and the set-up says so
@pytest.mark.parametrize("b,o", [(4, 1), (8, 2)])
def test_overflowing_blocks_are_refused(b, o):
    prob = I.thin_ellipse_stokes(N, kappa=1e308)
    with pytest.raises(sib.SibError, match="singular"):
        set_up(prob, b, o)
    S, _ = set_up(I.thin_ellipse_stokes(N, kappa=1e2), b, o)
    y = cu(np.zeros(3 * N * N))
    S.smooth(S.num_levels - 1, y, cu(rand(3 * N * N, 8400)), 1)
    assert torch.isfinite(y).all()
    S.close()
