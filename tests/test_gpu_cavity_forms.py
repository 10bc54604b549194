"""The two forms of the cavity's Vanka sweep (one launch, and residual, patches and update apart) and which levels take
which."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import TOL32, cu, host, rand, rel  # noqa: E402


def launches(S, f):
    before = S.launch_count
    f()
    return S.launch_count - before


# FP32 on both sides of the line against the FP64 form, sweeps and a V-cycle (its first sweeps start from zero), to
# the repository's bars; FP64 takes three launches everywhere, FP32 one below 256^2 (512^2 without a structure)
@pytest.mark.parametrize("kind,N,three", [("annulus", 32, False), ("annulus", 128, False), ("annulus", 256, True),
                                          ("none", 256, False), ("none", 512, True)])
def test_forms_of_the_sweep(kind, N, three):
    prob = I.paper_problem("annulus", N, 5.0) if kind == "annulus" else I.no_structure(N, rho=1.0, seed=4)
    S = sib.solver_for(prob, domain=sib.DOMAIN_CAVITY)
    l, n = S.num_levels - 1, N * N

    def field(seed, scale):   # values that FP32 holds, zero on the wall faces
        v = cu(rand(3 * n, seed, scale), torch.float32).reshape(3, N, N)
        v[0, :, 0] = 0
        v[1, 0, :] = 0
        return v.reshape(-1)

    x, b = field(8800 + N, 1.0), field(8900 + N, 1e4)
    x64, x32 = x.double(), x.clone()
    ib = launches(S, lambda: S.apply_ib(l, x64[: 2 * n]))
    assert launches(S, lambda: S.cavity_smooth(l, x64, b.double(), 2)) == 2 * (3 + ib)
    ib = launches(S, lambda: S.apply_ib(l, x32[: 2 * n]))
    assert launches(S, lambda: S.cavity_smooth(l, x32, b, 2)) == 2 * ((3 if three else 1) + ib)
    assert rel(host(x32), host(x64)) < TOL32
    assert rel(host(S.vcycle(b)), host(S.vcycle(b.double()))) < 1e-4
    S.close()
