"""sib_device_bytes counts what a context holds, not what it has allocated on the way."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import cu  # noqa: E402


# every smoother whose set-up takes temporaries (box inverses of all widths, the exact level solve), the time
# step's sequence of a new structure and a new set-up
@pytest.mark.parametrize("box,overlap", [(0, 0), (2, 1), (4, 1), (8, 2), (16, 4)])
def test_repeated_setup_holds_the_same(box, overlap):
    opts = dict(smoother=sib.SMOOTHER_RAS, box=box, box_overlap=overlap) if box else {}
    prob = I.paper_problem("annulus", 64, 50.0)
    st = prob.structure
    S = sib.solver_for(prob, **opts)
    held = S.device_bytes
    for _ in range(3):
        S.set_structure(cu(st.X), torch.as_tensor(st.edges, device="cuda"), cu(st.kappa))
        S.setup()
        assert S.device_bytes == held
    S.close()
