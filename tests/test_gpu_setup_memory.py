"""What a set-up holds at a time."""
import threading
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402


# 16 x 16 boxes of a thick structure: the low-rank matrices W of the levels' IB boxes (420 MB in FP64, as much in pairs of
# floats) and workspaces of twice a level's; with those of all levels at once the peak lay 0.9 GB above what stays
def test_wide_boxes_free_their_workspaces():
    torch.zeros(1, device="cuda")
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    prob = I.paper_problem("annulus", 256, 50.0)
    S = sib.Solver(prob.N)
    S.set_fluid(prob.rho, prob.mu, prob.dt)
    S.set_options(smoother=sib.SMOOTHER_RAS, box=16, box_overlap=4, restart=1, max_it=1)
    st = prob.structure
    args = [torch.as_tensor(a, device="cuda") for a in (st.X, st.edges, st.kappa)]
    S.set_structure(*args)
    lowest, stop = [torch.cuda.mem_get_info()[0]], []

    def watch():
        while not stop:
            lowest[0] = min(lowest[0], torch.cuda.mem_get_info()[0])
            time.sleep(0.0005)

    thread = threading.Thread(target=watch)
    thread.start()
    S.setup()
    torch.cuda.synchronize()
    stop.append(1)
    thread.join()
    now = torch.cuda.mem_get_info()[0]
    above, held = now - lowest[0], free - now
    assert above < 0.5 * held, (above >> 20, held >> 20)
    S.close()
