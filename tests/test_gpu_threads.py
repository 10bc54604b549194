"""Solvers of different sizes in different host threads of one process (contexts are independent of each other)."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import inputs as I  # noqa: E402
from paper_1612_02208_gb300 import sib  # noqa: E402

from tests.test_gpu_parity import cu, rand  # noqa: E402


def in_thread(f):
    """f() in a thread of its own; its result, or its exception raised here"""
    out = []

    def body():
        try:
            out.append((f(), None))
        except Exception as e:  # noqa: BLE001
            out.append((None, e))

    t = threading.Thread(target=body)
    t.start()
    t.join()
    value, error = out[0]
    if error is not None:
        raise error
    return value


class Work:
    """One sweep of the finest level, or (graphs off) one V-cycle, of a solver with the given options"""

    def __init__(self, N, what, dtype, **opts):
        self.S = sib.solver_for(I.paper_problem("circle", N, 50.0), use_graphs=0, **opts)
        self.what = what
        self.b = cu(rand(3 * N * N, 8000 + N), dtype)

    def __call__(self):
        if self.what == "vcycle":
            z = self.S.vcycle(self.b)
        else:
            z = self.S.smooth(self.S.num_levels - 1, torch.zeros_like(self.b), self.b, 1)
        torch.cuda.synchronize()
        return z


RAS = dict(smoother=sib.SMOOTHER_RAS)
PAIRS = {
    "16x16 f32": (lambda: Work(64, "smooth", torch.float32, box=16, box_overlap=4, **RAS),
                  lambda: Work(64, "smooth", torch.float32, box=16, box_overlap=0, **RAS)),
    "16x16 f64": (lambda: Work(64, "smooth", torch.float64, box=16, box_overlap=4, **RAS),
                  lambda: Work(64, "smooth", torch.float64, box=16, box_overlap=0, **RAS)),
    "split f64": (lambda: Work(64, "smooth", torch.float64, box=8, box_overlap=4, **RAS),
                  lambda: Work(64, "smooth", torch.float64, box=2, box_overlap=1, **RAS)),
    "cluster": (lambda: Work(32, "vcycle", torch.float32), lambda: Work(16, "vcycle", torch.float32)),
    "wide windows": (lambda: Work(256, "smooth", torch.float32, box=8, box_overlap=4, ras_tc=0, **RAS),
                     lambda: Work(256, "smooth", torch.float32, box=4, box_overlap=2, ras_tc=0, **RAS)),
}


# the larger case in this thread, the smaller one in another, the larger one again; set-ups in between included
@pytest.mark.parametrize("name", PAIRS)
def test_a_smaller_case_in_another_thread(name):
    large, small = PAIRS[name][0](), in_thread(PAIRS[name][1])
    ref = large()
    ref_small = in_thread(small)
    for _ in range(2):
        assert torch.equal(large(), ref)
        assert torch.equal(in_thread(small), ref_small)
    in_thread(lambda: large.S.setup())
    again = in_thread(PAIRS[name][1])
    large.S.set_options(omega=large.S.opts.omega)
    assert torch.equal(large(), ref)
    for w in (large, small, again):
        w.S.close()


# both at the same time
@pytest.mark.parametrize("name", ["split f64", "cluster"])
def test_side_by_side(name):
    works = [make() for make in PAIRS[name]]
    refs = [w() for w in works]
    errors = []

    def body(w, ref):
        try:
            for _ in range(200):
                if not torch.equal(w(), ref):
                    raise AssertionError("another result")
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=body, args=a) for a in zip(works, refs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w in works:
        w.S.close()
    assert not errors, errors[0]
