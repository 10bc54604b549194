"""The blocked Gauss-Jordan inversion that set-up uses for the coarsest grid and for the box smoothers' largest
subdomains, called by itself (a function of the library's internal C++ interface)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1612_02208_gb300 import sib  # noqa: E402


class Inversion:
    """Aug = [A | I] with `guard` rows of a known value before and behind it, and the pivot and information words."""

    def __init__(self, guard=2):
        lib = sib.load()
        self.run_ = getattr(lib, "_ZN3sib19launch_gauss_jordanEPdiPiS1_PvP11CUstream_st")
        self.run_.restype = None
        self.run_.argtypes = [ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 4
        self.bytes_ = getattr(lib, "_ZN3sib23gauss_jordan_work_bytesEi")
        self.bytes_.restype = ctypes.c_size_t
        self.bytes_.argtypes = [ctypes.c_int]
        self.guard = guard
        self.info = torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(self, A):
        """(inverse, pivot rows, whether the guard rows are as they were) of the n x n matrix A, n a multiple of 16"""
        n, g = A.shape[0], self.guard
        buf = torch.full((n + 2 * g, 2 * n), 7.0, dtype=torch.float64, device="cuda")
        buf[g:-g, :n] = torch.as_tensor(A, device="cuda")
        buf[g:-g, n:] = torch.eye(n, dtype=torch.float64, device="cuda")
        piv = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        work = torch.empty(self.bytes_(n), dtype=torch.uint8, device="cuda")
        self.run_(buf[g:].data_ptr(), n, self.info.data_ptr(), piv.data_ptr(), work.data_ptr(),
                  torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        whole = bool((buf[:g] == 7.0).all()) and bool((buf[-g:] == 7.0).all())
        return buf[g:-g, n:][piv.long().clamp(0, n - 1)].cpu().numpy(), piv.cpu().numpy(), whole


def matrix(n, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, n)) + 4 * np.sqrt(n) * np.eye(n)   # singular values from 2 sqrt(n) up


# both panels (up to 768 rows in registers, above in shared memory), with values that are not numbers in one
# column, one row or everywhere: every pivot row is one of the matrix's, each taken once, and nothing beside the
# matrix is written
@pytest.mark.parametrize("n", [16, 192, 768, 784, 1200])
@pytest.mark.parametrize("where", ["column", "row", "all", "nowhere"])
def test_pivot_rows(n, where):
    A = matrix(n, n)
    if where == "column":
        A[:, n // 2] = np.nan
    elif where == "row":
        A[n // 3] = np.inf
    elif where == "all":
        A[:] = np.nan
    inv, piv, whole = Inversion().run(A)
    assert whole
    assert np.array_equal(np.sort(piv), np.arange(n))
    if where == "nowhere":   # backward stable up to growth: a few n eps of condition number <= 3
        assert np.abs(inv @ A - np.eye(n)).max() < 64 * n * 2.0 ** -53


# A singular matrix (a zero column: its pivot is exactly zero) reports its column, and a regular one inverted
# after it with the same word leaves the report; both panels
@pytest.mark.parametrize("n", [48, 784])
def test_singular_report_stays(n):
    I = Inversion()
    I.run(matrix(n, 1))
    assert I.info.item() == 0
    A = matrix(n, 2)
    A[:, 20] = 0.0
    I.run(A)
    assert I.info.item() == 21
    I.run(matrix(n, 3))
    assert I.info.item() == 21
