"""Pivots and quotients at the ends of their ranges: a last pivot that is zero
or not a number, pivots that only their rounding makes zero, quotients that
overflow."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2307_16051_gb300 import nl
from paper_2307_16051_gb300 import workloads as W
from tests.test_gpu_batch import lu_grouped
from tests.test_gpu_kernels import T, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _last_pivot(N, value):
    """Column-wise dominant but for the last row and column, which hold the last pivot alone."""
    A = W.random_matrix(N, 90 + N)
    A += np.diag(np.abs(A).sum(axis=0) + np.abs(A).sum(axis=1))
    A[-1, :] = A[:, -1] = 0.0
    A[-1, -1] = value
    return A


def _lu64(A, nb, path):
    N = A.shape[0]
    Ad = T(A)
    ipiv = torch.full((N,), -1, device=dev(), dtype=torch.int32)
    info = nl.lu64(N, Ad, N, ipiv, nb=nb, path=path)
    return Ad.cpu().numpy(), ipiv.cpu().numpy(), info


@pytest.mark.parametrize("N,nb", [(1, 16), (32, 32), (33, 32), (64, 64), (100, 64), (128, 64), (128, 128)])
def test_lu64_zero_last_pivot(N, nb):
    """Singular in the last pivot alone, which no row lies below: info = N, as
    the oracle and the interchanging path say, whether or not the last block is a
    multiple of 32 wide.  Bound as in any double LU without growth."""
    A = _last_pivot(N, 0.0)
    LUo, ipivo, infoo = O.lu64(A)
    assert infoo == N
    for path in (0, 1):
        LU, ipiv, info = _lu64(A, nb, path)
        assert info == N and np.array_equal(ipiv, ipivo), (path, info)
        assert np.max(np.abs(LU - LUo)) <= 8 * N * 2.0 ** -53 * max(1.0, np.max(np.abs(LUo)))
    Ad, ipiv = T(A), torch.empty(N, device=dev(), dtype=torch.int32)  # (held: the call gets their addresses)
    assert nl.lib().nl_lu64(N, Ad.data_ptr(), N, ipiv.data_ptr(), nb, 0, None, None) == nl.NL_ESINGULAR


@pytest.mark.parametrize("N,nb", [(64, 64), (100, 64)])
def test_lu64_last_pivot_not_a_number(N, nb):
    """A last pivot that is not a number: the paths agree on info, pivots and factors."""
    A = _last_pivot(N, np.nan)
    ref, got = _lu64(A, nb, 1), _lu64(A, nb, 0)
    assert got[2] == ref[2] and np.array_equal(got[1], ref[1]) and np.isnan(got[0][-1, -1])
    assert np.max(np.abs((got[0] - ref[0]).ravel()[:-1])) <= 8 * N * 2.0 ** -53 * np.max(np.abs(A.ravel()[:-1]))


def test_lu_grouped_fp64_zero_last_pivot():
    """The grouped double LU leaves a matrix whose last pivot is zero to the
    interchanging path, at widths that are a multiple of 32 and at others."""
    Ns = [32, 64, 100, 128, 96]
    mats = [_last_pivot(N, 3.0 if N == 96 else 0.0) for N in Ns]
    _, flags = lu_grouped(mats, 64, 1, fp64=True)
    assert list(flags) == [1, 1, 1, 1, 0]
