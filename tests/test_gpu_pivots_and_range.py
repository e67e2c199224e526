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


@pytest.mark.parametrize("u00,u01,u11", [(1e-20, 1e290, 1.0), (1e-20, -1e300, 1e-20), (-1e-25, 1e300, 1e-8)])
def test_lusolve64_overflowing_inverse(u00, u01, u11):
    """A triangle whose inverse overflows: infinities with the signs the
    divisions give, not NaN."""
    LU = np.array([[u00, u01], [0.0, u11]])
    b = np.array([1.0, 1.0])
    with np.errstate(over="ignore"):
        z1 = b[1] / u11
        ref = np.array([(b[0] - u01 * z1) / u00, z1])
    assert np.isinf(ref[0])
    bd = T(b)
    nl.lusolve64(2, T(LU), 2, torch.arange(2, device=dev(), dtype=torch.int32), bd)
    assert np.array_equal(bd.cpu().numpy(), ref), bd


def test_div64_equals_ieee_division():
    """The quotients by corrected reciprocals against numpy's IEEE division, bit
    for bit (NaN by NaN): ordinary operands, quotients next to the middle of two doubles,
    every pair of exponents, and zeros, subnormal numbers, infinities and NaN of both signs
    against each other."""
    g = np.random.default_rng(64)
    n = 1 << 20
    a, b = g.standard_normal(n), g.standard_normal(n)
    k = n // 4
    # a = fl(m b) for m halfway between two doubles: the quotient lies next to the middle
    q = 1.0 + g.integers(0, 1 << 52, size=k) * 2.0 ** -52
    b[:k] = 1.0 + g.integers(0, 1 << 52, size=k) * 2.0 ** -52
    a[:k] = q * b[:k] + 2.0 ** -53 * b[:k] * g.integers(-2, 3, size=k)
    e = np.arange(-1074, 1024)
    ea, eb = np.meshgrid(e[::3], e[::5])
    sa, sb = (g.choice([-1.0, 1.0], ea.size) * (1.0 + g.random(ea.size)) for _ in range(2))
    edge = np.concatenate([[0.0, 5e-324, 2.0 ** -1022, 1e-30, 1e30, np.nextafter(1e-30, 0), np.nextafter(1e30, 1e31),
                            2.0 ** -900, np.nextafter(2.0 ** -900, 0), 2.0 ** 900, np.nextafter(2.0 ** 900, 0),
                            np.finfo(float).max, 1.0, 3.0, np.inf, np.nan]])
    edge = np.concatenate([edge, -edge])
    xa, xb = np.meshgrid(edge, edge)
    a = np.concatenate([a, np.ldexp(sa, ea.ravel()), xa.ravel()])
    b = np.concatenate([b, np.ldexp(sb, eb.ravel()), xb.ravel()])
    with np.errstate(all="ignore"):
        ref = a / b
    out = torch.empty(a.size, device=dev(), dtype=torch.float64)
    nl.k_div64(a.size, T(a), T(b), out)
    got = out.cpu().numpy()
    bad = ~((got.view(np.uint64) == ref.view(np.uint64)) | (np.isnan(got) & np.isnan(ref)))
    assert not bad.any(), (bad.sum(), a[bad][:5], b[bad][:5], got[bad][:5], ref[bad][:5])
