"""Pivots and quotients at the ends of their ranges: a last pivot that is zero
or not a number, pivots that only their rounding makes zero, quotients that
overflow."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2307_16051_gb300 import nl
from paper_2307_16051_gb300 import workloads as W
from tests.test_gpu_batch import lu_grouped
from tests.test_gpu_kernels import T, _lu16_gpu, dev

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


@pytest.mark.parametrize("to", ["zero", "infinity"])
@pytest.mark.parametrize("gemm", [1, 2])
@pytest.mark.parametrize("N,k", [(300, 1), (300, 7), (300, 8), (300, 127), (300, 299), (1200, 200), (1200, 1199)])
def test_lu16_pivot_leaves_binary16_by_rounding(N, k, gemm, to):
    """A pivot that single precision holds and its rounding to binary16 does not:
    -2^-34 (fl16(l u) - l u) becomes zero, 70000 becomes infinity, with only zeros
    below it, so that every check of the unrounded value passes.  Every path
    agrees bit for bit with the interchanging one, which names the zero pivot in
    info and, with the SIMT update, is the oracle's.  In the first and later
    columns of a block of eight and of a panel, in a ragged last panel, and in the
    matrix's last pivot."""
    nb = 128
    k0 = k // nb * nb  # the first column of k's panel: no rounding to storage in between
    A = 2.0 * np.eye(N) + W.random_matrix(N, 31) / (8.0 * N)
    A[[k0, k], :] = A[:, [k0, k]] = 0.0
    if to == "zero":
        l, u, a = 2.0 ** -1 * (1 + 2.0 ** -10), 2.0 ** -13 * (1 + 2.0 ** -10), 2.0 ** -14 * (1 + 2.0 ** -9)
        assert a - l * u == -(2.0 ** -34)
        A[k0, k0], A[k, k0], A[k0, k], A[k, k] = 1.0, l, u, a
    else:
        A[k0, k0], A[k, k0], A[k0, k], A[k, k] = 2.0, 1.0, -20000.0, 60000.0
    A16 = O.fl16(A)
    assert all(A16[i, j] == A[i, j] for i in (k0, k) for j in (k0, k))
    ref = _lu16_gpu(A16, nb, gemm, 1)
    assert ref[2] == (k + 1 if to == "zero" else 0) and abs(ref[0][k, k]) == (0.0 if to == "zero" else np.inf)
    for path in (0, 2, 4):
        got = _lu16_gpu(A16, nb, gemm, path)
        assert ref[2] == got[2] and np.array_equal(ref[1], got[1]), path
        assert np.array_equal(ref[0].view(np.uint64), got[0].view(np.uint64)), path
    if to == "zero" and gemm == 1 and N <= 300:
        LUo, ipivo, infoo, _ = O.lu16_dev(A16, nb)
        assert infoo == k + 1 and np.array_equal(ipivo, ref[1]) and np.array_equal(LUo, ref[0])


@pytest.mark.parametrize("kind", [1, 2, 3, 5])
def test_lu_grouped_pivot_leaves_binary16_by_rounding(kind):
    """The same in the grouped factorisations: such a matrix is flagged, its
    neighbours are not."""
    mats = []
    for N, k in ((200, 70), (200, 199), (64, 63), (130, 5), (96, -1)):
        A = 2.0 * np.eye(N) + W.random_matrix(N, 31) / (8.0 * N)
        if k >= 0:
            k0 = k // 64 * 64
            A[[k0, k], :] = A[:, [k0, k]] = 0.0
            A[k0, k0], A[k, k0], A[k0, k] = 1.0, 2.0 ** -1 * (1 + 2.0 ** -10), 2.0 ** -13 * (1 + 2.0 ** -10)
            A[k, k] = 2.0 ** -14 * (1 + 2.0 ** -9)
        mats.append(O.fl16(A))
    _, flags = lu_grouped(mats, 64, kind)
    assert list(flags) == [1, 1, 1, 1, 0]
