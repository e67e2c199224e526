"""Edges of the kernels' tiles and of the rules that choose between kernels:
sizes on both sides of each line, ragged remainders, unaligned leading
dimensions."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2307_16051_gb300 import nl
from paper_2307_16051_gb300 import workloads as W
from tests.test_gpu_batch import check_instance
from tests.test_gpu_kernels import T, _jacobian16, _lu16_gpu, dev, synthetic_factors

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,nb,gemm", [(129, 128, 2), (257, 128, 2), (384, 128, 2), (385, 128, 2), (1023, 128, 2),
                                       (1024, 128, 2), (1153, 128, 2), (2561, 128, 2), (1030, 64, 2), (145, 16, 1),
                                       (193, 48, 1), (1111, 128, 1), (203, 112, 1)])
def test_lu16_panels_equal_two_launches(N, nb, gemm):
    """The streaming panel, with and without the look-ahead and with the last
    panel's product formed inside it (nb 128 on the tensor cores), against the
    two-launch panel and one update: bitwise the same factors for every form
    of last panel and of trailing matrix (none, part of a tile, one tile and a
    column), below and above the size from which path 0 looks ahead."""
    J16 = _jacobian16(N, 0.99)
    ref = _lu16_gpu(J16, nb, gemm, 2)
    for path in (0, 4):
        got = _lu16_gpu(J16, nb, gemm, path)
        assert ref[2] == got[2] == 0 and np.array_equal(ref[1], got[1])
        assert np.array_equal(ref[0].view(np.uint64), got[0].view(np.uint64)), path


@pytest.mark.parametrize("big", [7e4, 1e-9])
@pytest.mark.parametrize("N,k", [(300, 0), (300, 130), (1200, 1100)])
def test_lu16_pivot_out_of_range(N, k, big):
    """A pivot that binary16 cannot hold (it rounds to infinity or to zero) in
    the first column, in a later panel and in the last one: the paths agree
    on pivots, info and factors, bit for bit."""
    A = 2.0 * np.eye(N) + W.random_matrix(N, 31) / (8.0 * N)
    A[k, :] = A[:, k] = 0.0
    A[k, k] = 60000.0 if big > 1 else 0.0
    if k > 0 and big > 1:  # column k of U: l_k0 u_0k = -10000 makes the pivot 70000
        A[0, k], A[k, 0] = -20000.0, 1.0
    A16 = O.fl16(A)
    ref = _lu16_gpu(A16, 128, 2, 2)
    for path in (0, 4):
        got = _lu16_gpu(A16, 128, 2, path)
        assert ref[2] == got[2] and np.array_equal(ref[1], got[1])
        assert np.array_equal(ref[0], got[0], equal_nan=True), path


@pytest.mark.parametrize("N,pad", [(129, 1), (1153, 64), (3071, 64), (3072, 64), (3073, 64), (3073, 1), (3200, 8)])
def test_lusolve16_kernel_choice(N, pad):
    """Both triangles at the last size of the cluster kernel and the first of
    the mailbox kernel, with full and ragged last blocks and with rows whose
    addresses are not aligned."""
    LUo, ipivo = synthetic_factors(N, 300 + N)
    b = W.random_vector(N, 400 + N).astype(np.float32)
    ref = O.lusolve_fly(LUo, ipivo, b).astype(np.float64)
    ld = (N + pad - 1) // pad * pad
    LUd = torch.zeros((N, ld), device=dev(), dtype=torch.float16)
    LUd[:, :N] = T(LUo.astype(np.float16))
    bd = T(b)
    nl.lusolve16(N, LUd, ld, T(ipivo), bd)
    got = bd.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.max(np.abs(ref)))


@pytest.mark.parametrize("N", [8, 33, 1216, 1217, 2432, 2433, 4864, 4865])
def test_residual_rows_per_block(N):
    """8, 16 or 32 rows of F per block, by the rows of the busiest
    multiprocessor: both sides of each line (152 multiprocessors) and ragged
    last blocks.  Bound: t_i = 1 - 1/r_i is a sum of N positive terms, so each
    side is within N 2^-53 of it and r_i within r_i^2 of that."""
    c = 0.95
    g = np.random.default_rng(N)
    x = 1.0 + g.uniform(0.0, 1.0, N)
    u = g.standard_normal(N) * 1e-3
    F, r, xo = (torch.empty(N, device=dev(), dtype=torch.float64) for _ in range(3))
    fn = torch.empty(1, device=dev(), dtype=torch.float64)
    for uu, dbl in ((None, False), (u.astype(np.float32), False), (u, True)):
        if uu is None:
            xn = x
            nl.k_residual(N, c, T(x), F, r, fn)
        else:
            xn = x + 0.5 * uu.astype(np.float64)
            nl.k_residual(N, c, T(x), F, r, fn, u=T(uu), u_is_double=dbl, scale=0.5, x_out=xo)
            assert np.array_equal(xo.cpu().numpy(), xn)
        Fo = O.F(N, c, xn)
        tol = (4 * N + 64) * 2.0 ** -53 * np.max(np.abs(xn - Fo)) ** 2
        assert np.max(np.abs(F.cpu().numpy() - Fo)) <= tol
        assert abs(fn.item() - np.linalg.norm(Fo)) <= tol * np.sqrt(N)


@pytest.mark.parametrize("N,nb", [(129, 128), (161, 32), (257, 64), (385, 128), (1217, 128), (1001, 48)])
@pytest.mark.parametrize("pad", [1, 64])
def test_lu64_edges(N, nb, pad):
    """Double precision without interchanges: last panels of one column,
    off-diagonal launches with a ragged last group of 32 lines, small and large
    update tiles, odd leading dimensions.  Column-wise dominance bounds the
    growth by 2, so both sides are within N 2^-53 times a few of the exact
    factors' scale."""
    A = W.random_matrix(N, 70 + N)
    A += np.diag(np.abs(A).sum(axis=0) + np.abs(A).sum(axis=1))
    ld = (N + pad - 1) // pad * pad
    Ad = torch.zeros((N, ld), device=dev(), dtype=torch.float64)
    Ad[:, :N] = T(A)
    ipiv = torch.empty(N, device=dev(), dtype=torch.int32)
    info = nl.lu64(N, Ad, ld, ipiv, nb=nb)
    LUo, ipivo, infoo = O.lu64(A)
    assert info == infoo == 0 and np.array_equal(ipiv.cpu().numpy(), ipivo)
    tol = 8 * N * 2.0 ** -53 * np.max(np.abs(LUo))
    assert np.max(np.abs(Ad.cpu().numpy()[:, :N] - LUo)) <= tol


def test_batch_jacobian_row_blocks():
    """The grouped Jacobian takes 32 rows of an instance per block: instances
    just below, at and above a block, of different widths in one launch, give
    the oracle's counts and solutions."""
    Ns = [31, 32, 33, 64, 65, 129, 257]
    cs = [0.5, 0.9, 0.99, 0.8, 0.95, 0.9, 0.99]
    with nl.Batch(Ns, cs, lu_nb=64) as B:
        xs, status = B.solve(tol=1e-10)
        stats = [B.stats(i) for i in range(len(Ns))]
    assert status == nl.NL_OK
    for N, c, x, st in zip(Ns, cs, xs, stats):
        xo, ro = O.newton(N, c, "IR16GM", tol=1e-10, lu_nb=64)
        check_instance(st, ro, x, xo)
