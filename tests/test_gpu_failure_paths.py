"""Failure paths of the C ABI on the GPU, made without faulting the device:
a bounded device-side wait that runs out (NL_ETIMEOUT, context intact), a
device allocation that fails (NL_ENOMEM, from the library's allocation test
hook), and the iterate returned when Newton does not converge (the one with
the smallest ||F||)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2307_16051_gb300 import nl
from tests.conftest import newton_counts_agree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _device():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    torch.cuda.init()


def _solve_raw(s, mode):
    x = np.empty(s.N)
    st = nl.lib().nl_solve(s._h, None, 1e-10, nl.MODES[mode], x.ctypes.data)
    return st, x


@pytest.mark.parametrize("cluster", [0, -1])
@pytest.mark.parametrize("mode", ["IR16", "GMRESIR16"])
def test_triangular_solve_wait_runs_out(cluster, mode):
    """wait_limit < 0 makes every wait of the half-precision triangular
    solves give up at once, whatever the producer does: the cluster solve
    (cluster = 0, N = 4096) and the global-memory solve (-1) record the
    timeout in their error word, every CTA returns, and the solve reports
    NL_ETIMEOUT.  The context stays usable: a solve on another handle, and
    on the same handle after its wait limit is restored, converge as the
    oracle does."""
    N, c = 4096, 0.9
    with nl.Solver(N, c, trsv_cluster=cluster, wait_limit=-1) as s:
        st, _ = _solve_raw(s, mode)
        assert st == nl.NL_ETIMEOUT, nl.STATUS_NAMES[st]
        assert "gave up" in nl.last_error()
        assert s.stats()["status"] == nl.NL_ETIMEOUT
    torch.cuda.synchronize()  # the device answers
    _, ro = O.newton(512, c, mode, tol=1e-10)
    with nl.Solver(512, c, trsv_cluster=cluster) as s:
        x, st = s.solve(tol=1e-10, mode=mode)
        assert st == nl.NL_OK and newton_counts_agree(s.stats()["newton_iters"], ro)


def test_allocation_failure_returns_enomem():
    """The allocation test hook fails the next device allocation: nl_create
    returns NL_ENOMEM and no handle; the first FP64-LU solve of a live handle
    (which allocates the double Jacobian) returns NL_ENOMEM and leaves the
    handle usable; with the hook spent both succeed."""
    L = nl.lib()
    h = nl._P()
    assert L.nl_debug_fail_allocs(1) == nl.NL_OK
    assert L.nl_create(256, 0.9, None, nl.ctypes.byref(h)) == nl.NL_ENOMEM
    assert not h.value
    assert "cudaMalloc" in nl.last_error()
    with nl.Solver(256, 0.9) as s:
        assert L.nl_debug_fail_allocs(1) == nl.NL_OK
        st, _ = _solve_raw(s, "FP64LU")
        assert st == nl.NL_ENOMEM
        x, st = s.solve(mode="FP64LU")
        assert st == nl.NL_OK
        x2, st = s.solve(mode="GMRESIR16")
        assert st == nl.NL_OK and np.max(np.abs(x - x2)) <= 1e-10 * np.max(np.abs(x))
    assert L.nl_debug_fail_allocs(0) == nl.NL_OK


@pytest.mark.parametrize("c,scale,maxit", [(0.999, 6.0, 7), (0.99, 4.5, 6), (0.9999, 1.0, 3)])
def test_best_iterate_on_not_converged(c, scale, maxit):
    """On NL_ENOTCONV the returned x is the iterate with the smallest ||F||
    of the history (far-from-solution starts make the history non-monotone):
    its residual, computed by the oracle's F in double, is the smallest
    entry of the history times ||F(x0)||, and nl_stats_t.fnorm is that
    norm."""
    N = 128
    x0 = scale * np.ones(N)
    with nl.Solver(N, c, newton_maxit=maxit) as s:
        x, st = s.solve(tol=1e-10, mode="GMRESIR16", x0=x0)
        S = s.stats()
    assert st == nl.NL_ENOTCONV and S["newton_iters"] == maxit
    h = np.array(S["hist"])
    best = int(np.argmin(h))
    fx = np.linalg.norm(O.F(N, c, x))
    assert abs(fx - h[best] * S["fnorm0"]) <= 1e-12 * S["fnorm0"] + 1e-9 * fx, (h, fx)
    assert abs(S["fnorm"] - h[best] * S["fnorm0"]) <= 1e-15 * S["fnorm0"]
    if best == 0:
        assert np.array_equal(x, x0)
    # the oracle returns its own best iterate by the same rule
    xo, ro = O.newton(N, c, "GMRESIR16", tol=1e-10, x0=x0, newton_maxit=maxit)
    fo = np.linalg.norm(O.F(N, c, xo))
    assert abs(fo - min(ro["hist"]) * np.linalg.norm(O.F(N, c, x0))) <= 1e-9 * fo + 1e-14


@pytest.mark.parametrize("gemm", [3, 5])
def test_persistent_grouped_lu_wait_runs_out(gemm):
    """The persistent grouped LU's dependency waits are bounded: with the poll
    limit set to give up at the first unmet poll, the off-diagonal tasks that
    start while their diagonal block is being factored give up, the launch
    completes, nl_lu_grouped returns NL_ETIMEOUT, and with the default limit
    the next call on the same context factors the same matrices correctly
    (bitwise the three-launch grouped LU with the same update)."""
    Ns = [1500, 300, 90]
    mats = [O.fl16(O.jacobian(N, 0.9, 1.0 + 0.3 * np.sin(np.arange(N)) ** 2).astype(np.float32).astype(np.float64))
            for N in Ns]

    def run(g):
        As, lds, ips = [], [], []
        for M in mats:
            N = M.shape[0]
            ld = ((N + 63) // 64) * 64
            a = np.zeros((N, ld), dtype=np.float16)
            a[:, :N] = M.astype(np.float16)
            As.append(torch.as_tensor(a, device="cuda"))
            lds.append(ld)
            ips.append(torch.empty(N, dtype=torch.int32, device="cuda"))
        flags = nl.lu_grouped(Ns, As, lds, ips, nb=64, gemm=g)
        torch.cuda.synchronize()
        return [A.cpu().numpy()[:, :n] for A, n in zip(As, Ns)], flags

    nl.grouped_wait_limit(-1)
    try:
        with pytest.raises(nl.NLError) as e:
            run(gemm)
        assert e.value.status == nl.NL_ETIMEOUT
    finally:
        nl.grouped_wait_limit(0)
    out, flags = run(gemm)
    ref, rflags = run(1 if gemm == 3 else 2)
    assert not flags.any() and not rflags.any()
    for a, b in zip(out, ref):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,cluster", [(256, 0), (1000, 8), (3072, 0), (4096, 4), (4096, 16)])
@pytest.mark.parametrize("limit", [-1, 1, 2])
def test_cluster_solve_waits_run_out_in_part(N, cluster, limit):
    """The one-launch cluster solve (both triangles) when its waits run out: all of
    them (-1), or those whose block has not arrived within one or two polls, so
    that some warps and CTAs give up and others do not.  The launch ends, the
    solve returns NL_ETIMEOUT or, if no wait ran out, the solution, and a
    handle with the default limit converges on the same context."""
    c = 0.9
    with nl.Solver(N, c, trsv_cluster=cluster) as s:
        xr, st = s.solve(tol=1e-10, mode="IR16")
        assert st == nl.NL_OK
    for _ in range(3):
        with nl.Solver(N, c, trsv_cluster=cluster, wait_limit=limit) as s:
            st, x = _solve_raw(s, "IR16")
            assert st == nl.NL_ETIMEOUT or (limit > 0 and st == nl.NL_OK and np.array_equal(x, xr)), nl.STATUS_NAMES[st]
            if st == nl.NL_ETIMEOUT:
                assert "gave up" in nl.last_error()
        torch.cuda.synchronize()  # the device answers
    with nl.Solver(N, c, trsv_cluster=cluster) as s:
        x, st = s.solve(tol=1e-10, mode="IR16")
        assert st == nl.NL_OK and np.array_equal(x, xr)


@pytest.mark.parametrize("call", ["lu_grouped", "lu_grouped_persistent", "batch", "solver", "gemv"])
def test_full_device_gives_kept_workspaces_back(call):
    """An allocation that finds the device full is tried again after the library
    has given its kept workspace memory back: each of a call's allocations in
    turn fails once and the call succeeds; when the second attempt fails too the
    call returns an error, and the next one succeeds."""
    L, d, N, ld = nl.lib(), torch.device("cuda:0"), 300, 320
    A32 = torch.eye(N, ld, device=d, dtype=torch.float32)
    b, u, r = (torch.ones(ld, device=d, dtype=torch.float32) for _ in range(3))
    fn = torch.zeros(1, device=d, dtype=torch.float64)
    A = torch.zeros((N, ld), device=d, dtype=torch.float16)
    ip = torch.empty(N, device=d, dtype=torch.int32)

    def keep():  # a workspace, released and kept
        nl.k_gemv_residual(N, A32, ld, b, u, r, fn)
        torch.cuda.synchronize()

    def run():
        if call.startswith("lu_grouped"):
            A[:, :N] = torch.eye(N, device=d, dtype=torch.float16)
            flags = nl.lu_grouped([N], [A], [ld], [ip], nb=64, gemm=5 if "persistent" in call else 2)
            assert not flags.any()
        elif call == "batch":
            with nl.Batch([64, N], [0.5, 0.9], lu_nb=64) as B:
                assert B.solve(tol=1e-10)[1] == nl.NL_OK
        elif call == "solver":
            with nl.Solver(N, 0.9) as s:
                assert s.solve(mode="FP64LU")[1] == nl.NL_OK
        else:
            nl.k_gemv_residual(N, A32, ld, b, u, r, fn)
            torch.cuda.synchronize()

    run()
    try:
        for skip in range(4):
            keep()
            assert L.nl_debug_device_full(skip, 1) == nl.NL_OK
            run()
        keep()
        assert L.nl_debug_device_full(0, 2) == nl.NL_OK
        with pytest.raises(nl.NLError):
            run()
    finally:
        assert L.nl_debug_device_full(0, 0) == nl.NL_OK
    run()


@pytest.mark.parametrize("N", [4096, 14000])
def test_released_workspaces_leave_the_device(N):
    """What a call's workspace leaves in the library's pool is at most 256 MB (N = 14000
    takes 784 MB) and goes back to the device on request; the call gives the same
    result after it."""
    d, ld = torch.device("cuda:0"), (N + 63) // 64 * 64
    J, A = (torch.empty((N, ld), device=d, dtype=t) for t in (torch.float32, torch.float16))
    r, ip = torch.ones(N, device=d, dtype=torch.float64), torch.empty(N, device=d, dtype=torch.int32)

    def run():
        nl.k_jacobian(N, 0.9, r, J, ld, A, ld)
        nl.lu16(N, A, ld, ip)
        torch.cuda.synchronize()
        return A.clone()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    first = run()
    nl.release_workspaces()
    torch.cuda.empty_cache()  # (what earlier tests left with torch's allocator)
    before = free()
    second = run()
    del second
    torch.cuda.empty_cache()
    kept = before - free()
    nl.release_workspaces()
    assert 0 < kept <= (256 << 20) + (64 << 20) and free() >= before  # (64 MB: the pool's granularity)
    third = run()
    assert torch.equal(first.view(torch.int16), third.view(torch.int16))


@pytest.mark.parametrize("N,nb,gemm,path,used", [(1100, 128, 2, 0, True), (1100, 64, 2, 0, True), (1000, 128, 2, 0, False),
                                                 (1100, 256, 2, 0, False), (1100, 512, 2, 4, False),
                                                 (1100, 96, 2, 0, False), (1100, 128, 1, 4, False),
                                                 (300, 128, 2, 4, True)])
def test_lu16_second_stream(N, nb, gemm, path, used):
    """nl_lu16 makes a second stream only where its look-ahead runs (outer block
    at most 128, tensor-core update, asked for or N >= 1024), and a failure to
    make it fails the call only if the look-ahead was asked for (path 4)."""
    d, ld, L = torch.device("cuda:0"), (N + 63) // 64 * 64, nl.lib()
    J32, A = (torch.empty((N, ld), device=d, dtype=t) for t in (torch.float32, torch.float16))
    r, ip = torch.ones(N, device=d, dtype=torch.float64), torch.empty(N, device=d, dtype=torch.int32)

    def run(p):
        nl.k_jacobian(N, 0.99, r, J32, ld, A, ld)
        st = L.nl_lu16(N, A.data_ptr(), ld, ip.data_ptr(), nb, gemm, p, None, None)
        torch.cuda.synchronize()
        return st, A.clone()

    st, ref = run(2)
    assert st == nl.NL_OK
    try:
        assert L.nl_debug_fail_streams(1) == nl.NL_OK
        st, got = run(path)
        assert st == (nl.NL_ECUDA if used and path == 4 else nl.NL_OK)
        if st == nl.NL_OK:
            assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
        # was the hook used up?  path 4 with a one-level tensor-core update always asks for a stream
        st = L.nl_lu16(128, A.data_ptr(), ld, ip.data_ptr(), 128, 2, 4, None, None)
        assert (st == nl.NL_ECUDA) == (not used)
    finally:
        assert L.nl_debug_fail_streams(0) == nl.NL_OK
    st, got = run(path)
    assert st == nl.NL_OK and torch.equal(got.view(torch.int16), ref.view(torch.int16))
