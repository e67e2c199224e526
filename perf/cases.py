"""What a user of this library has it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (the
handle, the inputs on the GPU), ``run`` makes one pass through the public entry points and returns
its outputs, ``work`` says what the pass cannot do without and ``exact`` what it should return, in
64 bits and without this library.

Kinds:
  newton    one Newton solve of the H-equation on a solver handle (nl_solve_device)
  sweep     the conditioning sweep: five handles solved at once, one host thread and stream each
  batch     many instances of different N and c in one batched solve (nl_batch_solve_device)
  factor    a caller's own loop: the Jacobian at an iterate and its binary16 LU
  linsolve  a caller's own loop: the refined linear solve with given factors (IR or GMRES-IR)
  residual  F(x) with the fused update, by the direct sum or the FFT
  gemv      r = b - J u with its norm, the residual of the refinement
"""
import math
import os
from concurrent.futures import ThreadPoolExecutor

import torch

# Read when the CUDA context is created: the sweep's streams (and each solve's look-ahead stream)
# get hardware queues of their own, as a program that solves concurrently sets it.
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

from paper_2307_16051_gb300 import nl, workloads  # noqa: E402

TOL = 1e-10


def listed():
    return [
        # serving: half of all requests have N = 256; IR16 with the GMRES fallback is the server's mode
        {"name": "newton_256", "kind": "newton", "N": 256, "c": 0.9, "mode": "IR16_GMRES", "lu_nb": 0, "scale": 0},
        # serving and library use: one solve on its own at the paper's N and its first c (Table 2)
        {"name": "newton_4096", "kind": "newton", "N": 4096, "c": 0.99, "mode": "GMRESIR16", "lu_nb": 0, "scale": 0},
        # the large configuration: one solve at N = 32768 with the two-level factorisation
        {"name": "newton_32768", "kind": "newton", "N": 32768, "c": 0.99, "mode": "GMRESIR16", "lu_nb": 512,
         "scale": 0},
        # the F64 column, the baseline that every three-precision run is compared with; an odd N
        {"name": "newton_f64_1001", "kind": "newton", "N": 1001, "c": 0.9, "mode": "FP64LU", "lu_nb": 0, "scale": 0},
        # the headline: the conditioning sweep of Tables 2 and 3, five solves side by side
        {"name": "sweep_4096", "kind": "sweep", "N": 4096, "mode": "GMRESIR16"},
        # the batched configuration: 512 instances, N log-uniform in [64, 2048]
        {"name": "batch_512", "kind": "batch", "count": 512, "n_lo": 64, "n_hi": 2048},
        # a caller's own Newton loop, factoring at a ragged and at a large size
        {"name": "factor_2049", "kind": "factor", "N": 2049, "c": 0.99, "scale": 0},
        {"name": "factor_8192", "kind": "factor", "N": 8192, "c": 0.9, "scale": 0},
        # the refinement with factors that are already there: a size past the cluster solve's range
        {"name": "linsolve_12000", "kind": "linsolve", "N": 12000, "c": 0.99, "solver": 2},
        # F(x) on its own, as a line search or a convergence test evaluates it: direct sum and FFT
        {"name": "residual_1001", "kind": "residual", "N": 1001, "c": 0.99, "fft": 0},
        {"name": "residual_fft_32768", "kind": "residual", "N": 32768, "c": 0.9, "fft": 1},
        # the residual of the refinement at a size that streams from HBM
        {"name": "gemv_16384", "kind": "gemv", "N": 16384, "c": 0.9},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["newton", "newton", "newton", "sweep", "batch", "factor", "factor", "linsolve", "residual", "gemv"])
    c = round(rng.uniform(0.5, 0.9999), 6)
    if kind == "newton":
        mode = rng.choice(["IR16_GMRES", "IR16_GMRES", "GMRESIR16", "GMRESIR16", "IR16", "FP64LU", "F32"])
        n = _log_int(rng, 64, 2048 if mode in ("FP64LU", "F32") else 16384)
        big = mode not in ("FP64LU", "F32")
        lu_nb = rng.choice([0, 0, 0, 64, 256 if n >= 512 else 0, 512 if n >= 1024 else 0]) if big else 0
        return {"kind": kind, "N": n, "c": c, "mode": mode, "lu_nb": lu_nb, "scale": int(big and rng.random() < 0.25)}
    if kind == "sweep":
        return {"kind": kind, "N": _log_int(rng, 256, 4096), "mode": rng.choice(["IR16", "GMRESIR16"])}
    if kind == "batch":
        lo = _log_int(rng, 32, 256)
        return {"kind": kind, "count": _log_int(rng, 8, 512), "n_lo": lo, "n_hi": _log_int(rng, 2 * lo, 2048)}
    if kind == "factor":
        return {"kind": kind, "N": _log_int(rng, 64, 8192), "c": c, "scale": rng.randrange(2)}
    if kind == "linsolve":
        return {"kind": kind, "N": _log_int(rng, 64, 12000), "c": c, "solver": rng.choice([0, 2])}
    if kind == "residual":
        fft = rng.randrange(2)
        return {"kind": kind, "N": _log_int(rng, 64, 32768 if fft else 4096), "c": c, "fft": fft}
    return {"kind": kind, "N": _log_int(rng, 64, 16384), "c": c}


# ------------------------------------------------------------------ inputs --


def _dev():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device="cpu")
    g.manual_seed(int(seed) % (1 << 31))
    return g


def _start(n, seed):
    """A starting iterate: ones, as the paper starts, within a tenth."""
    return (1.0 + 0.1 * (2.0 * torch.rand(n, generator=_gen(seed), dtype=torch.float64) - 1.0)).to(_dev())


def _hankel_transform(m, dev):
    length = 1 << max(2, (2 * m - 1).bit_length())
    h = torch.zeros(length, dtype=torch.float64, device=dev)
    h[: 2 * m - 1] = 1.0 / torch.arange(1, 2 * m, dtype=torch.float64, device=dev)
    return length, torch.fft.rfft(h)


def _rr(x, n, c, length, hf):
    """1 / (1 - (c / 2N) sum_j x_j mu_i / (mu_i + mu_j)) of eq. (3.2); x: (..., m), zero past each N."""
    m = x.shape[-1]
    s = torch.fft.irfft(hf * torch.conj(torch.fft.rfft(x, length)), length)[..., :m]
    i = torch.arange(m, dtype=torch.float64, device=x.device) + 0.5
    return 1.0 / (1.0 - (c / (2.0 * n)) * i * s)


def _r_at(x, c):
    n = x.numel()
    length, hf = _hankel_transform(n, x.device)
    return _rr(x, n, c, length, hf)


def _jacobian_rows(r, c, lo, hi):
    """Rows lo..hi of J in 64 bits."""
    n = r.numel()
    i = torch.arange(lo, hi, dtype=torch.float64, device=r.device)[:, None]
    j = torch.arange(n, dtype=torch.float64, device=r.device)[None, :]
    a = -(c / (2.0 * n)) * (r[lo:hi] ** 2)[:, None] * (i + 0.5) / (i + j + 1.0)
    a[torch.arange(hi - lo, device=r.device), torch.arange(lo, hi, device=r.device)] += 1.0
    return a


def _jacobian32(r, c, ld):
    n = r.numel()
    a = torch.zeros(n, ld, dtype=torch.float32, device=r.device)
    for lo in range(0, n, 2048):
        hi = min(n, lo + 2048)
        a[lo:hi, :n] = _jacobian_rows(r, c, lo, hi).float()
    return a


def _linear_system(case, seed):
    """J32 and the scaled right side -F/||F|| of a Newton step at a starting iterate."""
    n, c = case["N"], case["c"]
    x = _start(n, seed)
    r = _r_at(x, c)
    f = x - r
    return _jacobian32(r, c, _ld(n)), (-f / f.norm()).float()


def _ld(n):
    return (n + 63) // 64 * 64


def _gemv_inputs(case, seed):
    j32, b = _linear_system(case, seed)
    g = _gen(seed + 7)
    # a correction as the refinement holds it: b itself (J is near the identity), within a hundredth
    u = (b.cpu() * (1.0 + 0.01 * torch.randn(case["N"], generator=g))).to(b.device)
    return j32, b, u


def _residual_inputs(case, seed):
    n = case["N"]
    u = torch.randn(n, generator=_gen(seed + 3), dtype=torch.float32).to(_dev())
    return _start(n, seed), u, 0.02 / math.sqrt(n)


def _batch_instances(case):
    inst = workloads.batch_instances(count=case["count"], n_lo=case["n_lo"], n_hi=case["n_hi"])
    return [n for n, _ in inst], [c for _, c in inst]


def prepare(case, seed):
    kind = case["kind"]
    dev = _dev()
    if kind == "newton":
        n = case["N"]
        s = nl.Solver(n, case["c"], lu_nb=case["lu_nb"], scale_fp16=case["scale"])
        return {"kind": kind, "solver": s, "mode": case["mode"], "x0": _start(n, seed),
                "x": torch.empty(n, dtype=torch.float64, device=dev)}
    if kind == "sweep":
        n = case["N"]
        jobs = []
        for k, c in enumerate(workloads.SWEEP_C):
            s = nl.Solver(n, c, stream=(st := torch.cuda.Stream()))
            jobs.append((s, _start(n, seed * 5 + k), torch.empty(n, dtype=torch.float64, device=dev), st))
        return {"kind": kind, "jobs": jobs, "mode": case["mode"], "pool": ThreadPoolExecutor(len(jobs))}
    if kind == "batch":
        ns, cs = _batch_instances(case)
        # the outer block that the library's tuner takes for every larger bucket, so that no run depends on a timing
        return {"kind": kind, "batch": nl.Batch(ns, cs, lu_nb=64), "x0": _start(sum(ns), seed),
                "x": torch.empty(sum(ns), dtype=torch.float64, device=dev)}
    if kind == "factor":
        n, ld = case["N"], _ld(case["N"])
        return {"kind": kind, "N": n, "c": case["c"], "ld": ld, "scale": case["scale"],
                "r": _r_at(_start(n, seed), case["c"]),
                "J32": torch.empty(n, ld, dtype=torch.float32, device=dev),
                "J16": torch.empty(n, ld, dtype=torch.float16, device=dev),
                "rs": torch.empty(n, dtype=torch.float32, device=dev),
                "ipiv": torch.empty(n, dtype=torch.int32, device=dev)}
    if kind == "linsolve":
        n, ld = case["N"], _ld(case["N"])
        j32, b = _linear_system(case, seed)
        lu, ipiv = j32.half(), torch.empty(n, dtype=torch.int32, device=dev)
        nl.lu16(n, lu, ld, ipiv)
        return {"kind": kind, "N": n, "ld": ld, "J32": j32, "LU": lu, "ipiv": ipiv, "b": b, "solver": case["solver"],
                "u": torch.empty(n, dtype=torch.float32, device=dev)}
    if kind == "residual":
        x, u, scale = _residual_inputs(case, seed)
        out = [torch.empty_like(x) for _ in range(3)]
        return {"kind": kind, "N": x.numel(), "c": case["c"], "fft": case["fft"], "x": x, "u": u, "scale": scale,
                "out": out, "norm": torch.empty(1, dtype=torch.float64, device=dev)}
    j32, b, u = _gemv_inputs(case, seed)
    return {"kind": kind, "N": case["N"], "ld": _ld(case["N"]), "J32": j32, "b": b, "u": u, "r": torch.empty_like(b),
            "norm": torch.empty(1, dtype=torch.float64, device=dev)}


# --------------------------------------------------------------------- run --


def run(s):
    kind = s["kind"]
    if kind == "newton":
        s["solver"].solve_device(s["x"], tol=TOL, mode=s["mode"], x0=s["x0"])
        return s["x"]
    if kind == "sweep":
        mode = s["mode"]
        list(s["pool"].map(lambda j: j[0].solve_device(j[2], tol=TOL, mode=mode, x0=j[1]), s["jobs"]))
        return [x for _, _, x, _ in s["jobs"]]
    if kind == "batch":
        s["batch"].solve_device(s["x"], tol=TOL, x0=s["x0"])
        return s["x"]
    if kind == "factor":
        n, ld = s["N"], s["ld"]
        if s["scale"]:
            nl.k_jacobian_scaled(n, s["c"], s["r"], s["J32"], ld, s["J16"], ld, s["rs"])
        else:
            nl.k_jacobian(n, s["c"], s["r"], s["J32"], ld, s["J16"], ld)
        nl.lu16(n, s["J16"], ld, s["ipiv"])
        out = {"J32": s["J32"][:, :n], "LU": s["J16"][:, :n], "ipiv": s["ipiv"]}
        return out | {"rs": s["rs"]} if s["scale"] else out
    if kind == "linsolve":
        nl.linsolve16(s["N"], s["J32"], s["ld"], s["LU"], s["ld"], s["ipiv"], s["b"], s["u"], solver=s["solver"])
        return s["u"]
    if kind == "residual":
        f = nl.k_residual_fft if s["fft"] else nl.k_residual
        xo, F, r = s["out"]
        f(s["N"], s["c"], s["x"], F, r, s["norm"], u=s["u"], scale=s["scale"], x_out=xo)
        return {"x": xo, "F": F, "r": r, "norm": s["norm"]}
    nl.k_gemv_residual(s["N"], s["J32"], s["ld"], s["b"], s["u"], s["r"], s["norm"])
    return {"r": s["r"], "norm": s["norm"]}


# -------------------------------------------------------------------- work --


def _newton_steps(c):
    """Newton steps to 1e-10 (paper, Tables 2-3 and one step more): 3, 4, 6, 9, 11 for the sweep's c."""
    return 3 if c <= 0.6 else 4 if c <= 0.92 else 5 if c <= 0.98 else 6 if c <= 0.995 else 8 if c <= 0.9995 else 9 if c <= 0.99995 else 11


def _newton_flops(n, c):
    return _newton_steps(c) * (2.0 * n ** 3 / 3.0 + 6.0 * n * n)


def work(case):
    kind = case["kind"]
    if kind == "newton":
        n = case["N"]
        return {"bytes": 16.0 * n, "flops": _newton_flops(n, case["c"])}
    if kind == "sweep":
        n = case["N"]
        return {"bytes": 5 * 16.0 * n, "flops": sum(_newton_flops(n, c) for c in workloads.SWEEP_C)}
    if kind == "batch":
        ns, cs = _batch_instances(case)
        return {"bytes": 16.0 * sum(ns), "flops": sum(_newton_flops(n, c) for n, c in zip(ns, cs))}
    n = case["N"]
    if kind == "factor":  # r in, J32 and the factors out
        return {"bytes": 8.0 * n + 6.0 * n * n, "flops": 2.0 * n ** 3 / 3.0}
    if kind == "linsolve":  # J32 and the factors in
        return {"bytes": 6.0 * n * n + 8.0 * n, "flops": 4.0 * n * n}
    if kind == "residual":  # x and u in; x, F and r out; the sum as a convolution of length >= 2N
        length = 1 << (2 * n - 1).bit_length()
        return {"bytes": 36.0 * n, "flops": min(2.0 * n * n, 10.0 * length * math.log2(length))}
    return {"bytes": 4.0 * n * n + 12.0 * n, "flops": 2.0 * n * n}


# ------------------------------------------------------------------- exact --


def _fixed_point(ns, cs):
    """The solutions of eq. (3.2) for each (N, c), packed, by x <- 1/(1 - ...) in 64 bits.  It
    converges linearly from ones, at the rate (1 - s)/(1 + s), s = sqrt(1 - c)."""
    dev = _dev()
    m = max(ns)
    length, hf = _hankel_transform(m, dev)
    n = torch.tensor(ns, dtype=torch.float64, device=dev)[:, None]
    c = torch.tensor(cs, dtype=torch.float64, device=dev)[:, None]
    live = (torch.arange(m, device=dev)[None, :] < n).double()
    s = math.sqrt(1.0 - max(cs))
    steps = math.ceil(math.log(1e-17) / math.log((1.0 - s) / (1.0 + s)))
    x = live.clone()
    for _ in range(steps):
        x = _rr(x, n, c, length, hf) * live
    return [x[k, : ns[k]] for k in range(len(ns))]


def exact(case, seed):
    kind = case["kind"]
    if kind == "newton":
        return _fixed_point([case["N"]], [case["c"]])[0]
    if kind == "sweep":
        return _fixed_point([case["N"]] * len(workloads.SWEEP_C), list(workloads.SWEEP_C))
    if kind == "batch":
        return torch.cat(_fixed_point(*_batch_instances(case)))
    n, c = case["N"], case["c"]
    if kind == "factor":
        r = _r_at(_start(n, seed), c)
        j = torch.cat([_jacobian_rows(r, c, lo, min(n, lo + 2048)) for lo in range(0, n, 2048)])
        out = {"J32": j, "LU": None, "ipiv": None}
        if case["scale"]:
            # the largest power of two with 2^k (1 + c/(2N) r^2) <= 2^13
            k = torch.floor(torch.log2(2.0 ** 13 / (1.0 + c / (2.0 * n) * r * r)))
            out["rs"] = torch.pow(2.0, k)
            out["LU"] = torch.linalg.lu_factor(j * out["rs"][:, None])[0]
        else:
            out["LU"] = torch.linalg.lu_factor(j)[0]
        return out
    if kind == "linsolve":
        j32, b = _linear_system(case, seed)
        return torch.linalg.solve(j32[:, :n].double(), b.double())
    if kind == "residual":
        x, u, scale = _residual_inputs(case, seed)
        x = x + scale * u.double()
        r = _r_at(x, c)
        return {"x": x, "F": x - r, "r": r, "norm": (x - r).norm().reshape(1)}
    j32, b, u = _gemv_inputs(case, seed)
    r = torch.cat([b[lo:lo + 2048].double() - j32[lo:lo + 2048, :n].double() @ u.double() for lo in range(0, n, 2048)])
    return {"r": r, "norm": r.norm().reshape(1)}
