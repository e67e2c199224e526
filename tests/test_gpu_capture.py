"""Kernel-level entry points that neither synchronise nor read back, called
inside a stream capture as a process's first calls (each test in a process of its
own: what the library makes at its first call must not depend on an earlier one)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

SETUP = """
import sys
sys.path.insert(0, {root!r})
import torch
from paper_2307_16051_gb300 import nl
N, c, ld = 500, 0.9, 512
d = torch.device("cuda:0")
x = torch.linspace(1.0, 1.5, N, device=d, dtype=torch.float64)
F, r, F2, r2 = (torch.zeros_like(x) for _ in range(4))
fn, fn2 = (torch.zeros(1, device=d, dtype=torch.float64) for _ in range(2))
rin = torch.linspace(1.0, 2.0, N, device=d, dtype=torch.float64)
J32, J32b = (torch.zeros(N, ld, device=d, dtype=torch.float32) for _ in range(2))
J16, J16b = (torch.zeros(N, ld, device=d, dtype=torch.float16) for _ in range(2))
J64, J64b = (torch.zeros(N, ld, device=d, dtype=torch.float64) for _ in range(2))
A = torch.linspace(-1.0, 1.0, N * ld, device=d, dtype=torch.float32).reshape(N, ld)
b, u, g, g2 = (torch.linspace(0.0, 1.0, ld, device=d, dtype=torch.float32) for _ in range(4))
calls = {{
    "residual": (lambda s: nl.k_residual(N, c, x, F, r, fn, stream=s),
                 lambda: nl.k_residual(N, c, x, F2, r2, fn2), ((F, F2), (r, r2), (fn, fn2))),
    "residual_fft": (lambda s: nl.k_residual_fft(N, c, x, F, r, fn, stream=s),
                     lambda: nl.k_residual_fft(N, c, x, F2, r2, fn2), ((F, F2), (r, r2), (fn, fn2))),
    "jacobian": (lambda s: nl.k_jacobian(N, c, rin, J32, ld, J16, ld, stream=s),
                 lambda: nl.k_jacobian(N, c, rin, J32b, ld, J16b, ld), ((J32, J32b), (J16, J16b))),
    "jacobian64": (lambda s: nl.k_jacobian64(N, c, rin, J64, ld, stream=s),
                   lambda: nl.k_jacobian64(N, c, rin, J64b, ld), ((J64, J64b),)),
    "gemv": (lambda s: nl.k_gemv_residual(N, A, ld, b, u, g, fn, stream=s),
             lambda: nl.k_gemv_residual(N, A, ld, b, u, g2, fn2), ((g, g2), (fn, fn2))),
}}
captured, plain, outs = calls[{name!r}]
st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
torch.cuda.synchronize()
"""

FIRST_CALL = """
with torch.cuda.graph(graph, stream=st):
    captured(st)
for _ in range(2):
    graph.replay()
torch.cuda.synchronize()
"""

CHECK = """
plain()
torch.cuda.synchronize()
for got, ref in outs:
    assert torch.equal(got, ref)
print("equal")
"""


def _run(name, body):
    code = SETUP.format(root=ROOT, name=name) + body + CHECK
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "equal" in p.stdout, p.stderr[-2000:]


@pytest.mark.parametrize("name", ["residual", "residual_fft", "jacobian", "jacobian64", "gemv"])
def test_first_call_inside_a_capture(name):
    _run(name, FIRST_CALL)
