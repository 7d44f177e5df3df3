"""First FP64 calls of a process around a graph capture. The tables they need are
uploaded without disturbing a capture that another stream has going on; under
capture themselves they run on kernels that need none, where there is one."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SETUP = """
import torch
from paper_2302_08381_gb300 import api
gen = torch.Generator(device="cuda").manual_seed(3)
x = torch.randn(1000, 3, generator=gen, device="cuda", dtype=torch.float64)
new = lambda: (torch.empty(1000, 81, device="cuda", dtype=torch.float64),
               torch.empty(1000, 3, 81, device="cuda", dtype=torch.float64))
point, out, degree = new(), new(), new()
call = lambda o, **kw: api.spherical_harmonics(x, 8, True, gradients=True, out=o, **kw)
call(point, kernel="point_hc")  # needs no tables
count = torch.zeros(8, device="cuda")
count.add_(0.0)
other = torch.cuda.Stream()
graph = torch.cuda.CUDAGraph()
torch.cuda.synchronize()
same = lambda a, b: all(torch.equal(u, v) for u, v in zip(a, b))
"""

ELSEWHERE = """
with torch.cuda.graph(graph):  # captures in global mode
    count.add_(1.0)
    with torch.cuda.stream(other):
        call(out)
    count.add_(1.0)
other.synchronize()
graph.replay()
torch.cuda.synchronize()
call(degree, kernel="degree")
assert torch.all(count == 2) and same(out, degree) and not same(out, point)
"""

ITSELF = """
with torch.cuda.graph(graph):
    call(out)
graph.replay()
torch.cuda.synchronize()
call(degree, kernel="degree")
assert same(out, point) and not same(out, degree)
call(out)
torch.cuda.synchronize()
assert same(out, degree)
"""

# a kernel that needs tables, first called under capture: they are uploaded at once
NEEDED = """
z = torch.randn(70_000, 3, device="cuda")
mixed = lambda o, **kw: api.spherical_harmonics(z, 4, True, gradients=True, qprec="f64", out=o, **kw)
a, b = ((torch.empty(70_000, 25, device="cuda"), torch.empty(70_000, 3, 25, device="cuda")) for _ in range(2))
torch.cuda.synchronize()
with torch.cuda.graph(graph):
    mixed(a)
graph.replay()
torch.cuda.synchronize()
mixed(b, kernel="degree")
assert same(a, b)
"""


@pytest.mark.parametrize("body", [ELSEWHERE, ITSELF, NEEDED], ids=["elsewhere", "itself", "needed"])
def test_first_fp64_call(body):
    r = subprocess.run([sys.executable, "-c", SETUP + body], capture_output=True, text=True, cwd=ROOT, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
