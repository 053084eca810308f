"""A captured solve as the first call of a process, under a forced schedule (whose
applies of few planes run the direct i pass) and by the library's choice: every
kernel attribute that the captured step needs is set before the capture. u equals
that of the solve launched kernel by kernel, to the bit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
import torch
import workloads as W
from paper_2502_05507_gb300 import Context, Problem, set_conv_schedule
P = W.torus_helmholtz(128, kappa2=10.0)
set_conv_schedule(sys.argv[1])
ctx = Context(0)
prob = Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, P.kappa2, "double")
f = torch.from_numpy(P.f()).cuda()
g = torch.from_numpy(P.g_at(prob.boundary_points())).cuda()
u = [prob.solve(f, g, tol=1e-9, precision=sys.argv[2], use_graphs=graphs)[1] for graphs in (True, False)]
assert torch.equal(u[0], u[1])
"""


@pytest.mark.parametrize("schedule,precision", [("passes", "mixed"), ("passes", "fp64"), ("passes", "df64"), ("auto", "mixed"),
                                                ("auto", "fp64")])
def test_first_call_is_captured(schedule, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", CHILD, schedule, precision], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
