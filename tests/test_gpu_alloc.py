"""Device memory running short while a context is set up.

The NMC_DEBUG build lets the k-th allocation of nmc_create fail (NMC_FAIL_ALLOC=k: it asks for more memory than any
device has).  Each allocation in turn: set-up either reports NMC_ENOMEM or, for the tables that only make calls
faster, gives a context whose calls succeed with the usual results; no CUDA error stays pending for a later call.

The opacity lookup without its fixed-point tables is the FP64 form: 1e-13 as in test_gpu_interp_fixed.py.  Node
order, and the FP32 lookup, do not change a bit.  In a child process, so that the two builds do not share one.
"""

import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

CHILD = r"""
import os, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case, to_device
N = 2500                         # more nodes than resident blocks: the node order is in use
edges, g, tables, inp = make_case(10, 3.0, 1, 2, "profile", N, seed=41)
t = to_device(inp)
pts = [torch.tensor(x, device="cuda") for x in synthetic.make_interp_points(5000, g.eps, seed=2).values()]

def calls(ctx):
    o = ctx.collision_solve(nmc.default_params(), t["rho"], t["T"], t["Ye"], t["D"], t["I"], t["dt"], t["scale"])
    return o["J"], ctx.opacity_interp(0, 1, *pts, mixed=True), ctx.opacity_interp(0, 1, *pts)

whole = nmc.Context(edges, 1, 2, tables)
ref = calls(whole)
refused, served, exact, uses = 0, 0, 0, []
for k in range(1, 61):
    os.environ["NMC_FAIL_ALLOC"] = str(k)
    free = torch.cuda.mem_get_info()[0]
    try:
        ctx = nmc.Context(edges, 1, 2, tables)
    except nmc.NmcError as e:
        assert "code 3" in str(e), e                     # NMC_ENOMEM
        refused += 1
        calls(whole)                                     # no error is pending
        torch.ones(3, device="cuda").sum().item()
        continue
    assert ctx.last_error() == "", ctx.last_error()
    used = free - torch.cuda.mem_get_info()[0]
    got = calls(ctx)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    assert torch.max(torch.abs(got[2] - ref[2]) / ref[2]).item() <= 1e-13
    served += 1
    exact += int(torch.equal(got[2], ref[2]))
    uses.append((used, torch.equal(got[2], ref[2])))
    ctx.close()
del os.environ["NMC_FAIL_ALLOC"]
# the FP32 lookup's cells, 2 x 2 x 16 x 31 x 31 x 9 of 32 bytes, are one allocation (17.7 MB), the FP64 form's another
most = max(u for u, _ in uses)
no_cells = sum(1 for u, same in uses if same and u < most - (14 << 20))
print("ALLOC", refused, served, exact, no_cells)
"""


def test_each_allocation_failing_in_turn():
    from paper_2601_00976_gb300 import _build
    _build.build(debug=True)
    env = dict(os.environ, NMC_DEBUG="1")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, env=env, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    refused, served, exact, no_cells = (int(x) for x in r.stdout.split("ALLOC")[1].split())
    # the required tables, then those that are optional, then a k beyond the last allocation
    assert refused >= 20 and served - exact >= 5 and exact >= 5, (refused, served, exact)
    assert no_cells == 1, no_cells   # a context without the FP32 lookup's cells was served
