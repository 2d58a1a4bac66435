"""Setting a context up does not wait for work on other streams."""

import pytest
import torch

from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case

pytestmark = pytest.mark.gpu


def test_create_beside_a_busy_stream():
    edges, g, tables, _ = make_case(10, 3.0, 2, 2, "profile", 1)
    pts = [torch.tensor(x, device="cuda") for x in synthetic.make_interp_points(5000, g.eps, seed=2).values()]
    first = nmc.Context(edges, 2, 2, tables)     # loads the kernels
    ref = [first.opacity_interp(0, 1, *pts, mixed=m) for m in (False, True)]
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(int(4e9))              # about 2 s; a context takes some 10 ms
        done.record(side)
    ctx = nmc.Context(edges, 2, 2, tables)
    assert not done.query()
    for m in (False, True):                      # the tables are complete, for a call on any stream
        out = ctx.opacity_interp(0, 1, *pts, mixed=m)
        torch.cuda.current_stream().synchronize()
        assert torch.equal(out, ref[m])
    torch.cuda.synchronize()
    first.close()
    ctx.close()
