"""Node order of the persistent kernels (nmc_order.cu): longest nodes first.

A call with more nodes than resident blocks, up to 2^16, takes its nodes by falling rho dt; smaller and larger
calls in index order.  Every node's result is its own, so a batch must equal, bit for bit, the same nodes solved
in pieces small enough to be taken in index order.  Sizes at both ends of the rule; equal, invalid, zero and
extreme keys.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case, to_device

pytestmark = pytest.mark.gpu

PIECE = 150      # at most one node per SM: index order


@pytest.mark.parametrize("n", [153, 457, 609, 2501, 65536, 65537])
@pytest.mark.parametrize("velocity", [False, True])
def test_batch_equals_its_pieces(n, velocity):
    edges, g, tables, inp = make_case(10, 3.0, 1, 2, "core_tail", n, seed=95)
    rng = np.random.default_rng(4)
    odd = rng.permutation(n)[:40]
    inp["rho"][odd[:20]] = [np.nan, np.inf, 0.0, -1.0, 1e-300] * 4
    inp["dt"][odd[20:30]] = 0.0
    inp["rho"][odd[30:]] = 1e12
    inp["dt"][odd[30:]] = 1e-6
    t = to_device(inp)
    v = torch.tensor(synthetic.make_velocities("random", n, seed=3), device="cuda")
    ctx = nmc.Context(edges, 1, 2, tables)
    p = nmc.default_params(max_inner=12, max_outer=3)   # cut short: the order is what is tested

    def solve(i, j):
        x = [t[k][i:j].contiguous() for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
        if velocity:
            return ctx.collision_solve_v(p, *x[:3], v[i:j].contiguous(), *x[3:])
        return ctx.collision_solve(p, *x)
    whole = solve(0, n)
    for i in sorted({0, max(0, n // 2), max(0, n - PIECE)}):
        part = solve(i, min(n, i + PIECE))
        for k in part:
            a, b = part[k], whole[k][i:min(n, i + PIECE)]
            assert torch.equal(a.view(torch.int64 if a.dtype == torch.float64 else torch.int32),
                               b.contiguous().view(torch.int64 if a.dtype == torch.float64 else torch.int32)), (i, k)
    ctx.close()
