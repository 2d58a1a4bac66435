"""collision_adjoint's two register classes for blocks of up to 128 threads.

The narrow class serves batches of more nodes than the wide one's resident blocks, at shapes whose shared memory has
room for more; both are one source, and every node's gradient is its own, so a large batch must equal, bit for bit, the
same nodes taken in pieces of at most one node per SM (the wide class, compared with the oracle elsewhere).
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from gpu_helpers import make_case, to_device

pytestmark = pytest.mark.gpu

PIECE = 150
N = 2600      # above the wide class's resident blocks at every shape here (8 of 152 SMs' at most)


@pytest.mark.parametrize("n_elem,de1,nq,ns", [(10, 3.0, 1, 2), (16, 1.875, 1, 4), (20, 1.5, 1, 4), (12, 2.35, 2, 4),
                                              (8, 4.0, 2, 6), (16, 1.875, 2, 4)])
def test_batch_equals_its_pieces(n_elem, de1, nq, ns):
    edges, g, tables, inp = make_case(n_elem, de1, nq, ns, "profile", N, seed=51)
    ctx = nmc.Context(edges, nq, ns, tables)
    t = to_device(inp)
    p = nmc.default_params()
    x = [t[k] for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
    out = ctx.collision_solve(p, *x)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    cot = {"g" + k: torch.randn(out[k].shape, generator=gen, device="cuda", dtype=torch.float64) for k in ("J", "H", "Ye", "T")}

    def grad(i, j):
        s = lambda v: v[i:j].contiguous()  # noqa: E731
        return ctx.collision_adjoint(p, *[s(v) for v in x], s(out["J"]), s(out["T"]), **{k: s(v) for k, v in cot.items()})
    whole = grad(0, N)
    for i in range(0, N, PIECE):
        part = grad(i, min(N, i + PIECE))
        for k, v in part.items():
            a, b = v, whole[k][i:min(N, i + PIECE)].contiguous()
            as_bits = torch.int64 if v.dtype == torch.float64 else torch.int32
            assert torch.equal(a.view(as_bits), b.view(as_bits)), (i, k)
    ctx.close()


def test_first_call_under_capture():
    """Either class's first call can be recorded in a graph."""
    edges, g, tables, inp = make_case(12, 2.35, 2, 4, "profile", N, seed=52)
    ctx = nmc.Context(edges, 2, 4, tables)
    t = to_device(inp)
    p = nmc.default_params()
    x = [t[k] for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
    out = ctx.collision_solve(p, *x)
    gJ = torch.ones_like(out["J"])
    for n in (100, N):
        s = lambda v: v[:n].contiguous()  # noqa: E731
        a = [s(v) for v in x] + [s(out["J"]), s(out["T"])]
        c = s(gJ)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g1 = ctx.collision_adjoint(p, *a, gJ=c)
        graph.replay()
        g2 = ctx.collision_adjoint(p, *a, gJ=c)
        assert torch.equal(g1["J"], g2["J"])
    ctx.close()
