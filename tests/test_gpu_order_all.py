"""Node order of the persistent kernels (nmc_order.cu): every node of an ordered batch, around the rule's real lines.

collision_solve_noalloc takes nodes in index order whatever the batch; collision_solve orders them by falling rho dt
when the batch has more nodes than the launch has blocks.  The outputs must be the same bits at every node, and a node
that no block took would show: outputs are filled with a sentinel first.  The shape holds two blocks an SM (4 species,
32 energies in FP64), so that the line lies at 304 nodes on a 152-SM device; whether a batch was ordered is told by the
device's own limits.
"""

import ctypes

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case, to_device

pytestmark = pytest.mark.gpu

# more than two 128-thread blocks of 95-110 KB do not fit an SM's 228 KB
BLOCKS_PER_SM = 2
SENTINEL = -12345.0


def _outputs(n, ns, ne):
    f64 = lambda *s: torch.full(s, SENTINEL, dtype=torch.float64, device="cuda")  # noqa: E731
    i32 = lambda: torch.full((n,), -7, dtype=torch.int32, device="cuda")  # noqa: E731
    return dict(J=f64(n, ns, ne), H=f64(n, ns, ne, 3), Ye=f64(n), eps=f64(n), T=f64(n), n_outer=i32(), n_inner=i32(),
                status=i32())


def _same_bits(a, b):
    as_int = torch.int64 if a.dtype == torch.float64 else torch.int32
    return torch.equal(a.view(as_int), b.view(as_int))


def _keys(inp, n, kind):
    """rho and dt of the sort's kinds of keys: spread, equal, odd (invalid, zero, extreme) and over 64 octaves."""
    rng = np.random.default_rng(6)
    if kind == "equal":
        inp["rho"][:] = 1e11
        inp["dt"][:] = 1e-7
    elif kind == "wide":
        inp["dt"][:] = 10.0 ** rng.uniform(-300.0, -6.0, size=n)
    elif kind == "odd":
        k = rng.permutation(n)
        inp["rho"][k[:n // 4]] = np.resize([np.nan, np.inf, -np.inf, 0.0, -1.0, 5e-324, 1e-300, 1e300], n // 4)
        inp["dt"][k[n // 8:n // 3]] = np.resize([np.nan, np.inf, 0.0, -0.0, -1.0, 5e-324], n // 3 - n // 8)


@pytest.mark.parametrize("kind", ["spread", "equal", "wide", "odd"])
def test_fused_batch_equals_index_order(kind):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = BLOCKS_PER_SM * sms
    edges, g, tables, _ = make_case(16, 1.875, 2, 4, "profile", 1)
    ctx = nmc.Context(edges, 2, 4, tables)
    L = nmc.load_library()
    p = nmc.default_params(max_inner=6, max_outer=2)   # cut short: the order is what is tested
    for n in (line, line + 1, line + 2, 1023, 1025, 4097):
        ordered = line < n <= 65536
        assert ordered == (n != line)
        inp = synthetic.make_inputs("core_tail", n, g.eps, 4, seed=n)
        _keys(inp, n, kind)
        t = to_device(inp)
        x = [t[k] for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
        a, b = _outputs(n, 4, ctx.ne), _outputs(n, 4, ctx.ne)
        ctx.collision_solve(p, *x, out=a)
        ptr = lambda v: ctypes.c_void_p(v.data_ptr())  # noqa: E731
        rc = L.collision_solve_noalloc(ctx._h, ctypes.byref(p), n, *[ptr(v) for v in x],
                                       *[ptr(b[k]) for k in ("J", "H", "Ye", "eps", "T", "n_outer", "n_inner", "status")],
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == nmc.NMC_OK
        for k in a:
            assert _same_bits(a[k], b[k]), (n, k)
            assert not torch.any(a[k] == (SENTINEL if a[k].dtype == torch.float64 else -7)), (n, k)
    ctx.close()


@pytest.mark.parametrize("kind", ["spread", "odd"])
def test_velocity_batch_equals_its_pieces(kind):
    """The O(v/c) solve: every node against pieces of at most one node per SM, which are taken in index order."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * BLOCKS_PER_SM * sms + 5
    edges, g, tables, inp = make_case(16, 1.875, 2, 4, "core_tail", n, seed=9)
    _keys(inp, n, kind)
    t = to_device(inp)
    v = torch.tensor(synthetic.make_velocities("random", n, seed=3), device="cuda")
    ctx = nmc.Context(edges, 2, 4, tables)
    p = nmc.default_params(max_inner=6, max_outer=2)

    def solve(i, j):
        x = [t[k][i:j].contiguous() for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
        return ctx.collision_solve_v(p, *x[:3], v[i:j].contiguous(), *x[3:])
    whole = solve(0, n)
    for i in range(0, n, sms):
        part = solve(i, min(n, i + sms))
        for k in part:
            assert _same_bits(part[k], whole[k][i:min(n, i + sms)].contiguous()), (i, k)
    ctx.close()
