"""collision_adjoint with blocks of more than eight warps: six species and 33 to 64 energies (12 warps).

With matter held fixed the pairs do not know of one another, so a six-species gradient is that of a four-species context
(eight warps) pair by pair; the last pair, given the tables and moments of the second, must have its gradient.  Both
differentiate at the same moments.  Tolerance 1e-9 of the group's largest entry: one elimination of a system of condition
~dtau chi <= 1e4 in FP64 (1e-12), whatever warp holds a row.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from gpu_helpers import make_case, to_device

pytestmark = pytest.mark.gpu

NODES = 40


@pytest.mark.parametrize("n_elem,de1,nq", [(33, 2.0, 1), (17, 1.8, 2), (44, 1.0, 1)])
def test_six_species_equal_four(n_elem, de1, nq):
    edges, g, tables, inp = make_case(n_elem, de1, nq, 6, "profile", NODES, seed=81)
    tables = {k: (v.copy() if isinstance(v, np.ndarray) else v) for k, v in tables.items()}
    for k in ("emab", "iso", "nes"):
        tables[k][4:6] = tables[k][2:4]
    tables["pair"][2] = tables["pair"][1]
    for k in ("D", "I"):
        inp[k][:, 4:6] = inp[k][:, 2:4]
    four = dict(tables, **{k: np.ascontiguousarray(tables[k][:4]) for k in ("emab", "iso", "nes")},
                pair=np.ascontiguousarray(tables["pair"][:2]))
    p = nmc.default_params(frozen_matter=1, tol_inner=1e-12, max_inner=2000)
    t = to_device(inp)
    x = [t[k] for k in ("rho", "T", "Ye", "D", "I", "dt", "scale")]
    cut = lambda v, n: v[:, :n].contiguous()  # noqa: E731
    c6, c4 = nmc.Context(edges, nq, 6, tables), nmc.Context(edges, nq, 4, four)
    out = c6.collision_solve(p, *x)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    gJ, gH = (torch.randn(out[k].shape, generator=gen, device="cuda", dtype=torch.float64) for k in ("J", "H"))
    gJ[:, 4:6], gH[:, 4:6] = gJ[:, 2:4], gH[:, 2:4]
    a = c6.collision_adjoint(p, *x, out["J"], out["T"], gJ=gJ, gH=gH)
    b = c4.collision_adjoint(p, *x[:3], cut(x[3], 4), cut(x[4], 4), *x[5:], cut(out["J"], 4), out["T"], gJ=cut(gJ, 4),
                             gH=cut(gH, 4))
    assert torch.equal(a["status"], b["status"]) and not torch.any(a["status"] & ~nmc.TABLE_CLAMP)
    for k in ("J", "H"):
        ref = b[k]
        size = ref.abs().flatten(1).amax(1).view(-1, *[1] * (ref.dim() - 1))
        assert torch.all((a[k][:, :4] - ref).abs() <= 1e-9 * size), k
        assert torch.all((a[k][:, 4:6] - ref[:, 2:4]).abs() <= 1e-9 * size), k
    c6.close()
    c4.close()
