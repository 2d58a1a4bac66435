"""Warp sums, species votes and integer comparisons of the solve kernels at the edges of their shapes.

The fused and O(v/c) kernels form their block and species sums by recursive halving and vote on squared
thresholds; the plain per-iteration mode keeps one sum per species, a square root and FP64 compares.  Both
are compared over species groups of 2, 4, 8, 16 and 32 lanes, groups padded to 32 (20 energies) and groups
of several warps (40, 64 energies).

Tolerance: at tol 1e-12 both stop within tol (1 + dtau chi) of the root, dtau chi <= 1e4 on these states:
1e-8 in the W2 norm.  The two are separate compilations, so an inner loop may end one iteration apart.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case, to_device, wnorm_errors

pytestmark = pytest.mark.gpu

SHAPES = [(2, 60.0, 1, 2), (2, 60.0, 2, 4), (8, 4.0, 1, 6), (8, 4.0, 2, 2), (16, 1.875, 2, 4), (10, 3.0, 2, 4),
          (20, 1.5, 2, 4), (32, 1.0, 2, 2)]


@pytest.mark.parametrize("n_elem,de1,nq,ns", SHAPES)
def test_solves_match_the_plain_mode(n_elem, de1, nq, ns):
    edges, g, tables, inp = make_case(n_elem, de1, nq, ns, "profile", 33, seed=91)
    ctx = nmc.Context(edges, nq, ns, tables)
    t = to_device(inp)
    kw = dict(tol_inner=1e-12, tol_outer=1e-12)
    args = (t["rho"], t["T"], t["Ye"], t["D"], t["I"], t["dt"], t["scale"])
    plain = {k: v.cpu().numpy() for k, v in ctx.collision_solve(nmc.default_params(mode=nmc.MODE_PLAIN, **kw), *args).items()}
    fused = {k: v.cpu().numpy() for k, v in ctx.collision_solve(nmc.default_params(**kw), *args).items()}
    v0 = torch.zeros((33, 3), dtype=torch.float64, device="cuda")
    vel = {k: v.cpu().numpy() for k, v in ctx.collision_solve_v(nmc.default_params(**kw), t["rho"], t["T"], t["Ye"], v0,
                                                                *args[3:], freeze_velocity=True).items()}
    ctx.close()
    for o in (fused, vel):
        assert np.array_equal(o["status"], plain["status"])
        assert np.all(np.abs(o["n_inner"] - plain["n_inner"]) <= plain["n_outer"])
        eD, eI = wnorm_errors(o["J"], o["H"], plain["J"], plain["H"], g.W2)
        assert eD.max() <= 1e-8 and eI.max() <= 1e-8, (eD.max(), eI.max())
