"""Algorithm 2's FP32 filter (species_vote_fp64) on grids whose integration weights leave FP32's range.

Energies in units far from MeV (here 1e-20 and 1e14 of the usual grid, the kernel tables scaled so that the rates stay
the usual ones) give weights w eps^2 d eps that FP32 holds as 0 or infinity.  The votes must be those of FP64, as the
plain mode takes them.  Matter is held fixed: its exchange has no meaning on such grids.

Tolerance: at tol 1e-12 both stop within tol (1 + dtau chi) of the root, dtau chi <= 1e4 on these states: 1e-8 in the
W2 norm.  A node may be stopped by its cap where rounding keeps it from tol 1e-12 (iteration counts and that status bit
are decided by rounding); nodes where that happens in the plain mode, at most five, are left out.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from gpu_helpers import make_case, to_device, wnorm_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [1e-20, 1e14])
@pytest.mark.parametrize("n_elem,de1", [(16, 1.875), (20, 1.5)])
def test_votes_do_not_depend_on_the_energy_unit(n_elem, de1, unit):
    edges, g, tables, inp = make_case(n_elem, de1, 2, 2, "profile", 20, seed=61)
    tables = dict(tables, nes=tables["nes"] * unit ** -3, pair=tables["pair"] * unit ** -3)
    ctx = nmc.Context(edges * unit, 2, 2, tables)
    t = to_device(inp)
    kw = dict(tol_inner=1e-12, tol_outer=1e-12, max_inner=2000, frozen_matter=1)
    args = (t["rho"], t["T"], t["Ye"], t["D"], t["I"], t["dt"], t["scale"])
    num = lambda o: {k: v.cpu().numpy() for k, v in o.items()}  # noqa: E731
    plain = num(ctx.collision_solve(nmc.default_params(mode=nmc.MODE_PLAIN, **kw), *args))
    fused = num(ctx.collision_solve(nmc.default_params(**kw), *args))
    v0 = torch.zeros((20, 3), dtype=torch.float64, device="cuda")
    vel = num(ctx.collision_solve_v(nmc.default_params(**kw), t["rho"], t["T"], t["Ye"], v0, *args[3:], freeze_velocity=True))
    ctx.close()
    ok = plain["status"] == 0
    assert np.count_nonzero(ok) >= 15, plain["status"]
    for o in (fused, vel):
        eD, eI = wnorm_errors(o["J"][ok], o["H"][ok], plain["J"][ok], plain["H"][ok], g.W2)
        assert eD.max() <= 1e-8 and eI.max() <= 1e-8, (eD.max(), eI.max())
