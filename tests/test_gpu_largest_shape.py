"""The FP64 solve at the largest shape that its shared memory holds: 4 species and 65 energies, 232 KB a block."""

import numpy as np
import pytest

from paper_2601_00976_gb300 import nmc
from gpu_helpers import make_case, gpu_solve, wnorm_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m_inner", [3, 5])
def test_four_species_65_energies(m_inner):
    """Accepted, and within 1e-8 of the plain mode: at tol 1e-12 both stop within tol (1 + dtau chi) of the root,
    dtau chi <= 1e4 on these states."""
    edges, g, tables, inp = make_case(65, 0.9, 1, 4, "profile", 12, seed=71)
    ctx = nmc.Context(edges, 1, 4, tables)
    kw = dict(tol_inner=1e-12, tol_outer=1e-12, max_inner=2000, m_inner=m_inner)
    out, ref = gpu_solve(ctx, inp, **kw), gpu_solve(ctx, inp, mode=nmc.MODE_PLAIN, **kw)
    ctx.close()
    ok = ref["status"] == 0
    assert np.count_nonzero(ok) >= 9, ref["status"]
    eD, eI = wnorm_errors(out["J"][ok], out["H"][ok], ref["J"][ok], ref["H"][ok], g.W2)
    assert eD.max() <= 1e-8 and eI.max() <= 1e-8, (eD.max(), eI.max())
