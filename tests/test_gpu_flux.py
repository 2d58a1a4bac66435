"""Flux along one axis and in all directions (FP64 fused solve).

A node whose bins carry no flux off the first axis leaves the other two components out of its iterations; the
outputs must be those of the general form.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from gpu_helpers import make_case, gpu_solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_elem,de1", [(16, 1.875), (32, 1.0)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e308])
def test_non_finite_first_component(n_elem, de1, bad):
    """H[..., 0] not finite (or at the edge of the range) in one bin, the other two components zero: that bin's
    components are scaled by its own factor 1 / (1 + dtau kappa), so 0 stays 0, in the bin and everywhere else."""
    edges, g, tables, inp = make_case(n_elem, de1, 2, 4, "profile", 6, seed=33)
    inp["I"][1, 2, 5, 0] = bad
    ctx = nmc.Context(edges, 2, 4, tables)
    out = gpu_solve(ctx, inp)
    ctx.close()
    assert np.all(out["H"][..., 1:] == 0.0)
    assert out["status"][1] == (0 if np.isfinite(bad) else nmc.NONFINITE)
    assert np.isfinite(out["H"][1, 2, 5, 0]) == np.isfinite(bad)
    assert np.all(np.isfinite(np.delete(out["H"], 1, 0))) and np.all(np.delete(out["status"], 1) == 0)


def test_non_finite_factor():
    """A scale factor that makes kappa NaN: every component of every bin is NaN, as in the general form."""
    edges, g, tables, inp = make_case(16, 1.875, 2, 4, "profile", 3, seed=34)
    inp["scale"][1, 1] = np.nan
    ctx = nmc.Context(edges, 2, 4, tables)
    axis = gpu_solve(ctx, inp)
    inp["I"][1, 0, 0, 1] = 1e-30     # the general form
    general = gpu_solve(ctx, inp)
    ctx.close()
    for o in (axis, general):
        assert o["status"][1] & nmc.NONFINITE and np.all(np.isnan(o["H"][1]))
    assert np.all(axis["H"][[0, 2]][..., 1:] == 0.0)
