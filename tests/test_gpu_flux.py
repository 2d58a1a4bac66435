"""Flux along one axis and in all directions (FP64 fused solve).

A node whose bins carry no flux off the first axis leaves the other two components out of its iterations; the
outputs must be those of the general form.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from oracle import solver as osolver
from gpu_helpers import make_case, gpu_solve, compare_node
import oracle_pool

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


def _all_directions(inp, seed):
    d = np.random.default_rng(seed).normal(size=inp["I"].shape)
    inp["I"] = inp["I"][..., :1] * d / np.linalg.norm(d, axis=-1, keepdims=True)


@pytest.mark.parametrize("n_elem,de1,kind,N", [(16, 1.875, "profile", 10), (32, 1.0, "perturbed", 3)])
def test_flux_in_all_directions_matches_the_oracle(n_elem, de1, kind, N):
    """The general form at full physics: four species, 32 and 64 energies, randomly directed flux; to 1e-10, both sides
    at tol 1e-13."""
    edges, g, tables, inp = make_case(n_elem, de1, 2, 4, kind, N, seed=35)
    _all_directions(inp, 36)
    kw = dict(tol_inner=1e-13, tol_outer=1e-13, max_inner=2000, max_outer=100)
    ctx = nmc.Context(edges, 2, 4, tables)
    out = gpu_solve(ctx, inp, **kw)
    ctx.close()
    tasks = [dict(case=(n_elem, de1, 2, 4, 0), params=kw, x=oracle_pool.node_slice(inp, n)) for n in range(N)]
    for n, r in enumerate(oracle_pool.run(tasks, _node_solve)):
        compare_node(out, n, r, g.W2, 1e-10)


def _node_solve(task):
    g, tables = oracle_pool._grid_tables(*task["case"])
    x = task["x"]
    return osolver.solve_node(g, tables, osolver.Params(**task["params"]), x["rho"], x["T"], x["Ye"], x["D"], x["I"], x["dt"],
                              x["scale"])


@pytest.mark.parametrize("n_elem,de1", [(16, 1.875), (32, 1.0)])
def test_both_kinds_of_node_in_one_launch(n_elem, de1):
    """Nodes with flux along one axis and in all directions, mixed: blocks take one kind after the other, with the
    history registers of the one before; every node must equal, bit for bit, the same node in a launch in which each
    block takes one node."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 5 * sms + 3
    edges, g, tables, inp = make_case(n_elem, de1, 2, 4, "profile", n, seed=37)
    one_axis = inp["I"].copy()
    _all_directions(inp, 38)
    pick = np.random.default_rng(39).random(n) < 0.5
    inp["I"][pick] = one_axis[pick]
    inp["I"][3::17, :, :, 1:] *= -0.0        # signed zeros: along one axis too
    ctx = nmc.Context(edges, 2, 4, tables)
    whole = gpu_solve(ctx, inp)
    for i in range(0, n, sms):
        part = gpu_solve(ctx, {k: v[i:i + sms] for k, v in inp.items()})
        for k in part:
            assert np.array_equal(part[k], whole[k][i:i + sms]), (i, k)
    ctx.close()
    assert np.all(whole["status"] == 0)
