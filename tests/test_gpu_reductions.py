"""Warp sums, species votes and integer comparisons of the solve kernels at the edges of their shapes.

The fused and O(v/c) kernels form their block and species sums by recursive halving and decide Algorithm 2 in FP32
where that is certain; the plain per-iteration mode keeps one sum per species, a square root and FP64 compares.
Species groups of 2, 4, 8, 16 and 32 lanes, groups padded to 32 (20 energies) and groups of two warps (40, 64
energies), three (80) and, in the mixed path, four (128).
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc
from oracle import solver as osolver
from gpu_helpers import make_case, to_device, wnorm_errors

pytestmark = pytest.mark.gpu

SHAPES = [(2, 60.0, 1, 2), (2, 60.0, 2, 4), (8, 4.0, 1, 6), (8, 4.0, 2, 2), (16, 1.875, 2, 4), (10, 3.0, 2, 4),
          (20, 1.5, 2, 4), (32, 1.0, 2, 2), (40, 1.0, 2, 2)]


def _solve(ctx, t, velocity=False, **kw):
    args = (t["rho"], t["T"], t["Ye"], t["D"], t["I"], t["dt"], t["scale"])
    p = nmc.default_params(**kw)
    if velocity:
        v0 = torch.zeros((len(t["rho"]), 3), dtype=torch.float64, device="cuda")
        o = ctx.collision_solve_v(p, *args[:3], v0, *args[3:], freeze_velocity=True)
    else:
        o = ctx.collision_solve(p, *args)
    return {k: v.cpu().numpy() for k, v in o.items()}


@pytest.mark.parametrize("n_elem,de1,nq,ns", SHAPES)
def test_solves_match_the_plain_mode(n_elem, de1, nq, ns):
    """Steps of 1e-8 s: dtau chi <= 1e2, so the states converge without cycling at their rounding floor.  Tolerance: at
    tol 1e-12 both stop within tol (1 + dtau chi) ~ 1e-10 of the root; 1e-9 in the W2 norm.  A vote that passes too
    early misses that, one that passes too late shows in the iteration counts (the modes are separate compilations, so
    these are compared in total, to a fifth)."""
    edges, g, tables, inp = make_case(n_elem, de1, nq, ns, "profile", 33, seed=91)
    inp["dt"] *= 1e-2
    rng = np.random.default_rng(4)
    d = rng.normal(size=inp["I"].shape)
    inp["I"] = inp["I"][..., :1] * d / np.linalg.norm(d, axis=-1, keepdims=True)   # flux in all directions
    ctx = nmc.Context(edges, nq, ns, tables)
    t = to_device(inp)
    kw = dict(tol_inner=1e-12, tol_outer=1e-12, max_inner=500)
    plain = _solve(ctx, t, mode=nmc.MODE_PLAIN, **kw)
    outs = [_solve(ctx, t, **kw), _solve(ctx, t, velocity=True, **kw)]
    ctx.close()
    ok = plain["status"] & ~nmc.TABLE_CLAMP == 0
    assert np.count_nonzero(ok) >= 30, plain["status"]
    for o in outs:
        eD, eI = wnorm_errors(o["J"][ok], o["H"][ok], plain["J"][ok], plain["H"][ok], g.W2)
        assert eD.max() <= 1e-9 and eI.max() <= 1e-9, (eD.max(), eI.max())
        a, b = int(o["n_inner"][ok].sum()), int(plain["n_inner"][ok].sum())
        assert abs(a - b) <= b / 5, (a, b)


@pytest.mark.parametrize("n_elem,de1,nq,ns", [(2, 60.0, 2, 4), (10, 3.0, 2, 4), (40, 1.0, 2, 2), (64, 0.9, 2, 2)])
def test_mixed_solve_matches_the_oracle(n_elem, de1, nq, ns):
    """The FP32 votes over the same kinds of groups, to the mixed path's 1e-5."""
    edges, g, tables, inp = make_case(n_elem, de1, nq, ns, "profile", 4, seed=93)
    inp["dt"] *= 1e-2
    ctx = nmc.Context(edges, nq, ns, tables)
    o = _solve(ctx, to_device(inp), precision=nmc.MIXED, tol_inner=1e-11, tol_outer=1e-10, max_inner=500)
    ctx.close()
    ref = osolver.solve(g, tables, osolver.Params(tol_inner=1e-12, tol_outer=1e-12, max_inner=500), inp, nodes=range(4))
    for n, r in enumerate(ref):
        eD, eI = wnorm_errors(o["J"][n], o["H"][n], r["D"], r["I"], g.W2)
        assert eD.max() <= 1e-5 and eI.max() <= 1e-5, (n, eD, eI)


@pytest.mark.parametrize("n_elem,de1,nq,ns", SHAPES)
@pytest.mark.parametrize("velocity", [False, True])
def test_votes_at_the_threshold(n_elem, de1, nq, ns, velocity):
    """tol_inner set to a node's own first change, over the norm it is compared with, times 1 +- 1e-9 (far inside the
    band where the FP32 sums do not decide), 1 +- 4e-6 (its inside) and 1 +- 1e-4 (outside): one iteration is enough
    exactly when tol lies above.  The sums' own rounding, 1e-14, is far below 1e-9."""
    edges, g, tables, inp = make_case(n_elem, de1, nq, ns, "profile", 3, seed=92)
    rng = np.random.default_rng(5)
    d = rng.normal(size=inp["I"].shape)
    inp["I"] = inp["I"][..., :1] * d / np.linalg.norm(d, axis=-1, keepdims=True)
    ctx = nmc.Context(edges, nq, ns, tables)
    for n in range(3):
        node = {k: v[n:n + 1] for k, v in inp.items()}
        t = to_device(node)
        kw = dict(max_inner=1, max_outer=1, frozen_matter=1, velocity=velocity)
        o = _solve(ctx, t, tol_inner=1e-15, **kw)
        norm = lambda x: np.sqrt(np.sum(g.W2 * x ** 2, axis=-1))  # noqa: E731
        change = [norm(o["J"][0] - node["D"][0])] + [norm(o["H"][0, ..., c] - node["I"][0, ..., c]) for c in range(3)]
        r = float(np.max(np.stack(change) / norm(node["D"][0])))
        for e in (1e-9, 4e-6, 1e-4):
            above, below = (_solve(ctx, t, tol_inner=r * f, **kw)["status"][0] for f in (1.0 + e, 1.0 - e))
            assert above & nmc.NOT_CONVERGED_INNER == 0 and below & nmc.NOT_CONVERGED_INNER, (n, e, above, below)
    ctx.close()
