"""opacity_interp's fixed-point form against its FP64 form and against plain 64-bit numpy.

A context whose ln tables hold one value beyond the fixed-point range takes the FP64 form for every point, so
the same points, clean species, go through both.  Arguments: ordinary points, the axes' ends and beyond, table
nodes and their neighbours in the last bit, zero, denormal, negative, infinite and NaN coordinates (all clamped).

Tolerance 1e-13: ln chi is at most ~60 in magnitude here, FP64 rounds it by up to 60 * 2^-53 per operation over
about ten operations on the result's path (7e-14); the fixed-point form by less.
"""

import numpy as np
import pytest
import torch

from paper_2601_00976_gb300 import nmc, synthetic
from gpu_helpers import make_case

pytestmark = pytest.mark.gpu

TOL = 1e-13


def _points(rng, g, n):
    lo, hi, nr = synthetic.RHO_AXIS
    t0, t1, nt = synthetic.T_AXIS
    y0, y1, ny = synthetic.YE_AXIS
    rho, T = 10.0 ** rng.uniform(lo - 0.3, hi + 0.3, n), 10.0 ** rng.uniform(t0 - 0.3, t1 + 0.3, n)
    Ye, E = rng.uniform(y0 - 0.05, y1 + 0.05, n), np.exp(rng.uniform(np.log(g.eps[0]) - 1, np.log(g.eps[-1]) + 1, n))
    node = [10.0 ** np.linspace(lo, hi, nr), 10.0 ** np.linspace(t0, t1, nt), np.linspace(y0, y1, ny), g.eps]
    odd = np.array([0.0, -0.0, 5e-324, 1e-310, -1.0, np.inf, -np.inf, np.nan, 1.0, 1e300, 2.0 ** -1022])
    for x, nd in zip((rho, T, Ye, E), node):
        k = min(n, 4 * len(nd))
        x[:k] = np.nextafter(np.tile(nd, 4)[:k], rng.choice([-np.inf, 0.0, np.inf], k))
        rng.shuffle(x)
        j = rng.permutation(n)[:n // 5]
        x[j] = odd[rng.integers(0, len(odd), len(j))]
    return [torch.tensor(x, device="cuda") for x in (rho, T, Ye, E)]


def _reference(tables, which, s, pts):
    x = []
    with np.errstate(all="ignore"):
        rho, T, Ye, E = (p.cpu().numpy() for p in pts)
        for v, ax in ((np.log10(rho), tables["lrho"]), (np.log10(T), tables["lT"]), (Ye, tables["ye"])):
            c = (v - ax[0]) / (ax[1] - ax[0]) * (ax[2] - 1)
            c = np.clip(np.where(np.isnan(c), 0.0, c), 0.0, ax[2] - 1)
            i = np.minimum(c.astype(int), ax[2] - 2)
            x.append((i, c - i))
        le = np.log(E)
    ln = np.log(tables["energies"])
    le = np.clip(np.where(np.isnan(le), ln[0], le), ln[0], ln[-1])
    j = np.clip(np.searchsorted(ln, le, side="right") - 1, 0, len(ln) - 2)
    te = (le - ln[j]) / (ln[j + 1] - ln[j])
    (ir, tr), (it, tt), (iy, ty) = x
    tab, v = tables["emab" if which == 0 else "iso"][s], 0.0
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                w = (tr if a else 1 - tr) * (tt if b else 1 - tt) * (ty if c else 1 - ty)
                v = v + w * ((1 - te) * tab[iy + c, it + b, ir + a, j] + te * tab[iy + c, it + b, ir + a, j + 1])
    return np.exp(v)


@pytest.mark.parametrize("n_elem,de1,nq,ns,n", [(16, 1.875, 2, 4, 70001), (2, 60.0, 1, 2, 1), (2, 60.0, 1, 2, 513),
                                                (10, 3.0, 1, 6, 4097), (32, 1.0, 2, 2, 30000)])
def test_fixed_point_matches_fp64(n_elem, de1, nq, ns, n):
    edges, g, tables, _ = make_case(n_elem, de1, nq, ns, "profile", 1)
    wide = dict(tables, emab=tables["emab"].copy())
    wide["emab"][ns - 1, 0, 0, 0, 0] = -600.0     # the last species only: this context takes the FP64 form
    fixed, fp64 = nmc.Context(edges, nq, ns, tables), nmc.Context(edges, nq, ns, wide)
    pts = _points(np.random.default_rng(5), g, n)
    for which in (0, 1):
        for s in range(ns - 1):
            a, b = (c.opacity_interp(which, s, *pts).cpu().numpy() for c in (fixed, fp64))
            r = _reference(tables, which, s, pts)
            assert np.max(np.abs(a - b) / b) <= TOL
            assert np.max(np.abs(a - r) / r) <= TOL
            # no further from the plain values than the FP64 form, on the whole
            assert np.sqrt(np.mean(((a - r) / r) ** 2)) <= max(1.5 * np.sqrt(np.mean(((b - r) / r) ** 2)), 1e-15)
    fixed.close()
    fp64.close()


@pytest.mark.parametrize("n", [1, 255, 152 * 8 * 256, 152 * 16 * 256 - 1, 152 * 16 * 256 + 1, 1000003])
def test_points_do_not_depend_on_the_batch(n):
    """Sizes around one and two points a thread: every point's value is the one it has in a call of its own few
    thousand neighbours, bit for bit, in both precisions (each point is evaluated by itself)."""
    edges, g, tables, _ = make_case(10, 3.0, 2, 2, "profile", 1)
    ctx = nmc.Context(edges, 2, 2, tables)
    pts = [p.contiguous() for p in _points(np.random.default_rng(6), g, n)]
    for mixed in (False, True):
        whole = ctx.opacity_interp(1, 1, *pts, mixed=mixed)
        for i in sorted({0, max(0, n // 2 - 1000), max(0, n - 2000)}):
            part = ctx.opacity_interp(1, 1, *[p[i:i + 2000].contiguous() for p in pts], mixed=mixed)
            assert torch.equal(part, whole[i:i + 2000])
    ctx.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n", [1000, 700001])
def test_first_call_under_capture(n, mixed):
    """A context's first interpolation, recorded in a graph, gives the eager call's bits (either batch size's kernel)."""
    edges, g, tables, _ = make_case(10, 3.0, 2, 2, "profile", 1)
    ctx = nmc.Context(edges, 2, 2, tables)
    pts = [p.contiguous() for p in _points(np.random.default_rng(7), g, n)]
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.opacity_interp(0, 1, *pts, out=out, mixed=mixed)
    graph.replay()
    assert torch.equal(out, ctx.opacity_interp(0, 1, *pts, mixed=mixed))
    ctx.close()
