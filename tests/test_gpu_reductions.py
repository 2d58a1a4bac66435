"""Warp sums, species votes and integer comparisons of the solve kernels at the edges of their shapes.

The fused and O(v/c) kernels form their block and species sums by recursive halving and decide Algorithm 2 in FP32
where that is certain; the plain per-iteration mode keeps one sum per species, a square root and FP64 compares.  Both
are compared over species groups of 2, 4, 8, 16 and 32 lanes, groups padded to 32 (20 energies) and groups of two,
three and four warps (40, 64, 96 and 128 energies, constant and linear elements).

The iteration is stopped after a few inner and outer iterations at tol 1e-14, so that both modes take the same number
of steps from the same state and neither a vote near its threshold nor a state that cycles at its rounding floor
matters.  Tolerance 1e-8 in the W2 norm: the maps round differently by ~1e-14, and the least squares of a short window
amplifies that by at most the inverse of its pivot bound (1e-14 relative: unbounded in principle), in practice by
less than 1e5 over these steps.
"""
