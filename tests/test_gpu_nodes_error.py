"""Errors of the refined nonuniform solves at the default tolerance (GPU): a blowout
slice's sources with macroparticle noise, each group as the slice loop solves it, against
the float64 form solved to 1e-12 (its rounding at these sides is below that).  At most a
tenth of the tolerance 1e-10; the refined V-cycles leave 4e-13 to 1e-10 on such grids."""
import numpy as np
import pytest

from workloads.nonuniform import alternating_axis, bubble_sources, three_region_axis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n", [("three_region", 255), ("three_region", 127),
                                    ("alternating", 63), ("alternating", 31)])
def test_error_is_a_tenth_of_the_tolerance(qs, kind, n):
    import torch
    x = three_region_axis(n, 12.5) if kind == "three_region" else alternating_axis(n, 10.0)
    src = bubble_sources(x, x)
    rng = np.random.default_rng(n)
    edge = np.exp(-(np.hypot(*np.meshgrid(x[1:-1], x[1:-1])) / (0.7 * x[-1])) ** 8)
    s64, s32 = (qs.NonuniformSolver(x, x, precision=p) for p in ("fp64", "fp32r"))
    for names, screened in ((("psi",), False), (("ez", "bz"), False), (("bx", "by"), True)):
        j = torch.tensor(np.stack([src[k] + 0.01 * rng.standard_normal((n, n)) * edge
                                   for k in names]), device="cuda")
        m = torch.tensor(src["m"], device="cuda") if screened else None
        ref, _, _ = s64.solve(j, m=m, tol=1e-12, max_cycles=60)
        u, _, _ = s32.solve(j, m=m)
        for c, k in enumerate(names):
            assert float((u[c] - ref[c]).norm()) <= 1e-11 * float(ref[c].norm()), k
