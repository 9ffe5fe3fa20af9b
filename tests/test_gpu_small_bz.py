"""B_z of a weak driver (GPU, float64 form), orders of magnitude below E_z with which
it is solved: its residual against its own source, formed here from the particles
that the library returns at the window's last slice (which it does not push).

Bound: that of every solve, max(tol ||f||, 1e-13 ||u|| / h^2), and the rounding of
this file's source: f is a difference of j over h, j good to 8 roundings (four
corners, weights, velocity).  Sides: uneven halves, one line a block, and two."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle.qs_oracle import Grid, ddx, ddy, deposit, gather, laplacian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ppc", [(10, 4), (64, 4), (256, 4)])
def test_small_bz_meets_its_own_bound(qs, n, ppc):
    hw, n_xi, tol = 4.0, 4, 1e-13
    wl = W.Workload(name="z", n=n, half_width=hw, n_xi=n_xi, xi_len=0.8, ppc=ppc,
                    beams=(W.BeamSpec(amplitude=0.01, sigma_x=0.9, sigma_y=0.9, sigma_z=0.6,
                                      xi_c=0.4, n_particles=20000, seed=n),))
    ctx = qs.Context(qs.config_from_workload(wl, precision="fp64", mg_tol=tol, refine_k=1))
    ctx.init_plasma(ppc)
    ctx.step3d([qs.Beam(W.sample_beam(wl.beams[0]))])
    psi, ez, bz = (ctx.fields(f, device=False).numpy().reshape(n_xi, n, n)[-1]
                   for f in (qs.FIELD_PSI, qs.FIELD_EZ, qs.FIELD_BZ))
    pl = ctx.plasma()
    ctx.close()
    g = Grid.square(n, hw)
    a = 1.0 + gather(psi, pl["x"], pl["y"], g)
    jx = deposit(pl["x"], pl["y"], pl["w"] * pl["px"] / a, g)
    jy = deposit(pl["x"], pl["y"], pl["w"] * pl["py"] / a, g)
    rounding = 8 * 2.0 ** -53 * np.hypot(np.linalg.norm(jx), np.linalg.norm(jy)) / g.h
    for u, f in ((ez, -(ddx(jx, g.h, "zero") + ddy(jy, g.h, "zero"))),
                 (bz, ddx(jy, g.h, "zero") - ddy(jx, g.h, "zero"))):
        r = np.linalg.norm(f - laplacian(u, g.h))
        assert r <= max(tol * np.linalg.norm(f), 1e-13 * np.linalg.norm(u) / g.h ** 2) + rounding
    assert np.linalg.norm(bz) < 0.02 * np.linalg.norm(ez)
