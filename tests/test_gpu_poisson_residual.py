"""The residual that a step reports covers psi (GPU): psi of the window's last
slice against its source, n_* of the particles that the library returns (the last
slice does not push them) less the ions, at sides up to the largest that the
direct solves take.

The step's residual is the largest of any solve, so it is no smaller than psi's
to the rounding of two evaluations (the deposits differ by 1e-16 of n_*, here
below 1e-4 of the source's residual; 10 % allowed), and psi meets the bound that
every solve stops at: max(tol ||f||, 1e-13 ||u|| / h^2)."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle.qs_oracle import Grid, deposit, laplacian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,n,ppc", [("fp64", 64, 4), ("fp64", 512, 4), ("fp32r", 512, 4),
                                        ("fp32r", 640, 1), ("fp64", 2048, 1)])
def test_reported_residual_covers_psi(qs, form, n, ppc):
    hw = 4.0
    wl = W.Workload(name="p", n=n, half_width=hw, n_xi=2, xi_len=0.4, ppc=ppc,
                    beams=(W.BeamSpec(amplitude=2.0, sigma_x=0.8, sigma_y=0.6, sigma_z=0.6,
                                      xi_c=0.2, n_particles=20000, seed=n),))
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12, refine_k=1))
    ctx.init_plasma(ppc)
    start = ctx.plasma()
    st = ctx.step3d([qs.Beam(W.sample_beam(wl.beams[0]))])
    psi = ctx.fields(qs.FIELD_PSI, device=False).numpy().reshape(2, n, n)[1]
    end = ctx.plasma()
    ctx.close()
    g = Grid.square(n, hw)
    w = np.full(start["w"].shape, g.h ** 2 / ppc)
    f = (deposit(end["x"], end["y"], w, g) - deposit(start["x"], start["y"], w, g))
    r = np.linalg.norm(f - laplacian(psi, g.h))
    assert 0.9 * r / np.linalg.norm(f) <= st["max_relres"]
    assert r <= max(1e-12 * np.linalg.norm(f), 1e-13 * np.linalg.norm(psi) / g.h ** 2)
