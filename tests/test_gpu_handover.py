"""Solves that the iterations leave to the V-cycles (GPU): the cap on a solve's
iterations is below what they need, so that the staged cycles finish every
slice, and the next slice's iterations start after them.

Tolerances: those of the other parity tests (float64 1e-9, refined 2e-5)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "fp32r": 2e-5}


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
@pytest.mark.parametrize("n", [32, 64])
def test_cycles_finish_capped_iterations(qs, form, n):
    wl = W.Workload(name="h", n=n, half_width=3.0, n_xi=12, xi_len=2.4, ppc=4,
                    beams=(W.BeamSpec(amplitude=1.5, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                      xi_c=1.0, n_particles=3000, seed=n, x_c=0.3),))
    beams = [W.sample_beam(b) for b in wl.beams]
    pl, n_ion = O.plasma_from_workload(wl)
    ref = O.step3d(O.config_from_workload(wl), pl, n_ion, beams)
    counts = {}
    for cap in (4, 60):
        ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-10,
                                                 mg_max_vcycles=cap))
        ctx.init_plasma(wl.ppc)
        st = ctx.step3d([qs.Beam(b) for b in beams], schedule=list(ref.m))
        got = ctx.fields(qs.FIELD_ALL, device=False).numpy()
        ctx.close()
        counts[cap] = st["vcycles"][2]
        scale = np.linalg.norm(ref.history[0])
        for i in range(5):
            err = np.linalg.norm(got[i] - ref.history[i])
            assert err < TOL[form] * max(np.linalg.norm(ref.history[i]), scale), (cap, i)
    # at most four iterations a solve: more only with the cycles
    assert counts[4] > 4 * ref.slices
    # a cycle takes off about as much as an iteration: what the cap cuts off a
    # solve comes back as a cycle or two, not as another full set of them
    assert counts[4] <= counts[60] + 2 * ref.slices


def test_nonuniform_counts_the_iterations_too(qs):
    import torch
    x = np.linspace(-3.0, 3.0, 33)
    j = torch.randn((31, 31), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2))
    s = qs.NonuniformSolver(x, x, precision="fp32r")
    # below the rounding of the residual: the iterations stall, the cycles reach the cap
    _, cycles, relres = s.solve(j, tol=1e-18, max_cycles=9, raise_on_error=False)
    assert s.status == qs.QS_ERR_NOT_CONVERGED and relres[0] < 1e-12
    assert 9 < cycles <= 18  # the quarter of 36 iterations at most
