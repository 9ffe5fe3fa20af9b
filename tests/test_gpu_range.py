"""Sources at the ends of the number range and values that are not numbers (GPU).

The first slice is linear in the driver: a driver 2^k times as strong has 2^k
times the fields, to the solver's tolerance (1e-12 of the source, tens of times
that in the solution).  2^83 squares beyond float32's range; 2^116 is beyond what
the iterations hold, so that the V-cycles solve it (float64 form; the refined
form's own cycles are float32).  A source with a NaN has no solution: the call
says so."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _context(qs, form, n_xi=1, scale=1.0, cluster=0, n=32):
    wl = W.Workload(name="r", n=n, half_width=3.0, n_xi=n_xi, xi_len=1.0 * n_xi, ppc=4,
                    beams=(W.BeamSpec(amplitude=1.0, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                      xi_c=0.3, n_particles=3000, seed=3, x_c=0.3),))
    beam = W.sample_beam(wl.beams[0])
    beam["w"] = beam["w"] * scale
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12,
                                             cluster_size=cluster))
    ctx.init_plasma(wl.ppc)
    return ctx, qs.Beam(beam)


@pytest.mark.parametrize("form,k", [("fp64", 83), ("fp64", 116), ("fp32r", 83)])
def test_first_slice_is_linear_in_the_driver(qs, form, k):
    got = []
    for s in (1.0, 2.0 ** k):
        ctx, beam = _context(qs, form, scale=s)
        ctx.step3d([beam])
        got.append(ctx.fields(qs.FIELD_BX | qs.FIELD_BY, device=False).numpy() / s)
        ctx.close()
    assert np.linalg.norm(got[0]) > 0.0
    assert np.linalg.norm(got[1] - got[0]) < 1e-9 * np.linalg.norm(got[0])


@pytest.mark.parametrize("form,cluster", [("fp64", 0), ("fp32r", 0), ("fp64", 8), ("fp32r", 8)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_no_solution_is_reported(qs, form, cluster, bad):
    ctx, beam = _context(qs, form, n_xi=3, cluster=cluster)
    beam.t["w"][7] = bad
    with pytest.raises(qs.QsError) as e:
        ctx.step3d([beam])
    assert e.value.status == qs.QS_ERR_NOT_CONVERGED
    ctx.close()


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonuniform_solve_reports_no_solution(qs, form, bad):
    import torch
    x = np.linspace(-3.0, 3.0, 33)
    j = torch.zeros((2, 31, 31), dtype=torch.float64, device="cuda")
    j[0, 10, 12] = 1.0
    j[1, 10, 12] = bad
    s = qs.NonuniformSolver(x, x, precision=form)
    s.solve(j, max_cycles=20, raise_on_error=False)
    assert s.status == qs.QS_ERR_NOT_CONVERGED
    u, _, relres = s.solve(j[:1].contiguous(), max_cycles=40)  # the solver is fine after it
    assert relres[0] <= 1e-10 and bool(torch.isfinite(u).all())


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_envelope_reports_no_solution(qs, bad):
    import torch
    n, n_xi = 16, 3
    a = torch.ones((n_xi, n, n), dtype=torch.complex128, device="cuda")
    a[1, 3, 4] = bad
    chi = torch.zeros((n_xi, n, n), dtype=torch.float64, device="cuda")
    lz = qs.LaserEnvelope(n, 8.0, n_xi, 5.0, 1.0, 0.2)
    lz.advance(chi, a, raise_on_error=False)
    assert lz.status == qs.QS_ERR_NOT_CONVERGED


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
@pytest.mark.parametrize("k", [-300, -110, 120, 300])
def test_gradients_scale_with_the_cotangent(qs, form, k):
    import torch
    ctx, beam = _context(qs, form, n_xi=4)
    ctx.step3d([beam])
    g = torch.Generator(device="cuda").manual_seed(1)
    d = torch.randn((5, 4, 32, 32), dtype=torch.float64, device="cuda", generator=g)
    ref = ctx.step3d_adjoint(d)
    got = ctx.step3d_adjoint(d * 2.0 ** k)
    ctx.close()
    # two runs of one form: the order of the reductions, the solves' tolerance
    tol = 1e-9 if form == "fp64" else 1e-7
    for a, b in zip(got[:3], ref[:3]):
        assert float((a / 2.0 ** k - b).norm()) <= tol * float(b.norm()) and float(b.norm()) > 0


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
def test_nonuniform_residual_is_that_of_the_solution(qs, form):
    import torch
    from workloads.nonuniform import three_region_axis
    x = three_region_axis(255, 12.5)
    j = torch.randn((2, 255, 255), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2))
    s = qs.NonuniformSolver(x, x, precision=form)
    # below the rounding of the residual of a rounded solution, some 1e-14 here
    u, _, relres = s.solve(j, tol=1e-18, max_cycles=9, raise_on_error=False)
    assert s.status == qs.QS_ERR_NOT_CONVERGED
    for c in range(2):
        f = s.source(j[c].contiguous())
        r = float((f - s.apply(u[c].contiguous())).norm() / f.norm())
        # two evaluations of one residual at its rounding: within a factor
        assert r / 4 <= relres[c] <= 4 * r


def test_envelope_tolerance_below_rounding_is_not_met(qs):
    import torch
    n, n_xi = 32, 2
    a = torch.randn((n_xi, n, n), dtype=torch.complex128, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2))
    chi = torch.full((n_xi, n, n), 0.5, dtype=torch.float64, device="cuda")
    lz = qs.LaserEnvelope(n, 8.0, n_xi, 5.0, 1.0, 0.2)
    lz.advance(chi, a, tol=1e-19, max_cycles=9, raise_on_error=False)
    assert lz.status == qs.QS_ERR_NOT_CONVERGED
