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


@pytest.mark.parametrize("scale,power", [(1e4, 3), (1e5, 6)])
def test_envelope_cycles_finish_stalled_iterations(qs, scale, power):
    """A susceptibility so rough that the iterations make 48 steps (the first) or
    stall in a round of 24 (the second): 12 and 6 cycles' worth, then V-cycles, for
    every slice, each of which starts afresh."""
    import torch
    from oracle import qs_laser as QL
    from oracle.qs_oracle import Grid
    n, n_xi, width = 64, 3, 8.0
    rng = np.random.default_rng(int(power))
    a0 = rng.standard_normal((n_xi, n, n)) + 1j * rng.standard_normal((n_xi, n, n))
    chi = scale * rng.uniform(0.0, 1.0, (n_xi, n, n)) ** power
    ref = QL.envelope_advance(Grid.square(n, width / 2), a0, chi, 5.0, 1.0, 0.2, 1)
    a = torch.tensor(a0, device="cuda")
    _, cycles, relres = qs.LaserEnvelope(n, width, n_xi, 5.0, 1.0, 0.2).advance(
        torch.tensor(chi, device="cuda"), a, tol=1e-12, max_cycles=60)
    assert relres <= 1e-12 and cycles >= 7 * n_xi
    assert np.linalg.norm(a.cpu().numpy() - ref) < 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale,power", [(1e4, 3), (1e5, 6)])
def test_nonuniform_cycles_finish_stalled_iterations(qs, scale, power):
    """The same for GMRES: rounds of 8, so at least 2 cycles' worth before it gives up;
    the float64 form's V-cycles are the reference."""
    import torch
    n = 63
    x = np.linspace(-4.0, 4.0, n + 2)
    rng = np.random.default_rng(int(power))
    j = torch.tensor(rng.standard_normal((2, n, n)), device="cuda")
    m = torch.tensor(-scale * rng.uniform(0.0, 1.0, (n, n)) ** power, device="cuda")
    ref, alone, _ = qs.NonuniformSolver(x, x, precision="fp64").solve(j, m=m, max_cycles=60)
    u, cycles, relres = qs.NonuniformSolver(x, x, precision="fp32r").solve(j, m=m, max_cycles=60)
    assert max(relres) <= 1e-10 and cycles > 2
    assert float((u - ref).norm()) <= 1e-8 * float(ref.norm())


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
@pytest.mark.parametrize("settings", [dict(tile_x=16, tile_y=8, coarse_block_n=16),
                                      dict(tile_x=32, tile_y=32, pre_sweeps=2, post_sweeps=1),
                                      dict(coarse_block_n=32), dict(omega_pct=100)])
def test_settings_of_the_cycles_that_finish(qs, form, settings):
    """The multigrid's settings, on a side that takes it only after capped iterations:
    staged tiles of other shapes, other sweeps, more levels in one block, no
    over-relaxation."""
    n = 64
    wl = W.Workload(name="h", n=n, half_width=3.0, n_xi=6, xi_len=1.2, ppc=4,
                    beams=(W.BeamSpec(amplitude=1.5, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                      xi_c=0.6, n_particles=3000, seed=n, x_c=0.3),))
    beams = [W.sample_beam(b) for b in wl.beams]
    pl, n_ion = O.plasma_from_workload(wl)
    ref = O.step3d(O.config_from_workload(wl), pl, n_ion, beams)
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-10, mg_max_vcycles=4,
                                             **settings))
    ctx.init_plasma(wl.ppc)
    st = ctx.step3d([qs.Beam(b) for b in beams], schedule=list(ref.m))
    got = ctx.fields(qs.FIELD_ALL, device=False).numpy()
    ctx.close()
    assert st["vcycles"][2] > 4 * ref.slices  # more than the iterations alone
    scale = np.linalg.norm(ref.history[0])
    for i in range(5):
        err = np.linalg.norm(got[i] - ref.history[i])
        assert err < TOL[form] * max(np.linalg.norm(ref.history[i]), scale), i


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
def test_warm_starts_of_clustered_cycles_agree(qs, form):
    """Clusters on request keep the V-cycles, whose initial guesses the warm-start order
    sets: the same fields from each, from fewer cycles the higher the order."""
    wl = W.Workload(name="w", n=64, half_width=3.0, n_xi=16, xi_len=1.6, ppc=4,
                    beams=(W.BeamSpec(amplitude=0.5, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                      xi_c=0.8, n_particles=3000, seed=1),))
    got, cycles = [], []
    for order in (0, 1, 2):
        ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-10, cluster_size=8,
                                                 warm_start_order=order))
        ctx.init_plasma(wl.ppc)
        st = ctx.step3d([qs.Beam(W.sample_beam(b)) for b in wl.beams])
        got.append(ctx.fields(qs.FIELD_ALL, device=False).numpy())
        cycles.append(st["vcycles"][0])
        ctx.close()
    assert cycles[0] > cycles[2] > 2 * 16  # V-cycles: a direct solve counts one a slice
    for g in got[1:]:
        assert np.linalg.norm(g - got[0]) < TOL[form] * np.linalg.norm(got[0])


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
def test_residuals_are_complete_before_the_cycles(qs, form):
    """Two iterations are four phases, fewer than the parts in which idle blocks form
    the residuals of psi, E_z and B_z at 256^2; their partial sums lie where the cycles
    that follow put their tiles.  A wrong sum would be reported as not converged."""
    wl = W.Workload(name="p", n=256, half_width=4.0, n_xi=4, xi_len=0.8, ppc=1,
                    beams=(W.BeamSpec(amplitude=1.0, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                      xi_c=0.3, n_particles=3000, seed=2),))
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-6, mg_max_vcycles=2))
    ctx.init_plasma(wl.ppc)
    st = ctx.step3d([qs.Beam(W.sample_beam(wl.beams[0]))])
    ctx.close()
    assert st["vcycles"][2] > 2 * st["slices"] and st["max_relres"] <= 1e-6
