"""Field solves by sine transforms over the grid sides that change their route
(GPU): even sides with every odd factor the library takes (1, 3, 5, 7), the
smallest side of the direct path, sides one below it that keep the multigrid
cycles, sides whose lines span several rounds of a block, and a team of one
block in the batched launch.  The oracle solves the same discrete equations
with a sparse LU.

Tolerances: float64 1e-9 and refined 2e-5 relative, the forms' bounds in the
other parity tests (solver tolerance 1e-12, float32 particle rounding)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "fp32r": 2e-5}


def _workload(n, n_xi=6):
    return W.Workload(name="d", n=n, half_width=3.0, n_xi=n_xi, xi_len=2.4, ppc=4,
                      beams=(W.BeamSpec(amplitude=1.5, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                        xi_c=1.0, n_particles=3000, seed=n, x_c=0.3),))


def _reference(wl):
    cfg = O.config_from_workload(wl)
    pl, n_ion = O.plasma_from_workload(wl)
    beams = [W.sample_beam(b) for b in wl.beams]
    return beams, O.step3d(cfg, pl, n_ion, beams)


def _check(got, ref, tol):
    scale = np.linalg.norm(ref[0])
    for i in range(5):
        err = np.linalg.norm(got[i] - ref[i]) / max(np.linalg.norm(ref[i]), scale)
        assert err < tol, (i, err)


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
@pytest.mark.parametrize("n", [4, 6, 7, 8, 10, 12, 14, 20, 28, 48, 80, 112])
def test_grid_sides(qs, form, n):
    wl = _workload(n)
    beams, ref = _reference(wl)
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12))
    ctx.init_plasma(wl.ppc)
    # the refined form's float32 rounding may move a step count at the rule's edge
    st = ctx.step3d([qs.Beam(b) for b in beams], schedule=list(ref.m))
    assert st["slices"] == ref.slices
    _check(ctx.fields(qs.FIELD_ALL, device=False).numpy(), ref.history, TOL[form])
    ctx.close()


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
def test_one_block_teams_of_uneven_sides(qs, form):
    sides = (8, 40, 56, 96)
    wls = [_workload(n) for n in sides]
    refs = [_reference(wl) for wl in wls]
    ctxs = []
    for wl in wls:
        ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12))
        ctx.init_plasma(wl.ppc)
        ctxs.append(ctx)
    qs.step3d_batched(ctxs, [[qs.Beam(b) for b in beams] for beams, _ in refs], team_blocks=1)
    for ctx, (_, ref) in zip(ctxs, refs):
        m, _, _ = ctx.slice_diagnostics()
        assert np.array_equal(m, ref.m)
        _check(ctx.fields(qs.FIELD_ALL, device=False).numpy(), ref.history, TOL[form])
        ctx.close()
