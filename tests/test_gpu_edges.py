"""Sizes and places where the float-pair and direct-solve paths change (GPU).

Bunch pushes: macroparticles on and beside the walls, in the half cells along
them, at the ends of the window and outside of it, in a known wake (the
library's own stored slices, so that only the push is compared).  A push is
about a hundred operations in pairs of floats, 2^-47 relative each, on fields
that differ by up to the grid's contrast between neighbours: 1e-11 of the
largest change.

Nonuniform solves: the smallest and the largest side of the direct-solve
preconditioner and each number of rows a block can own (2, 4, 6, 6 with a second
turn on 152 SMs); the residual of the returned field against the float64
operator, which the solver must bring below tol, to the rounding of the two
evaluations (1e-12 of the source at these contrasts).

Envelope: sides with an odd factor of 7 and the smallest side of the direct
path, against the oracle's sparse LU at the bound of the other envelope tests.

Moments: particle counts that leave part of a warp idle."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import qs_laser as QL
from oracle.qs_oracle import Grid
from workloads.nonuniform import three_region_axis

pytestmark = pytest.mark.gpu


def _t(a, dtype=None):
    import torch
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype or torch.float64, device="cuda")


def _wake(n=16, n_xi=12, ppc=4):
    return W.Workload(name="e", n=n, half_width=3.0, n_xi=n_xi, xi_len=3.0, ppc=ppc,
                      beams=(W.BeamSpec(amplitude=1.0, sigma_x=0.6, sigma_y=0.6, sigma_z=0.5,
                                        xi_c=1.2, n_particles=3000, seed=5),))


@pytest.mark.parametrize("form", ["fp64", "fp32r"])
def test_push_at_walls_and_window_ends(qs, form):
    wl = _wake()
    ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12))
    ctx.init_plasma(wl.ppc)
    ctx.step3d([qs.Beam(W.sample_beam(b)) for b in wl.beams])
    hist = ctx.fields(qs.FIELD_ALL, device=False).numpy()
    hw, h, end = wl.half_width, 2 * wl.half_width / wl.n, wl.xi_len
    xs = [s * (hw - d) for s in (-1, 1) for d in (0.0, 1e-9, h / 4, h / 2, h)] + [0.0, 1.01 * hw]
    zs = [0.0, 1e-9, end / wl.n_xi / 2, end / 2, end * (1 - 1 / wl.n_xi), end - 1e-9, end,
          1.02 * end, -0.02 * end]
    X, Y, Z = (a.ravel() for a in np.meshgrid(xs, xs, zs))
    b = {k: np.resize(v, X.size).copy() if np.ndim(v) else v
         for k, v in W.sample_beam(wl.beams[0]).items()}
    b.update(x=X.copy(), y=Y.copy(), xi=Z.copy())
    beam = qs.Beam(b)
    ctx.push_beam([beam], 2.0)
    got = beam.numpy()
    ref = O.push_beam(O.config_from_workload(wl), hist, b, 2.0)
    ctx.close()
    for k in ("px", "py", "pz"):
        d = ref[k] - b[k]
        assert np.max(np.abs(got[k] - b[k] - d)) <= 1e-11 * np.max(np.abs(d)) + 1e-13 * np.max(
            np.abs(b[k])), k
    for k in ("x", "y", "xi"):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-12 * max(1.0, np.max(np.abs(ref[k]))), k


@pytest.mark.parametrize("n,nrhs", [(15, 1), (15, 4), (127, 3), (255, 3), (255, 4), (511, 1)])
@pytest.mark.parametrize("screened", [False, True])
def test_preconditioned_solve_meets_its_residual(qs, n, nrhs, screened):
    x = three_region_axis(n, 12.5)
    rng = np.random.default_rng(n + nrhs)
    X, Y = np.meshgrid(x[1:-1], x[1:-1])
    j = np.stack([np.exp(-((X - 0.3 * c) ** 2 + Y ** 2) / 4) * (1 + 0.1 * rng.standard_normal((n, n)))
                  for c in range(nrhs)])
    m = _t(-rng.uniform(0.0, 2.0, (n, n))) if screened else None
    s = qs.NonuniformSolver(x, x, correction=True, precision="fp32r")
    u, _, relres = s.solve(_t(j), m=m, tol=1e-10, max_cycles=60)
    assert max(relres) <= 1e-10
    for c in range(nrhs):
        f = s.source(_t(j[c])).cpu().numpy()
        r = f - s.apply(u[c].contiguous(), m).cpu().numpy()
        assert np.linalg.norm(r) <= (1e-10 + 1e-12) * np.linalg.norm(f), c


@pytest.mark.parametrize("n", [8, 28, 56])
def test_envelope_sides(qs, n):
    import torch
    width, n_xi = 8.0, 5
    rng = np.random.default_rng(n)
    x = -width / 2 + (np.arange(n) + 0.5) * width / n
    X, Y = np.meshgrid(x, x)
    a0 = (np.exp(-(X ** 2 + Y ** 2) / 4.0)[None]
          * (1.0 + 0.3j * rng.standard_normal((n_xi, n, n))))
    chi = rng.uniform(0.0, 2.0, (n_xi, n, n))
    ref = QL.envelope_advance(Grid.square(n, width / 2), a0, chi, 5.0, 1.0, 0.2, 2)
    a = _t(a0, torch.complex128)
    _, _, relres = qs.LaserEnvelope(n, width, n_xi, 5.0, 1.0, 0.2).advance(
        _t(chi), a, steps=2, tol=1e-13, max_cycles=60)
    assert relres <= 1e-13
    assert np.linalg.norm(a.cpu().numpy() - ref) < 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,ppc", [(4, 1), (6, 1), (10, 9)])
def test_moments_with_idle_lanes(qs, n, ppc):
    wl = _wake(n=n, n_xi=6, ppc=ppc)
    beams = [W.sample_beam(b) for b in wl.beams]
    cfg = O.config_from_workload(wl)
    pl, n_ion = O.plasma_from_workload(wl)
    ref = O.step3d(cfg, pl, n_ion, beams)
    ctx = qs.Context(qs.config_from_workload(wl, precision="fp32r", mg_tol=1e-12))
    ctx.init_plasma(wl.ppc)
    ctx.step3d([qs.Beam(b) for b in beams], schedule=list(ref.m))
    got = ctx.fields(qs.FIELD_ALL, device=False).numpy()
    ctx.close()
    scale = np.linalg.norm(ref.history[0])
    for i in range(5):
        err = np.linalg.norm(got[i] - ref.history[i])
        assert err < 2e-5 * max(np.linalg.norm(ref.history[i]), scale), i
