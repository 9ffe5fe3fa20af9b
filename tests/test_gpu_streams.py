"""Contexts, envelopes and nonuniform solvers made and used on a stream that does not
wait for the default one (GPU): the same results as on the default stream, to the bound
of two runs (float64 solves to 1e-10, the order of the reductions)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _results(qs, stream):
    import torch
    with torch.cuda.stream(stream):
        wl = W.Workload(name="s", n=32, half_width=3.0, n_xi=6, xi_len=1.2, ppc=4,
                        beams=(W.BeamSpec(amplitude=1.0, sigma_x=0.7, sigma_y=0.5, sigma_z=0.6,
                                          xi_c=0.6, n_particles=2000, seed=4),))
        ctx = qs.Context(qs.config_from_workload(wl, precision="fp64"))
        ctx.init_plasma(wl.ppc)
        ctx.step3d([qs.Beam(W.sample_beam(wl.beams[0]))])
        fields = ctx.fields(qs.FIELD_ALL, device=False).numpy()
        ctx.close()
        n, n_xi = 24, 4
        a = torch.ones((n_xi, n, n), dtype=torch.complex128, device="cuda")
        chi = torch.full((n_xi, n, n), 0.7, dtype=torch.float64, device="cuda")
        qs.LaserEnvelope(n, 8.0, n_xi, 5.0, 1.0, 0.2).advance(chi, a, steps=2)
        x = np.linspace(-3.0, 3.0, 33)
        j = torch.ones((31, 31), dtype=torch.float64, device="cuda")
        u, _, _ = qs.NonuniformSolver(x, x, precision="fp32r").solve(j)
        stream.synchronize()
        return fields, a.cpu().numpy(), u.cpu().numpy()


def test_a_stream_of_its_own(qs):
    import torch
    ref = _results(qs, torch.cuda.default_stream())
    got = _results(qs, torch.cuda.Stream())
    for a, b in zip(got, ref):
        assert np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)
