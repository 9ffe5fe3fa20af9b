"""How far a refined loss repeats (GPU).  The float32 moments are summed in the order in
which reductions arrive, so that two runs differ by float32 rounding averaged over the
plasma: 6e-8 of a momentum, 32 slices, some 1e4 particles that the witness feels, 4e-9; a
few times that at most (5e-8).  Against the float64 form the rounding does not average
over the runs: 2e-7.

A step that a gradient is taken of sums in float64: what differs is the solves' last
iterates, 1e-12 of the fields, which turn one in 1e4 roundings of momenta the other way:
a hundredth of the above, 2e-10."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("checkpoints,spread", [(0, 5e-8), (32, 2e-10), (8, 2e-10)])
def test_refined_gain_repeats(qs, checkpoints, spread):
    def gains(form, runs):
        wl = W.Workload(name="g", n=128, half_width=6.0, n_xi=32, xi_len=4.0, ppc=4,
                        beams=(W.BeamSpec(amplitude=2.0, sigma_x=0.4, sigma_y=0.4, sigma_z=0.6,
                                          xi_c=1.5, n_particles=50000, seed=1),))
        wit = W.sample_beam(W.BeamSpec(amplitude=0.5, sigma_x=0.3, sigma_y=0.3, sigma_z=0.3,
                                       xi_c=3.2, n_particles=20000, seed=2))
        ctx = qs.Context(qs.config_from_workload(wl, precision=form, mg_tol=1e-12, refine_k=1,
                                                 checkpoint_every=checkpoints))
        ctx.init_plasma(wl.ppc)
        out = []
        for _ in range(runs):
            beams = [qs.Beam(W.sample_beam(wl.beams[0])), qs.Beam(wit)]
            ctx.step3d(beams)
            out.append(ctx.beam_gain(beams[1], 10.0))
        ctx.close()
        return torch.tensor(out, dtype=torch.float64)

    refined, exact = gains("fp32r", 6), gains("fp64", 1)
    size = float(exact.abs()[0])
    assert float(refined.max() - refined.min()) <= spread * size
    assert float((refined - exact[0]).abs().max()) <= 2e-7 * size
