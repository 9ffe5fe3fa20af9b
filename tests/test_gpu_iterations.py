"""The envelope's and the nonuniform solver's iterations finish their solves by
themselves (GPU): a hand-over to the V-cycles gives the same fields, so that only the
count shows it.  A slice of the envelope needs 4 to 8 iterations at these sizes,
counted by fours (at most 3), a V-cycle solve 6 and more on top; a refined
nonuniform solve up to 20 (5), V-cycles 10 and more."""
import numpy as np
import pytest

from workloads.nonuniform import three_region_axis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 64, 256])
def test_envelope_iterations_converge(qs, n):
    import torch
    width, n_xi = 8.0, 4
    x = -width / 2 + (np.arange(n) + 0.5) * width / n
    X, Y = np.meshgrid(x, x)
    a0 = np.exp(-(X ** 2 + Y ** 2) / 4.0)[None] * np.ones((n_xi, 1, 1)) * (1.0 + 0.1j)
    chi = np.broadcast_to(1.0 - 0.5 * np.exp(-(X ** 2 + Y ** 2)), (n_xi, n, n))
    a = torch.tensor(a0, device="cuda")
    _, cycles, relres = qs.LaserEnvelope(n, width, n_xi, 5.0, 1.0, 0.2).advance(
        torch.tensor(np.ascontiguousarray(chi), device="cuda"), a, steps=2)
    assert relres <= 1e-10 and cycles <= 3 * 2 * n_xi


@pytest.mark.parametrize("n", [15, 127, 255])
def test_nonuniform_iterations_converge(qs, n):
    import torch
    x = three_region_axis(n, 12.5)
    X, Y = np.meshgrid(x[1:-1], x[1:-1])
    j = torch.tensor(np.exp(-((X - 0.3) ** 2 + Y ** 2) / 4), device="cuda")
    m = torch.tensor(-1.0 / (1.0 + 0.5 * np.exp(-X ** 2 - Y ** 2)), device="cuda")
    s = qs.NonuniformSolver(x, x, precision="fp32r")
    _, cycles, relres = s.solve(j, m=m)
    assert relres[0] <= 1e-10 and cycles <= 5


@pytest.mark.parametrize("kind", ["mirrored", "twin", "slanted", "two axes"])
def test_bases_of_other_axes(qs, kind):
    """The preconditioner's bases: of an axis that is its own mirror image (halved),
    with two fine regions whose eigenvalues agree to rounding, of one that is not, and
    of two different axes.  A basis that lacks a vector would leave GMRES stalled."""
    import torch
    n = 127
    t = np.linspace(-1.0, 1.0, n + 2)
    twin = t - 0.12 * np.sin(2 * np.pi * t) * np.abs(np.sin(np.pi * t))
    x = {"mirrored": t + 0.4 * t ** 3, "twin": twin, "slanted": t + 0.2 * t ** 2,
         "two axes": t + 0.4 * t ** 3}[kind]
    x, y = 6.0 * x, 6.0 * (t + 0.2 * t ** 2 if kind == "two axes" else x)
    X, Y = np.meshgrid(x[1:-1], y[1:-1])
    j = torch.tensor(np.exp(-((X - 0.3) ** 2 + Y ** 2)), device="cuda")
    u, cycles, relres = qs.NonuniformSolver(x, y, precision="fp32r").solve(j)
    ref, _, _ = qs.NonuniformSolver(x, y, precision="fp64").solve(j, tol=1e-11)
    assert relres[0] <= 1e-10 and cycles <= 6
    assert float((u - ref).norm()) <= 1e-9 * float(ref.norm())
