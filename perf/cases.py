"""The work that programs built on this library have it do, as measurable cases.

Kinds of case, each through the entry points that a user's program calls:

wake      one 3D step on the uniform grid (Context.step3d) and its fields: the
          quasi-static xi loop behind bi-Gaussian drivers, in both precisions,
          from 32^2 test problems to 512^2 channels
scan      many independent instances of uneven sizes in one batched call
          (parameter scans; step3d_batched)
grad      loss and gradient of the witness energy gain (forward and adjoint)
laser     the laser-driven 3D step: wake with |A|^2, then the envelope's step
envelope  the envelope advance alone with a given susceptibility
nodes     the five field solves of a slice on a nonuniform node grid
nodepic   the xi loop on the nonuniform node grid
push      the push of a driver bunch in the stored wake; with n_sub > 0 in the
          laser's own fields, sub-cycled

`exact` restates each of them in plain torch, float64, with direct solves (sine
transforms, block elimination) or solves iterated to rounding.
"""
import math

import torch

import paper_2012_00881_gb300 as qs

F64 = torch.float64
DEV = "cuda"


def listed():
    return [
        # a unit-test sized wake, the shortest complete step: launches and latency
        dict(name="wake32_fp64", kind="wake", n=32, half_width=4.0, n_xi=24, xi_len=6.0, ppc=4,
             form="fp64", channel=False, amplitude=0.5, sigma_r=0.6, sigma_z=0.8, beam_n=4000,
             witness_n=0),
        # the linear wake, the framework's correctness configuration, float64
        dict(name="wake64_fp64", kind="wake", n=64, half_width=6.0, n_xi=128, xi_len=12.0, ppc=4,
             form="fp64", channel=False, amplitude=0.3, sigma_r=0.5, sigma_z=1.0, beam_n=20000,
             witness_n=0),
        # the blowout with driver and witness, the headline configuration's grid
        # and bunches in its fast (refined) form, from the head into the bubble
        dict(name="wake256_fp32r", kind="wake", n=256, half_width=8.0, n_xi=160, xi_len=7.5,
             ppc=4, form="fp32r", channel=False, amplitude=5.0, sigma_r=0.3, sigma_z=0.7,
             beam_n=500000, witness_n=200000),
        # the same in float64, head of the window up to the driver's tail
        dict(name="wake256_fp64", kind="wake", n=256, half_width=8.0, n_xi=64, xi_len=3.0,
             ppc=4, form="fp64", channel=False, amplitude=5.0, sigma_r=0.3, sigma_z=0.7,
             beam_n=500000, witness_n=0),
        # the largest grid in use: a strong driver in a parabolic channel, nine
        # particles a cell, fine enough slices for the step rule to refine
        dict(name="channel512_fp32r", kind="wake", n=512, half_width=10.0, n_xi=80, xi_len=4.0,
             ppc=9, form="fp32r", channel=True, amplitude=10.0, sigma_r=1.0, sigma_z=1.21,
             beam_n=2000000, witness_n=0),
        # a parameter scan: instances of three sizes at once
        dict(name="scan12_fp32r", kind="scan", n=128, instances=12, n_xi=32, xi_len=2.0, ppc=4,
             form="fp32r", beam_n=100000),
        # driver and profile optimisation: one loss and gradient
        dict(name="grad256_fp32r", kind="grad", n=256, half_width=8.0, n_xi=64, xi_len=6.0, ppc=4,
             form="fp32r", amplitude=5.0, sigma_r=0.3, sigma_z=0.7, beam_n=500000,
             witness_n=200000, n_coef=16, dt=10.0),
        # a laser-driven step: wake and envelope
        dict(name="laser256_fp32r", kind="laser", n=256, half_width=12.0, n_xi=24, xi_len=5.0,
             ppc=4, form="fp32r", a0=2.0, w0=3.0, sigma_xi=2.0, xi_c=2.5, k0=20.0, dt=5.0),
        # the field solves of one slice on the three-region grid
        dict(name="nodes255_fp32r", kind="nodes", n=255, half_width=12.5, form="fp32r",
             axis="three_region"),
        # the slice loop on the node grid
        dict(name="nodepic127_fp32r", kind="nodepic", n=127, half_width=12.5, n_xi=24,
             xi_len=3.0, ppc=4, form="fp32r", axis="three_region", amplitude=3.0, sigma_r=0.5,
             sigma_z=0.7),
        # a whole driver bunch advanced in the wake
        dict(name="push500k", kind="push", n=256, half_width=8.0, n_xi=48, xi_len=4.5, ppc=4,
             form="fp64", amplitude=5.0, sigma_r=0.3, sigma_z=0.7, beam_n=500000, gamma=2000.0,
             dt=10.0, n_sub=0, a0=0.0, w0=3.0, sigma_xi=2.0, k0=20.0),
        # witness electrons in the laser's fields, sub-cycled
        dict(name="push200k_laser", kind="push", n=256, half_width=12.0, n_xi=48, xi_len=5.0,
             ppc=4, form="fp64", amplitude=0.5, sigma_r=0.5, sigma_z=0.7, beam_n=200000,
             gamma=20.0, dt=5.0, n_sub=50, a0=2.0, w0=3.0, sigma_xi=2.0, k0=20.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_side(rng, lo, hi):
    # every side the library takes coarsens by halves to at most 8
    sides = [b << k for b in (4, 5, 6, 7) for k in range(2, 8) if lo <= b << k <= hi]
    return rng.choice(sorted(sides))


def draw(rng):
    kind = rng.choice(["wake"] * 5 + ["scan", "grad", "laser", "envelope", "nodes", "nodepic",
                                      "push", "push"])
    form = rng.choice(["fp64", "fp32r"])
    if kind == "wake":
        n = _grid_side(rng, 32, 512)
        channel = rng.random() < 0.25
        top = 128 if n <= 128 else 64 if n <= 256 else 24
        n_xi = _log_int(rng, 12, top)
        h = 16.0 / n
        return dict(kind=kind, n=n, half_width=8.0, n_xi=n_xi,
                    xi_len=round(n_xi * h * rng.uniform(0.3, 0.8), 4), ppc=rng.choice([1, 4, 4, 9]),
                    form=form, channel=channel, amplitude=round(math.exp(rng.uniform(-1.5, 1.8)), 3),
                    sigma_r=round(rng.uniform(max(0.3, 3 * h), max(0.8, 5 * h)), 3),
                    sigma_z=round(rng.uniform(0.4, 1.0), 3), beam_n=_log_int(rng, 20000, 500000),
                    witness_n=0)
    if kind == "scan":
        return dict(kind=kind, n=_grid_side(rng, 32, 128), instances=rng.randint(2, 16),
                    n_xi=_log_int(rng, 8, 24), xi_len=round(rng.uniform(0.8, 2.0), 3), ppc=4,
                    form=form, beam_n=_log_int(rng, 20000, 100000))
    if kind == "grad":
        n = _grid_side(rng, 32, 160)
        return dict(kind=kind, n=n, half_width=6.0, n_xi=_log_int(rng, 12, 40), xi_len=6.0, ppc=4,
                    form=form, amplitude=round(rng.uniform(0.5, 2.0), 3), sigma_r=0.6,
                    sigma_z=round(rng.uniform(0.5, 0.8), 3), beam_n=_log_int(rng, 20000, 200000),
                    witness_n=20000, n_coef=rng.choice([1, 4, 16]), dt=round(rng.uniform(1, 10), 2))
    if kind in ("laser", "envelope"):
        n = _grid_side(rng, 32, 256)
        return dict(kind=kind, n=n, half_width=12.0, n_xi=_log_int(rng, 6, 24 if n > 128 else 48),
                    xi_len=round(rng.uniform(3.0, 5.0), 3), ppc=4, form=form,
                    a0=round(rng.uniform(0.5, 2.0), 3), w0=3.0, sigma_xi=2.0, xi_c=2.0,
                    k0=round(rng.uniform(10.0, 30.0), 2), dt=round(rng.uniform(1.0, 6.0), 2))
    if kind == "nodes":
        return dict(kind=kind, n=rng.choice([15, 31, 63, 127, 255]), form=form,
                    half_width=round(rng.uniform(8.0, 12.5), 2),
                    axis=rng.choice(["three_region", "uniform", "alternating"]))
    if kind == "nodepic":
        return dict(kind=kind, n=rng.choice([31, 63, 127]), half_width=round(rng.uniform(8, 12.5), 2),
                    n_xi=_log_int(rng, 8, 16), xi_len=1.5, ppc=rng.choice([1, 4]), form=form,
                    axis=rng.choice(["three_region", "uniform"]),
                    amplitude=round(rng.uniform(0.3, 2.0), 3), sigma_r=0.6, sigma_z=0.7)
    n = _grid_side(rng, 64, 256)
    sub = rng.choice([0, 0, _log_int(rng, 4, 50)])
    return dict(kind="push", n=n, half_width=12.0 if sub else 8.0, n_xi=32, xi_len=4.5, ppc=4,
                form="fp64", amplitude=round(rng.uniform(0.3, 2.0), 3), sigma_r=0.5, sigma_z=0.7,
                beam_n=_log_int(rng, 1000, 200000), gamma=round(rng.uniform(20.0, 2000.0), 1),
                dt=round(rng.uniform(2.0, 10.0), 2), n_sub=sub, a0=2.0 if sub else 0.0, w0=3.0,
                sigma_xi=2.0, k0=20.0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normals(seed, n):
    return torch.randn((3, n), dtype=F64, device=DEV, generator=_gen(seed))


def _uniforms(seed, k):
    g = torch.Generator()
    g.manual_seed(int(seed))
    return torch.rand(k, dtype=F64, generator=g).tolist()


def _bunch(seed, n, amplitude, sigma_r, sigma_z, xi_c, gamma=2000.0):
    """A cold bi-Gaussian electron bunch, n_b exp(-r^2/s_r^2 - (xi-xi_c)^2/s_z^2)."""
    z = _normals(seed, n)
    s2 = math.sqrt(2.0)
    total = amplitude * math.pi ** 1.5 * sigma_r * sigma_r * sigma_z
    zero = torch.zeros(n, dtype=F64, device=DEV)
    return dict(x=sigma_r / s2 * z[0], y=sigma_r / s2 * z[1], xi=xi_c + sigma_z / s2 * z[2],
                px=zero, py=zero.clone(), pz=zero + math.sqrt(gamma * gamma - 1.0),
                w=zero + total / n)


def _bunches(c, seed):
    """Driver three e-folding lengths behind the head; witness 4.5 behind it."""
    out = [_bunch(2 * seed, c["beam_n"], c["amplitude"], c["sigma_r"], c["sigma_z"],
                  3.0 * c["sigma_z"], c.get("gamma", 2000.0))]
    if c.get("witness_n"):
        out.append(_bunch(2 * seed + 1, c["witness_n"], 2.0, 0.3, 0.3, 3.0 * c["sigma_z"] + 4.5))
    return out


def _channel(half_width):
    r_max = half_width * math.sqrt(2.0)
    return [1.0 + 0.05 * (i * r_max / 256) ** 2 for i in range(257)], r_max


def _config(n, half_width, n_xi, xi_len, form, **more):
    return qs.default_config(nx=n, ny=n, x_min=-half_width, x_max=half_width, y_min=-half_width,
                             y_max=half_width, n_xi=n_xi, xi_min=0.0, xi_max=xi_len,
                             precision=qs.QS_FP64 if form == "fp64" else qs.QS_FP32_REFINED,
                             **more)


def _scan_instances(c):
    """(side, amplitude, sigma_r) of each instance: three sizes in turn, the
    driver's density and width rising through the scan."""
    k = c["instances"]
    sides = (c["n"], c["n"] * 3 // 2 if c["n"] % 2 == 0 and (c["n"] & (c["n"] - 1)) == 0 else c["n"],
             2 * c["n"])
    return [(sides[i % 3], 0.5 + 7.5 * i / max(1, k - 1), 0.5 + 0.3 * i / max(1, k - 1))
            for i in range(k)]


def _pulse(c, seed):
    """Envelope a0 exp(-r^2/w0^2 - (xi-xi_c)^2/s^2) with a weak phase front."""
    n, nx, hw = c["n"], c["n_xi"], c["half_width"]
    u = _uniforms(seed, 3)
    a0 = c["a0"] * (0.9 + 0.2 * u[0])
    x = -hw + (torch.arange(n, dtype=F64, device=DEV) + 0.5) * (2 * hw / n)
    xi = torch.arange(nx, dtype=F64, device=DEV) * (c["xi_len"] / nx)
    r2 = (x[None, :] - 0.1 * u[1]) ** 2 + x[:, None] ** 2
    env = torch.exp(-((xi - c.get("xi_c", 2.5)) / c["sigma_xi"]) ** 2)
    mag = a0 * env[:, None, None] * torch.exp(-r2 / c["w0"] ** 2)[None]
    return mag * torch.exp(1j * (0.05 + 0.05 * u[2]) * r2)[None]


def _susceptibility(c, seed):
    """chi of a synthetic blowout: a cavity with a compressed sheath."""
    n, nx, hw = c["n"], c["n_xi"], c["half_width"]
    rb0 = 3.0 + 2.0 * _uniforms(seed + 77, 1)[0]
    x = -hw + (torch.arange(n, dtype=F64, device=DEV) + 0.5) * (2 * hw / n)
    r = torch.sqrt(x[None, :] ** 2 + x[:, None] ** 2)[None]
    d = torch.arange(nx, dtype=F64, device=DEV) * (c["xi_len"] / nx) - c["xi_c"]
    rb = torch.sqrt(torch.clamp(rb0 ** 2 - (d - rb0) ** 2, min=0.0))[:, None, None]
    cavity = torch.sigmoid((r - rb) / 0.3)
    return (cavity * (1.0 + 2.0 * torch.exp(-((r - rb - 0.3) / 0.4) ** 2) * (rb > 0))).contiguous()


def _axis(c):
    """n + 2 node coordinates, walls included."""
    n, hw = c["n"], c["half_width"]
    if c["axis"] == "uniform":
        return torch.linspace(-hw, hw, n + 2, dtype=F64)
    if c["axis"] == "alternating":
        steps = torch.tensor([1.0, 2.0], dtype=F64).repeat((n + 1) // 2)
        x = torch.cat([torch.zeros(1, dtype=F64), torch.cumsum(steps, 0)])
        return x * (2 * hw / float(x[-1])) - hw
    # fine on the axis, coarser in the bubble, fine across its sheath, coarse outside
    m = 20001
    r = torch.linspace(0.0, hw, m, dtype=F64)
    kr = [0.0, 0.8, 1.3, 2.3, 2.8, 4.3, 4.8, 1e9]
    kh = [0.05, 0.05, 0.10, 0.10, 0.07, 0.07, 0.15, 0.15]
    s = torch.empty_like(r)
    for i in range(7):
        sel = (r >= kr[i]) & (r < kr[i + 1])
        s[sel] = kh[i] + (kh[i + 1] - kh[i]) * (r[sel] - kr[i]) / (kr[i + 1] - kr[i])
    inv = 1.0 / s
    q = torch.cat([torch.zeros(1, dtype=F64), torch.cumsum(0.5 * (inv[1:] + inv[:-1]) * (hw / (m - 1)), 0)])
    half = (n + 1) // 2
    t = torch.linspace(0.0, float(q[-1]), half + 1, dtype=F64)
    k = torch.clamp(torch.searchsorted(q, t), 1, m - 1)
    pos = r[k - 1] + (t - q[k - 1]) / (q[k] - q[k - 1]) * (r[k] - r[k - 1])
    pos[0], pos[-1] = 0.0, hw
    return torch.cat([-pos.flip(0), pos[1:]])


def _node_sources(c, seed):
    """Sources of one blowout slice on the nodes, with the noise of
    macroparticle deposits: psi, (E_z, B_z), (B_x, B_y) and M = -kappa."""
    xn = _axis(c).to(DEV)
    u = _uniforms(seed, 2)
    rad = 2.7 + 0.6 * u[0]
    x, y = xn[1:-1][None, :], xn[1:-1][:, None]
    r = torch.sqrt(x * x + y * y)
    noise = 0.01 * torch.randn((5,) + r.shape, dtype=F64, device=DEV, generator=_gen(seed))
    noise = noise * torch.exp(-(r / (0.7 * c["half_width"])) ** 8)
    ne = torch.sigmoid((r - rad) / 0.08) * (1.0 + (rad / math.sqrt(math.pi)) *
                                            torch.exp(-((r - rad - 0.15) / 0.25) ** 2))
    ring = torch.exp(-((r - rad) / 0.35) ** 2)
    well = 0.25 * rad * rad * torch.exp(-(r / rad) ** 4)
    psi = (ne - 1.0) * torch.exp(-(r / (2.2 * rad)) ** 8)
    j = torch.stack([psi, (r - rad) * ring, 0.1 * x * y * torch.exp(-r * r / 4.0), y * ring,
                     -x * ring]) + noise
    return j, (-ne / (1.0 + well)).contiguous()


def _node_driver(c, seed):
    """j_z of a bi-Gaussian driver at the nodes of every base slice."""
    xn = _axis(c).to(DEV)
    u = _uniforms(seed, 2)
    x, y = xn[1:-1][None, :] - 0.2 * u[0], xn[1:-1][:, None] - 0.2 * u[1]
    xi = torch.arange(c["n_xi"], dtype=F64, device=DEV) * (c["xi_len"] / c["n_xi"])
    prof = torch.exp(-((xi - 2.0 * c["sigma_z"]) / c["sigma_z"]) ** 2)
    return (c["amplitude"] * prof[:, None, None] *
            torch.exp(-(x * x + y * y) / c["sigma_r"] ** 2)[None]).contiguous()


def _grad_inputs(c, seed):
    u = _uniforms(seed, 4 + c["n_coef"])
    theta = [c["amplitude"], c["sigma_r"], c["sigma_r"], c["sigma_z"], 0.1 * u[0], 0.1 * u[1],
             3.0 * c["sigma_z"], 0.05 * u[2]]
    table = [1.0 + 0.1 * v for v in u[4:]]
    wit = _bunch(2 * seed + 1, c["witness_n"], 1.0, 0.3, 0.3, c["xi_len"] - 1.0)
    return theta, table, c["half_width"] * math.sqrt(2.0), _normals(2 * seed, c["beam_n"]), wit


# ---------------------------------------------------------------------------
# the library
# ---------------------------------------------------------------------------
def prepare(c, seed):
    k = c["kind"]
    if k in ("wake", "push"):
        # the wake that bunches are pushed in is an input: solved to rounding there
        ctx = qs.Context(_config(c["n"], c["half_width"], c["n_xi"], c["xi_len"], c["form"],
                                 mg_tol=1e-12 if k == "push" else 1e-10))
        if c.get("channel"):
            ctx.init_plasma(c["ppc"], *_channel(c["half_width"]))
        else:
            ctx.init_plasma(c["ppc"])
        beams = [qs.Beam(b) for b in _bunches(c, seed)]
        s = dict(case=c, ctx=ctx, beams=beams)
        if k == "push":
            if c["n_sub"]:
                s["env0"] = _pulse(c, seed).contiguous()
                s["env1"] = (s["env0"] * torch.exp(torch.tensor(0.02j, device=DEV))).contiguous()
                ctx.step3d_laser(beams, (s["env0"].abs() ** 2).contiguous())
            else:
                ctx.step3d(beams)
        return s
    if k == "scan":
        ctxs, beams = [], []
        for i, (n, amp, sr) in enumerate(_scan_instances(c)):
            ctx = qs.Context(_config(n, 8.0, c["n_xi"], c["xi_len"], c["form"]))
            ctx.init_plasma(c["ppc"])
            ctxs.append(ctx)
            beams.append([qs.Beam(_bunch(seed + 1000 * i, c["beam_n"], amp, sr, 0.5, 1.0))])
        return dict(case=c, ctxs=ctxs, beams=beams)
    if k == "grad":
        theta, table, r_max, z, wit = _grad_inputs(c, seed)
        ctx = qs.Context(_config(c["n"], c["half_width"], c["n_xi"], c["xi_len"], c["form"],
                                 mg_tol=1e-12, checkpoint_every=c["n_xi"]))
        return dict(case=c, ctx=ctx, theta=torch.tensor(theta, dtype=F64),
                    table=torch.tensor(table, dtype=F64), r_max=r_max, z=z, witness=qs.Beam(wit))
    if k == "laser":
        ctx = qs.Context(_config(c["n"], c["half_width"], c["n_xi"], c["xi_len"], c["form"]))
        ctx.init_plasma(c["ppc"])
        env = qs.LaserEnvelope(c["n"], 2 * c["half_width"], c["n_xi"], c["k0"], c["dt"],
                               c["xi_len"] / c["n_xi"])
        return dict(case=c, ctx=ctx, laser=env, a=_pulse(c, seed).contiguous())
    if k == "envelope":
        env = qs.LaserEnvelope(c["n"], 2 * c["half_width"], c["n_xi"], c["k0"], c["dt"],
                               c["xi_len"] / c["n_xi"])
        return dict(case=c, laser=env, a=_pulse(c, seed).contiguous(), chi=_susceptibility(c, seed))
    if k == "nodes":
        j, m = _node_sources(c, seed)
        ax = _axis(c).numpy()
        return dict(case=c, solver=qs.NonuniformSolver(ax, ax, precision=c["form"]),
                    j=[j[:1].contiguous(), j[1:3].contiguous(), j[3:].contiguous()], m=m)
    if k == "nodepic":
        ax = _axis(c).numpy()
        pic = qs.NonuniformPIC(ax, ax, c["n_xi"], c["xi_len"], precision=c["form"])
        pic.init_plasma(c["ppc"])
        return dict(case=c, pic=pic, jzb=_node_driver(c, seed))
    raise ValueError(k)


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "wake":
        st = s["ctx"].step3d(s["beams"])
        return dict(fields=s["ctx"].fields(), slices=st["slices"])
    if k == "scan":
        st = qs.step3d_batched(s["ctxs"], s["beams"])
        return dict(fields=[x.fields() for x in s["ctxs"]], slices=[t["slices"] for t in st])
    if k == "grad":
        theta = s["theta"].clone().requires_grad_(True)
        table = s["table"].clone().requires_grad_(True)
        gain = qs.witness_gain(s["ctx"], theta, table, s["z"], 2000.0, s["witness"], c["dt"],
                               c["ppc"], s["r_max"])
        gain.backward()
        return dict(gain=gain.detach(), theta=theta.grad, table=table.grad)
    if k == "laser":
        a = s["a"].clone()
        st = s["ctx"].laser_step3d(s["laser"], a)
        return dict(fields=s["ctx"].fields(), envelope=a, slices=st["slices"])
    if k == "envelope":
        return dict(envelope=s["laser"].advance(s["chi"], s["a"].clone())[0])
    if k == "nodes":
        so = s["solver"]
        return [so.solve(s["j"][0])[0], so.solve(s["j"][1])[0], so.solve(s["j"][2], m=s["m"])[0]]
    if k == "nodepic":
        hist, st = s["pic"].step3d(s["jzb"])
        return dict(fields=hist, slices=st["slices"])
    b = s["beams"][0]
    bunch = qs.Beam({key: b.t[key].clone() for key in qs.Beam.KEYS}, b.charge, b.q_over_m)
    if c["n_sub"]:
        s["ctx"].push_beam_dla([bunch], c["dt"], s["env0"], s["env1"], c["k0"], c["n_sub"])
    else:
        s["ctx"].push_beam([bunch], c["dt"])
    return {key: bunch.t[key] for key in ("x", "y", "xi", "px", "py", "pz")}


def work(c):
    """Inputs read once and outputs written once; the flops of the particle
    updates, the sources and one direct solve per field."""
    k = c["kind"]

    def loop(n, n_xi, ppc, particles):
        cells = n * n
        flops = n_xi * cells * (ppc * 300.0 + 150.0 + 5 * 20.0 * math.log2(n))
        return 8.0 * (5 * n_xi * cells + 5 * ppc * cells + 7 * particles), flops

    if k == "wake":
        b, f = loop(c["n"], c["n_xi"], c["ppc"], c["beam_n"] + c["witness_n"])
    elif k == "scan":
        parts = [loop(n, c["n_xi"], c["ppc"], c["beam_n"]) for n, _, _ in _scan_instances(c)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif k == "grad":
        b, f = loop(c["n"], c["n_xi"], c["ppc"], c["beam_n"] + c["witness_n"])
        b, f = 2 * b, 3 * f
    elif k in ("laser", "envelope"):
        cells = c["n"] ** 2 * c["n_xi"]
        b, f = loop(c["n"], c["n_xi"], c["ppc"], 0) if k == "laser" else (0.0, 0.0)
        b, f = b + 40.0 * cells, f + cells * 40.0 * math.log2(c["n"])
    elif k == "nodes":
        b, f = 8.0 * 11 * c["n"] ** 2, 5 * 40.0 * c["n"] ** 2 * math.log2(c["n"])
    elif k == "nodepic":
        b, f = loop(c["n"], c["n_xi"], c["ppc"], 0)
        b += 8.0 * c["n_xi"] * c["n"] ** 2
    else:
        near = min(c["n"] ** 2 * c["n_xi"], 8 * c["beam_n"])
        b = 8.0 * (13 * c["beam_n"] + 5 * near) + (32.0 * near if c["n_sub"] else 0.0)
        f = c["beam_n"] * max(1, c["n_sub"]) * (700.0 if c["n_sub"] else 300.0)
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------
# the same in plain torch, float64
# ---------------------------------------------------------------------------
class _Screened(torch.autograd.Function):
    """u with (lap - kappa) u = f for a stack of f; reverse mode by the same solve."""

    @staticmethod
    def forward(ctx, f, kappa, g):
        u = g._pcg(f, kappa)
        ctx.g = g
        ctx.save_for_backward(u, kappa)
        return u

    @staticmethod
    def backward(ctx, gu):
        u, kappa = ctx.saved_tensors
        mu = ctx.g._pcg(gu, kappa)
        return mu, (mu * u).sum(0), None


class _Cells:
    """Cell-centred square grid: CIC, differences, direct solves."""

    def __init__(self, n, half_width):
        self.n, self.lo, self.hi, self.h = n, -half_width, half_width, 2.0 * half_width / n
        k = torch.arange(1, n + 1, dtype=F64, device=DEV)
        i = torch.arange(n, dtype=F64, device=DEV) + 0.5
        s = torch.sin(math.pi * k[:, None] * i[None, :] / n) * math.sqrt(2.0 / n)
        s[-1] *= math.sqrt(0.5)
        self.S = s
        lam = -(2.0 - 2.0 * torch.cos(math.pi * k / n)) / (self.h * self.h)
        self.lam = lam[:, None] + lam[None, :]
        self.v0 = self.h

    def _axis(self, s):
        t = s - 0.5
        a = torch.floor(t.detach())
        f = t - a
        a = a.long()
        b = a + 1
        a = torch.where(a < 0, -1 - a, a).clamp(0, self.n - 1)
        b = torch.where(b > self.n - 1, 2 * self.n - 1 - b, b).clamp(0, self.n - 1)
        return (a, 1.0 - f), (b, f)

    def stencil(self, x, y):
        ax, ay = self._axis((x - self.lo) / self.h), self._axis((y - self.lo) / self.h)
        return [(iy * self.n + ix, wy * wx) for iy, wy in ay for ix, wx in ax]

    def deposit(self, st, q):
        out = torch.zeros(self.n * self.n, dtype=F64, device=DEV)
        for i, w in st:
            out = out.index_add(0, i, q * w)
        return (out / (self.h * self.h)).reshape(self.n, self.n)

    def gather(self, u, st):
        v = u.reshape(-1)
        return sum(v[i] * w for i, w in st)

    def _pad(self, u, ghost, dim):
        a, b = u.select(dim, 0).unsqueeze(dim), u.select(dim, -1).unsqueeze(dim)
        s = {"zero": 0.0, "odd": -1.0, "even": 1.0}[ghost]
        return torch.cat([s * a, u, s * b], dim)

    def ddx(self, u, ghost):
        p = self._pad(u, ghost, -1)
        return (p[..., 2:] - p[..., :-2]) / (2.0 * self.h)

    def ddy(self, u, ghost):
        p = self._pad(u, ghost, -2)
        return (p[..., 2:, :] - p[..., :-2, :]) / (2.0 * self.h)

    def lap(self, u):
        px, py = self._pad(u, "odd", -1), self._pad(u, "odd", -2)
        return (px[..., 2:] + px[..., :-2] + py[..., 2:, :] + py[..., :-2, :] - 4.0 * u) / self.h ** 2

    def _modes(self, f, d):
        s = self.S if not f.is_complex() else self.S.to(f.dtype)
        return s.T @ ((s @ f @ s.T) / d) @ s

    def poisson(self, f):
        return self._modes(f, self.lam)

    def _pcg(self, f, kappa):
        kb = 0.5 * (kappa.max() + kappa.min())
        d = self.lam - kb
        f2 = (f * f).sum((-2, -1), keepdim=True)
        u = self._modes(f, d)
        r = f - self.lap(u) + kappa * u
        z = self._modes(r, d)
        p, rz = z, (r * z).sum((-2, -1), keepdim=True)
        for it in range(120):
            ap = self.lap(p) - kappa * p
            den = (p * ap).sum((-2, -1), keepdim=True)
            al = torch.where(den == 0, 0.0, rz / torch.where(den == 0, 1.0, den))
            u = u + al * p
            r = r - al * ap
            if it % 4 == 3 and bool(((r * r).sum((-2, -1), keepdim=True) <= 1e-29 * f2).all()):
                break
            z = self._modes(r, d)
            new = (r * z).sum((-2, -1), keepdim=True)
            p = z + torch.where(rz == 0, 0.0, new / torch.where(rz == 0, 1.0, rz)) * p
            rz = new
        return u

    def screened(self, f, kappa):
        return _Screened.apply(f, kappa, self)

    def lattice(self, ppc):
        s = int(round(math.sqrt(ppc)))
        m = torch.arange(self.n * s, dtype=F64, device=DEV)
        x = self.lo + (torch.floor(m / s) + (m % s + 0.5) / s) * self.h
        X, Y = x[None, :].expand(len(x), -1).reshape(-1), x[:, None].expand(-1, len(x)).reshape(-1)
        return X.clone(), Y.clone(), torch.full_like(X, self.h * self.h / ppc)


class _Nodes:
    """Vertex-centred tensor grid: the corrected 9-point operator, block
    elimination along y."""

    def __init__(self, xn):
        xn = xn.to(DEV)
        self.xn, self.n = xn, len(xn) - 2
        self.lo, self.hi = float(xn[0]), float(xn[-1])
        hm, hp = xn[1:-1] - xn[:-2], xn[2:] - xn[1:-1]
        ha = hm + hp
        s = 2.0 / (hm * hp * ha)
        self.D2 = torch.diag(-s * ha) + torch.diag((s * hp)[1:], -1) + torch.diag((s * hm)[:-1], 1)
        a, b = hm / (ha * hp), hp / (ha * hm)
        self.D1 = torch.diag(b - a) + torch.diag(-b[1:], -1) + torch.diag(a[:-1], 1)
        self.c = (hp - hm) / 3.0
        self.B = torch.eye(self.n, dtype=F64, device=DEV) + self.c[:, None] * self.D1
        v = 0.5 * ha
        v[0] += 0.5 * hm[0]
        v[-1] += 0.5 * hp[-1]
        self.area = v[:, None] * v[None, :]
        self.v0 = float((xn[1:] - xn[:-1]).min())
        self._free = None

    def _axis(self, x):
        x = x.clamp(self.lo, self.hi)
        k = (torch.searchsorted(self.xn, x, right=True) - 1).clamp(0, self.n)
        f = (x - self.xn[k]) / (self.xn[k + 1] - self.xn[k])
        return ((k - 1).clamp(0, self.n - 1), 1.0 - f), (k.clamp(0, self.n - 1), f)

    def stencil(self, x, y):
        return [(iy * self.n + ix, wy * wx) for iy, wy in self._axis(y) for ix, wx in self._axis(x)]

    gather = _Cells.gather

    def deposit(self, st, q):
        out = torch.zeros(self.n * self.n, dtype=F64, device=DEV)
        for i, w in st:
            out = out.index_add(0, i, q * w)
        return out.reshape(self.n, self.n) / self.area

    def ddx(self, u, ghost):
        return u @ self.D1.T

    def ddy(self, u, ghost):
        return self.D1 @ u

    def _block(self, j, i, m):
        """Coefficients of row j of nodes on row i."""
        out = self.D2[j, i] * self.B + self.c[j] * self.D1[j, i] * self.D2
        if i == j:
            out = out + self.D2
        if m is not None:
            out = out + self.c[j] * self.D1[j, i] * torch.diag(m[i])
            if i == j:
                out = out + self.B * m[j][None, :]
        return out

    def _factor(self, m):
        inv = []
        for j in range(self.n):
            d = self._block(j, j, m)
            if j:
                d = d - self._block(j, j - 1, m) @ inv[-1] @ self._block(j - 1, j, m)
            inv.append(torch.linalg.inv(d))
        return inv

    def _apply(self, u, m):
        v = u @ self.D2.T
        w = v if m is None else v + m * u
        out = self.D2 @ u @ self.B.T + w + self.c[:, None] * (self.D1 @ w)
        return out if m is None else out + (m * u) @ (self.c[:, None] * self.D1).T

    def _sweep(self, f, inv, m):
        y = torch.empty_like(f)
        for j in range(self.n):
            t = f[:, j] if j == 0 else f[:, j] - y[:, j - 1] @ self._block(j, j - 1, m).T
            y[:, j] = t @ inv[j].T
        for j in range(self.n - 2, -1, -1):
            y[:, j] -= (y[:, j + 1] @ self._block(j, j + 1, m).T) @ inv[j].T
        return y

    def solve(self, f, m=None):
        f = f.reshape(-1, self.n, self.n)
        f = f + f @ (self.c[:, None] * self.D1).T + self.c[:, None] * (self.D1 @ f)
        if m is None:
            self._free = self._free or self._factor(None)
        inv = self._free if m is None else self._factor(m)
        u = self._sweep(f, inv, m)
        return u + self._sweep(f - self._apply(u, m), inv, m)

    def poisson(self, f):
        return self.solve(f).reshape(f.shape)

    def screened(self, f, kappa):
        return self.solve(f, -kappa)

    def lattice(self, ppc):
        s = int(round(math.sqrt(ppc)))
        off = (torch.arange(s, dtype=F64, device=DEV) + 0.5) / s
        d = self.xn[1:] - self.xn[:-1]
        x = (self.xn[:-1, None] + d[:, None] * off[None, :]).reshape(-1)
        w = d.repeat_interleave(s) / s
        X, Y = x[None, :].expand(len(x), -1).reshape(-1), x[:, None].expand(-1, len(x)).reshape(-1)
        return X.clone(), Y.clone(), (w[:, None] * w[None, :]).reshape(-1)


def _slice(g, p, n_ion, jzb, a2):
    """Fields of one slice from the particles; also grad psi and kappa."""
    x, y, px, py, w = p
    st = g.stencil(x, y)
    n_star = g.deposit(st, w)
    psi = g.poisson(n_star - n_ion)
    a = (1.0 + g.gather(psi, st)).clamp(min=1e-3)
    half_a2 = 0.0 if a2 is None else 0.5 * g.gather(a2, st)
    gam = (1.0 + px * px + py * py + a * a + half_a2) / (2.0 * a)
    vx, vy = px / a, py / a
    jx, jy, txx, txy, tyy, G = (g.deposit(st, w * q) for q in
                                (vx, vy, vx * vx, vx * vy, vy * vy, gam))
    ez = g.poisson(-(g.ddx(jx, "zero") + g.ddy(jy, "zero")))
    bz = g.poisson(g.ddx(jy, "zero") - g.ddy(jx, "zero"))
    ag = (1.0 + psi).clamp(min=1e-3)
    jz = G / ag - n_star + jzb
    kappa = n_star / ag
    gx, gy = g.ddx(psi, "odd"), g.ddy(psi, "odd")
    sx = (g.ddx(jz, "zero") - g.ddx(txx, "zero") - g.ddy(txy, "zero") - jy * bz / ag
          + G * gx / ag ** 2 - jx * ez / ag - (txx * gx + txy * gy) / ag)
    sy = (g.ddy(jz, "zero") - g.ddx(txy, "zero") - g.ddy(tyy, "zero") + jx * bz / ag
          + G * gy / ag ** 2 - jy * ez / ag - (txy * gx + tyy * gy) / ag)
    fx = fy = None
    if a2 is not None:
        fx, fy = g.ddx(0.25 * a2, "even"), g.ddy(0.25 * a2, "even")
        sx, sy = sx - n_star * fx / ag ** 2, sy - n_star * fy / ag ** 2
    b = g.screened(torch.stack([sy, -sx]), kappa)
    return st, half_a2, (psi, ez, bz, b[0], b[1]), (gx, gy, fx, fy), kappa


def _push(g, p, sl, dxi):
    x, y, px, py, w = p
    st, half_a2, (psi, _, bz_g, bx_g, by_g), (gx_g, gy_g, fx_g, fy_g), _ = sl
    a = (1.0 + g.gather(psi, st)).clamp(min=1e-3)
    gx, gy, bx, by, bz = (g.gather(u, st) for u in (gx_g, gy_g, bx_g, by_g, bz_g))
    fx = 0.0 if fx_g is None else g.gather(fx_g, st)
    fy = 0.0 if fy_g is None else g.gather(fy_g, st)
    d = 0.5 * dxi
    gam = (1.0 + px * px + py * py + a * a + half_a2) / (2.0 * a)
    qx, qy = px + d * ((gam * gx - fx) / a - by), py + d * ((gam * gy - fy) / a + bx)
    t = d * bz / a
    ux, uy = qx - t * qy, qy + t * qx
    s = 2.0 * t / (1.0 + t * t)
    qx, qy = qx - s * uy, qy + s * ux
    gam = (1.0 + qx * qx + qy * qy + a * a + half_a2) / (2.0 * a)
    px, py = qx + d * ((gam * gx - fx) / a - by), qy + d * ((gam * gy - fy) / a + bx)
    vmax = (torch.sqrt(px.detach() ** 2 + py.detach() ** 2) / a.detach()).max()
    x, y = x + dxi * px / a, y + dxi * py / a
    px = torch.where((x > g.hi) | (x < g.lo), -px, px)
    py = torch.where((y > g.hi) | (y < g.lo), -py, py)
    x = torch.where(x > g.hi, 2 * g.hi - x, torch.where(x < g.lo, 2 * g.lo - x, x))
    y = torch.where(y > g.hi, 2 * g.hi - y, torch.where(y < g.lo, 2 * g.lo - y, y))
    return (x, y, px, py, w), float(vmax)


def _loop(g, p, n_ion, jzb, dxi0, a2=None):
    """The xi loop; returns (history [5, n_xi, n, n], slices, kappa per slice)."""
    n_xi = jzb.shape[0]
    zero = torch.zeros((g.n, g.n), dtype=F64, device=DEV)
    hist, kap, m, slices = [], [], 1, 0
    for j in range(n_xi):
        vmax = 0.0
        for q in range(m):
            f = q / m
            mix = lambda v: v[j] if q == 0 else (1 - f) * v[j] + f * (v[j + 1] if j + 1 < n_xi else zero)  # noqa: E731
            sl = _slice(g, p, n_ion, mix(jzb), None if a2 is None else mix(a2))
            slices += 1
            if q == 0:
                hist.append(torch.stack(sl[2]))
                kap.append(sl[4])
            if j < n_xi - 1:
                p, vmax = _push(g, p, sl, dxi0 / m)
        v0 = g.v0 / dxi0
        m = 1 if vmax <= v0 else int(min(8, max(1, math.ceil(vmax / v0))))
    return torch.stack(hist, 1), slices, kap


def _driver_current(g, bunches, n_xi, dxi0):
    n = g.n
    out = torch.zeros(n_xi * n * n, dtype=F64, device=DEV)
    for b in bunches:
        q = b["w"] * b["pz"] / torch.sqrt(1.0 + b["px"] ** 2 + b["py"] ** 2 + b["pz"] ** 2)
        ok0 = (b["x"] >= g.lo) & (b["x"] <= g.hi) & (b["y"] >= g.lo) & (b["y"] <= g.hi)
        s = b["xi"] / dxi0
        j0 = torch.floor(s.detach())
        f = s - j0
        for jj, wj in ((j0.long(), 1.0 - f), (j0.long() + 1, f)):
            ok = ok0 & (jj >= 0) & (jj < n_xi)
            for i, w in g.stencil(b["x"], b["y"]):
                out = out.index_add(0, (jj * n * n + i)[ok], (q * wj * w)[ok])
    return (out / (g.h * g.h * dxi0)).reshape(n_xi, n, n)


def _table(r, table, r_max):
    m = len(table)
    if m == 1:
        return table[0] * torch.ones_like(r)
    s = (r / r_max * (m - 1)).clamp(max=float(m - 1))
    i = torch.floor(s).long().clamp(max=m - 2)
    f = s - i
    return table[i] * (1.0 - f) + table[i + 1] * f


def _plasma(g, ppc, table=None, r_max=1.0):
    x, y, w = g.lattice(ppc)
    if table is not None:
        w = w * _table(torch.sqrt(x * x + y * y), table, r_max)
    z = torch.zeros_like(x)
    return (x, y, z, z.clone(), w), g.deposit(g.stencil(x, y), w)


def _at_particles(g, grids, x, y, xi, dxi0):
    """Grids [n_xi, n, n] at particles: CIC in x, y; linear in xi; zero outside."""
    n_xi, nn = grids[0].shape[0], g.n * g.n
    ok0 = (x >= g.lo) & (x <= g.hi) & (y >= g.lo) & (y <= g.hi)
    s = xi / dxi0
    j0 = torch.floor(s)
    f = s - j0
    st = g.stencil(x.clamp(g.lo, g.hi), y.clamp(g.lo, g.hi))
    out = [0.0] * len(grids)
    for jj, wj in ((j0.long(), 1.0 - f), (j0.long() + 1, f)):
        ok = ok0 & (jj >= 0) & (jj < n_xi)
        base, wj = jj.clamp(0, n_xi - 1) * nn, torch.where(ok, wj, 0.0)
        for k, u in enumerate(grids):
            v = u.reshape(-1)
            out[k] = out[k] + wj * sum(v[base + i] * w for i, w in st)
    return out


def _boris(b, e, m, dt):
    d = -0.5 * dt
    u = torch.stack([b["px"], b["py"], b["pz"]]) + d * e
    t = d * m / torch.sqrt(1.0 + (u * u).sum(0))
    v = u + torch.linalg.cross(u, t, dim=0)
    u = u + torch.linalg.cross(v, t, dim=0) * (2.0 / (1.0 + (t * t).sum(0))) + d * e
    gam = torch.sqrt(1.0 + (u * u).sum(0))
    return dict(x=b["x"] + dt * u[0] / gam, y=b["y"] + dt * u[1] / gam,
                xi=b["xi"] + dt * (1.0 - u[2] / gam), px=u[0], py=u[1], pz=u[2])


def _wake_fields(g, hist, b, dxi0):
    grads = (g.ddx(hist[0], "odd"), g.ddy(hist[0], "odd"))
    ez, bz, bx, by, gx, gy = _at_particles(g, [hist[1], hist[2], hist[3], hist[4], *grads],
                                           b["x"], b["y"], b["xi"], dxi0)
    return torch.stack([-gx + by, -gy - bx, ez]), torch.stack([bx, by, bz])


def _push_bunch(g, hist, b, dt, dxi0, n_sub, env=None, k0=0.0):
    if not n_sub:
        return _boris(b, *_wake_fields(g, hist, b, dxi0), dt)
    grads = (g.ddx(hist[0], "odd"), g.ddy(hist[0], "odd"))
    pad = torch.zeros_like(env[0][:1])
    both = []
    for a in env:
        p = torch.cat([pad, a, pad])
        both += [a, (p[2:] - p[:-2]) / (2.0 * dxi0), g.ddx(a, "odd"), g.ddy(a, "odd")]
    grids = [hist[1], hist[2], hist[3], hist[4], *grads, *both]
    for s in range(n_sub):
        ez, bz, bx, by, gx, gy, *v = _at_particles(g, grids, b["x"], b["y"], b["xi"], dxi0)
        f = s / n_sub
        a, axi, ax, ay = ((1 - f) * v[i] + f * v[4 + i] for i in range(4))
        ph = torch.exp(-1j * k0 * b["xi"])
        exl = (-(((v[4] - v[0]) / dt + axi) - 1j * k0 * a) * ph).real
        byl = ((-axi + 1j * k0 * a) * ph).real
        e = torch.stack([-gx + by + exl, -gy - bx, ez + (-ax * ph).real])
        b = _boris(b, e, torch.stack([bx, by + byl, bz + (-ay * ph).real]), dt / n_sub)
    return b


def _envelope_step(g, a, chi, k0, dt, dxi):
    """Time-centred step of the envelope, slice by slice from the head."""
    q = 4.0 / (dt * dxi)
    c = 4.0j * k0 / dt - q
    new = torch.zeros_like(a)
    for j in range(a.shape[0]):
        f = (c + chi[j]) * a[j] - g.lap(a[j])
        if j:
            f = f - q * (new[j - 1] - a[j - 1])
        kb = 0.5 * (chi[j].max() + chi[j].min())
        d = g.lam - kb + c
        u = g._modes(f, d)
        for _ in range(80):
            r = f - g.lap(u) + (chi[j] - c) * u
            e = g._modes(r, d)
            u = u + e
            if float(e.abs().max()) <= 1e-15 * float(u.abs().max()):
                break
        new[j] = u
    return new


def exact(c, seed):
    k = c["kind"]
    if k in ("wake", "push"):
        g = _Cells(c["n"], c["half_width"])
        dxi0 = c["xi_len"] / c["n_xi"]
        bunches = _bunches(c, seed)
        table, r_max = _channel(c["half_width"]) if c.get("channel") else (None, 1.0)
        p, n_ion = _plasma(g, c["ppc"], None if table is None else torch.tensor(table, dtype=F64, device=DEV), r_max)
        env = _pulse(c, seed) if c.get("n_sub") else None
        jzb = _driver_current(g, bunches, c["n_xi"], dxi0)
        hist, slices, _ = _loop(g, p, n_ion, jzb, dxi0, None if env is None else env.abs() ** 2)
        if k == "wake":
            return dict(fields=hist, slices=slices)
        env1 = None if env is None else (env, env * torch.exp(torch.tensor(0.02j, device=DEV)))
        return _push_bunch(g, hist, bunches[0], c["dt"], dxi0, c["n_sub"], env1, c["k0"])
    if k == "scan":
        fields, slices = [], []
        for i, (n, amp, sr) in enumerate(_scan_instances(c)):
            g = _Cells(n, 8.0)
            p, n_ion = _plasma(g, c["ppc"])
            dxi0 = c["xi_len"] / c["n_xi"]
            b = _bunch(seed + 1000 * i, c["beam_n"], amp, sr, 0.5, 1.0)
            h, s, _ = _loop(g, p, n_ion, _driver_current(g, [b], c["n_xi"], dxi0), dxi0)
            fields.append(h)
            slices.append(s)
        return dict(fields=fields, slices=slices)
    if k == "grad":
        th, tb, r_max, z, wit = _grad_inputs(c, seed)
        theta = torch.tensor(th, dtype=F64, device=DEV, requires_grad=True)
        table = torch.tensor(tb, dtype=F64, device=DEV, requires_grad=True)
        g = _Cells(c["n"], c["half_width"])
        dxi0, nd, s2 = c["xi_len"] / c["n_xi"], z.shape[1], math.sqrt(2.0)
        xi = theta[6] + theta[3] / s2 * z[2]
        zero = torch.zeros(nd, dtype=F64, device=DEV)
        drv = dict(x=theta[4] + theta[7] * (xi - theta[6]) + theta[1] / s2 * z[0],
                   y=theta[5] + theta[2] / s2 * z[1], xi=xi, px=zero, py=zero,
                   pz=zero + math.sqrt(2000.0 ** 2 - 1.0),
                   w=zero + theta[0] * math.pi ** 1.5 * theta[1] * theta[2] * theta[3] / nd)
        p, n_ion = _plasma(g, c["ppc"], table, r_max)
        hist, _, _ = _loop(g, p, n_ion, _driver_current(g, [drv, wit], c["n_xi"], dxi0), dxi0)
        after = _boris(wit, *_wake_fields(g, hist, wit, dxi0), c["dt"])
        gamma = lambda b: torch.sqrt(1.0 + b["px"] ** 2 + b["py"] ** 2 + b["pz"] ** 2)  # noqa: E731
        gain = (gamma(after) - gamma(wit)).mean()
        dth, dtb = torch.autograd.grad(gain, (theta, table))
        return dict(gain=gain.detach().cpu(), theta=dth.cpu(), table=dtb.cpu())
    if k in ("laser", "envelope"):
        g = _Cells(c["n"], c["half_width"])
        dxi0, a = c["xi_len"] / c["n_xi"], _pulse(c, seed)
        if k == "envelope":
            return dict(envelope=_envelope_step(g, a, _susceptibility(c, seed), c["k0"], c["dt"], dxi0))
        p, n_ion = _plasma(g, c["ppc"])
        hist, slices, kap = _loop(g, p, n_ion, torch.zeros(a.shape, dtype=F64, device=DEV), dxi0,
                                  a.abs() ** 2)
        return dict(fields=hist, envelope=_envelope_step(g, a, kap, c["k0"], c["dt"], dxi0),
                    slices=slices)
    if k == "nodes":
        g = _Nodes(_axis(c))
        j, m = _node_sources(c, seed)
        return [g.solve(j[:1]), g.solve(j[1:3]), g.solve(j[3:], m)]
    g = _Nodes(_axis(c))
    p, n_ion = _plasma(g, c["ppc"])
    hist, slices, _ = _loop(g, p, n_ion, _node_driver(c, seed), c["xi_len"] / c["n_xi"])
    return dict(fields=hist, slices=slices)
