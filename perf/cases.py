"""Performance cases: the work a user of this package has it do, through its public entry points.

Three groups: whole runs and their gradients on a handle (forward runs, field-level
inference, parameter gradients, batches), the single-kernel entry points that callers chain
themselves (sweeps, particle-mesh force, spectra), and the learned closure (inside a run, and
its training gradient). Sizes and parameters are those of the benchmark, the tests and the
default parameter block, with odd and non-power-of-two grids among them.

Losses and parameter derivatives leave the library as float64 device scalars built from
float32 partial sums; `run` hands them on as the float32 values an optimiser steps with.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2502_02294_gb300 as dh

GAMMA = 5.0 / 3.0
# the benchmark's subgrid settings
SUBGRID = dict(subgrid_on=1, delta_c=100.0, Pi0=0.05, E0=0.03, T_c=3.0e4, w_delta=5.0,
               w_T=1500.0, T0_uv=1.0e4, gamma_uv=1.4)
# sweep forms the autotuner picks on this GPU for grids of 48 cells and more, pinned so that
# every run of a case does the same arithmetic
TUNED = ([1, 5, 5], [4, 4, 4])
NORM = ([0.15, 0.0, 0.0, 0.0, 5e-4], [0.05, 0.01, 0.01, 0.01, 5e-4],
        [1e-4, 1e-5, 1e-5, 1e-5, 1e-7])
LAYERS = ((5, 16), (16, 16), (16, 16), (16, 5))


def listed():
    return [
        # the default parameter block's grid and schedule, replayed as a graph: a small run
        # inside a loop over seeds, where launches and latency count
        dict(name="run_32", kind="run", n=32, steps=20, subgrid=True, graphs=True, tuned=False,
             closure=False, batch=1),
        # one step and its reverse pass on an odd grid, called one by one (a custom loop)
        dict(name="step_grad_45", kind="step_grad", n=45),
        # gradient of a density loss to the noise and the parameters on the P(k) inference
        # grid: the plain calls run / loss_density / run_adjoint without graphs
        dict(name="grad_64", kind="grad", n=64, steps=20, batch=1, graphs=False, stars=True),
        # field-level inference, the headline workload: posterior and gradient at 128^3
        dict(name="posterior_128", kind="posterior", n=128, steps=100, observable=0),
        # large forward run (state beyond L2), built-in sweep forms
        dict(name="run_256", kind="run", n=256, steps=10, subgrid=True, graphs=True, tuned=False,
             closure=False, batch=1),
        # parameter sampling: a batch of instances with their own cosmology, forward and
        # parameter gradients
        dict(name="batch_grad_48", kind="grad", n=48, steps=20, batch=16, graphs=True,
             stars=False),
        # hydro alone (the blast-wave validation): three sweeps in Strang order
        dict(name="sweeps_128", kind="sweeps", n=128),
        # the three sweeps' adjoints, called directly (a user's own reverse pass)
        dict(name="sweep_adjoint_96", kind="sweep_adjoint", n=96),
        # particle-mesh force: deposit, Poisson, readout, and the force's adjoint
        dict(name="pm_force_128", kind="pm", n=128),
        # P(k) likelihood: spectrum, its adjoint, and the correlation coefficient
        dict(name="spectra_128", kind="spectra", n=128, nbins=64),
        # solver in the loop: a run with the learned closure after every step
        dict(name="closure_run_128", kind="run", n=128, steps=10, subgrid=False, graphs=True,
             tuned=True, closure=True, batch=1),
        # the closure's training gradient at the training set's grid and batch
        dict(name="closure_grad_64", kind="closure_grad", n=64, batch=2),
    ]


def _size(rng, lo, hi):
    """A grid size spread over the logarithm of [lo, hi], any parity."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "step_grad", "grad", "posterior", "sweeps", "sweep_adjoint", "pm",
                       "spectra", "closure_run", "closure_grad"])
    if kind == "run":
        return dict(kind="run", n=_size(rng, 16, 192), steps=rng.randint(3, 20),
                    subgrid=rng.random() < 0.7, graphs=rng.random() < 0.6,
                    tuned=rng.random() < 0.5, closure=False, batch=1)
    if kind == "step_grad":
        return dict(kind="step_grad", n=_size(rng, 16, 144))
    if kind == "grad":
        batch = rng.choice([1, 1, 2, 5, 16])
        return dict(kind="grad", n=_size(rng, 16, 96 if batch < 5 else 48),
                    steps=rng.randint(4, 16), batch=batch, graphs=rng.random() < 0.5,
                    stars=rng.random() < 0.5)
    if kind == "posterior":
        return dict(kind="posterior", n=_size(rng, 24, 128), steps=rng.randint(5, 30),
                    observable=rng.randint(0, 1))
    if kind in ("sweeps", "sweep_adjoint"):
        return dict(kind=kind, n=_size(rng, 16, 200))
    if kind == "pm":
        return dict(kind="pm", n=_size(rng, 16, 200))
    if kind == "spectra":
        n = _size(rng, 16, 200)
        return dict(kind="spectra", n=n, nbins=max(4, rng.randint(n // 4, n // 2)))
    if kind == "closure_run":
        return dict(kind="run", n=_size(rng, 24, 160), steps=rng.randint(2, 8), subgrid=False,
                    graphs=True, tuned=True, closure=True, batch=1)
    return dict(kind="closure_grad", n=_size(rng, 16, 96), batch=rng.randint(1, 3))


# ------------------------------------------------------------------------------ inputs
def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + what)


def _randn(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _smooth(x):
    for ax in (-3, -2, -1):
        x = (torch.roll(x, 1, ax) + 2 * x + torch.roll(x, -1, ax)) / 4
    return x


def _gas(n, gen, batch=0):
    """Gas state(s) [(batch,) 5, n, n, n]: density around the mean gas density with 30 %
    scatter, velocities of 5 km/s, positive pressure; smooth on a few cells, so that the
    limiter meets both smooth runs and extrema."""
    lead = (batch,) if batch else ()
    z = _smooth(_randn(lead + (5, n, n, n), gen))
    c = z.unbind(-4)
    rho = 0.16 * (1 + 0.3 * torch.tanh(c[0]))
    v = [0.05 * q for q in c[1:4]]
    P = 1e-4 * (1 + 0.5 * torch.tanh(c[4]))
    eps = P / (GAMMA - 1) + 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
    return torch.stack([rho] + [rho * q for q in v] + [eps], dim=-4).contiguous()


def _displacements(n, gen):
    """Particle displacements [3, n^3] in cells: a coherent flow (several cells, varying
    over a quarter of the box) with cell-scale scatter on top, as late in a run."""
    k = torch.fft.fftfreq(n, d=1.0 / n, device="cuda")
    kr = torch.fft.rfftfreq(n, d=1.0 / n, device="cuda")
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kr[None, None, :] ** 2
    s = torch.fft.irfftn(torch.fft.rfftn(_randn((3, n, n, n), gen), dim=(-3, -2, -1))
                         * torch.exp(-k2 / 16.0), s=(n, n, n), dim=(-3, -2, -1))
    s = 3.0 * s / s.std() + 0.3 * _randn((3, n, n, n), gen)
    return s.reshape(3, n ** 3).float().contiguous()


def _params(case, seed):
    n, steps = case["n"], case["steps"]
    kind = case["kind"]
    if kind == "run" and not case["closure"] and n <= 64:  # the default block's schedule
        p = dict(n=n, box=float(n), n_steps=steps, a_start=0.1, a_end=0.1 + 0.02 * steps)
    elif kind == "grad" and case["stars"]:  # the P(k) inference boxes: stars form at z > 3
        p = dict(n=n, box=n / 8.0, n_steps=steps, a_start=0.05, a_end=0.05 + 0.01 * steps,
                 ckpt_every=10, **dict(SUBGRID, delta_c=1.0))
    else:
        p = dict(n=n, box=float(n), n_steps=steps, a_start=0.05, a_end=0.05 + 0.0095 * steps,
                 ckpt_every=10)
    if kind != "run" or case["subgrid"]:
        for key, v in SUBGRID.items():
            p.setdefault(key, v)
    out = []
    for b in range(case.get("batch", 1)):
        q = dict(p, seed=1 + int(seed) % 1000 + b)
        if case.get("batch", 1) > 1:  # spread of the parameter study
            u = (b + 0.5) / case["batch"]
            q.update(omega_m=0.25 + 0.1 * u, sigma8=0.9 - 0.2 * u, Pi0=0.01 + 0.09 * u,
                     T0_uv=5e3 + 1.5e4 * u, delta_c=p["delta_c"] * (0.5 + 1.5 * u))
        out.append(dh.default_params(**q))
    return out


def _weights(seed):
    w = np.random.default_rng(int(seed)).standard_normal(sum(27 * i * o + o for i, o in LAYERS))
    return (0.05 * w).astype(np.float32)


def _field(n, gen, lead=()):
    """A positive density field around the mean gas density (the observed map)."""
    return (0.1633 * torch.exp(0.3 * _smooth(_randn(lead + (n, n, n), gen)))).contiguous()


def _sweep_inputs(case, seed):
    n = case["n"]
    u = _gas(n, _gen(seed, 1))
    lam = _randn((5, n, n, n), _gen(seed, 2))
    return u, lam


def _pm_inputs(case, seed):
    n = case["n"]
    return _displacements(n, _gen(seed, 1)), _smooth(_randn((3, n, n, n), _gen(seed, 2))).contiguous()


def _spectra_inputs(case, seed):
    n = case["n"]
    a = _field(n, _gen(seed, 1))
    b = (a + 0.03 * _randn((n, n, n), _gen(seed, 2))).contiguous()
    w = torch.randn(case["nbins"], generator=_gen(seed, 3), device="cuda", dtype=torch.float64)
    return a, b, w


def _closure_inputs(case, seed):
    n, B = case["n"], case["batch"]
    gas = _gas(n, _gen(seed, 1), batch=B)
    scale = torch.tensor(NORM[2], device="cuda")[:, None, None, None]
    target = (gas + scale * _smooth(_randn((B, 5, n, n, n), _gen(seed, 2)))).contiguous()
    return gas, target


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    st = dict(case=case, kind=kind, n=n)
    if kind in ("run", "grad", "posterior"):
        plist = _params(case, seed)
        B = len(plist)
        lead = (B,) if B > 1 else ()
        noise = _randn(lead + (n, n, n), _gen(seed, 1))
        sim = dh.Simulation(plist if B > 1 else plist[0], noise)
        if kind != "run" or case["tuned"]:
            sim.set_sweep_variants(*TUNED)
        if kind == "run" and case["closure"]:
            st["closure"] = dh.Closure(_weights(seed))
            st["closure"].set_norm(*NORM)
            sim.set_closure(st["closure"])
        if case.get("graphs", True):
            sim.set_graphs(True)
        st.update(sim=sim, noise=noise)
        if kind != "run":
            target = _field(n, _gen(seed, 2), lead)
            if case.get("observable", 0) == 1:  # an internal energy density map
                target = (target * 2e-3).contiguous()
            st.update(target=target, sigma=0.1 * float(target.std()), c=1.0 / n ** 3,
                      out=torch.empty(lead + (5, n, n, n), device="cuda"),
                      grad=torch.empty_like(noise),
                      loss=torch.empty(B, dtype=torch.float64, device="cuda"))
    elif kind == "step_grad":
        p = dh.default_params(n=n, box=float(n), n_steps=8, a_start=0.1, a_end=0.3, **SUBGRID)
        sim = dh.Simulation(p, _randn((n, n, n), _gen(seed, 1)))
        sim.set_sweep_variants(*TUNED)
        st.update(sim=sim, lam_gas=_randn((5, n, n, n), _gen(seed, 2)),
                  lam_part=_randn((6, n ** 3), _gen(seed, 3)))
    elif kind in ("sweeps", "sweep_adjoint"):
        st["u"], st["lam"] = _sweep_inputs(case, seed)
    elif kind == "pm":
        st["s"], st["lam"] = _pm_inputs(case, seed)
    elif kind == "spectra":
        st["a"], st["b"], st["w"] = _spectra_inputs(case, seed)
    else:
        st["gas"], st["target"] = _closure_inputs(case, seed)
        st["closure"] = dh.Closure(_weights(seed))
        st["closure"].set_norm(*NORM)
    return st


NU = 1.0       # dtau / dx of the direct sweeps: a Courant number near 0.2 for _gas
AXES = (0, 1, 2)


def run(st):
    kind, n = st["kind"], st["n"]
    if kind == "run":
        sim = st["sim"]
        sim.reset()
        sim.run()
        s = sim.state()
        return {k: s[k] for k in ("gas", "s", "p", "star")}
    if kind == "grad":
        sim = st["sim"]
        sim.reset()
        sim.run()
        dL, loss = sim.loss_density(st["target"], st["c"], out=st["out"], loss=st["loss"])
        dnoise, dpar = sim.run_adjoint(dL)
        return {"dnoise": dnoise, "dparams": dpar.float(), "loss": loss.float()}
    if kind == "posterior":
        loss, grad = st["sim"].posterior(st["noise"], st["target"], st["sigma"], grad=st["grad"],
                                         loss=st["loss"], observable=st["case"]["observable"])
        return {"loss": loss.float(), "grad": grad}
    if kind == "step_grad":
        sim = st["sim"]
        sim.reset()
        sim.step()
        lg, lp = st["lam_gas"].clone(), st["lam_part"].clone()
        dpar = torch.zeros(dh.NPARAMS, dtype=torch.float64, device="cuda")
        sim.step_adjoint(lg, lp, dpar)
        s = sim.state()
        return {"gas": s["gas"], "p": s["p"], "lam_gas": lg, "lam_part": lp,
                "dparams": dpar.float()}
    if kind == "sweeps":
        u = st["u"]
        for ax in AXES:
            u = dh.sweep(u, ax, NU, GAMMA)
        return u
    if kind == "sweep_adjoint":
        lam, dnu = st["lam"], []
        for ax in AXES:
            lam, d = dh.sweep_adjoint(st["u"], lam, ax, NU, GAMMA)
            dnu.append(d)
        return {"lam": lam, "dnu": torch.cat(dnu).float()}
    if kind == "pm":
        box = float(n)
        grid = dh.deposit_cic(st["s"], n, box)
        g = dh.gravity(grid, box, 1.5)
        gp = dh.interp_cic(g, st["s"], n, box)
        lam = dh.gravity_adjoint(st["lam"], box, 1.5)
        return {"grid": grid, "g": g, "gp": gp, "lam": lam}
    if kind == "spectra":
        box, nb = float(n), st["case"]["nbins"]
        k, pk, nm = dh.power_spectrum(st["a"], box, nb)
        da = dh.power_spectrum_adjoint(st["a"], box, nb, st["w"])
        _, rc, _ = dh.cross_correlation(st["a"], st["b"], box, nb)
        return {"k": k, "pk": pk, "nmodes": nm, "da": da, "rc": rc}
    loss, grad = st["closure"].gradient(st["gas"], st["target"])
    return {"loss": np.float32(loss), "grad": grad}


# ------------------------------------------------------------------------------- work
# Per cell (one particle per cell): state = 5 gas fields + 6 particle components.
STEP_BYTES = 88          # the state read and written once
STEP_FLOPS = 1650        # three sweeps, CIC, transforms, kicks, subgrid
CLOSURE_FLOPS = 2 * 27 * sum(i * o for i, o in LAYERS)


def work(case):
    kind, n3 = case["kind"], case["n"] ** 3
    B = case.get("batch", 1)
    if kind == "run":
        b, f = STEP_BYTES, STEP_FLOPS
        if case["closure"]:
            b, f = b + 40, f + CLOSURE_FLOPS
        return {"bytes": b * n3 * case["steps"] * B, "flops": f * n3 * case["steps"] * B}
    if kind in ("grad", "posterior"):
        # forward, then the reverse pass: the step's states read, their adjoints read and written
        return {"bytes": (STEP_BYTES + 44 + 88) * n3 * case["steps"] * B,
                "flops": 3 * STEP_FLOPS * n3 * case["steps"] * B}
    if kind == "step_grad":
        return {"bytes": (STEP_BYTES + 44 + 88) * n3, "flops": 3 * STEP_FLOPS * n3}
    if kind == "sweeps":
        return {"bytes": 3 * 40 * n3, "flops": 3 * 350 * n3}
    if kind == "sweep_adjoint":
        return {"bytes": 3 * 60 * n3, "flops": 3 * 1000 * n3}
    if kind == "pm":
        # deposit 16, force 16, readout 36, force adjoint 16; five transforms
        return {"bytes": 84 * n3, "flops": (150 + 8 * 2.5 * 3 * math.log2(case["n"])) * n3}
    if kind == "spectra":
        # a read, a read and da written, a and b read; five transforms
        return {"bytes": 20 * n3, "flops": (60 + 5 * 2.5 * 3 * math.log2(case["n"])) * n3}
    return {"bytes": 40 * n3 * B, "flops": 3 * CLOSURE_FLOPS * n3 * B}


# ------------------------------------------------------------------- values in 64 bits
def _split64(U, f):
    rho, eps = U[0], U[4]
    v = U[f] / rho
    P = (GAMMA - 1) * (eps - (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / (2 * rho))
    cs2 = GAMMA * P / rho
    pos = cs2 > 0
    c = v.abs() + torch.where(pos, torch.where(pos, cs2, torch.ones_like(cs2)).sqrt(), 0 * cs2)
    F = [U[f]] + [U[k] * v + (P if k == f else 0.0) for k in (1, 2, 3)] + [(eps + P) * v]
    F = torch.stack(F)
    return 0.5 * (c * U + F), 0.5 * (c * U - F)


def _limit64(a, b):
    ab, s = a * b, a + b
    num = torch.where(ab > 0, ab, torch.zeros_like(ab))
    return 2 * num / (s + torch.copysign(torch.full_like(s, 1e-30), s.detach()))


def _sweep64(U, axis, nu):
    dim = 3 - axis

    def nb(x, k):
        return torch.roll(x, -k, dim)

    R, L = _split64(U, 1 + axis)
    F = R - nb(L, 1)
    R, L = _split64(U - 0.5 * nu * (F - nb(F, -1)), 1 + axis)
    L1, L2 = nb(L, 1), nb(L, 2)
    F = R + _limit64(0.5 * (R - nb(R, -1)), 0.5 * (nb(R, 1) - R)) \
        - (L1 - _limit64(0.5 * (L1 - L), 0.5 * (L2 - L1)))
    return U - nu * (F - nb(F, -1))


def _modes(n):
    k = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    kr = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    return k[:, None, None], k[None, :, None], kr[None, None, :]


def _cic64(s, n, box):
    t = s.double() * (n / box)
    i = torch.arange(n ** 3, device="cuda")
    q = torch.stack([i % n, (i // n) % n, i // (n * n)])
    fl = torch.floor(t)
    base, f = q + fl.long(), t - fl
    for c in range(8):
        o = (c & 1, (c >> 1) & 1, (c >> 2) & 1)
        w = 1.0
        for j in range(3):
            w = w * (f[j] if o[j] else 1.0 - f[j])
        ix, iy, iz = ((base[j] + o[j]) % n for j in range(3))
        yield (iz * n + iy) * n + ix, w


def _grad_operator64(n, box):
    kz, ky, kx = _modes(n)
    k2 = kx ** 2 + ky ** 2 + kz ** 2
    inv = torch.where(k2 > 0, 1.0 / k2.clamp_min(1), torch.zeros_like(k2))
    kf = 2 * math.pi / box
    ks = []
    for k in (kx, ky, kz):  # gradient factors, zero at the Nyquist index
        ks.append(torch.where(k.abs() * 2 == n, torch.zeros_like(k), k) * inv / kf)
    return ks


def _pm64(case, seed):
    n, box = case["n"], float(case["n"])
    s, lam = _pm_inputs(case, seed)
    grid = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    for idx, w in _cic64(s, n, box):
        grid.index_add_(0, idx, w)
    dk = torch.fft.rfftn(grid.reshape(n, n, n))
    ks = _grad_operator64(n, box)
    g = torch.stack([torch.fft.irfftn(1j * k * 1.5 * dk, s=(n, n, n)) for k in ks])
    gp = torch.zeros(3, n ** 3, dtype=torch.float64, device="cuda")
    for idx, w in _cic64(s, n, box):
        gp += w * g.reshape(3, -1)[:, idx]
    yk = sum(-1j * k * 1.5 * torch.fft.rfftn(lam[j].double()) for j, k in enumerate(ks))
    return {"grid": grid.reshape(n, n, n), "g": g, "gp": gp,
            "lam": torch.fft.irfftn(yk, s=(n, n, n))}


def _spectra64(case, seed):
    n, nb = case["n"], case["nbins"]
    box = float(n)
    a, b, w = _spectra_inputs(case, seed)
    ak, bk = torch.fft.rfftn(a.double()), torch.fft.rfftn(b.double())
    kz, ky, kx = _modes(n)
    kk = (kx ** 2 + ky ** 2 + kz ** 2).sqrt()
    binno = torch.round(kk).long()
    wt = torch.where((kx == 0) | (kx * 2 == n), 1.0, 2.0) * torch.ones_like(kk)
    inside = (binno >= 1) & (binno <= nb)
    j = (binno[inside] - 1)

    def total(v):
        return torch.zeros(nb, dtype=torch.float64, device="cuda").index_add_(0, j, (wt * v)[inside])

    nm = total(torch.ones_like(kk))
    norm = box ** 3 / float(n) ** 6
    paa, pbb = total(ak.abs() ** 2), total(bk.abs() ** 2)
    pab = total(ak.real * bk.real + ak.imag * bk.imag)
    c = torch.zeros_like(kk)
    c[inside] = (2 * norm * w / nm)[j]
    da = torch.fft.irfftn(ak * c, s=(n, n, n)) * float(n) ** 3
    return {"k": 2 * math.pi / box * total(kk) / nm, "pk": norm * paa / nm, "nmodes": nm,
            "da": da, "rc": pab / (paa * pbb).sqrt()}


def _closure64(case, seed):
    """The training loss and its gradient of the network as defined (weights and activations
    rounded to bfloat16, the rounding taken as the identity in the derivative)."""
    gas, target = _closure_inputs(case, seed)
    mu, sigma, scale = (torch.tensor(v, device="cuda", dtype=torch.float32).double()[:, None, None, None]
                        for v in NORM)
    flat = torch.tensor(_weights(seed), device="cuda").double().requires_grad_(True)

    def q(x):
        return x + (x.detach().to(torch.bfloat16).double() - x.detach())

    h = q(((gas.double() - mu) / sigma).movedim(1, -1))  # [B, z, y, x, channel]
    o = 0
    for l, (ci, co) in enumerate(LAYERS):
        W = q(flat[o:o + 27 * ci * co].reshape(27, ci, co))
        o += 27 * ci * co
        z = flat[o:o + co]
        o += co
        for t in range(27):
            off = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
            z = z + torch.roll(h, tuple(-d for d in off), dims=(1, 2, 3)) @ W[t]
        h = q(0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))) if l < 3 else z
    t64 = ((target.double() - gas.double()) / scale).movedim(1, -1)
    loss = ((h - t64) ** 2).mean()
    (g,) = torch.autograd.grad(loss, flat)
    return {"loss": loss.detach(), "grad": g}


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "sweeps":
        u = _sweep_inputs(case, seed)[0].double()
        for ax in AXES:
            u = _sweep64(u, ax, NU)
        return u
    if kind == "sweep_adjoint":
        u, lam = (t.double() for t in _sweep_inputs(case, seed))
        dnu = []
        for ax in AXES:
            x = u.clone().requires_grad_(True)
            nu = torch.tensor(NU, dtype=torch.float64, device="cuda", requires_grad=True)
            lam, d = torch.autograd.grad(_sweep64(x, ax, nu), (x, nu), lam)
            dnu.append(d.reshape(1))
        return {"lam": lam, "dnu": torch.cat(dnu)}
    if kind == "pm":
        return _pm64(case, seed)
    if kind == "spectra":
        return _spectra64(case, seed)
    if kind == "closure_grad":
        return _closure64(case, seed)
    # whole steps and runs: hundreds of coupled kernels and random draws, no closed form
    return None
