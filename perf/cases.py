"""What a user of this framework has it do, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes what a user's program has
in hand (initial states made from a seed, solver handles), ``run`` makes one
pass through the public entry points, ``work`` counts what the path cannot do
without, and ``exact`` gives the same outputs in 64 bits from plain torch.

Keys of a case
  path    "step"   Solver.rk3_step with the CFL step (or a fixed one)
          "run"    Solver.run, `steps` steps in one call
          "batch"  Batch.step, `steps` steps of simulations of uneven sizes
          "vjp"    autograd.rk3_step and its vector-Jacobian product
          "grad"   autograd.rollout of `steps` steps, the density loss, backward
          "train"  learned_flux.Trainer.loss_and_grad
  flow    the initial state (_flow)
  nx, ny, nz, dtype, bc ("p" periodic, "o" open, "w" wall per axis), viscous,
  flux, recon, speeds, integrator: as in jf.Solver
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2203_13760_gb300 import autograd, jf, learned_flux

GAMMA, R_GAS, PR, CFL, EPS = 1.4, 1.0, 0.72, 0.5, 1e-6
HIDDEN = 32


def _case(name, path, flow, nx, ny=1, nz=1, dtype="f32", bc="ppp", viscous=False, flux="hllc", recon="weno5-js",
          speeds="einfeldt", integrator="rk3", **more):
    case = dict(path=path, flow=flow, nx=nx, ny=ny, nz=nz, dtype=dtype, bc=bc, viscous=viscous, flux=flux,
                recon=recon, speeds=speeds, integrator=integrator, **more)
    return dict(name=name, **case) if name else case


def listed():
    return [
        # the smallest call: one FP64 CFL step of the 200-cell Sod tube; latency and launches are all there is
        _case("tube200_f64", "step", "tube", 200, dtype="f64", bc="ooo"),
        # an ordinary 2D run: a viscous shear layer advanced by several CFL steps in one call
        _case("shear1024_f32", "run", "shear", 1024, 1024, viscous=True, steps=5),
        # a 3D grid of odd sizes with open ends in z
        _case("waves_odd_f32", "step", "waves", 107, 61, 45, bc="ppo", viscous=True),
        # the benchmark grid: viscous Taylor-Green vortex, FP32
        _case("vortex256_f32", "step", "vortex", 256, 256, 256, viscous=True),
        # the largest single grid of the benchmark: inviscid turbulence
        _case("turbulence384_f32", "step", "turbulence", 384, 384, 384),
        # the FP64 variant of the vortex, for runs held to round-off
        _case("vortex128_f64", "step", "vortex", 128, 128, 128, dtype="f64", viscous=True),
        # the ROE setup (characteristic flux splitting) on the vortex
        _case("vortex128_roe_f32", "step", "vortex", 128, 128, 128, viscous=True, flux="roe"),
        # many 2D Riemann problems of uneven sizes advanced together
        _case("quadrants64_f32", "batch", "quadrants", 512, bc="ooo", nsim=64, pick=2203, steps=5),
        # gradient of a loss at the end of a 2D trajectory, checkpoints every 20 steps
        _case("shear256_grad_f32", "grad", "shear", 256, 256, viscous=True, steps=24),
        # one differentiable 3D step, forward and backward
        _case("turbulence128_vjp_f32", "vjp", "turbulence", 128, 128, 128, viscous=True),
        # one training step of the learned flux: 20 windows of 15 steps on 32 x 32 cells
        _case("train32_f32", "train", "implosion", 32, 32, bc="wwo", flux="rusanov-nn", recon="weno3-js",
              integrator="rk2", nsim=20, steps=15),
        # its ground truth: the fine implosion in a walled box, FP64, one sample
        _case("implosion128_f64", "run", "implosion", 128, 128, dtype="f64", bc="wwo", recon="weno3-js",
              integrator="rk2", steps=4, dt=2.5e-4),
    ]


def _between(rng, lo, hi):
    """A size between lo and hi, even in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "shear", "waves", "vortex", "turbulence", "roe", "quadrants", "grad", "vjp", "train",
                       "implosion"])
    dtype = "f64" if rng.random() < 0.25 else "f32"
    small = dtype == "f64"  # FP64 cells cost some fifty times as much
    if kind == "tube":
        return _case("", "step", "tube", _between(rng, 50, 20000), dtype=dtype, bc="ooo")
    if kind == "shear":
        return _case("", "run", "shear", _between(rng, 64, 512 if small else 2048),
                     _between(rng, 64, 512 if small else 1024), dtype=dtype, viscous=True, steps=rng.randint(1, 6))
    if kind == "waves":
        flux, recon = rng.choice([("hllc", "weno5-js"), ("hllc", "weno5-js"), ("hll", "weno5-z"),
                                  ("rusanov", "weno5-js")])
        n = [_between(rng, 20, 110 if small else 160) for _ in range(3)]
        return _case("", "step", "waves", *n, dtype=dtype, bc=rng.choice(["ppp", "ppo", "poo", "ooo"]),
                     viscous=rng.random() < 0.7, flux=flux, recon=recon)
    if kind in ("vortex", "turbulence", "roe", "vjp"):
        n = _between(rng, 24, {"vortex": 288, "turbulence": 352, "roe": 160, "vjp": 144}[kind] if not small
                     else 48 if kind == "vjp" else 96)
        return _case("", "vjp" if kind == "vjp" else "step", "turbulence" if kind in ("turbulence", "vjp") else "vortex",
                     n, n, n, dtype=dtype, viscous=kind != "turbulence", flux="roe" if kind == "roe" else "hllc")
    if kind == "quadrants":
        return _case("", "batch", "quadrants", 128 if small else rng.choice([128, 256, 512]), dtype=dtype, bc="ooo",
                     nsim=rng.randint(3, 20 if small else 64), pick=rng.randint(1, 10**6), steps=rng.randint(1, 5))
    if kind == "grad":
        n = [_between(rng, *((48, 128) if small else (128, 320))) for _ in range(2)]
        return _case("", "grad", "shear", *n, dtype=dtype, viscous=rng.random() < 0.8,
                     steps=rng.randint(5, 10 if small else 24))
    if kind == "train":
        n = rng.choice([24, 32, 32, 40])
        return _case("", "train", "implosion", n, n, bc="wwo", flux="rusanov-nn", recon="weno3-js", integrator="rk2",
                     nsim=rng.randint(4, 24), steps=rng.randint(4, 16))
    n = _between(rng, 64, 256)
    return _case("", "run", "implosion", n, n, dtype=dtype, bc="wwo", recon="weno3-js", integrator="rk2",
                 steps=rng.randint(2, 8), dt=0.032 / n)


# ---------------------------------------------------------------------------
# inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _type(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _domain(case):
    """Edge lengths of the domain and the viscosity of the flow."""
    if case["flow"] in ("vortex", "turbulence"):
        return (2 * math.pi,) * 3, 1.0 / 1600.0
    return (1.0,) * 3, 1e-4 if case["flow"] == "shear" else 2e-3


def _axes(case):
    """The axes along which the case has more than one cell."""
    return [0, 1] if case["path"] == "batch" else [a for a, k in enumerate(("nx", "ny", "nz")) if case[k] > 1]


def _sides(case):
    """Grid sizes (nx, ny, nz) of every simulation of the case."""
    if case["path"] == "batch":  # squares of 64, 128, .. up to nx
        sides = [s for s in (64, 128, 256, 512) if s <= case["nx"]]
        pick = np.random.default_rng(case["pick"])
        return [(s, s, 1) for s in (sides[int(pick.integers(len(sides)))] for _ in range(case["nsim"]))]
    if case["path"] == "train":
        return [(case["nx"], case["ny"], 1)] * case["nsim"]
    return [(case["nx"], case["ny"], case["nz"])]


def _flow(flow, n, length, rng):
    """Conservative state (5, nz, ny, nx) in 64 bits; rng draws its parameters."""
    dev = _device()
    x, y, z = (((torch.arange(n[a], device=dev, dtype=torch.float64) + 0.5) * (length[a] / n[a]))
               .reshape([-1 if b == 2 - a else 1 for b in range(3)]) for a in range(3))
    u = v = w = torch.zeros(1, dtype=torch.float64, device=dev)
    if flow == "tube":  # a shock tube with states near Sod's
        left = x <= 0.5 + rng.uniform(-0.05, 0.05)
        rho = torch.where(left, rng.uniform(0.9, 1.1), rng.uniform(0.11, 0.14))
        p = torch.where(left, rng.uniform(0.9, 1.1), rng.uniform(0.09, 0.11))
    elif flow == "shear":  # a double shear layer with a perturbation of four modes
        a, phi = rng.uniform(0, 1, 4), rng.uniform(0, 2 * math.pi, 4)
        u = 0.5 * (torch.tanh((y - 0.25) / 0.05) - torch.tanh((y - 0.75) / 0.05) - 1.0)
        mode = sum(a[k] * torch.sin(2 * math.pi * (k + 1) * x + phi[k]) for k in range(4)) / a.sum()
        v = 1e-2 * mode * (torch.exp(-((y - 0.25) / 0.05) ** 2) + torch.exp(-((y - 0.75) / 0.05) ** 2))
        rho, p = 1.0 + 0.05 * mode * torch.cos(2 * math.pi * y), 2.5 + 0 * mode
    elif flow == "vortex":  # Taylor-Green at Mach 0.1, shifted and with an uneven amplitude
        s = rng.uniform(0, 2 * math.pi, 3)
        x, y, z = x + s[0], y + s[1], z + s[2]
        amp = rng.uniform(0.9, 1.1)
        p0 = 1.0 / (GAMMA * 0.01)
        u = amp * torch.sin(x) * torch.cos(y) * torch.cos(z)
        v = -amp * torch.cos(x) * torch.sin(y) * torch.cos(z)
        w = 0.05 * torch.sin(2 * x) * torch.sin(2 * y) * torch.ones_like(z)
        p = p0 + amp**2 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
        rho = p / p0
    elif flow == "turbulence":  # solenoidal modes |k| <= 5, rms Mach number 0.3
        vel = [0.0, 0.0, 0.0]
        for _ in range(12):
            k = rng.integers(-3, 4, 3).astype(float)
            k = k if k.any() else np.array([1.0, 2.0, 0.0])
            a = np.cross(rng.normal(size=3), k / np.linalg.norm(k))
            wave = torch.cos(k[0] * x + rng.uniform(0, 2 * math.pi) + k[1] * y + k[2] * z)
            vel = [vel[c] + float(a[c]) * wave for c in range(3)]
        rms = torch.sqrt(sum((c * c).mean() for c in vel))
        u, v, w = (0.3 * c / rms for c in vel)
        rho = torch.ones_like(u)
        p = rho / GAMMA
    elif flow == "quadrants":  # four constant states that meet in the middle
        states = np.stack([rng.uniform(0.1, 1.5, 4), rng.uniform(-1, 1, 4), rng.uniform(-1, 1, 4),
                           rng.uniform(0.1, 1.5, 4)])
        q = (x > 0.5).long() + 2 * (y > 0.5).long() + 0 * z.long()
        rho, u, v, p = (torch.as_tensor(s, device=dev)[q] for s in states)
    elif flow == "implosion":  # low pressure in a corner of a box, and a weak wave
        c, phi = rng.uniform(0.15, 0.5), rng.uniform(0, 2 * math.pi, 2)
        inner = (x + y <= c) & (z > -1)
        wave = torch.sin(2 * math.pi * x + phi[0]) * torch.sin(2 * math.pi * y + phi[1]) + 0 * z
        rho = torch.where(inner, 0.14, 1.0) * (1 + 0.05 * wave)
        p = torch.where(inner, 0.125, 1.0) * (1 + 0.07 * wave)
        u, v = 0.05 * torch.sin(math.pi * x) * torch.cos(math.pi * y), 0.05 * torch.sin(math.pi * y) + 0 * x
    else:  # "waves": every field a sum of a few modes
        field = []
        for _ in range(5):
            f = 0.0
            for _ in range(3):
                k, ph = rng.integers(1, 4, 3), rng.uniform(0, 2 * math.pi, 3)
                f = f + (torch.sin(2 * math.pi * float(k[0]) * x + ph[0]) * torch.cos(2 * math.pi * float(k[1]) * y + ph[1])
                         * torch.cos(2 * math.pi * float(k[2]) * z + ph[2]))
            field.append(f / 3)
        rho, p = 1 + 0.4 * field[0], 1 + 0.4 * field[4]
        u, v, w = (0.4 * f for f in field[1:4])
    E = p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w)
    shape = (n[2], n[1], n[0])
    return torch.stack([f.expand(shape) for f in (rho, rho * u, rho * v, rho * w, E)])


def _inputs(case, seed):
    """The tensors of the case in its own type: states, and what else the path takes."""
    rng = np.random.default_rng([seed, 7])
    length, _ = _domain(case)
    t = _type(case)
    got = {"U": [_flow(case["flow"], n, length, rng).to(t) for n in _sides(case)] if case["path"] != "train" else []}
    U = got["U"][0] if got["U"] else None
    if case["path"] == "vjp":
        gen = torch.Generator(device=_device()).manual_seed(int(seed))
        got["lam"] = torch.randn(U.shape, generator=gen, device=U.device, dtype=t)
    if case["path"] in ("vjp", "grad"):  # a fixed step near the CFL limit of a Mach number below 1
        fastest = 11.5 if case["flow"] == "vortex" else 2.5
        got["dt"] = 0.4 * min(length[a] / n for a, n in enumerate(_sides(case)[0]) if n > 1) / fastest
    if case["path"] == "grad":
        phi = rng.uniform(0, 2 * math.pi, 2)  # a target density away from the flow's
        x, y = (torch.linspace(0, 2 * math.pi, n + 1, device=U.device)[:n] for n in (case["nx"], case["ny"]))
        got["target"] = U[0] * (1 + 0.3 * torch.sin(x + phi[0]) * torch.cos(2 * y + phi[1]).reshape(-1, 1)).to(t)
    if case["path"] == "train":
        # a coarse reference run: an implosion whose fields drift from sample to sample
        n, samples = _sides(case)[0], 3 * case["steps"] + case["nsim"]
        a, b = (_flow("implosion", n, length, rng) for _ in range(2))
        s = torch.linspace(0, 1, samples, device=a.device, dtype=torch.float64).reshape(-1, 1, 1, 1, 1)
        got["cg"] = (a + 0.1 * s * (b - a)).to(t).contiguous()
        got["starts"] = [int(k) for k in rng.permutation(samples - case["steps"] - 1)[:case["nsim"]]]
        layers = [rng.normal(0, math.sqrt(2 / 4), (HIDDEN, 4)), rng.normal(0, 0.1, HIDDEN)]
        for _ in range(2):
            layers += [rng.normal(0, math.sqrt(2 / HIDDEN), (HIDDEN, HIDDEN)), rng.normal(0, 0.1, HIDDEN)]
        layers += [rng.normal(0, 0.1 / math.sqrt(HIDDEN), HIDDEN), np.array([math.log(2.0)])]
        got["theta"] = np.concatenate([a.ravel() for a in layers])
    return got


_BC = {"p": jf.PERIODIC, "o": jf.ZERO_GRADIENT, "w": jf.WALL}


def _options(case):
    _, mu = _domain(case)
    return dict(gamma=GAMMA, R=R_GAS, mu=mu if case["viscous"] else 0.0, Pr=PR, dtype=case["dtype"], eps=EPS, cfl=CFL,
                viscous=case["viscous"], heat=case["viscous"], flux=case["flux"], recon=case["recon"],
                speeds=case["speeds"], integrator=case["integrator"])


def prepare(case, seed):
    got = _inputs(case, seed)
    length, _ = _domain(case)
    bc = tuple(_BC[b] for b in case["bc"] for _ in range(2))
    state = dict(got, case=case)
    if case["path"] == "train":
        state["trainer"] = learned_flux.Trainer(got["cg"], got["theta"], batch=case["nsim"], unroll=case["steps"],
                                                dtype=case["dtype"])
    elif case["path"] == "batch":
        state["batch"] = jf.Batch([jf.make_grid(n, hi=length, bc=bc) for n in _sides(case)], **_options(case))
    else:
        s = state["solver"] = jf.Solver(_sides(case)[0], hi=length, bc=bc, **_options(case))
        state["dt"] = s.scalar(case.get("dt", got.get("dt", 0.0)))
        state["U"] = got["U"][0].contiguous()
    return state


def run(state):
    case, path = state["case"], state["case"]["path"]
    if path == "train":
        loss, grad = state["trainer"].loss_and_grad(state["starts"])
        return [loss, grad]
    if path == "batch":
        state["batch"].step(state["U"], case["steps"])
        return state["U"]
    s, U, dt = state["solver"], state["U"], state["dt"]
    if path == "step":
        used = s.scalar()
        s.rk3_step(U, None, used)
        return [U, used]
    if path == "run":
        return [s.run(U, case["steps"], dt if "dt" in case else None)]
    U = U.detach().requires_grad_(True)
    if path == "vjp":
        out = autograd.rk3_step(s, U, dt)
        return [out.detach(), torch.autograd.grad(out, U, state["lam"])[0]]
    out = autograd.rollout(s, U, case["steps"], dt, ckpt_every=20)
    loss = autograd.density_l2(s, out, state["target"])
    loss.backward()
    return [loss.detach(), U.grad]


# Operations of one right-hand side and stage combination per cell, each face
# once: (axes, viscous) -> HLLC with WENO5-JS; the ROE setup; WENO3-JS.
_OPS = {(1, False): 864, (1, True): 923, (2, False): 1694, (2, True): 1932, (3, False): 2524, (3, True): 3061}
_OPS_ROE = {(1, False): 1783, (1, True): 1842, (2, False): 3532, (2, True): 3770, (3, False): 5281, (3, True): 5818}


def work(case):
    size = 8 if case["dtype"] == "f64" else 4
    axes = len(_axes(case))
    cells = sum(a * b * c for a, b, c in _sides(case))
    ops = (_OPS_ROE if case["flux"] == "roe" else _OPS)[axes, bool(case["viscous"])]
    if case["recon"] == "weno3-js":
        ops = 754
    net = 2 * (4 * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN) * axes if case["flux"] == "rusanov-nn" else 0
    stages = case.get("steps", 1) * {"rk3": 3, "rk2": 2}[case["integrator"]]
    state = 5 * cells * size
    if case["path"] in ("step", "run", "batch"):
        return {"bytes": 2 * state, "flops": cells * stages * ops}
    if case["path"] == "train":  # forward, and twice that for the reverse of each product
        return {"bytes": state * 2 + state * case["steps"], "flops": 3 * cells * stages * (ops + net)}
    arrays = 4 if case["path"] == "vjp" else 2.2
    return {"bytes": arrays * state, "flops": 3 * cells * stages * ops}


# ---------------------------------------------------------------------------
# the same in 64 bits: the scheme written with plain torch operations


def _pad(U, bc, axes):
    """Three ghost cells on every active axis; a wall mirrors and turns the normal momentum."""
    for a in axes:
        n, dim = U.shape[3 - a], 3 - a
        i = torch.arange(-3, n + 3, device=U.device)
        if bc[a] == "p":
            U = U.index_select(dim, i % n)
        elif bc[a] == "o":
            U = U.index_select(dim, i.clamp(0, n - 1))
        else:
            U = U.index_select(dim, torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i)))
            turn = torch.ones(5, n + 6, device=U.device, dtype=U.dtype)
            turn[1 + a, :3] = turn[1 + a, -3:] = -1
            U = U * turn.reshape([5] + [n + 6 if d == dim else 1 for d in (1, 2, 3)])
    return U


def _weno(v, recon):
    """Left-biased value at the face between v[2] and v[3]; v holds the cells in order."""
    if recon == "weno3-js":
        a, b, c = v[1:4]
        q = (0.5 * (3 * b - a), 0.5 * (b + c))
        beta, d = ((b - a) ** 2, (c - b) ** 2), (1 / 3, 2 / 3)
    else:
        a, b, c, e, f = v[:5]
        q = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * e) / 6, (2 * c + 5 * e - f) / 6)
        beta = (13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2,
                13 / 12 * (b - 2 * c + e) ** 2 + 0.25 * (b - e) ** 2,
                13 / 12 * (c - 2 * e + f) ** 2 + 0.25 * (3 * c - 4 * e + f) ** 2)
        d = (0.1, 0.6, 0.3)
    if recon == "weno5-z":
        tau = (beta[0] - beta[2]).abs()
        alpha = [dk * (1 + tau / (EPS + bk)) for dk, bk in zip(d, beta)]
    else:
        alpha = [dk / (EPS + bk) ** 2 for dk, bk in zip(d, beta)]
    return sum(x * y for x, y in zip(alpha, q)) / sum(alpha)


def _sides_of(cells, recon):
    """Left and right values of every face from the six cells around it, a component at a time where they are large."""
    def both(c):
        return _weno(c, recon), _weno(c[::-1], recon)
    if cells[0].numel() < 1 << 24:
        return both(cells)
    parts = [both([c[m] for c in cells]) for m in range(cells[0].shape[0])]
    return torch.stack([p[0] for p in parts]), torch.stack([p[1] for p in parts])


def _flux_of(W, E, d):
    un = W[1 + d]
    F = [W[0] * un, W[0] * un * W[1], W[0] * un * W[2], W[0] * un * W[3], un * (E + W[4])]
    F[1 + d] = F[1 + d] + W[4]
    return F


def _energy(W):
    return W[4] / (GAMMA - 1) + 0.5 * W[0] * (W[1] ** 2 + W[2] ** 2 + W[3] ** 2)


def _conserved(W, E):
    return [W[0], W[0] * W[1], W[0] * W[2], W[0] * W[3], E]


def _riemann(WL, WR, d, flux, net):
    EL, ER = _energy(WL), _energy(WR)
    UL, UR, FL, FR = _conserved(WL, EL), _conserved(WR, ER), _flux_of(WL, EL, d), _flux_of(WR, ER, d)
    cL, cR = torch.sqrt(GAMMA * WL[4] / WL[0]), torch.sqrt(GAMMA * WR[4] / WR[0])
    uL, uR = WL[1 + d], WR[1 + d]
    if flux in ("rusanov", "rusanov-nn"):
        if flux == "rusanov":
            a = torch.maximum(uL.abs() + cL, uR.abs() + cR)
        else:
            sL, sR = ((torch.log(W[4]) - GAMMA * torch.log(W[0])) / (GAMMA - 1) for W in (WL, WR))
            h = torch.stack([(uR - uL).abs(), 0.5 * (uL + uR), 0.5 * (cL + cR), (sR - sL).abs()], dim=-1)
            for w, b in net[:-1]:
                h = torch.relu(h @ w.T + b)
            a = torch.exp(h @ net[-1][0] + net[-1][1])
        return [0.5 * (f + g) - 0.5 * a * (v - u) for f, g, u, v in zip(FL, FR, UL, UR)]
    # Einfeldt's speeds from Roe averages
    rL, rR = torch.sqrt(WL[0]), torch.sqrt(WR[0])
    mean = lambda a, b: (rL * a + rR * b) / (rL + rR)  # noqa: E731
    vel = [mean(WL[k], WR[k]) for k in (1, 2, 3)]
    H = mean((EL + WL[4]) / WL[0], (ER + WR[4]) / WR[0])
    c = torch.sqrt((GAMMA - 1) * (H - 0.5 * sum(q * q for q in vel)))
    SL, SR = torch.minimum(uL - cL, vel[d] - c), torch.maximum(uR + cR, vel[d] + c)
    if flux == "hll":
        return [torch.where(SL >= 0, f, torch.where(SR <= 0, g, (SR * f - SL * g + SL * SR * (v - u)) / (SR - SL)))
                for f, g, u, v in zip(FL, FR, UL, UR)]
    mL, mR = WL[0] * (SL - uL), WR[0] * (SR - uR)
    S = (WR[4] - WL[4] + mL * uL - mR * uR) / (mL - mR)

    def star(W, E, U, F, SK, m):
        k = m / (SK - S)
        V = [k, k * W[1], k * W[2], k * W[3], k * (E / W[0] + (S - W[1 + d]) * (S + W[4] / m))]
        V[1 + d] = k * S
        return [f + SK * (a - b) for f, a, b in zip(F, V, U)]
    left, right = star(WL, EL, UL, FL, SL, mL), star(WR, ER, UR, FR, SR, mR)
    return [torch.where(SL >= 0, f, torch.where(S >= 0, a, torch.where(SR > 0, b, g)))
            for f, a, b, g in zip(FL, left, right, FR)]


def _roe(cells, d):
    """Flux splitting in the characteristic fields of the Roe average of the two cells beside the face."""
    t1, t2 = (d + 1) % 3, (d + 2) % 3
    WL, WR = cells[2], cells[3]
    rL, rR = torch.sqrt(WL[0]), torch.sqrt(WR[0])
    mean = lambda a, b: (rL * a + rR * b) / (rL + rR)  # noqa: E731
    u = [mean(WL[k], WR[k]) for k in (1, 2, 3)]
    H = mean((_energy(WL) + WL[4]) / WL[0], (_energy(WR) + WR[4]) / WR[0])
    q2 = sum(a * a for a in u)
    c = torch.sqrt((GAMMA - 1) * (H - 0.5 * q2))
    b1 = (GAMMA - 1) / c**2
    b2 = 0.5 * b1 * q2

    def project(X):
        s = b2 * X[0] - b1 * (u[0] * X[1] + u[1] * X[2] + u[2] * X[3]) + b1 * X[4]
        e = (u[d] * X[0] - X[1 + d]) / c
        return [0.5 * (s + e), X[0] - s, X[1 + t1] - u[t1] * X[0], X[1 + t2] - u[t2] * X[0], 0.5 * (s - e)]
    lam = [(u[d] - c).abs(), u[d].abs(), u[d].abs(), u[d].abs(), (u[d] + c).abs()]
    up, down = [], []
    for W in cells:
        E = _energy(W)
        V, G = project(_conserved(W, E)), project(_flux_of(W, E, d))
        up.append([0.5 * (g + a * v) for g, a, v in zip(G, lam, V)])
        down.append([0.5 * (g - a * v) for g, a, v in zip(G, lam, V)])
    G = [_weno([s[k] for s in up], "weno5-js") + _weno([s[k] for s in down[::-1]], "weno5-js") for k in range(5)]
    S, D = G[0] + G[1] + G[4], G[4] - G[0]
    F = [S, u[0] * S, u[1] * S, u[2] * S, None]
    F[1 + d] = F[1 + d] + c * D
    F[1 + t1], F[1 + t2] = F[1 + t1] + G[2], F[1 + t2] + G[3]
    F[4] = H * (G[0] + G[4]) + u[d] * c * D + 0.5 * q2 * G[1] + u[t1] * G[2] + u[t2] * G[3]
    return F


def _viscous_flux(W, T, d, axes, n, h, mu, heat):
    """Dissipative flux of the faces normal to d from the padded velocities and temperature."""
    dim = lambda a: 2 - a  # noqa: E731

    def at(f, s, off=None, t=0):
        """f at the cell s of every face (0: the left one), t cells along the tangent off."""
        f = f.narrow(dim(d), 2 + s, n[d] + 1)
        for a in axes:
            if a != d:
                f = f.narrow(dim(a), 3 + (t if a == off else 0), n[a])
        return f
    face = lambda v: (-v[0] + 9 * v[1] + 9 * v[2] - v[3]) / 16  # noqa: E731

    def along(f, e):
        if e == d:
            v = [at(f, s) for s in (-1, 0, 1, 2)]
            return (v[0] - 27 * v[1] + 27 * v[2] - v[3]) / (24 * h[e])
        return face([(at(f, s, e, -2) - 8 * at(f, s, e, -1) + 8 * at(f, s, e, 1) - at(f, s, e, 2)) / (12 * h[e])
                     for s in (-1, 0, 1, 2)])
    grad = {(a, a): along(W[1 + a], a) for a in axes}
    div = sum(grad.values())
    tau, power = [None] * 3, 0.0
    for a in range(3):
        t = along(W[1 + a], d)
        if a in axes and a != d:
            t = t + along(W[1 + d], a)
        tau[a] = mu * t if a != d else mu * (2 * grad[d, d] - 2 / 3 * div)
        power = power + face([at(W[1 + a], s) for s in (-1, 0, 1, 2)]) * tau[a]
    return [0.0, *tau, power + heat * along(T, d)]


def _rhs(U, case, length, mu, net):
    n, axes = [U.shape[3], U.shape[2], U.shape[1]], _axes(case)
    h = [length[a] / n[a] for a in range(3)]
    U = _pad(U, case["bc"], axes)
    vel = [U[k] / U[0] for k in (1, 2, 3)]
    p = (GAMMA - 1) * (U[4] - 0.5 * U[0] * sum(q * q for q in vel))
    W = torch.stack([U[0], *vel, p])
    T = p / (U[0] * R_GAS)
    out = 0.0
    for d in axes:
        V = W
        for a in axes:
            if a != d:
                V = V.narrow(3 - a, 3, n[a])

        def faces(V, W, T, d=d):
            cells = [V.narrow(3 - d, j, n[d] + 1) for j in range(6)]
            F = _roe(cells, d) if case["flux"] == "roe" else _riemann(*_sides_of(cells, case["recon"]), d,
                                                                      case["flux"], net)
            if case["viscous"]:
                heat = mu * GAMMA * R_GAS / ((GAMMA - 1) * PR)
                F = [f - v for f, v in zip(F, _viscous_flux(W, T, d, axes, n, h, mu, heat))]
            F = torch.stack(F)
            return (F.narrow(3 - d, 0, n[d]) - F.narrow(3 - d, 1, n[d])) / h[d]
        if torch.is_grad_enabled():
            out = out + torch.utils.checkpoint.checkpoint(faces, V, W, T, use_reentrant=False)
        else:
            out = out + faces(V, W, T)
    return out


def _dt(U, case, length, mu):
    n, axes = [U.shape[3], U.shape[2], U.shape[1]], _axes(case)
    h = min(length[a] / n[a] for a in axes)
    vel = [U[k] / U[0] for k in (1, 2, 3)]
    c = torch.sqrt(GAMMA * (GAMMA - 1) * (U[4] - 0.5 * U[0] * sum(q * q for q in vel)) / U[0])
    dt = h / max(float((vel[a].abs() + c).max()) for a in axes)
    if case["viscous"]:
        cv = R_GAS / (GAMMA - 1)
        k = max(mu, mu * GAMMA * R_GAS / ((GAMMA - 1) * PR) / cv)
        dt = min(dt, 3 / 14 * h * h / (k / float(U[0].min())))
    return CFL * dt


def _advance(U, dt, case, net=None):
    length, mu = _domain(case)
    f = lambda V: V + dt * _rhs(V, case, length, mu, net)  # noqa: E731
    if case["integrator"] == "rk2":
        return 0.5 * U + 0.5 * f(f(U))
    return U / 3 + 2 / 3 * f(0.75 * U + 0.25 * f(f(U)))


def _layers(theta):
    sizes, net, at = [(HIDDEN, 4), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (1, HIDDEN)], [], 0
    for rows, cols in sizes:
        w, b = theta[at:at + rows * cols].reshape(rows, cols), theta[at + rows * cols:at + rows * cols + rows]
        net.append((w, b) if rows > 1 else (w[0], b[0]))
        at += rows * cols + rows
    return net


def exact(case, seed):
    got, path = _inputs(case, seed), case["path"]
    length, mu = _domain(case)
    dev = _device()
    if path == "train":
        t = torch.float64 if case["dtype"] == "f64" else torch.float32
        theta = torch.tensor(got["theta"], dtype=t, device=dev).double().requires_grad_(True)
        net, cg = _layers(theta), got["cg"].double()
        # the windows stand side by side along z, which is none of the case's axes
        U, total = torch.cat([cg[s] for s in got["starts"]], dim=1), 0.0

        def prim(U):
            vel = [U[k] / U[0] for k in (1, 2, 3)]
            return torch.stack([U[0], vel[0], vel[1], (GAMMA - 1) * (U[4] - 0.5 * U[0] * sum(q * q for q in vel))])
        for k in range(1, case["steps"] + 1):
            U = torch.utils.checkpoint.checkpoint(_advance, U, 1e-3, case, net, use_reentrant=False)
            ref = torch.cat([cg[s + k] for s in got["starts"]], dim=1)
            total = total + ((prim(U) - prim(ref)) ** 2).mean()
        loss = total / case["steps"]
        return [loss.detach(), torch.autograd.grad(loss, theta)[0]]
    Us = [u.double() for u in got["U"]]
    if path == "vjp":
        U = Us[0].requires_grad_(True)
        out = _advance(U, got["dt"], case)
        return [out.detach(), torch.autograd.grad(out, U, got["lam"].double())[0]]
    if path == "grad":
        U0 = U = Us[0].requires_grad_(True)
        for _ in range(case["steps"]):
            U = torch.utils.checkpoint.checkpoint(_advance, U, got["dt"], case, use_reentrant=False)
        volume = math.prod(length[a] / n for a, n in enumerate(_sides(case)[0]) if n > 1)
        loss = ((U[0] - got["target"].double()) ** 2).sum() * volume
        return [loss.detach(), torch.autograd.grad(loss, U0)[0]]
    with torch.no_grad():
        if case["flux"] == "roe" and Us[0].numel() > 5 * 180**3:
            return None  # the projected stencils do not fit
        done, dts = [], []
        for U in Us:
            for _ in range(case.get("steps", 1)):
                dt = case.get("dt") or _dt(U, case, length, mu)
                U = _advance(U, dt, case)
            done.append(U)
            dts.append(dt)
        dts = torch.tensor(dts, dtype=torch.float64, device=dev)
        return {"step": [done[0], dts], "run": [done[0]], "batch": done}[path]
